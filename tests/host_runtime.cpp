// The library's host code (runtime.cu, grammar.cpp) on a stand-in for the CUDA
// runtime, for what cannot be shown on a GPU without reaching the fault:
// the order of work across streams, and calls that fail part-way.
//
// Device memory is host memory.  Copies run at the call, but are numbered per
// stream with vector clocks, so that the program knows which other work each
// one is ordered after: by its stream, by an event that its stream waited
// for, or because the host waited.  A use of memory that is not ordered
// after its last write, after its allocation, or before its release, is a
// violation.  The kernels only check the arrays that they are given and leave
// the loop's counters as a terminal initialisation of `rows` rows and `pairs`
// pairs per non-terminal, and a closure that adds nothing, would.
//
// usage: host_runtime <scenario>; prints what went wrong, exits 0 if nothing.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <string>
#include <vector>

#include "cflr.h"
#include "kernels.cuh"

using namespace cflr;

// ---------------------------------------------------------------------------
// the stand-in
// ---------------------------------------------------------------------------

namespace {

typedef std::vector<uint64_t> Clock;            // per stream: work done up to this number

struct Stream {
    size_t id;
    Clock seen;                                 // what the stream's next work is ordered after
};
struct Event {
    Clock at;
};
struct Mark {                                   // a piece of work: stream and number
    size_t stream;
    uint64_t seq;
};
struct Block {                                  // an allocation
    char *p;
    size_t n;
    bool live, pinned;
    Mark made;
    std::vector<Mark> writes, uses;
};

std::vector<Stream *> g_streams;                // by id; null once destroyed
Clock g_host;                                   // what the host has waited for
std::map<char *, Block> g_blocks;
int g_bad = 0;
uint64_t g_rows = 1000, g_pairs = 10;           // of an initialisation
uint64_t g_maps = 0;                            // launches of the row map
std::function<bool(size_t)> g_fail_alloc;       // device allocation of so many bytes
std::string g_fail_launch;                      // name of the launch that fails next
bool g_fail_captured = false;                   // ... when it is captured into a graph
uint32_t g_iters = 1;                           // iterations of a closure
unsigned g_overflow = 0;                        // OVF_* bits that stop the next iteration
bool g_capturing = false;
cudaError_t g_last = cudaSuccess;

void bad(const std::string &what) {
    std::printf("violation: %s\n", what.c_str());
    g_bad++;
}
void expect(bool ok, const std::string &what) {
    if (!ok) bad(what);
}

void merge(Clock &a, const Clock &b) {
    if (a.size() < b.size()) a.resize(b.size(), 0);
    for (size_t k = 0; k < b.size(); k++) a[k] = std::max(a[k], b[k]);
}
bool covers(const Clock &c, Mark m) { return m.stream < c.size() && c[m.stream] >= m.seq; }

Stream *of(cudaStream_t s) {
    if (s != cudaStreamPerThread) return (Stream *)s;
    // (the one of the only thread here)
    static Stream *mine = nullptr;
    if (!mine) {
        if (g_streams.empty()) g_streams.push_back(nullptr);
        mine = new Stream{g_streams.size(), {}};
        g_streams.push_back(mine);
    }
    return mine;
}
Mark enqueue(cudaStream_t st) {
    Stream *s = of(st);
    merge(s->seen, g_host);
    if (s->seen.size() <= s->id) s->seen.resize(s->id + 1, 0);
    return Mark{s->id, ++s->seen[s->id]};
}
bool idle(cudaStream_t st) {                    // the host has waited for all of it
    Stream *s = of(st);
    return s->seen.size() <= s->id || covers(g_host, Mark{s->id, s->seen[s->id]}) ||
           s->seen[s->id] == 0;
}

Block *block_of(const void *p) {
    auto it = g_blocks.upper_bound((char *)p);
    if (it == g_blocks.begin()) return nullptr;
    --it;
    return (char *)p < it->second.p + it->second.n ? &it->second : nullptr;
}
// work `m` on stream st uses [p, p + n)
void use(const char *what, const void *p, size_t n, cudaStream_t st, Mark m, bool writes) {
    if (!n || g_capturing) return;
    Block *b = block_of(p);
    if (!b) {
        if (p == nullptr || writes) bad(std::string(what) + ": not an allocation");
        return;                                 // (host memory of the caller)
    }
    expect(b->live, std::string(what) + ": released memory");
    expect((char *)p + n <= b->p + b->n, std::string(what) + ": past the end of the allocation");
    const Clock &seen = of(st)->seen;
    expect(covers(seen, b->made), std::string(what) + ": not ordered after its allocation");
    for (Mark w : b->writes)
        expect(covers(seen, w), std::string(what) + ": not ordered after a write");
    if (writes) {
        for (Mark w : b->uses)
            expect(covers(seen, w), std::string(what) + ": written while in use");
        b->writes.assign(1, m);
    }
    b->uses.push_back(m);
}
void launch(const char *name, cudaStream_t st) {
    if (!g_capturing) enqueue(st);
    if (g_fail_launch == name && g_fail_captured == g_capturing) {
        g_fail_launch.clear();
        g_last = cudaErrorLaunchOutOfResources;
    }
}
// a kernel's argument: at least n elements on the device
template <class T>
void arg(const char *what, T *p, uint64_t n, cudaStream_t st) {
    use(what, p, n * sizeof(T), st, Mark{of(st)->id, of(st)->seen[of(st)->id]}, false);
}

void *make_block(size_t n, bool pinned, Mark m) {
    char *p = (char *)std::malloc(n ? n : 1);
    std::memset(p, 0xAB, n);
    g_blocks[p] = Block{p, n, true, pinned, m, {}, {}};
    return p;                                   // (never reused: stale pointers show)
}

}  // namespace

extern "C" {

cudaError_t cudaGetDeviceCount(int *n) { return *n = 1, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int) {
    std::memset(p, 0, sizeof *p);
    p->multiProcessorCount = 4;
    p->sharedMemPerBlockOptin = 227 << 10;
    return cudaSuccess;
}
const char *cudaGetErrorString(cudaError_t) { return "(stand-in)"; }
cudaError_t cudaGetLastError() {
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *) {
    return *p = (cudaMemPool_t)1, cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t, cudaStream_t st) {
    if (g_fail_alloc && g_fail_alloc(n)) return g_last = cudaErrorMemoryAllocation;
    *p = make_block(n, false, enqueue(st));
    return cudaSuccess;
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t st) {
    enqueue(st);
    Block *b = block_of(p);
    if (!b || !b->live || b->p != p) {
        bad("free: not an allocation");
        return cudaSuccess;
    }
    for (Mark m : b->uses)
        expect(covers(of(st)->seen, m), "free: not ordered after a use");
    b->live = false;
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) {
    *p = make_block(n, true, Mark{0, 0});
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void **p, size_t n) { return cudaHostAlloc(p, n, 0); }
cudaError_t cudaFreeHost(void *p) {
    Block *b = block_of(p);
    for (Mark m : b->uses) expect(covers(g_host, m), "free of pinned memory that a copy reads");
    b->live = false;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
    if (g_streams.empty()) g_streams.push_back(nullptr);     // 0: no stream
    Stream *x = new Stream{g_streams.size(), {}};
    g_streams.push_back(x);
    return *s = (cudaStream_t)x, cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
    expect(idle(s), "stream destroyed with work pending");
    g_streams[of(s)->id] = nullptr;
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    expect(!g_capturing, "a wait inside a capture");
    return merge(g_host, of(s)->seen), cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    if (!g_capturing) merge(of(s)->seen, ((Event *)e)->at);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) {
    return *e = (cudaEvent_t) new Event(), cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    if (g_capturing) return cudaSuccess;
    enqueue(s);
    return ((Event *)e)->at = of(s)->seen, cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) {
    return merge(g_host, ((Event *)e)->at), cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
    return *ms = 0, cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *to, const void *from, size_t n, cudaMemcpyKind k,
                            cudaStream_t st) {
    const Mark m = enqueue(st);
    const bool to_dev = k != cudaMemcpyDeviceToHost, from_dev = k != cudaMemcpyHostToDevice;
    if (from_dev || block_of(from)) use("copy from", from, n, st, m, false);
    if (to_dev || block_of(to)) use("copy to", to, n, st, m, true);
    std::memcpy(to, from, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t st) {
    use("memset", p, n, st, enqueue(st), true);
    std::memset(p, v, n);
    return cudaSuccess;
}
// (a graph is captured but never launched here)
cudaError_t cudaGraphCreate(cudaGraph_t *g, unsigned) { return *g = (cudaGraph_t)1, cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle *h, cudaGraph_t, unsigned,
                                             unsigned) {
    return *h = 1, cudaSuccess;
}
cudaError_t cudaGraphAddNode(cudaGraphNode_t *, cudaGraph_t, const cudaGraphNode_t *,
                             const cudaGraphEdgeData *, size_t, cudaGraphNodeParams *p) {
    static cudaGraph_t body = (cudaGraph_t)2;
    return p->conditional.phGraph_out = &body, cudaSuccess;
}
cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t, cudaGraph_t, const cudaGraphNode_t *,
                                          const cudaGraphEdgeData *, size_t,
                                          cudaStreamCaptureMode) {
    return g_capturing = true, cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *) {
    return g_capturing = false, cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **, const void *) { return cudaErrorNotSupported; }

}  // extern "C"

// ---------------------------------------------------------------------------
// the kernels' launches (those that no scenario reaches are not defined)
// ---------------------------------------------------------------------------

namespace cflr {

static void check_work(const char *what, const WorkBufs &W, cudaStream_t st) {
    const std::string w = what;
    for (int q = 0; q < 2; q++) arg((w + ": touched").c_str(), W.touched[q], W.touched_cap, st);
    for (int b = 0; b < N_BINS; b++)
        arg((w + ": groups").c_str(), W.groups[b], W.group_cap[b], st);
    arg((w + ": cand_key").c_str(), W.cand_key, W.cand_cap, st);
    arg((w + ": cand_slot").c_str(), W.cand_slot, W.cand_cap, st);
    arg((w + ": cand_pos").c_str(), W.cand_pos, W.cand_cap, st);
    if (W.cand_wit) arg((w + ": cand_wit").c_str(), W.cand_wit, W.cand_cap, st);
    arg((w + ": big_rows").c_str(), W.big_rows, W.big_cap, st);
    arg((w + ": cnt").c_str(), W.cnt, 1, st);
}

void prepare_launch_attributes() {}
void launch_symbolic(const SlotTab &, const ProdTab &P, const WorkBufs &W, int, const Tuning &,
                     int, cudaStream_t st) {
    launch("symbolic", st);
    check_work("symbolic", W, st);
    arg("use_off", P.use_off, 1, st);
    if (P.use_off && block_of(P.use_off))
        expect(P.use_off[0] == 0, "production tables not written");
}
void launch_spgemm(int bin, const SlotTab &, const ProdTab &, const WorkBufs &W, uint32_t,
                   const Tuning &, int, cudaStream_t st) {
    launch(("bin" + std::to_string(bin)).c_str(), st);
    check_work("product", W, st);
}
void launch_commit(const SlotTab &, const WorkBufs &W, uint32_t, int, cudaStream_t st) {
    launch("commit", st);
    check_work("commit", W, st);
}
void launch_iter_begin(const SlotTab &, const InstTab &, const WorkBufs &, uint32_t, uint32_t,
                       cudaStream_t st) {
    launch("iter_begin", st);
}
void launch_iter_end(const SlotTab &S, const InstTab &I, const WorkBufs &W, LoopCtl *ctl,
                     uint32_t n_slots, uint32_t n_inst, bool count, cudaGraphConditionalHandle,
                     bool, cudaStream_t st) {
    launch("iter_end", st);
    if (g_capturing) return;
    if (count && g_overflow) {
        ctl->status = g_overflow;
        g_overflow = 0;
        W.cnt->cand = W.cand_cap + 1;
        for (int b = 0; b < N_BINS; b++) W.cnt->groups[b] = W.group_cap[b] + 1;
        for (uint32_t s = 0; s < n_slots; s++) S.cand[s] = S.hmask[s];
        for (uint32_t k = 0; k < n_inst; k++) I.pool_top[k] = I.pool_cap[k] + 1;
        return;
    }
    const int par = *W.parity;
    const uint64_t rows =
        count && ctl->iter + 1 >= g_iters ? 0 : std::min<uint64_t>(g_rows, W.touched_cap);
    W.touched_n[par] = 0;
    W.touched_n[par ^ 1] = rows;
    for (uint64_t q = 0; q < rows; q++) W.touched[par ^ 1][q] = make_uint2(0, 0);
    *W.parity = par ^ 1;
    ctl->status = 0;
    ctl->iter++;
    ctl->last_delta = rows;
    for (uint32_t s = 0; s < n_slots; s++) S.nnz[s] = g_pairs;
    for (uint32_t k = 0; k < n_inst; k++) I.active[k] = rows != 0;
}
void launch_check_reset(const SlotTab &, const WorkBufs &, uint32_t, bool, int, cudaStream_t st) {
    launch("check_reset", st);
}
void launch_capacity(const SlotTab &, const InstTab &, const WorkBufs &, int, cudaStream_t st) {
    launch("capacity", st);
}
void launch_capacity_big(const SlotTab &, const InstTab &, const WorkBufs &, uint32_t, int,
                         cudaStream_t st) {
    launch("capacity_big", st);
}
void launch_scatter(const SlotTab &, const WorkBufs &, int, cudaStream_t st) {
    launch("scatter", st);
}
void launch_pack(const SlotTab &, const WorkBufs &, int, cudaStream_t st) { launch("pack", st); }
void launch_init_edges(const uint32_t *, const uint32_t *, const uint32_t *, unsigned long long,
                       const uint32_t *, const uint32_t *, uint32_t, const WorkBufs &W, int,
                       cudaStream_t st) {
    launch("init_edges", st);
    check_work("initialisation", W, st);
}
void launch_clear_sets(const SlotTab &, uint32_t, unsigned long long, int, cudaStream_t st) {
    launch("clear_sets", st);
}
void launch_clear_rows(uint4 *, uint2 *, uint32_t *, uint32_t, uint32_t, int, cudaStream_t st) {
    launch("clear_rows", st);
}
void launch_rehash(const unsigned long long *old_tab, const uint2 *old_val,
                   unsigned long long old_cap, unsigned long long *new_tab, uint2 *new_val,
                   unsigned long long new_cap, unsigned *, int, cudaStream_t st) {
    launch("rehash", st);
    arg("rehash from", old_tab, old_cap, st);
    arg("rehash to", new_tab, new_cap, st);
    expect(!old_val == !new_val, "rehash: witnesses");
    if (old_val) arg("rehash from", old_val, old_cap, st);
    if (new_val) arg("rehash to", new_val, new_cap, st);
}
unsigned long long set_chunks(unsigned long long cap, int) { return cap / 1024; }
void launch_rehash_many(const GrownSet *sets, uint32_t count, unsigned long long,
                        unsigned long long, unsigned *err, int sms, cudaStream_t st) {
    arg("grown sets", sets, count + 1, st);
    for (uint32_t k = 0; k < count; k++)
        launch_rehash(sets[k].old_tab, sets[k].old_val, sets[k].old_cap, sets[k].new_tab,
                      sets[k].new_val, sets[k].new_cap, err, sms, st);
}
void launch_permute_ids(uint32_t *, unsigned long long, const uint32_t *, int, cudaStream_t st) {
    launch("permute_ids", st);
}
void launch_remap_touched(const uint2 *in, unsigned long long n, uint32_t slot_base, uint2 *out,
                          cudaStream_t st) {
    launch("remap_touched", st);
    arg("remap: a context's delta rows", in, n, st);
    arg("remap: the batch's delta rows", out, n, st);
    for (unsigned long long q = 0; q < n; q++)
        out[q] = make_uint2(in[q].x + 2 * slot_base, in[q].y);
}
void extract_plan(uint32_t count, uint32_t n, const uint64_t *, int, uint32_t *rows_per,
                  unsigned long long *first) {
    for (uint32_t k = 0; k <= count; k++) first[k] = k;
    for (uint32_t k = 0; k < count; k++) rows_per[k] = n;
}
void launch_row_map(const ExtractList &L, const uint32_t *, uint32_t, uint32_t *map, int,
                    cudaStream_t st) {
    launch("row_map", st);
    arg("row map", map, (uint64_t)L.count * ((L.n + 31) / 32), st);
    g_maps++;
}
void launch_extract_count(const ExtractList &L, unsigned long long *units, unsigned long long *,
                          unsigned long long *total, int, cudaStream_t st) {
    launch("extract_count", st);
    arg("units", units, L.units + 1, st);
    for (unsigned long long u = 0; u < L.units; u++) units[u] = u * g_pairs;
    *total = L.count * g_pairs;
}
void launch_extract_write(const ExtractList &L, uint32_t *, uint32_t *, const unsigned long long *,
                          uint4 *big, unsigned long long big_cap, unsigned long long *, uint32_t *,
                          unsigned *, int, cudaStream_t st) {
    launch("extract_write", st);
    arg("read-out ids", L.nts, L.count, st);
    arg("long rows", big, big_cap, st);
}

}  // namespace cflr

// ---------------------------------------------------------------------------
// scenarios
// ---------------------------------------------------------------------------

namespace {

const char GRAMMAR[] = "S -> A B | S S\nA -> a\nB -> b\n";

struct Context {
    cflr_ctx *c = nullptr;
    explicit Context(std::function<void(cflr_config &)> set = nullptr,
                     const std::string &text = GRAMMAR) {
        cflr_config cfg;
        cflr_default_config(&cfg);
        if (set) set(cfg);
        expect(cflr_create(&c, &cfg) == CFLR_OK, "cflr_create");
        expect(cflr_load_grammar(c, text.data(), text.size()) == CFLR_OK, "cflr_load_grammar");
    }
    ~Context() { cflr_destroy(c); }
    int load(uint32_t n = 100, uint64_t m = 300) {
        std::vector<uint32_t> s(m), l(m), d(m);
        for (uint64_t e = 0; e < m; e++) s[e] = e % n, d[e] = e * 7 % n, l[e] = e % 2;
        return cflr_load_graph(c, n, m, s.data(), l.data(), d.data());
    }
};

int batch(std::vector<cflr_ctx *> cx) {
    std::vector<cflr_stats> st(cx.size());
    return cflr_solve_batch(cx.data(), (int)cx.size(), st.data());
}

// Contexts with private streams, loaded or reset and at once solved together,
// led by one of them or by a context with nothing to do.
void batch_across_streams() {
    Context lead, a, b;
    g_rows = 0;
    expect(lead.load() == CFLR_OK && cflr_solve(lead.c, nullptr) == CFLR_OK, "leader");
    g_rows = 1000;
    for (int round = 0; round < 3; round++) {
        if (round == 0) expect(a.load() == CFLR_OK && b.load() == CFLR_OK, "load");
        else expect(cflr_reset(a.c) == CFLR_OK && cflr_reset(b.c) == CFLR_OK, "reset");
        expect(batch(round == 1 ? std::vector<cflr_ctx *>{b.c, a.c}
                                : std::vector<cflr_ctx *>{lead.c, a.c, b.c}) == CFLR_OK, "batch");
    }
    // a single active context, whose list needs no split
    expect(cflr_reset(a.c) == CFLR_OK && batch({lead.c, a.c}) == CFLR_OK, "one of a batch");
}

cudaStream_t new_stream() {
    cudaStream_t s;
    cudaStreamCreateWithFlags(&s, 0);
    return s;
}
// fails the k-th device allocation from now on (k = 1, 2, ...), or that and all
// later ones
std::function<bool(size_t)> nth(uint64_t k) {
    return [k](size_t) mutable { return k && --k == 0; };
}
std::function<bool(size_t)> from(uint64_t k) {
    return [k](size_t) mutable { return k <= 1 || (--k, false); };
}

// Read-outs that run out of memory at each allocation in turn: the call's tables
// are copied from memory that the next call writes, so nothing may be pending
// on return.
void failed_readouts() {
    const uint32_t ids[2] = {0, 1};
    for (int host = 0; host < 2; host++) {
        int failed = 0, rc = CFLR_ENOMEM;
        for (uint64_t k = 1; rc != CFLR_OK && k < 50; k++) {
            const cudaStream_t st = new_stream();
            Context x([&](cflr_config &c) { c.stream = st; });
            expect(x.load() == CFLR_OK && cflr_solve(x.c, nullptr) == CFLR_OK, "solve");
            std::vector<uint32_t> s(2 * g_pairs), d(2 * g_pairs);
            // (stands for device arrays too: no kernel writes them here)
            uint64_t off[3];
            auto read = [&]() {
                return host ? cflr_get_pairs_many(x.c, 2, ids, s.data(), d.data(), s.size(), off)
                            : cflr_get_pairs_device_many(x.c, 2, ids, s.data(), d.data(), s.size(),
                                                         off);
            };
            g_fail_alloc = from(k);
            rc = read();
            g_fail_alloc = nullptr;
            failed += rc == CFLR_ENOMEM;
            expect(rc == CFLR_OK || rc == CFLR_ENOMEM, "read-out: code");
            expect(idle(st), "read-out: work pending after the call");
            expect(read() == CFLR_OK, "read-out after a failed one");
        }
        expect(rc == CFLR_OK && failed >= 4, "read-out: allocations reached");
    }
}

// A launch that fails while the product bins run on several streams, or while
// they are captured: nothing may be running when the call returns, and the
// streams do not go to another context.
void failed_products() {
    for (int captured = 0; captured < 2; captured++) {
        for (const char *at : {"bin3", "bin2", "bin1", "bin0"}) {
            const std::string what = std::string(at) + (captured ? " (captured)" : "");
            const cudaStream_t st = new_stream();
            const size_t first = g_streams.size();
            {
                Context x([&](cflr_config &c) {
                    c.stream = st;
                    c.form = CFLR_FORM_GRAPH;
                });
                expect(x.load() == CFLR_OK, "load");
                expect(g_streams.size() > first, "streams of its own");
                g_iters = 3;                    // the second iteration is captured
                g_fail_launch = at;
                g_fail_captured = captured;
                expect(cflr_solve(x.c, nullptr) == CFLR_ECUDA, what + ": code");
                expect(g_fail_launch.empty() && !g_capturing, what + ": launch reached");
                g_fail_captured = false;
                g_iters = 1;
                for (Stream *s : g_streams)
                    if (s) expect(idle((cudaStream_t)s), what + ": work pending");
            }
            for (size_t k = first; k < g_streams.size(); k++)
                expect(!g_streams[k], what + ": a stream is kept for another context");
        }
    }
}

// A context stays usable after CFLR_ENOMEM, whichever allocation of a load or of
// a solve whose buffers overflow it was: the next graph's kernels get arrays
// that hold what they are said to (the launches look at each).
void failed_buffers() {
    for (int witness = 0; witness < 2; witness++) {
        for (int solving = 0; solving < 2; solving++) {
            int failed = 0, rc = CFLR_ENOMEM;
            for (uint64_t k = 1; rc != CFLR_OK && k < 100; k++) {
                Context x([&](cflr_config &c) { c.witness = witness; });
                expect(x.load() == CFLR_OK && cflr_solve(x.c, nullptr) == CFLR_OK, "solve");
                if (solving) {
                    expect(x.load() == CFLR_OK, "load");
                    g_overflow = OVF_CAND | OVF_GROUPS;
                }
                g_fail_alloc = from(k);
                // (100,000 edges: more initial pairs than the first buffers hold)
                rc = solving ? cflr_solve(x.c, nullptr) : x.load(5000, 100000);
                g_fail_alloc = nullptr;
                g_overflow = 0;
                failed += rc == CFLR_ENOMEM;
                expect(rc == CFLR_OK || rc == CFLR_ENOMEM, "code");
                if (rc != CFLR_OK)
                    expect(cflr_solve(x.c, nullptr) == CFLR_ESTATE, "no graph after a failure");
                for (int more = 0; more < 2; more++)
                    expect(x.load() == CFLR_OK && cflr_solve(x.c, nullptr) == CFLR_OK, "next graph");
            }
            expect(rc == CFLR_OK && failed >= 6, "allocations reached");
        }
    }
}

// A batch larger than the leader's tables hold, whose allocations fail in turn:
// the leader's next solve by itself has its production tables.
void failed_batch_tables() {
    int failed = 0, rc = CFLR_ENOMEM;
    for (uint64_t k = 1; rc != CFLR_OK && k < 50; k++) {
        Context lead;
        std::vector<Context> more(8);
        std::vector<cflr_ctx *> cx(1, lead.c);
        expect(lead.load() == CFLR_OK, "load");
        for (auto &x : more) {
            expect(x.load() == CFLR_OK, "load");
            cx.push_back(x.c);
        }
        g_fail_alloc = nth(k);
        rc = batch(cx);
        g_fail_alloc = nullptr;
        failed += rc == CFLR_ENOMEM;
        expect(rc == CFLR_OK || rc == CFLR_ENOMEM, "code");
        for (cflr_ctx *c : cx) expect(rc == CFLR_OK || cflr_reset(c) == CFLR_ESTATE, "dropped");
        expect(lead.load() == CFLR_OK && cflr_solve(lead.c, nullptr) == CFLR_OK, "leader again");
    }
    expect(rc == CFLR_OK && failed >= 1, "allocations reached");
}

// A device without room for the map of non-empty rows, which a read-out can do
// without, or without room for what comes after it beside it.
void readout_without_map() {
    const uint32_t n = 10000, ids[2] = {0, 1};
    const size_t map = 2 * ((n + 31) / 32) * 4;
    for (int host = 0; host < 2; host++) {
        for (int beside = 0; beside < 2; beside++) {
            const cudaStream_t st = new_stream();
            Context x([&](cflr_config &c) { c.stream = st; });
            expect(x.load(n, 300) == CFLR_OK && cflr_solve(x.c, nullptr) == CFLR_OK, "solve");
            std::vector<uint32_t> s(2 * g_pairs), d(2 * g_pairs);
            uint64_t off[3];
            int failed = 0;
            g_fail_alloc = [&](size_t bytes) {
                bool fail = bytes == map && !beside;
                if (beside)                       // whatever it is, while the map is there
                    for (auto &b : g_blocks) fail |= b.second.n == map && b.second.live;
                failed += fail;
                return fail;
            };
            expect((host ? cflr_get_pairs_many(x.c, 2, ids, s.data(), d.data(), s.size(), off)
                         : cflr_get_pairs_device_many(x.c, 2, ids, s.data(), d.data(), s.size(),
                                                      off)) == CFLR_OK,
                   "read-out without room for the map");
            g_fail_alloc = nullptr;
            expect(failed == 1, "one allocation failed");
        }
    }
}

// Read-outs under a memory budget that fail again and again leave what the
// context is said to hold as it was.
void budget_after_failed_readouts() {
    Context x([](cflr_config &c) { c.mem_budget_bytes = 64 << 20; });
    const uint64_t few = g_pairs;
    g_pairs = 100000;
    expect(x.load(1000, 3000) == CFLR_OK && cflr_solve(x.c, nullptr) == CFLR_OK, "solve");
    std::vector<uint32_t> s(g_pairs), d(g_pairs);
    uint64_t got = 0;
    auto read = [&]() { return cflr_get_pairs(x.c, 0, s.data(), d.data(), s.size(), &got); };
    const size_t staging = 2 * g_pairs * 4;       // two buffers of sources, two of targets
    for (int turn = 0; turn < 200; turn++) {
        int seen = 0;                             // the second array of the pair fails
        g_fail_alloc = [&](size_t bytes) { return bytes == staging && ++seen % 2 == 0; };
        expect(read() == CFLR_ENOMEM && seen >= 2, "read-out without room");
        g_fail_alloc = nullptr;
    }
    expect(read() == CFLR_OK && got == g_pairs, "read-out after failed ones");
    g_pairs = few;
}

// Growths of the pair sets and of the row pool that run out of memory at each
// allocation in turn (sets one at a time under a budget, together without one):
// nothing stays allocated once the contexts are gone, and the next graph works.
void failed_growths() {
    for (unsigned bits : {OVF_HASH, OVF_POOL}) {
        for (int witness = 0; witness < 2; witness++) {
            for (int budget = 0; budget < 2; budget++) {
                int failed = 0, rc = CFLR_ENOMEM;
                for (uint64_t k = 1; rc != CFLR_OK && k < 50; k++) {
                    Context x([&](cflr_config &c) {
                        c.witness = witness;
                        c.mem_budget_bytes = budget ? 1ull << 32 : 0;
                    });
                    expect(x.load() == CFLR_OK, "load");
                    g_overflow = bits;
                    g_fail_alloc = from(k);
                    rc = cflr_solve(x.c, nullptr);
                    g_fail_alloc = nullptr;
                    failed += rc == CFLR_ENOMEM;
                    expect(rc == CFLR_OK || rc == CFLR_ENOMEM, "code");
                    expect(x.load() == CFLR_OK && cflr_solve(x.c, nullptr) == CFLR_OK,
                           "next graph");
                }
                expect(rc == CFLR_OK && failed >= 1, "allocations reached");
            }
        }
    }
    for (auto &b : g_blocks)
        expect(b.second.pinned || !b.second.live, "device memory left allocated");
}

// A device without room for roomy first pair sets, or for the rest of a load
// beside them: the load takes small ones.
void load_without_roomy_sets() {
    const size_t sets = 3 * (512u << 10);         // of the three named non-terminals
    for (int beside = 0; beside < 2; beside++) {
        Context x;
        int failed = 0, seen = 0;
        g_fail_alloc = [&](size_t bytes) {
            seen += bytes == sets;
            bool fail = bytes == sets && !beside;
            if (beside)
                for (auto &b : g_blocks) fail |= b.second.n == sets && b.second.live;
            failed += fail;
            return fail;
        };
        expect(x.load() == CFLR_OK && cflr_solve(x.c, nullptr) == CFLR_OK, "small first sets");
        g_fail_alloc = nullptr;
        expect(seen == 1 && failed == 1, "one allocation failed");
        expect(x.load() == CFLR_OK && cflr_solve(x.c, nullptr) == CFLR_OK, "with room again");
    }
}

// cudaStreamPerThread is another stream in every thread, though one handle: the
// next call may come from another thread, so nothing may be pending.
void per_thread_stream() {
    Context x([](cflr_config &c) { c.stream = cudaStreamPerThread; });
    expect(x.load() == CFLR_OK && idle(cudaStreamPerThread), "pending after a load");
    expect(cflr_solve(x.c, nullptr) == CFLR_OK && idle(cudaStreamPerThread), "after a solve");
    expect(cflr_reset(x.c) == CFLR_OK && idle(cudaStreamPerThread), "pending after a reset");
}

const std::map<std::string, void (*)()> SCENARIOS = {
    {"per_thread_stream", per_thread_stream},
    {"load_without_roomy_sets", load_without_roomy_sets},
    {"failed_growths", failed_growths},
    {"budget_after_failed_readouts", budget_after_failed_readouts},
    {"readout_without_map", readout_without_map},
    {"failed_batch_tables", failed_batch_tables},
    {"failed_buffers", failed_buffers},
    {"failed_products", failed_products},
    {"batch_across_streams", batch_across_streams},
    {"failed_readouts", failed_readouts},
};

}  // namespace

int main(int argc, char **argv) {
    const auto it = SCENARIOS.find(argc > 1 ? argv[1] : "");
    if (it == SCENARIOS.end()) return 2;
    it->second();
    return g_bad ? 1 : 0;
}
