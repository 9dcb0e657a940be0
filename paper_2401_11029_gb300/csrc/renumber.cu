// Vertex renumbering on the device (cflr_load_graph).
//
// The order is the breadth-first order of the edges taken as undirected that
// a one-thread queue search gives: components in the order of their smallest
// vertex, each searched from that vertex, the neighbours of a vertex in edge
// order (the edge index, then its source side before its destination side;
// the two entries a self-loop gives are the same vertex).  Consecutive ids
// then go to vertices that reach one another, so a closure row falls into
// few 32-bit words of the tile lists.
//
// Steps: an undirected adjacency (CSR) whose lists hold (edge index << 32 |
// neighbour) and are sorted; connected components by hooking the larger of
// two roots under the smaller and pointer jumping, so every component's root
// is its smallest vertex; a breadth-first search from all roots at once.  In
// level L the frontier is sorted by root and, within a root, by the order of
// the search.  An unseen neighbour v goes to the frontier vertex that reaches
// it first in that order: the smallest key (frontier position << 32 | list
// position) that claims it.  Each frontier vertex then writes the vertices it
// won, in list order, at a scanned offset, so the next frontier keeps the
// order the queue search would give it.  A vertex's final position is its
// component's offset, plus the vertices of its component in earlier levels,
// plus its rank in its component's part of its level; per-root tables of the
// frontier segments (first, end, earlier count), kept for two levels, give
// both without a pass of their own.
#include "kernels.cuh"

#include <cooperative_groups.h>

#include <mutex>

namespace cflr {

namespace {

constexpr uint32_t RN_UNSEEN = 0xFFFFFFFFu;

inline int rn_grid(unsigned long long items, int per_block, int sms, int mult) {
    unsigned long long g = (items + per_block - 1) / per_block;
    const unsigned long long cap = (unsigned long long)sms * mult;
    if (g > cap) g = cap;
    return g < 1 ? 1 : (int)g;
}

// Degrees of the undirected graph (a self-loop counts twice) and the largest.
__global__ void k_rn_degree(const uint32_t *src, const uint32_t *dst, unsigned long long m,
                            uint32_t *deg) {
    for (unsigned long long e = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; e < m;
         e += (unsigned long long)gridDim.x * blockDim.x) {
        atomicAdd(&deg[src[e]], 1u);
        atomicAdd(&deg[dst[e]], 1u);
    }
}

__global__ void k_rn_max(const uint32_t *deg, uint32_t n, uint32_t *out) {
    uint32_t mx = 0;
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
        mx = max(mx, deg[v]);
    mx = __reduce_max_sync(0xFFFFFFFFu, mx);
    if ((threadIdx.x & 31) == 0) atomicMax(out, mx);
}

// Adjacency entries (edge << 32 | neighbour), in any order within a list.
__global__ void k_rn_fill(const uint32_t *src, const uint32_t *dst, unsigned long long m,
                          unsigned long long *cur, unsigned long long *adj) {
    for (unsigned long long e = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; e < m;
         e += (unsigned long long)gridDim.x * blockDim.x) {
        const uint32_t s = src[e], d = dst[e];
        adj[atomicAdd(&cur[s], 1ull)] = (e << 32) | d;
        adj[atomicAdd(&cur[d], 1ull)] = (e << 32) | s;
    }
}

// Sort the lists of up to 32 entries in registers (a warp per list); longer
// ones are listed for k_rn_sort_big.
__global__ void __launch_bounds__(256) k_rn_sort_small(const unsigned long long *off, uint32_t n,
                                                       unsigned long long *adj, uint32_t *big,
                                                       uint32_t *big_n) {
    const int lane = threadIdx.x & 31;
    const uint32_t warps = gridDim.x * (blockDim.x >> 5);
    for (uint32_t v = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); v < n; v += warps) {
        const unsigned long long a = off[v], d = off[v + 1] - a;
        if (d <= 1) continue;
        if (d > 32) {
            if (lane == 0) big[atomicAdd(big_n, 1u)] = v;
            continue;
        }
        unsigned long long x = (unsigned long long)lane < d ? adj[a + lane] : ~0ull;
#pragma unroll
        for (uint32_t k = 2; k <= 32; k <<= 1) {
#pragma unroll
            for (uint32_t j = k >> 1; j > 0; j >>= 1) {
                const unsigned long long y = __shfl_xor_sync(0xFFFFFFFFu, x, j);
                const bool up = (lane & k) == 0, lower = (lane & j) == 0;
                x = (lower == up) ? min(x, y) : max(x, y);
            }
        }
        if ((unsigned long long)lane < d) adj[a + lane] = x;
    }
}

// Sort the listed longer lists, a CTA each, by a bitonic sort of P entries in
// shared memory (P: the next power of two, at most the launch's size).
__global__ void __launch_bounds__(256) k_rn_sort_big(const unsigned long long *off,
                                                     unsigned long long *adj, const uint32_t *big,
                                                     const uint32_t *big_n) {
    extern __shared__ unsigned long long sk[];
    const uint32_t nb = *big_n;
    for (uint32_t r = blockIdx.x; r < nb; r += gridDim.x) {
        const uint32_t v = big[r];
        const unsigned long long a = off[v];
        const uint32_t d = (uint32_t)(off[v + 1] - a);
        uint32_t P = 64;
        while (P < d) P <<= 1;
        for (uint32_t t = threadIdx.x; t < P; t += blockDim.x) sk[t] = t < d ? adj[a + t] : ~0ull;
        __syncthreads();
        for (uint32_t k = 2; k <= P; k <<= 1) {
            for (uint32_t j = k >> 1; j > 0; j >>= 1) {
                for (uint32_t q = threadIdx.x; q < P / 2; q += blockDim.x) {
                    const uint32_t t = ((q & ~(j - 1)) << 1) | (q & (j - 1));
                    const unsigned long long x = sk[t], y = sk[t | j];
                    const bool up = (t & k) == 0;
                    if ((x > y) == up) {
                        sk[t] = y;
                        sk[t | j] = x;
                    }
                }
                __syncthreads();
            }
        }
        for (uint32_t t = threadIdx.x; t < d; t += blockDim.x) adj[a + t] = sk[t];
        __syncthreads();
    }
}

__global__ void k_rn_init(uint32_t n, uint32_t *parent, uint32_t *lvl, unsigned long long *key,
                          uint32_t *iperm) {
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        parent[v] = v;
        lvl[v] = RN_UNSEEN;
        key[v] = ~0ull;
        iperm[v] = RN_UNSEEN;
    }
}

// Pointer jumping: every vertex to its root (parents always have smaller
// ids, so the chains end).  *more is set when a chain was left unfinished.
__global__ void k_rn_compress(uint32_t *parent, uint32_t n, unsigned *more) {
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        uint32_t x = parent[v];
        for (int it = 0; it < 4096 && parent[x] != x; it++) x = parent[x];
        if (parent[x] != x) *more = 1;
        parent[v] = x;
    }
}

// Hooking: for an edge between two components, the larger root goes under
// the smaller (a root that another edge hooked in the same pass may lose that
// link; its edge then hooks again in the next pass).
__global__ void k_rn_hook(const uint32_t *src, const uint32_t *dst, unsigned long long m,
                          uint32_t *parent, unsigned *more) {
    for (unsigned long long e = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; e < m;
         e += (unsigned long long)gridDim.x * blockDim.x) {
        const uint32_t ru = parent[src[e]], rv = parent[dst[e]];
        if (ru != rv) {
            atomicMin(&parent[max(ru, rv)], min(ru, rv));
            *more = 1;
        }
    }
}

// Component sizes (by root) and the root flags.
__global__ void k_rn_count(const uint32_t *parent, uint32_t n, uint32_t *cnt, uint32_t *is_root) {
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        atomicAdd(&cnt[parent[v]], 1u);
        is_root[v] = parent[v] == v ? 1u : 0u;
    }
}

// Level 0: the roots in id order, each first in its component.
__global__ void k_rn_roots(const uint32_t *parent, uint32_t n, const unsigned long long *roff,
                           const unsigned long long *comp_off, uint32_t *F, uint32_t *lvl,
                           uint32_t *sf, uint32_t *se, uint32_t *pc, uint32_t *perm,
                           uint32_t *iperm) {
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        if (parent[v] != v) continue;
        const uint32_t q = (uint32_t)roff[v];
        F[q] = v;
        lvl[v] = 0;
        sf[v] = q;
        se[v] = q + 1;
        pc[v] = 0;
        const uint32_t pos = (uint32_t)comp_off[v];
        iperm[pos] = v;
        perm[v] = pos;
    }
}

// Claims of one level: every unseen neighbour takes the smallest key.
__global__ void __launch_bounds__(256) k_rn_claim(const uint32_t *F, uint32_t fsize,
                                                  const unsigned long long *off,
                                                  const unsigned long long *adj,
                                                  const uint32_t *lvl, unsigned long long *key) {
    const int lane = threadIdx.x & 31;
    const uint32_t warps = gridDim.x * (blockDim.x >> 5);
    for (uint32_t q = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); q < fsize; q += warps) {
        const uint32_t u = F[q];
        const unsigned long long a = off[u], b = off[u + 1];
        for (unsigned long long j = a + lane; j < b; j += 32) {
            const uint32_t v = (uint32_t)adj[j];
            if (lvl[v] == RN_UNSEEN)
                atomicMin(&key[v], ((unsigned long long)q << 32) | (uint32_t)(j - a));
        }
    }
}

// The vertices each frontier vertex won.
__global__ void __launch_bounds__(256) k_rn_won(const uint32_t *F, uint32_t fsize,
                                                const unsigned long long *off,
                                                const unsigned long long *adj,
                                                const uint32_t *lvl,
                                                const unsigned long long *key, uint32_t *won) {
    const int lane = threadIdx.x & 31;
    const uint32_t warps = gridDim.x * (blockDim.x >> 5);
    for (uint32_t q = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); q < fsize; q += warps) {
        const uint32_t u = F[q];
        const unsigned long long a = off[u], b = off[u + 1];
        uint32_t c = 0;
        for (unsigned long long j = a + lane; j < b; j += 32) {
            const uint32_t v = (uint32_t)adj[j];
            c += lvl[v] == RN_UNSEEN &&
                 key[v] == (((unsigned long long)q << 32) | (uint32_t)(j - a));
        }
        c = __reduce_add_sync(0xFFFFFFFFu, c);
        if (lane == 0) won[q] = c;
    }
}

// The next frontier (won vertices in list order from woff[q]) and the final
// positions of its vertices; the segment-start warp of each root carries the
// root's segment table to the next level.
__global__ void __launch_bounds__(256) k_rn_write(
    const uint32_t *F, uint32_t fsize, const unsigned long long *off,
    const unsigned long long *adj, uint32_t *lvl, const unsigned long long *key,
    const unsigned long long *woff, uint32_t *F2, uint32_t level, const uint32_t *parent,
    const unsigned long long *comp_off, const uint32_t *sf, const uint32_t *se,
    const uint32_t *pc, uint32_t *sf2, uint32_t *se2, uint32_t *pc2, uint32_t *perm,
    uint32_t *iperm, uint32_t n) {
    const int lane = threadIdx.x & 31;
    const uint32_t warps = gridDim.x * (blockDim.x >> 5);
    for (uint32_t q = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); q < fsize; q += warps) {
        const uint32_t u = F[q], r = parent[u];
        const uint32_t s0 = sf[r], s1 = se[r];
        const unsigned long long wbase = woff[s0];
        if (q == s0 && lane == 0) {
            sf2[r] = (uint32_t)wbase;
            se2[r] = (uint32_t)woff[s1];
            pc2[r] = pc[r] + (s1 - s0);
        }
        // first final position of the root's vertices of the next level
        const unsigned long long pos0 = comp_off[r] + pc[r] + (s1 - s0);
        unsigned long long t = woff[q];
        const unsigned long long a = off[u], b = off[u + 1];
        for (unsigned long long jb = a; jb < b; jb += 32) {
            const unsigned long long j = jb + lane;
            uint32_t v = 0;
            bool w = false;
            if (j < b) {
                v = (uint32_t)adj[j];
                w = lvl[v] == RN_UNSEEN &&
                    key[v] == (((unsigned long long)q << 32) | (uint32_t)(j - a));
            }
            const unsigned m = __ballot_sync(0xFFFFFFFFu, w);
            if (w) {
                // (positions stay below n whenever the component counts are
                // right; k_rn_check reports a position left unwritten)
                const unsigned long long tt = t + __popc(m & ((1u << lane) - 1));
                const unsigned long long pos = pos0 + (tt - wbase);
                lvl[v] = level + 1;
                if (tt < n) F2[tt] = v;
                if (pos < n) {
                    iperm[pos] = v;
                    perm[v] = (uint32_t)pos;
                }
            }
            t += __popc(m);
        }
    }
}

// The levels of a small frontier by one cluster of RN_CTAS CTAs, without the
// host: claim, count and write as above, with cluster barriers between them.
// A level of a few thousand vertices is all latency: seven launches and a
// read of the next size by the host took 28 us of it, and a program-shaped
// graph has about a hundred levels.  Eight lanes take a frontier vertex (the
// lists hold about eleven entries; those of more than RN_LONG take the warp),
// each group a contiguous run of them, so the offsets are a scan of the
// groups' counts: over the CTA in shared memory, over the cluster through the
// other CTAs' totals.  Larger frontiers, where
// eight SMs are too few, go back to the host's launches.
// The loop ends when the frontier is empty or larger than `limit`, at the
// latest after n levels (each places a vertex); the barriers are the
// hardware's.
constexpr uint32_t RN_CTAS = 8, RN_THREADS = 1024, RN_GROUPS = RN_THREADS / 8;
constexpr uint32_t RN_LONG = 64;

__global__ void __cluster_dims__(RN_CTAS, 1, 1) __launch_bounds__(RN_THREADS, 1)
    k_rn_levels(RnLoop *loop, RnTables T, uint32_t n, uint32_t limit) {
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    auto cluster_sync = [&]() {
        __syncwarp();                          // (the groups of a warp meet again)
        cl.sync();
    };
    __shared__ uint32_t run_sum[RN_GROUPS];    // won by each group's run, then their scan
    __shared__ uint32_t warp_sum[RN_GROUPS / 32];
    __shared__ uint32_t cta_won;
    const uint32_t rank = cl.block_rank();
    const uint32_t g = threadIdx.x >> 3, gl = threadIdx.x & 7, lane = threadIdx.x & 31;
    const uint32_t gsh = lane & ~7u, gmask = 0xFFu << gsh;
    uint32_t fsize = loop->fsize, level = loop->level, b = loop->which, placed = 0;
    while (fsize && fsize <= limit && level <= n) {
        const uint32_t *F = T.F[b];
        uint32_t *F2 = T.F[b ^ 1];
        const unsigned long long gid = (unsigned long long)rank * RN_GROUPS + g;
        const uint32_t q0 = (uint32_t)(fsize * gid / (RN_CTAS * RN_GROUPS));
        const uint32_t q1 = (uint32_t)(fsize * (gid + 1) / (RN_CTAS * RN_GROUPS));
        // work(q, u, a, e, first lane, lanes, mask) for every vertex of the
        // run: short lists by the group, then the long ones of the warp's four
        // runs by the whole warp
        auto each = [&](auto &&work) {
            bool any_long = false;
            for (uint32_t q = q0; q < q1; q++) {
                const uint32_t u = F[q];
                const unsigned long long a = T.off[u], e = T.off[u + 1];
                if (e - a > RN_LONG) any_long = true;
                else work(q, u, a, e, gl, 8u, gmask);
            }
            if (!__any_sync(0xFFFFFFFFu, any_long)) return;
            for (uint32_t w = 0; w < 32; w += 8) {
                const uint32_t w0 = __shfl_sync(0xFFFFFFFFu, q0, w);
                const uint32_t w1 = __shfl_sync(0xFFFFFFFFu, q1, w);
                for (uint32_t q = w0; q < w1; q++) {
                    const uint32_t u = F[q];
                    const unsigned long long a = T.off[u], e = T.off[u + 1];
                    if (e - a > RN_LONG) work(q, u, a, e, lane, 32u, 0xFFFFFFFFu);
                }
            }
            __syncwarp();
        };
        each([&](uint32_t q, uint32_t, unsigned long long a, unsigned long long e, uint32_t l0,
                 uint32_t lanes, uint32_t) {
#pragma unroll 4
            for (unsigned long long j = a + l0; j < e; j += lanes) {
                const uint32_t v = (uint32_t)T.adj[j];
                if (T.lvl[v] == RN_UNSEEN)
                    atomicMin(&T.key[v], ((unsigned long long)q << 32) | (uint32_t)(j - a));
            }
        });
        cluster_sync();
        each([&](uint32_t q, uint32_t, unsigned long long a, unsigned long long e, uint32_t l0,
                 uint32_t lanes, uint32_t mask) {
            uint32_t c = 0;
#pragma unroll 4
            for (unsigned long long j = a + l0; j < e; j += lanes) {
                const uint32_t v = (uint32_t)T.adj[j];
                c += T.lvl[v] == RN_UNSEEN &&
                     T.key[v] == (((unsigned long long)q << 32) | (uint32_t)(j - a));
            }
            for (uint32_t d = lanes / 2; d > 0; d >>= 1) c += __shfl_xor_sync(mask, c, d);
            if (l0 == 0) T.woff[q] = c;
        });
        // the run's counts into positions from its start
        uint32_t sum = 0;
        if (gl == 0) {
            for (uint32_t q = q0; q < q1; q++) {
                const uint32_t c = (uint32_t)T.woff[q];
                T.woff[q] = sum;
                sum += c;
            }
        }
        if (gl == 0) run_sum[g] = sum;
        __syncthreads();
        if (threadIdx.x < RN_GROUPS) {         // four whole warps
            uint32_t x = run_sum[threadIdx.x];
            const uint32_t own = x;
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, d);
                if (lane >= (uint32_t)d) x += y;
            }
            if (lane == 31) warp_sum[threadIdx.x >> 5] = x;
            run_sum[threadIdx.x] = x - own;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t t = 0;
            for (uint32_t w = 0; w < RN_GROUPS / 32; w++) {
                const uint32_t x = warp_sum[w];
                warp_sum[w] = t;
                t += x;
            }
            cta_won = t;
        }
        cluster_sync();                        // (orders the CTA's threads too)
        uint32_t before = 0, won = 0;
        for (uint32_t r = 0; r < RN_CTAS; r++) {
            const uint32_t x = *cl.map_shared_rank(&cta_won, r);
            if (r < rank) before += x;
            won += x;
        }
        before += warp_sum[g >> 5] + run_sum[g];
        if (gl == 0)
            for (uint32_t q = q0; q < q1; q++) T.woff[q] += before;
        if (rank == 0 && threadIdx.x == 0) T.woff[fsize] = won;
        cluster_sync();
        each([&](uint32_t q, uint32_t u, unsigned long long a, unsigned long long e, uint32_t l0,
                 uint32_t lanes, uint32_t mask) {
            const uint32_t r = T.parent[u], sh = lanes == 8 ? gsh : 0u;
            const uint32_t s0 = T.sf[b][r], s1 = T.se[b][r], p0 = T.pc[b][r];
            const unsigned long long wbase = T.woff[s0];
            if (q == s0 && l0 == 0) {
                T.sf[b ^ 1][r] = (uint32_t)wbase;
                T.se[b ^ 1][r] = (uint32_t)T.woff[s1];
                T.pc[b ^ 1][r] = p0 + (s1 - s0);
            }
            const unsigned long long pos0 = T.comp_off[r] + p0 + (s1 - s0);
            unsigned long long t = T.woff[q];
            for (unsigned long long jb = a; jb < e; jb += lanes) {
                const unsigned long long j = jb + l0;
                uint32_t v = 0;
                bool w = false;
                if (j < e) {
                    v = (uint32_t)T.adj[j];
                    w = T.lvl[v] == RN_UNSEEN &&
                        T.key[v] == (((unsigned long long)q << 32) | (uint32_t)(j - a));
                }
                const unsigned m = (__ballot_sync(mask, w) & mask) >> sh;
                if (w) {
                    const unsigned long long tt = t + __popc(m & ((1u << l0) - 1));
                    const unsigned long long pos = pos0 + (tt - wbase);
                    T.lvl[v] = level + 1;
                    if (tt < n) F2[tt] = v;
                    if (pos < n) {
                        T.iperm[pos] = v;
                        T.perm[v] = (uint32_t)pos;
                    }
                }
                t += __popc(m);
            }
        });
        cluster_sync();
        placed += fsize;
        fsize = won;
        level++;
        b ^= 1;
    }
    if (rank == 0 && threadIdx.x == 0) {
        loop->fsize = fsize;
        loop->level = level;
        loop->which = b;
        loop->placed += placed;
    }
}

// *bad = 1 unless perm and iperm are inverse permutations of 0..n-1.
__global__ void k_rn_check(const uint32_t *perm, const uint32_t *iperm, uint32_t n,
                           unsigned *bad) {
    for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const uint32_t v = iperm[k];
        if (v >= n || perm[v] != k) *bad = 1;
    }
}

}  // namespace

void launch_rn_adjacency(const uint32_t *src, const uint32_t *dst, unsigned long long m,
                         uint32_t n, uint32_t *deg, uint32_t *max_deg, int sms, cudaStream_t st) {
    cudaMemsetAsync(deg, 0, (size_t)n * 4, st);
    cudaMemsetAsync(max_deg, 0, 4, st);
    if (m) k_rn_degree<<<rn_grid(m, 256, sms, 8), 256, 0, st>>>(src, dst, m, deg);
    if (n) k_rn_max<<<rn_grid(n, 256, sms, 4), 256, 0, st>>>(deg, n, max_deg);
}

void launch_rn_fill(const uint32_t *src, const uint32_t *dst, unsigned long long m, uint32_t n,
                    const unsigned long long *off, unsigned long long *cur,
                    unsigned long long *adj, uint32_t *big, uint32_t *big_n, uint32_t max_deg,
                    int sms, cudaStream_t st) {
    cudaMemcpyAsync(cur, off, (size_t)n * 8, cudaMemcpyDeviceToDevice, st);
    cudaMemsetAsync(big_n, 0, 4, st);
    if (m) k_rn_fill<<<rn_grid(m, 256, sms, 8), 256, 0, st>>>(src, dst, m, cur, adj);
    if (!n) return;
    k_rn_sort_small<<<rn_grid(n, 8, sms, 16), 256, 0, st>>>(off, n, adj, big, big_n);
    if (max_deg > 32) {
        uint32_t P = 64;
        while (P < max_deg) P <<= 1;
        static std::mutex mu;
        static bool done[64] = {};
        int dev = 0;
        cudaGetDevice(&dev);
        {
            std::lock_guard<std::mutex> lock(mu);
            if (dev >= 0 && dev < 64 && !done[dev]) {
                cudaFuncSetAttribute(k_rn_sort_big, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)(RENUM_LIST_MAX * 8));
                done[dev] = true;
            }
        }
        k_rn_sort_big<<<sms * 2, 256, (size_t)P * 8, st>>>(off, adj, big, big_n);
    }
}

void launch_rn_init(uint32_t n, uint32_t *parent, uint32_t *lvl, unsigned long long *key,
                    uint32_t *iperm, int sms, cudaStream_t st) {
    if (n) k_rn_init<<<rn_grid(n, 256, sms, 4), 256, 0, st>>>(n, parent, lvl, key, iperm);
}

void launch_rn_cc_pass(const uint32_t *src, const uint32_t *dst, unsigned long long m,
                       uint32_t n, uint32_t *parent, unsigned *more, int sms, cudaStream_t st) {
    cudaMemsetAsync(more, 0, 4, st);
    if (n) k_rn_compress<<<rn_grid(n, 256, sms, 4), 256, 0, st>>>(parent, n, more);
    if (m) k_rn_hook<<<rn_grid(m, 256, sms, 8), 256, 0, st>>>(src, dst, m, parent, more);
}

void launch_rn_count(const uint32_t *parent, uint32_t n, uint32_t *cnt, uint32_t *is_root,
                     int sms, cudaStream_t st) {
    cudaMemsetAsync(cnt, 0, (size_t)n * 4, st);
    if (n) k_rn_count<<<rn_grid(n, 256, sms, 4), 256, 0, st>>>(parent, n, cnt, is_root);
}

void launch_rn_roots(const uint32_t *parent, uint32_t n, const unsigned long long *roff,
                     const unsigned long long *comp_off, uint32_t *F, uint32_t *lvl, uint32_t *sf,
                     uint32_t *se, uint32_t *pc, uint32_t *perm, uint32_t *iperm, int sms,
                     cudaStream_t st) {
    if (n)
        k_rn_roots<<<rn_grid(n, 256, sms, 4), 256, 0, st>>>(parent, n, roff, comp_off, F, lvl, sf,
                                                             se, pc, perm, iperm);
}

void launch_rn_claim(const uint32_t *F, uint32_t fsize, const unsigned long long *off,
                     const unsigned long long *adj, const uint32_t *lvl, unsigned long long *key,
                     uint32_t *won, int sms, cudaStream_t st) {
    if (!fsize) return;
    const int g = rn_grid(fsize, 8, sms, 16);
    k_rn_claim<<<g, 256, 0, st>>>(F, fsize, off, adj, lvl, key);
    k_rn_won<<<g, 256, 0, st>>>(F, fsize, off, adj, lvl, key, won);
}

void launch_rn_write(const uint32_t *F, uint32_t fsize, const unsigned long long *off,
                     const unsigned long long *adj, uint32_t *lvl, const unsigned long long *key,
                     const unsigned long long *woff, uint32_t *F2, uint32_t level,
                     const uint32_t *parent, const unsigned long long *comp_off,
                     const uint32_t *sf, const uint32_t *se, const uint32_t *pc, uint32_t *sf2,
                     uint32_t *se2, uint32_t *pc2, uint32_t *perm, uint32_t *iperm, uint32_t n,
                     int sms, cudaStream_t st) {
    if (!fsize) return;
    k_rn_write<<<rn_grid(fsize, 8, sms, 16), 256, 0, st>>>(F, fsize, off, adj, lvl, key, woff, F2,
                                                          level, parent, comp_off, sf, se, pc,
                                                          sf2, se2, pc2, perm, iperm, n);
}

void launch_rn_levels(RnLoop *loop, const RnTables &T, uint32_t n, uint32_t limit,
                      cudaStream_t st) {
    k_rn_levels<<<RN_CTAS, RN_THREADS, 0, st>>>(loop, T, n, limit);
}

void launch_rn_check(const uint32_t *perm, const uint32_t *iperm, uint32_t n, unsigned *bad,
                     int sms, cudaStream_t st) {
    cudaMemsetAsync(bad, 0, 4, st);
    if (n) k_rn_check<<<rn_grid(n, 256, sms, 4), 256, 0, st>>>(perm, iperm, n, bad);
}

}  // namespace cflr
