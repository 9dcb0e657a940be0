"""What a user of the CFL-reachability solver has it do, as measured cases.

A case is one program analysis (or one batch of them): a grammar, a program-
shaped graph made from a seed, and the way the calling program uses the solver:

  resident   the graph stays loaded; a pass is cflr_reset, cflr_solve and the
             read-out of every named non-terminal into device arrays
  reload     the context stays, a pass loads the graph from host arrays, solves
             and reads out into device arrays
  oneshot    a pass creates the context, compiles the grammar, loads, solves,
             reads out and destroys the context again
  batch      many resident contexts, reset, solved together and read out
  requests   a server's work on a burst of requests: every request is loaded
             into a context of its own, all advance together in ticks led by
             a context that stays, and each is read out and destroyed

The graphs have the shapes of the package's own generators (procedures of 64
vertices, Zipf source weights and field indices, rare long edges, reversed
edges where the grammar has barred labels), drawn on the GPU because the host
generators take seconds at the larger sizes.  Closure sizes differ several
times over between random structures of one size, so a case's structure is
its own and the seed gives the vertex ids and the order of the edges.
"""
import math

import numpy as np
import torch

from paper_2401_11029_gb300 import cflr, gen

# kind -> (grammar, pairs of the closure per input edge, from the recorded
# results of the full-size workloads; only used to estimate output bytes)
KINDS = {"alias": ("fica", 84.6), "points_to": ("fsjpt", 30.7), "field_alias": ("fsca", 16.2),
         "value_flow": ("cscvf", 3.5), "dyck1": ("dyck1", 359.0), "dyck3": ("dyck3", 1.4)}

WINDOW, LONG_BLOCKS, P_LONG, K_MAX = (gen.DEFAULT_WINDOW, 64, gen.DEFAULT_P_LONG,
                                      gen.DEFAULT_K_MAX)


def _case(name, kind, mode, n, form="graph", out="device", index=0, witness=False, count=1):
    """index: the largest value of the grammar's index variable (fields, call
    sites); count: instances of a batch or requests of a burst, whose vertex
    counts are log-uniform up to n."""
    c = {"kind": kind, "mode": mode, "n": n, "form": form, "out": out, "index": index,
         "witness": witness, "count": count}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # balanced words on a small random digraph: the smallest closure, bound
        # by the launches and host steps of each iteration
        _case("dyck1_1000", "dyck1", "resident", 1000),
        # one function-sized alias query from a tool that keeps nothing: the
        # latency of the whole call sequence
        _case("alias_613_oneshot", "alias", "oneshot", 613, out="host"),
        # a module-sized alias analysis as the quick start runs it, but in the
        # default execution form, results to plain host arrays
        _case("alias_20011_oneshot", "alias", "oneshot", 20_011, form="default", out="host"),
        # alias analysis that keeps a derivation step for every pair
        # (single-path semantics), for tools that explain their reports
        _case("alias_50021_witness", "alias", "resident", 50_021, witness=True),
        # a build server's next revision: a new graph into a context that stays
        _case("alias_99991_reload", "alias", "reload", 99_991),
        # the headline workload: whole-program alias analysis
        _case("alias_200000", "alias", "resident", 200_000),
        # field-sensitive points-to of a medium program, from nothing
        _case("points_to_61001_oneshot", "points_to", "oneshot", 61_001, index=63),
        # field-sensitive points-to of a large program, 386 named non-terminals
        _case("points_to_500000", "points_to", "resident", 500_000, index=63),
        # field-sensitive C alias analysis of the imagick graph's shape: many
        # iterations with few new pairs each
        _case("field_alias_41652", "field_alias", "resident", 41_652, index=141),
        # context-sensitive value flow: more than 1500 non-terminals, most of
        # them nearly empty
        _case("value_flow_100000", "value_flow", "resident", 100_000, index=511),
        # independent Dyck-3 instances solved as one batch
        _case("dyck3_batch_64", "dyck3", "batch", 50_000, count=64),
        # a server's burst of ten alias requests of mixed sizes
        _case("alias_requests_10", "alias", "requests", 40_000, count=10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    pick = rng.randrange(8)
    if pick == 0:
        return _case(None, "dyck1", "resident", rng.randrange(200, 1400))
    if pick <= 2:       # alias in every way of use
        mode = rng.choice(["resident", "reload", "oneshot"])
        hi = 200_000 if mode == "resident" else 100_000
        witness = rng.random() < 0.2
        form = rng.choice(["graph", "graph", "default"])
        n = _log_int(rng, 400, 60_000 if witness else hi)
        out = rng.choice(["host", "device"]) if n < 30_000 else "device"
        return _case(None, "alias", mode, n, form=form, out=out, witness=witness)
    if pick <= 4:
        mode = rng.choice(["resident", "reload", "oneshot"])
        n = _log_int(rng, 1000, 250_000 if mode == "resident" else 100_000)
        return _case(None, "points_to", mode, n, index=rng.choice([7, 31, 63]))
    if pick == 5:
        return _case(None, "field_alias", rng.choice(["resident", "oneshot"]),
                     _log_int(rng, 500, 45_000), index=rng.choice([7, 63, 141]))
    if pick == 6:
        return _case(None, "value_flow", rng.choice(["resident", "oneshot"]),
                     _log_int(rng, 2000, 100_000), index=rng.choice([63, 255, 511]))
    if rng.random() < 0.5:
        return _case(None, "dyck3", "batch", rng.randrange(5000, 50_001),
                     count=rng.randrange(4, 65))
    return _case(None, "alias", "requests", rng.randrange(6000, 40_001), count=rng.randrange(2, 11))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

class _Draw:
    """Integer draws on the GPU from one seed."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed))

    def below(self, hi, size):
        return torch.randint(0, int(hi), (int(size),), generator=self.g, device="cuda")

    def perm(self, n):
        return torch.randperm(int(n), generator=self.g, device="cuda")

    def zipf(self, s, k_max, size):
        """Indices 0..k_max-1 with weights (k + 1)^-s."""
        w = [max(1, int(round((1 << 40) * math.pow(k, -s)))) for k in range(1, k_max + 1)]
        cdf = torch.tensor(w, dtype=torch.int64, device="cuda").cumsum(0)
        return torch.searchsorted(cdf, self.below(int(cdf[-1]), size), right=True)


class _Procedures:
    """Forward edges inside blocks of WINDOW positions of a random order,
    a few into the next LONG_BLOCKS blocks; sources by Zipf weights."""

    def __init__(self, rnd, m):
        self.rnd, self.m = rnd, m
        self.order = rnd.perm(m)                      # position -> vertex
        self.pos = torch.empty_like(self.order)
        self.pos[self.order] = torch.arange(m, device="cuda")
        self.cw = (rnd.zipf(gen.ZIPF_S, K_MAX, m) + 1).cumsum(0)
        self.top = int(self.cw[-1])

    def edges(self, size):
        rnd, m = self.rnd, self.m
        si = torch.searchsorted(self.cw, rnd.below(self.top, size), right=True)
        far = rnd.below(1 << 32, size) < int(P_LONG * (1 << 32))
        r = rnd.below(1 << 62, size)
        p = self.pos[si]
        end = ((p // WINDOW + 1) * WINDOW).clamp(max=m)
        near_n = end - 1 - p
        far_n = (end + LONG_BLOCKS * WINDOW).clamp(max=m) - end
        ok = torch.where(far, far_n > 0, near_n > 0)
        t = torch.where(far, end + r % far_n.clamp(min=1), p + 1 + r % near_n.clamp(min=1))
        return si[ok], self.order[t.clamp(max=m - 1)[ok]]


def _distinct(rnd, n, labels, want, sample):
    """The first `want` distinct (src, label, dst) triples of the draws of
    sample(size) -> (src, label, dst)."""
    keys = None
    for _ in range(64):
        have = 0 if keys is None else keys.numel()
        if have >= want:
            break
        s, l, d = sample(max(1024, int((want - have) * 1.25) + 16))
        k = (s * labels + l) * n + d
        k = k if keys is None else torch.cat([keys, k])
        srt, at = torch.sort(k, stable=True)
        first = torch.ones_like(srt, dtype=torch.bool)
        first[1:] = srt[1:] != srt[:-1]
        keys = k[torch.sort(at[first]).values]
    keys = keys[:want]
    return torch.stack([keys // n // labels, keys // n % labels, keys % n])


def _graph(rnd, n, labels, parts, reverse=0):
    """The edges of all parts, vertices and edges in the order rnd gives them;
    labels 0..reverse-1 also get their reversed edges under the labels that
    follow the forward ones."""
    e = torch.cat(parts, dim=1)
    if reverse:
        f = e[:, e[1] < reverse]
        e = torch.cat([e, torch.stack([f[2], f[1] + reverse, f[0]])], dim=1)
    ids = rnd.perm(n)
    e = torch.stack([ids[e[0]], e[1], ids[e[2]]])[:, rnd.perm(e.shape[1])]
    src, lab, dst = e.to(torch.int32).cpu().numpy().view(np.uint32)
    return gen.Graph(n=n, labels=labels, src=np.ascontiguousarray(src),
                     lab=np.ascontiguousarray(lab), dst=np.ascontiguousarray(dst))


def _make_graph(kind, n, index, seed):
    rnd, ids = _Draw(1000 * n + index), _Draw(seed)
    if kind == "dyck1":
        def er(size):
            return rnd.below(n, size), rnd.below(2, size), rnd.below(n, size)
        return _graph(ids, n, ["a", "b"], [_distinct(rnd, n, 2, 3 * n, er)])
    proc = _Procedures(rnd, n if kind != "points_to" else n - n // 10)

    def with_label(label):
        def sample(size):
            s, d = proc.edges(size)
            return s, torch.full_like(s, label) if isinstance(label, int) else label(s.numel()), d
        return sample

    if kind == "alias":
        parts = [_distinct(rnd, n, 2, 2 * n, with_label(0)),
                 _distinct(rnd, n, 2, 3 * n // 4, with_label(1))]
        return _graph(ids, n, ["a", "d", "a_r", "d_r"], parts, reverse=2)
    if kind == "dyck3":
        labels = ["a_1", "b_1", "a_2", "b_2", "a_3", "b_3"]
        return _graph(ids, n, labels,
                      [_distinct(rnd, n, 6, 3 * n, with_label(lambda k: rnd.below(6, k)))])
    F = index + 1
    if kind == "field_alias":
        m, L = 55_775 * n // 41_652, 2 + F
        fields = [_distinct(rnd, n, L, m * 30 // 100,
                            with_label(lambda k: 2 + rnd.zipf(1.0, F, k)))]
        parts = [_distinct(rnd, n, L, m * 45 // 100, with_label(0)),
                 _distinct(rnd, n, L, m * 25 // 100, with_label(1))] + fields
        fwd = ["a", "d"] + [f"f_{i}" for i in range(F)]
        rev = ["a_r", "d_r"] + [f"f_r_{i}" for i in range(F)]
        return _graph(ids, n, fwd + rev, parts, reverse=L)
    if kind == "value_flow":
        m, L = 168 * n // 100, 1 + 2 * F
        blocks = -(-n // WINDOW)
        caller = rnd.below(blocks, F)
        callee = (rnd.zipf(1.0, blocks, F) + rnd.below(blocks, F)) % blocks
        lo = caller * WINDOW
        length = (lo + WINDOW).clamp(max=n) - lo
        at = lo + rnd.below(1 << 62, F) % length
        back = at + rnd.below(1 << 62, F) % (lo + length - at)
        entry = callee * WINDOW
        leave = (entry + WINDOW).clamp(max=n) - 1
        i = torch.arange(F, device="cuda")
        calls = torch.stack([proc.order[at], 1 + i, proc.order[entry]])
        rets = torch.stack([proc.order[leave], 1 + F + i, proc.order[back]])
        labels = ["a"] + [f"call_{k}" for k in range(F)] + [f"ret_{k}" for k in range(F)]
        flow = _distinct(rnd, n, L, max(m - 2 * F, n // 2), with_label(0))
        return _graph(ids, n, labels, [flow, calls, rets])
    # points-to: a tenth of the vertices (the highest ids) are objects
    m, L, n_var = 4 * n, 2 + 2 * F, n - n // 10
    n_obj = n - n_var
    rank, per = rnd.perm(n_obj), max(1, n_obj * WINDOW // n_var)

    def alloc(size):
        s, _ = proc.edges(size)
        near = (proc.pos[s] // WINDOW * per + rnd.below(per, s.numel())) % n_obj
        far = rnd.below(1 << 32, s.numel()) < int(P_LONG * (1 << 32))
        o = rank[torch.where(far, rnd.below(n_obj, s.numel()), near)]
        return s, torch.ones_like(s), n_var + o

    parts = [_distinct(rnd, n, L, m * 4 // 10, with_label(0)), _distinct(rnd, n, L, m // 10, alloc),
             _distinct(rnd, n, L, m // 4, with_label(lambda k: 2 + rnd.zipf(1.0, F, k))),
             _distinct(rnd, n, L, m // 4, with_label(lambda k: 2 + F + rnd.zipf(1.0, F, k)))]
    fwd = ["assign", "alloc"] + [f"load_{k}" for k in range(F)] + [f"store_{k}" for k in range(F)]
    rev = ["assign_r", "alloc_r"] + [f"load_r_{k}" for k in range(F)] + \
          [f"store_r_{k}" for k in range(F)]
    return _graph(ids, n, fwd + rev, parts, reverse=L)


def _text(case):
    return gen.grammar_text(KINDS[case["kind"]][0], case["index"] or None)


def _sizes(case):
    """Vertex counts of a batch or burst: an even spread of the logarithm from
    an eighth (Dyck-3: a fiftieth) of n to n, so the work hardly depends on the
    seed."""
    k, n = case["count"], case["n"]
    ratio = 50.0 if case["kind"] == "dyck3" else 8.0
    return [int(n / ratio * math.pow(ratio, (i + 0.5) / k)) for i in range(k)]


def _config(case):
    cfg = {} if case["form"] == "default" else {"form": cflr.CFLR_FORM_GRAPH}
    if case["witness"]:
        cfg["witness"] = 1
    return cfg


class _State:
    """The graphs and contexts a user's program holds; frees the contexts."""

    def __init__(self, case, seed):
        self.case, self.text = dict(case), _text(case)
        kind, mode = case["kind"], case["mode"]
        self.graphs, self.solvers, self.leader = [], [], None
        if mode in ("batch", "requests"):
            self.graphs = [_make_graph(kind, n, case["index"], seed * 1000 + i)
                           for i, n in enumerate(_sizes(case))]
        else:
            self.graphs = [_make_graph(kind, case["n"], case["index"], seed)]
        if mode in ("resident", "reload", "batch"):
            for g in self.graphs:
                s = cflr.Solver(self.text, **_config(case))
                self.solvers.append(s)
                if mode != "reload":
                    s.load(g)
        if mode == "requests":
            # the context that leads the ticks and lends its work buffers
            self.leader = cflr.Solver(self.text, max_iterations=16, stop_on_first_converged=1,
                                      **_config(case))
            cflr.cflr_load_graph(self.leader.ctx, 1, [], [], [])
            self.leader.solve()

    def __del__(self):
        for s in self.solvers + [self.leader]:
            if s is not None and s.ctx is not None:
                s.close()


def prepare(case, seed):
    return _State(case, seed)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _read_device(s):
    """Every named non-terminal's pairs in device arrays of the right size."""
    ids = np.arange(s.n_named, dtype=np.uint32)
    total = int(cflr.cflr_get_pairs_many(s.ctx, ids, count_only=True)[-1])
    src = torch.empty(total, dtype=torch.int32, device="cuda")
    dst = torch.empty(total, dtype=torch.int32, device="cuda")
    off = cflr.cflr_get_pairs_device_many(s.ctx, ids, src.data_ptr(), dst.data_ptr(), total)
    return src, dst, off.astype(np.int64)


def _read(s, out):
    if out == "device":
        return _read_device(s)
    src, dst, off = cflr.cflr_get_pairs_many(s.ctx, np.arange(s.n_named, dtype=np.uint32))
    return src.view(np.int32), dst.view(np.int32), off.astype(np.int64)


def _requests(state):
    """The loads and ticks of a server on one burst; results by request."""
    active, done = [], {}
    for i, g in enumerate(state.graphs):
        s = cflr.Solver(state.text, size_hint=90, **_config(state.case))
        s.load(g)
        active.append((i, s))
    while active:
        stats = cflr.cflr_solve_batch([state.leader.ctx] + [s.ctx for _, s in active],
                                      allow_limit=True)
        still = []
        for (i, s), st in zip(active, stats[1:]):
            if st["converged"]:
                done[i] = _read(s, state.case["out"])
                s.close()
            else:
                still.append((i, s))
        active = still
    return [done[i] for i in range(len(state.graphs))]


def run(state):
    case = state.case
    mode = case["mode"]
    if mode == "requests":
        return _requests(state)
    if mode == "oneshot":
        with cflr.Solver(state.text, **_config(case)) as s:
            s.load(state.graphs[0])
            s.solve()
            return _read(s, case["out"])
    if mode == "batch":
        for s in state.solvers:
            cflr.cflr_reset(s.ctx)
        cflr.cflr_solve_batch([s.ctx for s in state.solvers])
        # one array of each kind for the whole batch keeps the outputs few
        got = [_read(s, case["out"]) for s in state.solvers]
        return (torch.cat([g[0] for g in got]), torch.cat([g[1] for g in got]),
                np.concatenate([g[2] for g in got]))
    s = state.solvers[0]
    if mode == "reload":
        s.load(state.graphs[0])
    else:
        cflr.cflr_reset(s.ctx)
    s.solve()
    return _read(s, case["out"])


def _edges(kind, n):
    per = {"alias": 5.5, "points_to": 8.0, "field_alias": 2.678, "value_flow": 1.68, "dyck1": 3.0,
           "dyck3": 3.0}
    return per[kind] * n


def work(case):
    """Each edge read once (source, label, destination), each pair written
    once (source, destination); boolean work only, so no flops."""
    kind = case["kind"]
    sizes = _sizes(case) if case["mode"] in ("batch", "requests") else [case["n"]]
    total = 0.0
    for n in sizes:
        m = _edges(kind, n)
        # the random digraph's closure grows with the square of n
        pairs = 1.08 * n * n if kind == "dyck1" else KINDS[kind][1] * m
        total += 12 * m + 8 * pairs
    return {"bytes": total, "flops": 0}


# ---------------------------------------------------------------------------
# small closures in dense 64-bit arithmetic
# ---------------------------------------------------------------------------

# named non-terminals in order of appearance, productions over them and the
# labels (a label's matrix is its edges)
DENSE = {
    "dyck1": (["S", "S1", "A", "B"],
              [("S", "A", "B"), ("S", "A", "S1"), ("S", "S", "S"), ("S1", "S", "B")],
              [("A", "a"), ("B", "b")]),
    "alias": (["M", "N1", "N2", "N3", "AM"],
              [("M", "N1", "N3"), ("M", "N2", "N3"), ("N1", "N1", "a_r"), ("N1", "N2", "a_r"),
               ("N2", "N1", "M"), ("N3", "a", "N3"), ("N3", "AM", "N3"), ("AM", "a", "M")],
              [("N1", "d_r"), ("N3", "d")]),
}


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    if kind not in DENSE or n > 1500 or case["mode"] in ("batch", "requests"):
        return None
    g = _make_graph(kind, n, case["index"], seed)
    names, binary, terminal = DENSE[kind]
    m = {x: torch.zeros(n, n, dtype=torch.float64, device="cuda") for x in names + g.labels}
    for i, x in enumerate(g.labels):
        e = g.lab == i
        m[x][torch.from_numpy(g.src[e].astype(np.int64)).cuda(),
             torch.from_numpy(g.dst[e].astype(np.int64)).cuda()] = 1.0
    for c, x in terminal:
        m[c] = torch.maximum(m[c], m[x])
    before = -1.0
    while True:
        for c, a, b in binary:
            m[c] = torch.maximum(m[c], (m[a] @ m[b] > 0).double())
        now = float(sum(m[x].sum() for x in names))
        if now == before:
            break
        before = now
    pairs = [torch.nonzero(m[x]).to(torch.int32) for x in names]
    src, dst = (torch.cat([p[:, k] for p in pairs]).contiguous() for k in (0, 1))
    off = np.cumsum([0] + [p.shape[0] for p in pairs]).astype(np.int64)
    if case["out"] == "host":
        return src.cpu().numpy(), dst.cpu().numpy(), off
    return src, dst, off
