"""The work this library is measured by, through its public Python entry points.

Five kinds of pass, each the way a program uses the library:

  update   resident graph, previous ranks known: a batch arrives (deletions and
           insertions), is applied and followed by one update, the ranks are
           read; then the batch is retracted, followed by an update and a read
           again.  The retraction returns the graph to where it was, so a pass
           can be repeated.  The batches hold what real ones hold: repeated
           edges, insertions of edges that exist, self-loops among the draws.
  solve    Static PageRank of a resident graph from scratch (first ranks, or
           the periodic exact refresh).
  load     a graph built from a device edge list, solved once, read, closed.
  group    many independent graphs, one batch each, one group update
           (Group.apply_batches_device + Group.update), then the retraction.
  serve    a request loop over resident graphs: a burst of one request per
           graph is submitted and drained, then its retraction.

Graphs are R-MAT (a, b, c, d = 0.57, 0.19, 0.19, 0.05) with scrambled ids or a
stream graph (heavy-tailed endpoints, a quarter of the edges repeats), in
place of the paper's static graphs with random batches (80 % insertions, 20 %
deletions) and of its temporal streams (insertions only).
"""
import math

import numpy as np
import torch

import paper_2401_15870_gb300 as pr

ALPHA, TAU, TOL = 0.85, 1e-10, 1e-6
CHUNK = 1 << 27          # edges handled at a time where whole-graph temporaries would be large


def listed():
    return [
        # the smallest call: one request on a graph of 16K vertices, everything through host arrays
        dict(name="tiny dfp host", kind="update", graph="rmat", n=1 << 14, edges=1 << 18, method="dfp", batch=262,
             host=True),
        # first ranks of the same small graph
        dict(name="tiny static", kind="solve", graph="rmat", n=1 << 14, edges=1 << 18),
        # a ragged small graph, no pruning (DF), a batch of 1e-3 of its edges
        dict(name="small df", kind="update", graph="rmat", n=70001, edges=1300003, method="df", batch=1300, host=False),
        # a million vertices, a small batch (1e-5 of the edges)
        dict(name="mid dfp", kind="update", graph="rmat", n=1 << 20, edges=1 << 24, method="dfp", batch=168,
             host=False),
        # the traversal comparator: reachability, then sweeps of the reachable set
        dict(name="mid dt", kind="update", graph="rmat", n=1 << 21, edges=1 << 25, method="dt", batch=336, host=False),
        # the temporal stream: insertions only, 1e-4 of 63M timestamped edges per batch
        dict(name="stream dfp", kind="update", graph="stream", n=2600000, edges=56700000, method="dfp", batch=6300,
             host=False),
        # a large batch (1e-2 of the edges: rows overflow and are repacked) followed by Naive-dynamic
        dict(name="bulk nd", kind="update", graph="rmat", n=1 << 23, edges=1 << 28, method="nd", batch=2684355,
             host=False),
        # the large graph with 1.07e9 edges: the benchmark's batch (1e-4 of the edges) and a very small one (1e-7)
        dict(name="large dfp", kind="update", graph="rmat", n=1 << 25, edges=1 << 30, method="dfp", batch=107374,
             host=False),
        dict(name="large dfp few", kind="update", graph="rmat", n=1 << 25, edges=1 << 30, method="dfp", batch=107,
             host=False),
        # the batched workload: 64 uneven graphs of 2^12 to 2^21 vertices, 1e-4 of the edges per batch
        dict(name="group dfp", kind="group", count=64, lo=12.0, hi=21.0, method="dfp", share=1e-4),
        # a burst of requests of 10 to 1e5 edges over 12 resident graphs, small and large ones
        dict(name="serve burst", kind="serve", count=12, lo=15.0, hi=21.0, method="dfp", small=10, big=100000),
        # a graph of 2M vertices and 33M edges built, solved and read
        dict(name="load", kind="load", graph="rmat", n=1 << 21, edges=1 << 25),
    ]


def draw(rng):
    """One more case of the same kinds: sizes over the whole range on a logarithmic scale, odd ones among them."""
    kind = rng.choice(["update"] * 6 + ["solve", "load", "group", "serve"])
    if kind == "group":
        lo = rng.uniform(8.0, 13.0)
        return dict(kind=kind, count=rng.randint(3, 40), lo=lo, hi=lo + rng.uniform(2.0, 7.0),
                    method=rng.choice(["dfp", "dfp", "df"]), share=10.0 ** rng.uniform(-4.5, -3.0))
    if kind == "serve":
        return dict(kind=kind, count=rng.randint(3, 14), lo=13.0, hi=rng.uniform(16.0, 21.0), method="dfp", small=10,
                    big=int(10.0 ** rng.uniform(2.0, 5.0)))
    n = int(2.0 ** rng.uniform(12.0, 23.0)) | rng.randint(0, 1)
    edges = int(n * rng.uniform(8.0, 32.0))
    graph = rng.choice(["rmat", "rmat", "stream"])
    if kind in ("solve", "load"):
        return dict(kind=kind, graph=graph, n=n, edges=edges)
    batch = max(1, int(edges * 10.0 ** rng.uniform(-6.0, -2.0)))
    return dict(kind=kind, graph=graph, n=n, edges=edges, method=rng.choice(["dfp", "dfp", "dfp", "df", "nd", "dt"]),
                batch=batch, host=rng.random() < 0.25)


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _scramble(n, gen):
    return torch.randperm(n, generator=gen, device="cuda").to(torch.int32)


def _rmat(n, m, gen):
    """R-MAT endpoints before the scramble; n need not be a power of two (endpoints are folded into range)."""
    bits = max(1, math.ceil(math.log2(n)))
    a, b, c = 0.57, 0.19, 0.19
    u = torch.zeros(m, dtype=torch.int32, device="cuda")
    v = torch.zeros(m, dtype=torch.int32, device="cuda")
    for _ in range(bits):
        r = torch.rand(m, generator=gen, device="cuda")
        right = r >= a + b
        u.mul_(2).add_(right)
        v.mul_(2).add_(torch.where(right, r >= a + b + c, r >= a))
    if n != 1 << bits:
        u.remainder_(n)
        v.remainder_(n)
    return u, v


def _stream(n, m, gen):
    """Heavy-tailed endpoints; a quarter of the edges repeat earlier ones."""
    def ends():
        x = torch.rand(m, generator=gen, device="cuda")
        return (x * x * x * n).to(torch.int32).clamp_(max=n - 1)

    u, v = ends(), ends()
    if m > 1:
        back = (torch.rand(m, generator=gen, device="cuda") * torch.arange(m, device="cuda")).to(torch.int64)
        rep = torch.rand(m, generator=gen, device="cuda") < 0.25
        u, v = torch.where(rep, u[back], u), torch.where(rep, v[back], v)
    return u, v


def _graph_edges(graph, n, m, gen):
    u, v = torch.empty(m, dtype=torch.int32, device="cuda"), torch.empty(m, dtype=torch.int32, device="cuda")
    perm = _scramble(n, gen)
    make = _rmat if graph == "rmat" else _stream
    for i in range(0, m, CHUNK):
        k = min(CHUNK, m - i)
        a, b = make(n, k, gen)
        u[i:i + k] = perm.index_select(0, a)
        v[i:i + k] = perm.index_select(0, b)
    return u, v, perm


def _keys(u, v):
    return (u.to(torch.int64) << 32) | v.to(torch.int64)


def _split(keys):
    return (keys >> 32).to(torch.int32), (keys & 0xFFFFFFFF).to(torch.int32)


def _in_graph(keys, u, v):
    """Which of the sorted distinct keys are edges of the list (u, v)."""
    found = torch.zeros(keys.numel(), dtype=torch.bool, device="cuda")
    if keys.numel() == 0:
        return found
    for i in range(0, u.numel(), CHUNK):
        k = _keys(u[i:i + CHUNK], v[i:i + CHUNK])
        at = torch.searchsorted(keys, k).clamp_(max=keys.numel() - 1)
        found[at[keys[at] == k]] = True
    return found


def _batch(graph, n, size, u, v, perm, gen):
    """A batch (del_src, del_dst, ins_src, ins_dst) and the one that retracts its effective change."""
    if graph == "stream":
        n_del = 0
    else:
        n_del = size - int(round(0.8 * size))
    n_ins = size - n_del
    at = torch.randint(u.numel(), (n_del,), generator=gen, device="cuda")
    ds, dd = u[at], v[at]
    if graph == "stream":   # the stream's next edges
        a, b = _stream(n, n_ins, gen)
        a, b = perm.index_select(0, a), perm.index_select(0, b)
        old = torch.randint(u.numel(), (n_ins,), generator=gen, device="cuda")
        rep = torch.rand(n_ins, generator=gen, device="cuda") < 0.25
        is_, id_ = torch.where(rep, u[old], a), torch.where(rep, v[old], b)
    else:
        is_ = torch.randint(n, (n_ins,), generator=gen, device="cuda", dtype=torch.int32)
        id_ = torch.randint(n, (n_ins,), generator=gen, device="cuda", dtype=torch.int32)
    ik, dk = torch.unique(_keys(is_, id_)[is_ != id_]), torch.unique(_keys(ds, dd)[ds != dd])
    eff_ins = ik[~_in_graph(ik, u, v)]
    eff_del = dk[~torch.isin(dk, ik)]
    back = _split(eff_ins) + _split(eff_del)
    return tuple(t.contiguous() for t in (ds, dd, is_, id_)), tuple(t.contiguous() for t in back)


def _members(case):
    """The graphs of a group or a server: (n, edges, batch size), sizes log-uniform, edge factors 8 to 32."""
    r = np.random.RandomState(case["count"])
    out = []
    for i in range(case["count"]):
        x = case["lo"] + (case["hi"] - case["lo"]) * (i + r.random_sample()) / case["count"]
        n = int(2.0 ** x) | 1
        m = int(n * (r.uniform(8.0, 32.0) if case["kind"] == "group" else 16.0))
        if case["kind"] == "group":
            size = max(1, int(round(case["share"] * m)))
        else:
            size = int(case["small"] * (case["big"] / case["small"]) ** r.random_sample())
        out.append((n, m, size))
    return out


def _one(graph, n, m, size, gen):
    u, v, perm = _graph_edges(graph, n, m, gen)
    fwd, back = _batch(graph, n, size, u, v, perm, gen) if size else (None, None)
    return u, v, fwd, back


def _host(batch):
    return tuple(t.cpu().numpy() for t in batch)


def prepare(case, seed):
    gen = _gen(seed)
    kind = case["kind"]
    if kind in ("update", "solve", "load"):
        n = case["n"]
        u, v, fwd, back = _one(case["graph"], n, case["edges"], case.get("batch", 0), gen)
        if kind == "load":
            return dict(kind=kind, n=n, u=u, v=v)
        torch.cuda.empty_cache()
        g = pr.Graph.from_edges(n, u, v, device=True)
        del u, v
        torch.cuda.empty_cache()
        if kind == "solve":
            return dict(kind=kind, g=g, n=n)
        g.update("static")
        s = dict(kind=kind, g=g, n=n, method=case["method"], host=case["host"])
        if case["host"]:
            s.update(r0=g.ranks(), fwd=_host(fwd), back=_host(back))
        else:
            s.update(r0=g.ranks_device(torch.empty(n, dtype=torch.float64, device="cuda")), fwd=fwd, back=back)
        return s
    graphs, r0, fwd, back, first = [], [], [], [], [0]
    for n, m, size in _members(case):
        u, v, f, b = _one("rmat", n, m, size, gen)
        g = pr.Graph.from_edges(n, u, v, device=True)
        del u, v
        g.update("static")
        graphs.append(g)
        r0.append(g.ranks_device(torch.empty(n, dtype=torch.float64, device="cuda")))
        fwd.append(f if kind == "group" else _host(f))
        back.append(b if kind == "group" else _host(b))
        first.append(first[-1] + n)
    torch.cuda.empty_cache()
    s = dict(kind=kind, graphs=graphs, r0=r0, fwd=fwd, back=back, first=first, method=case["method"])
    if kind == "group":
        s["group"] = pr.Group(graphs)
    return s


# ------------------------------------------------------------------ one pass

def _counts(st):
    return [st.iterations, st.vertices_ever_affected, st.edges_processed, st.vertices_processed, st.eff_deletions,
            st.eff_insertions]


def _ranks(s, g, n):
    if s.get("host"):
        return g.ranks()
    return g.ranks_device(torch.empty(n, dtype=torch.float64, device="cuda"))


def _all_ranks(s):
    out = torch.empty(s["first"][-1], dtype=torch.float64, device="cuda")
    for g, a, b in zip(s["graphs"], s["first"], s["first"][1:]):
        g.ranks_device(out[a:b])
    return out


def run(s):
    kind = s["kind"]
    if kind == "update":
        g = s["g"]
        (g.set_ranks if s["host"] else g.set_ranks_device)(s["r0"])
        apply = g.apply_batch if s["host"] else g.apply_batch_device
        ranks, counts = [], []
        for batch in (s["fwd"], s["back"]):
            apply(*batch)
            counts.append(_counts(g.update(s["method"])))
            ranks.append(_ranks(s, g, s["n"]))
        return dict(ranks=ranks, counts=np.array(counts, np.int64))
    if kind == "solve":
        st = s["g"].update("static")
        return dict(ranks=[_ranks(s, s["g"], s["n"])], iterations=st.iterations)
    if kind == "load":
        g = pr.Graph.from_edges(s["n"], s["u"], s["v"], device=True)
        st = g.update("static")
        out = dict(ranks=[_ranks(s, g, s["n"])], iterations=st.iterations, edges=g.m)
        g.close()
        return out
    for g, r in zip(s["graphs"], s["r0"]):
        g.set_ranks_device(r)
    ranks, counts = [], []
    if kind == "group":
        q = s["group"]
        for batches in (s["fwd"], s["back"]):
            q.apply_batches_device(batches)
            counts.append([_counts(st) for st in q.update(s["method"])])
            ranks.append(_all_ranks(s))
        return dict(ranks=ranks, counts=np.array(counts, np.int64))
    srv = pr.Server(s["graphs"], method=s["method"])
    for batches in (s["fwd"], s["back"]):
        tickets = [srv.submit(i, *b) for i, b in enumerate(batches)]
        counts.append([_counts(srv.wait(t).stats) for t in tickets])
    srv.close()
    return dict(ranks=[_all_ranks(s)], counts=np.array(counts, np.int64))


def work(case):
    """Every edge of the graph once (a 4-byte id) with its source's 8-byte contribution at least once per vertex,
    ranks read and written, the batch read; an update of a pass with a retraction counts twice.  Two operations per
    edge, ten per vertex."""
    if case["kind"] in ("group", "serve"):
        parts = [(n, m, k, 2) for n, m, k in _members(case)]
    else:
        parts = [(case["n"], case["edges"], case.get("batch", 0), 2 if case["kind"] == "update" else 1)]
    nbytes = flops = 0
    for n, m, k, times in parts:
        nbytes += times * (4 * m + 32 * n + 8 * k) + (8 * m if case["kind"] == "load" else 0)
        flops += times * (2 * m + 10 * n)
    return dict(bytes=nbytes, flops=flops)


# ------------------------------------------------------------------ the same in plain torch, 64 bits

class _Plain:
    """An edge set (self-loop on every vertex) and the methods of the paper in synchronous order."""

    def __init__(self, n, u, v):
        loops = torch.arange(n, device="cuda", dtype=torch.int64)
        self.n = n
        keys = torch.empty(u.numel() + n, dtype=torch.int64, device="cuda")
        keys[:u.numel()] = _keys(u, v)
        keys[u.numel():] = (loops << 32) | loops
        self.set(torch.unique(keys))

    def set(self, keys):
        self.keys = keys
        self.u, self.v = _split(keys)
        first = torch.arange(self.n + 1, device="cuda", dtype=torch.int64) << 32
        self.d = torch.searchsorted(keys, first).diff()

    def edit(self, ds, dd, is_, id_):
        """Deletions first, then insertions; self-loops stay.  Returns the sources of the effective change."""
        dk = torch.unique(_keys(ds, dd)[ds != dd])
        ik = torch.unique(_keys(is_, id_))
        dk = dk[~torch.isin(dk, ik)]

        def has(k):
            at = torch.searchsorted(self.keys, k).clamp_(max=self.keys.numel() - 1)
            return self.keys[at] == k

        dk, ik = dk[has(dk)], ik[~has(ik)]
        before = (self.keys, self.u, self.v)
        keep = torch.ones(self.keys.numel(), dtype=torch.bool, device="cuda")
        keep[torch.searchsorted(self.keys, dk)] = False
        keys = torch.cat([self.keys[keep], ik])
        del keep
        self.set(torch.sort(keys)[0])
        touched = torch.cat([dk, ik]) >> 32
        self.lost = _split(dk)
        self.before = before
        return touched

    def _spread(self, mark, u, v):
        """Out-neighbours of the marked vertices."""
        out = torch.zeros(self.n, dtype=torch.bool, device="cuda")
        for i in range(0, u.numel(), CHUNK):
            hit = mark.index_select(0, u[i:i + CHUNK])
            out[v[i:i + CHUNK][hit].long()] = True
        return out

    def _sums(self, x):
        c = torch.zeros(self.n, dtype=torch.float64, device="cuda")
        for i in range(0, self.u.numel(), CHUNK):
            c.index_add_(0, self.v[i:i + CHUNK], x.index_select(0, self.u[i:i + CHUNK]))
        return c

    def update(self, method, r, touched=None, max_iter=500):
        n, d = self.n, self.d.double()
        c0 = (1.0 - ALPHA) / n
        inside = torch.ones(n, dtype=torch.bool, device="cuda")
        if method == "static":
            r = torch.full((n,), 1.0 / n, dtype=torch.float64, device="cuda")
        elif method in ("df", "dfp", "dt"):
            start = torch.zeros(n, dtype=torch.bool, device="cuda")
            start[touched] = True
            if method == "dt":
                inside = self._reach(start, self.u, self.v) | self._reach(start, *self.before[1:])
            else:
                inside = self._spread(start, self.u, self.v)
                inside[self.lost[1].long()] = True
        for _ in range(max_iter):
            x = r / d
            c = self._sums(x)
            if method == "dfp":
                new = (c0 + ALPHA * (c - x)) / (1.0 - ALPHA / d)
            else:
                new = c0 + ALPHA * c
            dr = torch.where(inside, (new - r).abs(), torch.zeros((), dtype=torch.float64, device="cuda"))
            if method in ("df", "dfp"):
                rel = dr / torch.maximum(new, r)
                out = inside & (rel > TOL)
                stay = inside & (rel > TOL) if method == "dfp" else inside
            r = torch.where(inside, new, r)
            if dr.max().item() <= TAU:
                break
            if method in ("df", "dfp"):
                inside = stay | self._spread(out, self.u, self.v)
        return r

    def _reach(self, start, u, v):
        seen, wave = start.clone(), start
        while True:
            wave = self._spread(wave, u, v) & ~seen
            if not wave.any().item():
                return seen
            seen |= wave


def _plain_update(graph, n, m, size, method, gen):
    u, v, fwd, back = _one(graph, n, m, size, gen)
    p = _Plain(n, u, v)
    del u, v
    r = p.update("static", None)
    out = []
    for batch in (fwd, back):
        r = p.update(method, r, p.edit(*batch))
        out.append(r)
    return out


def exact(case, seed):
    gen = _gen(seed)
    kind = case["kind"]
    if kind == "update":
        ranks = _plain_update(case["graph"], case["n"], case["edges"], case["batch"], case["method"], gen)
        if case["host"]:
            ranks = [r.cpu().numpy() for r in ranks]
        return dict(ranks=ranks, counts=None)
    if kind in ("solve", "load"):
        u, v, _, _ = _one(case["graph"], case["n"], case["edges"], 0, gen)
        p = _Plain(case["n"], u, v)
        out = dict(ranks=[p.update("static", None)], iterations=None)
        return dict(out, edges=None) if kind == "load" else out
    both = [[], []]
    for n, m, size in _members(case):
        for to, r in zip(both, _plain_update("rmat", n, m, size, case["method"], gen)):
            to.append(r)
    ranks = [torch.cat(rs) for rs in both]
    return dict(ranks=ranks if kind == "group" else ranks[1:], counts=None)
