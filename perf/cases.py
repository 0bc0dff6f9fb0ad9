"""Timed workloads of the dynamic graph store, run through its Python API.

Every case is what a program that uses the store does between two answers it
needs: look edges up, apply a batch and bring BFS, SSSP and the components up
to date, load a graph, rank its vertices, count its triangles, size its hash
tables.  Graphs are R-MAT graphs (a, b, c = .57, .19, .19, self-loops and
repeated pairs dropped) or road-like grids, of the sizes the benchmark and the
tests of this repository use; sources are the vertex of the largest
out-degree (R-MAT) or the corner vertex (grid).

Deleted pairs are never reused by the store, so a program that keeps updating
one graph loads it anew from time to time.  The update cases do that when a
quarter of the edges have been deleted: it is part of the pass it falls in,
and each pass leaves the edge set as it found it.
"""
from __future__ import annotations

import math

import torch

import paper_2305_17813_gb300 as mk
from paper_2305_17813_gb300 import sizing

DEVICE = "cuda"
LOAD_FACTOR = 0.7


def listed():
    return [
        # a few lookups on a graph that fits the caches: launch and latency
        {"name": "query_small", "kind": "query", "scale": 14, "degree": 16, "n": 1003, "weights": True},
        # the benchmark's lookups on its graph: half present, stored weights asked for
        {"name": "query_large", "kind": "query", "scale": 20, "degree": 16, "n": 2097169, "weights": True},
        # a service's round: many small insert, delete and query requests, then BFS and SSSP brought up to date
        {"name": "requests", "kind": "requests", "scale": 17, "degree": 16, "requests": 48, "edges": 200},
        # a small batch on a middling graph: insert, commit, delete, commit, every algorithm after each, lookups
        {"name": "step_small", "kind": "step", "scale": 18, "degree": 16, "batch": 4099, "batches": 1, "fresh": False},
        # the benchmark's graph and batch: load it, run every algorithm, then three whole steps
        {"name": "step_large", "kind": "step", "scale": 20, "degree": 16, "batch": 1 << 20, "batches": 3, "fresh": True},
        # raw edge list (repeats and self-loops in it) to a committed graph sized by the load-factor rule
        {"name": "load", "kind": "load", "scale": 21, "degree": 16},
        # BFS, SSSP and components from scratch, after an epoch that none of them followed
        {"name": "static", "kind": "static", "scale": 20, "degree": 16},
        # road grid: ordered SSSP from scratch after links closed and opened, then incrementally as they change back
        {"name": "road", "kind": "road", "side": 1024, "batch": 8192, "delta": 4000},
        # ranks from the uniform start
        {"name": "pagerank", "kind": "pagerank", "scale": 20, "degree": 16, "warm": False},
        # triangles of an undirected graph, and the change that its last batch made
        {"name": "triangles", "kind": "triangles", "scale": 17, "degree": 16, "batch": 20011},
        # the unweighted layout's whole life: sized, loaded, searched, updated, queried
        {"name": "set_graph", "kind": "set", "scale": 19, "degree": 16, "batch": 1 << 18},
        # learned sizing: features, targets, one training gradient, bucket counts for every vertex
        {"name": "sizing", "kind": "sizing", "vertices": 1 << 22, "sample": 1 << 18},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["query", "query", "requests", "step", "step", "load", "static", "road", "pagerank", "triangles",
                       "set", "sizing"])
    degree = rng.randint(4, 16)
    if kind == "query":
        return {"kind": kind, "scale": rng.randint(12, 20), "degree": degree, "n": _log_int(rng, 100, 1 << 21),
                "weights": rng.random() < 0.7}
    if kind == "requests":
        return {"kind": kind, "scale": rng.randint(12, 17), "degree": degree, "requests": rng.randint(4, 64),
                "edges": _log_int(rng, 16, 1000)}
    if kind == "step":
        scale = rng.randint(13, 20)
        most = (degree << scale) // 8
        if rng.random() < 0.5:
            return {"kind": kind, "scale": scale, "degree": degree, "batch": _log_int(rng, 256, most // 8),
                    "batches": 1, "fresh": False}
        return {"kind": kind, "scale": scale, "degree": degree, "batch": _log_int(rng, most // 16, most),
                "batches": rng.randint(1, 2), "fresh": True}
    if kind == "load":
        return {"kind": kind, "scale": rng.randint(14, 21), "degree": degree}
    if kind == "static":
        return {"kind": kind, "scale": rng.randint(14, 20), "degree": degree}
    if kind == "road":
        return {"kind": kind, "side": _log_int(rng, 100, 1024), "batch": _log_int(rng, 64, 1024),
                "delta": rng.choice([0, 1500, 4000])}
    if kind == "pagerank":
        return {"kind": kind, "scale": rng.randint(13, 20), "degree": degree, "warm": rng.random() < 0.5}
    if kind == "triangles":
        return {"kind": kind, "scale": rng.randint(12, 17), "degree": degree, "batch": _log_int(rng, 200, 20000)}
    if kind == "set":
        scale = rng.randint(13, 19)
        return {"kind": kind, "scale": scale, "degree": degree, "batch": _log_int(rng, 256, (degree << scale) // 16)}
    return {"kind": kind, "vertices": _log_int(rng, 10000, 1 << 22), "sample": _log_int(rng, 2000, 1 << 18)}


# ------------------------------------------------------------------ inputs

def _generator(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    return g


def _rmat(scale, n, gen):
    """n R-MAT pairs of 2^scale vertices, as 64-bit ids."""
    src = torch.zeros(n, dtype=torch.int64, device=DEVICE)
    dst = torch.zeros(n, dtype=torch.int64, device=DEVICE)
    for _ in range(scale):
        u = torch.rand(n, generator=gen, device=DEVICE)
        src.mul_(2).add_(u >= 0.76)
        dst.mul_(2).add_(((u >= 0.57) & (u < 0.76)) | (u >= 0.95))
    return src, dst


def _shuffled(x, gen):
    return x[torch.randperm(x.numel(), generator=gen, device=DEVICE)]


def _keys(scale, n, gen):
    """Sorted distinct pairs (src << scale | dst) of n R-MAT draws, self-loops dropped."""
    s, d = _rmat(scale, n, gen)
    return torch.unique(((s << scale) | d)[s != d])


def _absent(keys, sorted_keys):
    at = torch.searchsorted(sorted_keys, keys).clamp_(max=sorted_keys.numel() - 1)
    return sorted_keys[at] != keys


def _new_keys(scale, want, keys, gen):
    """`want` distinct pairs that are not among `keys` (fewer only if the graph is nearly complete)."""
    got = keys[:0]
    for _ in range(20):
        more = _keys(scale, 2 * want + 64, gen)
        got = torch.unique(torch.cat([got, more[_absent(more, keys)]]))
        if got.numel() >= want:
            break
    return _shuffled(got, gen)[:want]


def _split(keys, scale):
    return (keys >> scale).int(), (keys & ((1 << scale) - 1)).int()


def _weights(n, gen, hi=100):
    return torch.randint(1, hi + 1, (n,), generator=gen, device=DEVICE, dtype=torch.int32)


def _uniform(n, hi, gen):
    return torch.randint(0, hi, (n,), generator=gen, device=DEVICE, dtype=torch.int64)


def _half_present(keys, scale, n, gen):
    """n lookups, half of them pairs of `keys`, the rest uniform pairs."""
    half = n // 2
    q = torch.cat([keys[_uniform(half, keys.numel(), gen)], _uniform(n - half, 1 << (2 * scale), gen)])
    return _split(_shuffled(q, gen), scale)


def _rmat_base(case, gen):
    """Edge list of the case's graph in random order: (sorted keys, src, dst, w, hub)."""
    scale = case["scale"]
    keys = _keys(scale, case["degree"] << scale, gen)
    src, dst = _split(_shuffled(keys, gen), scale)
    hub = int(torch.bincount(src, minlength=1 << scale).argmax())
    return keys, src, dst, _weights(src.numel(), gen), hub


def _open(V, src, dst, w, spare=0):
    """A committed graph of these edges, sized by the load-factor rule, with
    pool room for `spare` more pairs."""
    g = mk.Graph(V, edge_capacity_hint=src.numel() + spare, buckets=mk.bucket_rule(V, src, LOAD_FACTOR))
    g.insert(src, dst, w, flags=False)
    g.commit()
    return g


# ------------------------------------------------------------------- kinds

class _Query:
    def __init__(self, case, gen):
        keys, src, dst, w, _ = _rmat_base(case, gen)
        self.g = _open(1 << case["scale"], src, dst, w)
        self.weights = case["weights"]
        self.q = _half_present(keys, case["scale"], case["n"], gen)

    def run(self):
        bitmap, w = self.g.query(*self.q, weights=self.weights)
        return (bitmap, w) if self.weights else bitmap


class _Updates:
    """A graph and the batches of one cycle: batch k inserts pairs that the
    graph lacks (beside some that it holds and some repeats) and deletes the
    new ones again.  After a cycle, a quarter of the edges deleted, the graph
    is loaded anew."""

    def __init__(self, case, gen, batch, cycle=None):
        scale = case["scale"]
        self.V = 1 << scale
        self.keys, self.src, self.dst, self.w, self.hub = _rmat_base(case, gen)
        E = self.src.numel()
        held, again = batch // 16, batch // 64
        new = batch - held - again
        self.cycle = cycle or max(1, min(E // 4 // new, 4096))
        fresh = _new_keys(scale, self.cycle * new, self.keys, gen)
        self.cycle = max(1, fresh.numel() // new)
        fresh = fresh[: self.cycle * new].view(self.cycle, -1)
        pick = torch.cat([fresh, self.keys[_uniform(self.cycle * held, E, gen)].view(self.cycle, held),
                          fresh[:, :again]], 1)
        pick = pick[:, torch.randperm(pick.shape[1], generator=gen, device=DEVICE)].contiguous()
        self.ins = _split(pick, scale)
        self.ins_w = _weights(pick.numel(), gen).view(pick.shape)
        self.dele = _split(fresh.contiguous(), scale)
        self.spare = 2 * self.cycle * new
        self.g, self.k = None, 0

    def reload(self):
        if self.g is not None:
            self.g.close()
        self.g, self.k = _open(self.V, self.src, self.dst, self.w, self.spare), 0

    def answers(self):
        return self.g.bfs(self.hub), self.g.sssp(self.hub), self.g.wcc()


class _Step(_Updates):
    def __init__(self, case, gen):
        self.fresh, self.batches = case["fresh"], case["batches"]
        super().__init__(case, gen, case["batch"], cycle=case["batches"] if case["fresh"] else None)
        n = case["batch"]
        q = _half_present(self.keys, case["scale"], n * self.cycle, gen)
        self.q = [x.view(self.cycle, n) for x in q]
        if not self.fresh:
            self.reload()
            self.answers()

    def step(self):
        g, k = self.g, self.k
        out = [g.insert(self.ins[0][k], self.ins[1][k], self.ins_w[k]), self.answers()]
        g.commit()
        out += [g.delete(self.dele[0][k], self.dele[1][k]), self.answers()]
        g.commit()
        out.append(g.query(self.q[0][k], self.q[1][k]))
        self.k += 1
        return out

    def run(self):
        if not self.fresh and self.k + self.batches <= self.cycle:
            return [self.step() for _ in range(self.batches)]
        self.reload()
        first = self.answers()
        steps = [self.step() for _ in range(min(self.batches, self.cycle))]
        return [first] + steps if self.fresh else steps


class _Requests(_Updates):
    def __init__(self, case, gen):
        # uneven requests, from a twentieth to twice the mean
        n = case["requests"]
        sizes = [max(1, case["edges"] * (1 + 39 * (7 * i % n) // n) // 20) for i in range(n)]
        super().__init__(case, gen, sum(sizes))
        cut = lambda total: [0] + [min(total, sum(sizes[: i + 1])) for i in range(len(sizes))]  # noqa: E731
        self.cut_ins, self.cut_del = cut(self.ins[0].shape[1]), cut(self.dele[0].shape[1])
        q = _half_present(self.keys, case["scale"], sum(sizes), gen)
        self.queries = [(q[0][a:b], q[1][a:b]) for a, b in zip(self.cut_ins, self.cut_ins[1:])]
        self.wanted = [("sssp", self.hub), ("bfs", self.hub)]
        self.reload()

    def reload(self):
        super().reload()
        self.g.incr_multi(self.wanted)

    def run(self):
        if self.k >= self.cycle:
            self.reload()
        g, k = self.g, self.k
        (s, d), w, (ds, dd) = self.ins, self.ins_w, self.dele
        ups = [("insert", s[k, a:b], d[k, a:b], w[k, a:b]) for a, b in zip(self.cut_ins, self.cut_ins[1:])]
        found = g.update_multi(ups), g.query_multi(self.queries), g.incr_multi(self.wanted)
        g.commit()
        ups = [("delete", ds[k, a:b], dd[k, a:b]) for a, b in zip(self.cut_del, self.cut_del[1:])]
        gone = g.update_multi(ups), g.incr_multi(self.wanted)
        g.commit()
        self.k += 1
        # one tensor for each kind of answer
        flags, answers, trees = found
        return [torch.cat(flags), torch.cat([b for b, _ in answers]), torch.cat([x for _, x in answers]), trees,
                torch.cat(gone[0]), gone[1]]


class _Load:
    def __init__(self, case, gen):
        self.V = 1 << case["scale"]
        s, d = _rmat(case["scale"], case["degree"] << case["scale"], gen)
        self.src, self.dst, self.w = s.int(), d.int(), _weights(s.numel(), gen)

    def run(self):
        buckets = mk.bucket_rule(self.V, self.src, LOAD_FACTOR)
        g = mk.Graph(self.V, edge_capacity_hint=self.src.numel(), buckets=buckets)
        flags = g.insert(self.src, self.dst, self.w)
        g.commit()
        g.close()
        return buckets, flags


class _Static:
    def __init__(self, case, gen):
        _, src, dst, w, self.hub = _rmat_base(case, gen)
        self.g = _open(1 << case["scale"], src, dst, w)
        self.seen = src[:1000].clone(), dst[:1000].clone(), w[:1000].clone()

    def run(self):
        flags = self.g.insert(*self.seen)  # edges that the graph holds: an epoch without a change
        self.g.commit()
        return flags, self.g.bfs(self.hub), self.g.sssp(self.hub), self.g.wcc()


class _Road:
    def __init__(self, case, gen):
        n = case["side"]
        self.V, self.delta = n * n, case["delta"]
        v = torch.arange(n * n, device=DEVICE).view(n, n)
        a = torch.cat([v[:, :-1].reshape(-1), v[:-1].reshape(-1)])
        b = torch.cat([v[:, 1:].reshape(-1), v[1:].reshape(-1)])
        grid = _shuffled(torch.cat([a * self.V + b, b * self.V + a]), gen)
        far = _uniform(max(1, grid.numel() // 1000), self.V * self.V, gen)
        keys = torch.unique(torch.cat([grid, far[far // self.V != far % self.V]]))
        E = keys.numel()
        keys = _shuffled(keys, gen)
        self.src, self.dst, self.w = (keys // self.V).int(), (keys % self.V).int(), _weights(E, gen, 1000)
        # batch k closes links and opens diagonals
        B = case["batch"]
        self.cycle = max(1, min(E // 8 // B, 256))
        self.shut = torch.randperm(E, generator=gen, device=DEVICE)[: self.cycle * B].view(self.cycle, -1)
        corner = v[:-1, :-1].reshape(-1)
        corner = _shuffled(corner, gen)[: self.shut.numel()]
        self.cycle = min(self.cycle, corner.numel() // B)
        corner = corner[: self.cycle * B].view(self.cycle, B)
        self.open = corner.int(), (corner + n + 1).int()
        self.open_w = _weights(corner.numel(), gen, 1000).view(corner.shape)
        self.g = None
        self.reload()

    def reload(self):
        if self.g is not None:
            self.g.close()
        self.g = mk.Graph(self.V, edge_capacity_hint=2 * self.src.numel(), buckets=1)
        self.g.set_sssp_delta(self.delta, 0)
        self.g.insert(self.src, self.dst, self.w, flags=False)
        self.g.commit()
        self.g.sssp(0)
        self.k = 0

    def run(self):
        if self.k >= self.cycle:
            self.reload()
        g, k = self.g, self.k
        at = self.shut[k]
        links, diagonals = (self.src[at], self.dst[at]), (self.open[0][k], self.open[1][k])
        out = [g.delete(*links), g.insert(*diagonals, self.open_w[k])]
        g.commit()  # the tree has not followed this epoch
        out.append(g.sssp(0))
        out += [g.delete(*diagonals), g.insert(*links, self.w[at])]
        out.append(g.sssp(0))
        g.commit()
        self.k += 1
        return out


class _PageRank:
    def __init__(self, case, gen):
        keys, self.src, self.dst, w, _ = _rmat_base(case, gen)
        self.V = 1 << case["scale"]
        more = _new_keys(case["scale"], max(1, self.src.numel() // 64), keys, gen)
        self.more = _split(more, case["scale"])
        self.g = _open(self.V, self.src, self.dst, w, more.numel())
        self.before = self.g.pagerank()[0] if case["warm"] else None
        self.g.insert(*self.more, flags=False)
        self.g.commit()

    def run(self):
        # warm: the ranks before the last batch
        return self.g.pagerank(None if self.before is None else self.before.clone())


class _Triangles:
    def __init__(self, case, gen):
        scale = case["scale"]
        self.V = 1 << scale
        s, d = _rmat(scale, case["degree"] << scale, gen)
        lo, hi = torch.minimum(s, d), torch.maximum(s, d)
        pairs = _shuffled(torch.unique(((lo << scale) | hi)[lo != hi]), gen)
        last = pairs[: min(case["batch"], pairs.numel() // 2)]
        src, dst = self.both(pairs, scale)
        self.g = _open(self.V, src, dst, None)
        self.batch = self.both(last, scale)
        self.upd = _open(self.V, *self.batch, None)

    @staticmethod
    def both(pairs, scale):
        a, b = _split(pairs, scale)
        return torch.cat([a, b]), torch.cat([b, a])

    def run(self):
        return self.g.triangles(), self.g.triangle_delta(self.upd, *self.batch, False)


class _Set:
    def __init__(self, case, gen):
        scale = case["scale"]
        self.V = 1 << scale
        s, d = _rmat(scale, case["degree"] << scale, gen)
        keys, n = torch.unique((s << scale) | d), case["batch"]
        self.src, self.dst = s.int(), d.int()
        self.hub = int(torch.bincount(s, minlength=self.V).argmax())
        self.dele = _split(keys[torch.randperm(keys.numel(), generator=gen, device=DEVICE)[:n]], scale)
        self.ins = _split(_new_keys(scale, n, keys, gen), scale)
        self.q = _half_present(keys, scale, n, gen)

    def run(self):
        g = mk.SetGraph(self.V, edge_capacity_hint=2 * self.src.numel(),
                        buckets=mk.set_bucket_rule(self.V, self.src, LOAD_FACTOR))
        out = [g.insert(self.src, self.dst), g.bfs(self.hub), g.wcc()]
        out += [g.delete(*self.dele), g.insert(*self.ins), g.query(*self.q), g.bfs(self.hub), g.wcc()]
        g.close()
        return out


class _Sizing:
    horizon = 8.0

    def __init__(self, case, gen):
        V = case["vertices"]
        # heavy-tailed degrees that grew over the last five batches
        growth = torch.rand(V, generator=gen, device=DEVICE).add_(1e-4).pow_(-0.7).mul_(4).long()
        self.trace = sizing.DegreeTrace(V)
        for k in range(5):
            part = torch.rand(V, generator=gen, device=DEVICE).mul_(0.1).add_(0.9 - 0.15 * k)
            self.trace.hist[k] = (growth * part).int()
        self.trace.out_deg.copy_(self.trace.hist[0])
        self.trace.in_deg.copy_(_shuffled(growth, gen).int())
        self.later = (growth * 2).int()
        self.count = (self.trace.out_deg / (LOAD_FACTOR * 15)).ceil().clamp_(min=1).int()
        scale = torch.cat([torch.full((512,), (2 / 8) ** 0.5), torch.zeros(64), torch.full((4096,), (2 / 64) ** 0.5),
                           torch.zeros(64), torch.full((64,), (2 / 64) ** 0.5), torch.zeros(1)]).to(DEVICE)
        self.params = torch.randn(4801, generator=gen, device=DEVICE) * scale
        self.model = sizing.SizingModel()
        self.model.set_params(self.params.cpu().numpy())
        self.rows = torch.randperm(V, generator=gen, device=DEVICE)[: min(case["sample"], V)]

    def run(self):
        X = self.trace.features(self.count)
        T = sizing.growth_targets(self.trace.hist[4], self.later, self.horizon)
        grad, sse = self.model.gradient(X[self.rows].contiguous(), T[self.rows].contiguous())
        buckets, y = self.model.buckets(X, self.trace.out_deg, self.horizon, LOAD_FACTOR)
        return X, T, grad, (sse / self.rows.numel()).float(), buckets, y


KINDS = {"query": _Query, "requests": _Requests, "step": _Step, "load": _Load, "static": _Static, "road": _Road,
         "pagerank": _PageRank, "triangles": _Triangles, "set": _Set, "sizing": _Sizing}


def prepare(case, seed):
    return KINDS[case["kind"]](case, _generator(seed))


def run(state):
    return state.run()


# -------------------------------------------------------------------- work

def work(case):
    """Bytes of one pass: its batches and their flags or answers, 8 bytes for
    each stored edge that it has to read or write, its result arrays.  Each
    graph is counted once for each pass over all of it that no incremental
    state can save (from-scratch runs, components after a delete)."""
    kind, flops = case["kind"], 0.0
    if "scale" in case:
        V = 1 << case["scale"]
        E = case["degree"] * V
    tree = 8  # distance and parent
    if kind == "query":
        n = case["n"]
        moved = n * (8 + 8 + (4 if case["weights"] else 0)) + n / 8
    elif kind == "requests":
        n = case["requests"] * case["edges"]
        moved = n * (12 + 1 + 8) + n * (8 + 1 + 8) + n * (8 + 8 + 4) + n / 8 + 4 * tree * V
    elif kind == "step":
        n = case["batch"]
        moved = n * (12 + 1 + 8) + n * (8 + 1 + 8) + n * (8 + 8 + 4) + n / 8 + 2 * (2 * tree + 4) * V + 8 * E
        moved *= case["batches"]
        if case["fresh"]:
            moved += E * (12 + 8) + 8 * E + (2 * tree + 4) * V
    elif kind == "load":
        moved = E * (12 + 1 + 8) + 4 * V
    elif kind == "static":
        moved = 8 * E + (2 * tree + 4) * V
    elif kind == "road":
        V = case["side"] ** 2
        moved = 2 * case["batch"] * (8 + 1 + 8 + 12 + 1 + 8) + 8 * 4 * V + 2 * tree * V
    elif kind == "pagerank":
        moved = 8 * E + 4 * V * (2 if case["warm"] else 1)
    elif kind == "triangles":
        moved = 8 * 2 * E + 2 * case["batch"] * 8
    elif kind == "set":
        n = case["batch"]
        moved = E * (8 + 1 + 4) + 2 * n * (8 + 1 + 4) + n * 12 + 2 * (4 * E + (tree + 4) * V)
    else:
        V, n = case["vertices"], case["sample"]
        moved = V * (5 * 4 + 4 + 4 + 32) + V * 12 + n * 36 + V * (4 + 4 + 4) + 4801 * 8
        flops = 2.0 * 4672 * (V + 3 * n)
    return {"bytes": float(moved), "flops": flops}


# ------------------------------------------------------------------- exact

def _pagerank64(src, dst, V, damping=0.85, eps=1e-7, most=100):
    s, d = src.long(), dst.long()
    out = torch.bincount(s, minlength=V).double()
    pr = torch.full((V,), 1.0 / V, dtype=torch.float64, device=DEVICE)
    delta, steps = 0.0, 0
    while steps < most:
        share = torch.where(out > 0, pr / out.clamp(min=1), torch.zeros_like(pr))
        into = torch.zeros_like(pr).index_add_(0, d, share[s])
        new = (1 - damping) / V + damping * (into + pr[out == 0].sum() / V)
        delta = float((new - pr).abs().sum())
        pr, steps = new, steps + 1
        if delta <= eps:
            break
    return pr, steps, delta


def _sizing64(state):
    """Features, targets, gradient, mean squared error and prediction in 64
    bits, of the network's parameters rounded to bfloat16."""
    t = state.trace
    log1p = lambda x: torch.log1p(x.clamp(min=0))  # noqa: E731
    hist, into = t.hist.double(), t.in_deg.double()
    cols = [log1p(hist[0])] + [log1p(hist[0] - hist[k]) for k in range(1, 5)]
    cols += [log1p(into), log1p(into) - log1p(hist[0]), hist[0] / (15.0 * state.count.double())]
    X = torch.stack(cols, 1)
    T = log1p((state.later.double() - hist[4]) / state.horizon)
    P = state.params.bfloat16().double()
    W1, b1, W2, b2, w3, b3 = P.split([512, 64, 4096, 64, 64, 1])
    W1, W2 = W1.view(8, 64), W2.view(64, 64)

    def forward(x):
        h1 = (x @ W1 + b1).clamp(min=0)
        h2 = (h1 @ W2 + b2).clamp(min=0)
        return h1, h2, h2 @ w3 + b3

    # the network's inputs are 32-bit features
    x, n = X.float()[state.rows].double(), state.rows.numel()
    h1, h2, y = forward(x)
    e = y - T.float()[state.rows].double()
    dy = 2 * e / n
    dz2 = (h2 > 0) * (dy[:, None] * w3)
    dz1 = (h1 > 0) * (dz2 @ W2.T)
    grad = torch.cat([(x.T @ dz1).reshape(-1), dz1.sum(0), (h1.T @ dz2).reshape(-1), dz2.sum(0), h2.T @ dy,
                      dy.sum().view(1)])
    every = torch.cat([forward(part.double())[2] for part in X.float().split(1 << 19)])
    return X, T, grad, (e * e).sum() / n, None, every


def exact(case, seed):
    """64-bit values of the computed outputs; the other kinds return whole
    numbers, which have to be equal."""
    if case["kind"] == "pagerank" and not case["warm"]:
        state = prepare(case, seed)
        src, dst = torch.cat([state.src, state.more[0]]), torch.cat([state.dst, state.more[1]])
        return _pagerank64(src, dst, state.V)
    if case["kind"] == "sizing":
        return _sizing64(prepare(case, seed))
    return None
