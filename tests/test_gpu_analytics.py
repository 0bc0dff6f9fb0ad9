"""PageRank and triangle counting on the GPU against the oracle.

PageRank: the device works in 64-bit fixed point (scale 2^48) and stops
when the L1 change of a super-step is <= 1e-7; the oracle iterates in
double precision to 1e-13.  The distance to the common fixpoint is then at
most about 1e-7 * d / (1 - d) = 5.7e-7 (d = 0.85) on the device side, plus
its rounding (below 2^-48 per added term, and the float32 output: 2^-24
relative per rank, at most 6e-8 in L1), so the test bound is an L1
distance of 1e-5 between the two rank vectors.  Results are bit-identical
from run to run (integer atomics).  Triangle counts are exact integers:
static counts and the running count after insert and delete batches
(inclusion-exclusion over the batch) equal the oracle's brute-force count.
"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
L1_TOL = 1e-5


def _mk():
    import paper_2305_17813_gb300 as mk

    mk.load()
    return mk


def test_pagerank_static_incremental_decremental(cuda_lib):
    import torch

    mk = _mk()
    G = synth.powerlaw_graph(scale=14, draws=1 << 18)
    b = mk.bucket_rule(G.V, G.src, 0.7)
    g = mk.Graph(G.V, edge_capacity_hint=len(G.src) * 2, buckets=b)
    g.insert(G.src, G.dst, G.w)
    g.commit()
    o = oracle.OracleGraph(G.V)
    o.insert(G.src, G.dst, G.w)
    pr, it_static, delta = g.pagerank(eps=1e-7, max_iter=300)
    assert delta <= 1e-7 and it_static < 300
    ref, _ = o.pagerank(eps=1e-13, max_iter=3000)
    assert np.abs(pr.cpu().numpy().astype(np.float64) - ref).sum() <= L1_TOL
    assert abs(float(pr.double().sum()) - 1.0) < 1e-4
    # the same bits on a second run
    pr2, it2, _ = g.pagerank(eps=1e-7, max_iter=300)
    assert it2 == it_static and torch.equal(pr, pr2)
    S = synth.PowerlawStream(G, max_batch=1 << 12)
    bt = S.batch(1 << 12)
    for step in ("insert", "delete"):
        if step == "insert":
            g.insert(bt.ins_src, bt.ins_dst, bt.ins_w)
            o.insert(bt.ins_src, bt.ins_dst, bt.ins_w)
        else:
            g.delete(bt.del_src, bt.del_dst)
            o.delete(bt.del_src, bt.del_dst)
        g.commit()
        # warm start from the ranks before the batch (the dynamic case)
        pr, it_warm, _ = g.pagerank(pr, eps=1e-7, max_iter=300)
        ref, _ = o.pagerank(eps=1e-13, max_iter=3000)
        assert np.abs(pr.cpu().numpy().astype(np.float64) - ref).sum() <= L1_TOL, step
        assert it_warm < it_static, (step, it_warm, it_static)
    assert g.last_error() == mk.MK_OK


def _undirected(s, d):
    keep = s != d
    s, d = s[keep], d[keep]
    a = np.concatenate([s, d]).astype(np.uint32)
    b = np.concatenate([d, s]).astype(np.uint32)
    return a, b


def test_triangles_static_and_after_batches(cuda_lib):
    mk = _mk()
    G = synth.powerlaw_graph(scale=12, draws=1 << 15)
    V = G.V
    s, d = _undirected(G.src, G.dst)
    b = mk.bucket_rule(V, s, 0.7)
    g = mk.Graph(V, edge_capacity_hint=len(s) * 3, buckets=b)
    g.insert(s, d)
    g.commit()
    o = oracle.OracleGraph(V)
    o.insert(s, d)
    count = g.triangles()
    assert count == o.triangles() and count > 1000
    rng = np.random.default_rng(3)
    es, ed, _ = o.export()
    for k in range(4):
        deletion = k % 2 == 1
        if not deletion:
            # new edges: random pairs, plus a K4 on four vertices and a fan,
            # so that triangles with two and three new edges occur
            bs = rng.integers(0, V, 3000)
            bd = rng.integers(0, V, 3000)
            q = rng.choice(V, 6, replace=False)
            k4 = [(q[i], q[j]) for i in range(4) for j in range(i + 1, 4)]
            fan = [(q[4], x) for x in (q[0], q[1], q[5])]
            bs = np.concatenate([bs, [a for a, _ in k4 + fan]]).astype(np.uint32)
            bd = np.concatenate([bd, [c for _, c in k4 + fan]]).astype(np.uint32)
            us, ud = _undirected(bs, bd)
            f = g.insert(us, ud).cpu().numpy().astype(bool)
            assert np.array_equal(f, o.insert(us, ud).astype(bool))
        else:
            es, ed, _ = o.export()
            pick = rng.choice(len(es), 2000, replace=False)
            us, ud = _undirected(es[pick], ed[pick])
            f = g.delete(us, ud).cpu().numpy().astype(bool)
            assert np.array_equal(f, o.delete(us, ud).astype(bool))
        # the batch's applied edges, both directions, and a graph of just them
        ns, nd = us[f], ud[f]
        upd = mk.Graph(V, edge_capacity_hint=len(ns) + 64, buckets=1)
        upd.insert(ns, nd)
        delta = g.triangle_delta(upd, ns, nd, deletion)
        upd.close()
        count += delta
        assert count == o.triangles(), (k, delta)
        assert g.triangles() == count
        g.commit()
    assert g.last_error() == mk.MK_OK


def test_analytics_degenerate_graphs(cuda_lib):
    """No edges: every vertex dangles, the teleport term alone gives ranks
    1 / V.  A grid (no triangles) counts 0, and an empty batch changes
    nothing."""
    mk = _mk()
    g = mk.Graph(1000, edge_capacity_hint=16, buckets=1)
    pr, it, _ = g.pagerank(eps=1e-7)
    assert np.allclose(pr.cpu().numpy(), 1e-3, rtol=1e-6) and it <= 2
    g.close()
    s, d = synth.grid_pairs(30, 30)
    grid = mk.Graph(900, edge_capacity_hint=len(s) * 2, buckets=2)
    grid.insert(s, d)
    assert grid.triangles() == 0
    upd = mk.Graph(900, edge_capacity_hint=16, buckets=1)
    assert grid.triangle_delta(upd, np.zeros(0, np.uint32), np.zeros(0, np.uint32), False) == 0
    lib = mk.load()
    assert lib.mk_l2_window(grid.handle, 7, None, None) == mk.MK_ERR_INVALID_ARG
    assert grid.last_error() == mk.MK_OK
    upd.close()
    grid.close()


@pytest.mark.parametrize("V", [5000, (1 << 20) + 9])  # bitmaps, hash sets
@pytest.mark.parametrize("buckets", [1, "rule"])
def test_triangles_neighbourhood_sizes(cuda_lib, V, buckets):
    """Vertices with 2 to 1,500 neighbours ranked above them (one warp up to
    32, then one block, which takes hash sets 1,024 at a time): a clique of 90,
    a hub joined to 1,500 vertices, sparse edges among those."""
    mk = _mk()
    rng = np.random.default_rng(V)
    name = np.sort(rng.choice(V, 1600, replace=False)).astype(np.uint32)
    i, j = np.triu_indices(90, 1)
    a = [i, np.zeros(1500, np.int64), rng.integers(0, 1600, 6000)]
    b = [j, np.arange(1, 1501), rng.integers(0, 1600, 6000)]
    pairs = np.unique(np.sort(np.stack([np.concatenate(a), np.concatenate(b)], 1), 1), axis=0)
    s, d = _undirected(name[pairs[:, 0]], name[pairs[:, 1]])
    o = oracle.OracleGraph(V)
    o.insert(s, d, np.ones(len(s), np.uint32))
    nb = 1 if buckets == 1 else mk.bucket_rule(V, s, 0.7)
    g = mk.Graph(V, edge_capacity_hint=2 * len(s), buckets=nb)
    g.insert(s, d)
    g.commit()
    assert g.triangles() == o.triangles()
    assert g.last_error() == mk.MK_OK
    g.close()


@pytest.mark.parametrize("V", [700, 70000, 3000000])  # one bin; bins of packed edges; of wide ones
def test_pagerank_binned_and_pushed(cuda_lib, V):
    """A call of three super-steps at most pushes, one of more bins its edges:
    both against double precision within the float32 rounding of the ranks
    (2^-24 of each) and 2^-48 for each of the in-degree + 3 terms of a step,
    and stopping after the same step with the same delta."""
    mk = _mk()
    rng = np.random.default_rng(V)
    n = min(8 * V, 400000)
    s = rng.integers(0, V, n).astype(np.uint32)
    d = (rng.integers(0, V, n) * rng.random(n) ** 3).astype(np.uint32)  # some vertices with many in-edges
    g = mk.Graph(V, edge_capacity_hint=2 * n, buckets=mk.bucket_rule(V, s, 0.7))
    g.insert(s, d)
    g.commit()
    pushed, it, _ = g.pagerank(eps=1e-30, max_iter=3)
    binned, it4, _ = g.pagerank(eps=1e-30, max_iter=4)
    assert (it, it4) == (3, 4)
    # the oracle's steps in double precision
    k = np.unique(s.astype(np.int64) * V + d)
    us, ud = k // V, k % V
    out = np.bincount(us, minlength=V)
    pr, damp = np.full(V, 1.0 / V), float(np.float32(0.85))
    for step in range(4):
        share = np.where(out > 0, pr / np.maximum(out, 1), 0.0)
        pr = (1 - damp) / V + damp * (np.bincount(ud, share[us], minlength=V) + pr[out == 0].sum() / V)
        if step == 2:
            three = pr.copy()
    term = (np.bincount(ud, minlength=V) + 3) * 4 * 2.0 ** -48
    for got, want in ((pushed, three), (binned, pr)):
        err = np.abs(got.cpu().numpy().astype(np.float64) - want)
        assert (err <= want * 2.0 ** -24 + term.max() + term).all()
    # the stop after the same step with both forms
    _, i3, d3 = g.pagerank(eps=0.5, max_iter=3)
    _, i9, d9 = g.pagerank(eps=0.5, max_iter=9)
    assert i3 == i9 and d3 == d9
    assert g.last_error() == mk.MK_OK
    g.close()


@pytest.mark.parametrize("buckets", [1, 3])
def test_triangles_without_work_arrays(cuda_lib, buckets):
    """The count over the slab lists themselves, used where the neighbours'
    copy does not fit: vertices with one slab and with chains, deleted pairs."""
    from paper_2305_17813_gb300._native import MK_DEBUG_NO_SCRATCH

    mk = _mk()
    rng = np.random.default_rng(buckets)
    V = 400
    i, j = np.triu_indices(40, 1)
    a = np.concatenate([i, np.zeros(V - 1, np.int64), rng.integers(0, V, 4000)])
    b = np.concatenate([j, np.arange(1, V), rng.integers(0, V, 4000)])
    pairs = np.unique(np.sort(np.stack([a, b], 1), 1), axis=0)
    pairs = pairs[pairs[:, 0] != pairs[:, 1]]
    s, d = _undirected(*pairs.T.astype(np.uint32))
    o = oracle.OracleGraph(V)
    g = mk.Graph(V, edge_capacity_hint=2 * len(s), buckets=buckets)
    o.insert(s, d, np.ones(len(s), np.uint32))
    g.insert(s, d)
    cut = _undirected(*pairs[rng.permutation(len(pairs))[:300]].T.astype(np.uint32))
    o.delete(*cut)
    g.delete(*cut)
    g.commit()
    mk.check(mk.load().mk_debug_set(g.handle, MK_DEBUG_NO_SCRATCH, 1), "mk_debug_set")
    assert g.triangles() == o.triangles()
    mk.check(mk.load().mk_debug_set(g.handle, MK_DEBUG_NO_SCRATCH, 0), "mk_debug_set")
    assert g.triangles() == o.triangles()
    assert g.last_error() == mk.MK_OK
    g.close()


@pytest.mark.parametrize("V", [1 << 21, (1 << 24) + 5])
def test_pagerank_at_the_limits_of_its_forms(cuda_lib, V):
    """2^21 vertices: a source and its place in a bin fill all bits of a word.
    More than 2^24: the bins' sums no longer fit, calls of any length push."""
    test_pagerank_binned_and_pushed(cuda_lib, V)
