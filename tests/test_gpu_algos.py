"""GPU parity of incremental / decremental BFS and SSSP trees and of WCC
labels with the CPU oracle (which recomputes from scratch after every batch):
distances, min-id tight parents and min-id component labels, bit-exact."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _mk():
    import paper_2305_17813_gb300 as mk

    mk.load()
    return mk


def check_algos(g, o, sources, wcc=True):
    mk = _mk()
    for src in sources:
        d, p = g.sssp(src)
        od, op = o.sssp(src)
        assert np.array_equal(mk.to_numpy_u32(d), od), "sssp dist from %d" % src
        assert np.array_equal(mk.to_numpy_u32(p), op), "sssp parent from %d" % src
        d, p = g.bfs(src)
        od, op = o.bfs(src)
        assert np.array_equal(mk.to_numpy_u32(d), od), "bfs dist from %d" % src
        assert np.array_equal(mk.to_numpy_u32(p), op), "bfs parent from %d" % src
    if wcc:
        assert np.array_equal(mk.to_numpy_u32(g.wcc()), o.wcc()), "wcc labels"
    assert g.last_error() == mk.MK_OK


def test_tiny_workload_incremental_sequence(cuda_lib):
    mk = _mk()
    w = synth.tiny_workload()
    g = mk.Graph(w.V, edge_capacity_hint=16384, buckets=1)
    o = oracle.OracleGraph(w.V)
    g.insert(w.g_src, w.g_dst, w.g_w)
    o.insert(w.g_src, w.g_dst, w.g_w)
    g.commit()
    check_algos(g, o, [0])          # static
    g.commit()
    g.insert(w.ins_src, w.ins_dst, w.ins_w)
    o.insert(w.ins_src, w.ins_dst, w.ins_w)
    check_algos(g, o, [0])          # incremental
    g.commit()
    g.delete(w.del_src, w.del_dst)
    o.delete(w.del_src, w.del_dst)
    check_algos(g, o, [0])          # decremental (WCC recomputes)
    g.commit()


@pytest.mark.parametrize("buckets", [1, 4])
@pytest.mark.parametrize("seed", [0, 1, 2])
def test_mixed_epochs_match_recompute(cuda_lib, buckets, seed):
    """Random insert / delete batches; the algorithms run after every batch
    and sometimes twice inside one epoch, commits between some batches."""
    mk = _mk()
    rng = np.random.default_rng(10 + seed)
    V = 600
    g = mk.Graph(V, edge_capacity_hint=50000, buckets=buckets)
    o = oracle.OracleGraph(V)
    s = rng.integers(0, V, 3000).astype(np.uint32)
    d = rng.integers(0, V, 3000).astype(np.uint32)
    w = rng.integers(1, 50, 3000).astype(np.uint32)
    g.insert(s, d, w)
    o.insert(s, d, w)
    srcs = [0, int(rng.integers(0, V))]
    check_algos(g, o, srcs)
    for step in range(8):
        n = int(rng.integers(1, 400))
        if step % 3 == 1:
            ls, ld, _ = o.export()
            pick = rng.integers(0, len(ls), n)
            g.delete(ls[pick], ld[pick])
            o.delete(ls[pick], ld[pick])
        else:
            s = rng.integers(0, V, n).astype(np.uint32)
            d = rng.integers(0, V, n).astype(np.uint32)
            w = rng.integers(1, 50, n).astype(np.uint32)
            g.insert(s, d, w)
            o.insert(s, d, w)
        check_algos(g, o, srcs, wcc=step % 2 == 0)
        if step % 2 == 1:
            g.commit()


def test_delete_then_reinsert_tree_edge(cuda_lib):
    mk = _mk()
    V = 6
    g = mk.Graph(V, buckets=1)
    o = oracle.OracleGraph(V)
    s = np.array([0, 1, 2, 0, 3, 4], np.uint32)
    d = np.array([1, 2, 3, 3, 4, 5], np.uint32)
    w = np.array([1, 1, 1, 10, 1, 1], np.uint32)
    for x in (g, o):
        x.insert(s, d, w)
    check_algos(g, o, [0])
    g.commit()
    for x in (g, o):
        x.delete([1], [2])            # tree edge: 2, 3, 4, 5 lose their paths
    check_algos(g, o, [0])
    for x in (g, o):
        x.insert([1], [2], [2])       # same edge, new weight, same epoch
    check_algos(g, o, [0])
    g.commit()
    for x in (g, o):
        x.delete([0, 0], [1, 3])      # source cut off from everything
    check_algos(g, o, [0])


def test_grid_closed_form_and_single_component(cuda_lib):
    mk = _mk()
    rows, cols = 64, 96
    s, d = synth.grid_pairs(rows, cols)
    g = mk.Graph(rows * cols, buckets=1)
    g.insert(s, d, np.ones(len(s), np.uint32))
    r, c = np.divmod(np.arange(rows * cols), cols)
    dist, _ = g.bfs(0)
    assert np.array_equal(mk.to_numpy_u32(dist), r + c)
    dist, _ = g.sssp(0)
    assert np.array_equal(mk.to_numpy_u32(dist), r + c)
    assert np.all(mk.to_numpy_u32(g.wcc()) == 0)


def test_power_law_with_bucket_rule(cuda_lib):
    """R-MAT scale 14 with the load-factor bucket rule (many buckets for hubs):
    static, then an insert batch and a delete batch with recomputation."""
    mk = _mk()
    G = synth.powerlaw_graph(scale=14, draws=1 << 18)
    b = mk.bucket_rule(G.V, G.src, 0.7)
    g = mk.Graph(G.V, edge_capacity_hint=len(G.src) * 2, buckets=b)
    o = oracle.OracleGraph(G.V)
    g.insert(G.src, G.dst, G.w)
    o.insert(G.src, G.dst, G.w)
    g.commit()
    src = int(np.argmax(o.out_degree()))
    check_algos(g, o, [src])
    g.commit()
    B = synth.PowerlawStream(G, max_batch=1 << 14).batch(1 << 14)
    g.insert(B.ins_src, B.ins_dst, B.ins_w)
    o.insert(B.ins_src, B.ins_dst, B.ins_w)
    check_algos(g, o, [src])
    g.commit()
    g.delete(B.del_src, B.del_dst)
    o.delete(B.del_src, B.del_dst)
    check_algos(g, o, [src])
    g.commit()
    bm, _ = g.query(B.q_src, B.q_dst)
    assert np.array_equal(mk.to_numpy_u32(bm), o.query(B.q_src, B.q_dst)[0])


def test_long_path_and_mixed_frontier_sizes(cuda_lib):
    """A 9,000-vertex path (thousands of one-list rounds, more than one
    solo phase of the round kernel) feeding a dense random block (frontiers
    of thousands of lists), then a delete that cuts the path in the middle."""
    mk = _mk()
    P = 9000
    B = 4000
    rng = np.random.default_rng(5)
    V = P + B
    ps = np.arange(P - 1, dtype=np.uint32)
    pd = ps + 1
    bs = rng.integers(P, V, 120000).astype(np.uint32)
    bd = rng.integers(P, V, 120000).astype(np.uint32)
    s = np.concatenate([ps, [P - 1], bs]).astype(np.uint32)
    d = np.concatenate([pd, [P], bd]).astype(np.uint32)
    w = rng.integers(1, 9, len(s)).astype(np.uint32)
    g = mk.Graph(V, edge_capacity_hint=len(s) * 2, buckets=1)
    o = oracle.OracleGraph(V)
    g.insert(s, d, w)
    o.insert(s, d, w)
    check_algos(g, o, [0], wcc=True)
    g.commit()
    for x in (g, o):
        x.delete([P // 2], [P // 2 + 1])
    check_algos(g, o, [0], wcc=True)
    g.commit()
    for x in (g, o):
        x.insert([P // 2], [P // 2 + 1], [3])
    check_algos(g, o, [0], wcc=True)


@pytest.mark.parametrize("delta", [7, 300])
def test_near_far_sssp_power_law_stream(cuda_lib, delta):
    """Near-Far ordered SSSP on R-MAT batches of inserts and deletes of live
    edges: the tree equals the oracle's after every batch, BFS (never
    ordered) too, and switching the ordering off mid-stream keeps it."""
    mk = _mk()
    G = synth.powerlaw_graph(scale=13, draws=1 << 17)
    S = synth.PowerlawStream(G, max_batch=1 << 12)
    src = int(np.argmax(np.bincount(G.src, minlength=G.V)))
    g = mk.Graph(G.V, edge_capacity_hint=len(G.src) + (1 << 16), buckets=mk.bucket_rule(G.V, G.src, 0.7))
    g.set_sssp_delta(delta, delta)
    o = oracle.OracleGraph(G.V)
    g.insert(G.src, G.dst, G.w, flags=False)
    o.insert(G.src, G.dst, G.w)
    g.commit()
    for k in range(6):
        if k == 4:
            g.set_sssp_delta(0, 0)
        b = S.batch(1 << 12)
        g.insert(b.ins_src, b.ins_dst, b.ins_w, flags=False)
        o.insert(b.ins_src, b.ins_dst, b.ins_w)
        for fn, ofn in ((g.sssp, o.sssp), (g.bfs, o.bfs)):
            d, p = fn(src)
            od, op = ofn(src)
            assert np.array_equal(mk.to_numpy_u32(d), od) and np.array_equal(mk.to_numpy_u32(p), op), k
        g.commit()
        g.delete(b.del_src, b.del_dst, flags=False)
        o.delete(b.del_src, b.del_dst)
        d, p = g.sssp(src)
        od, op = o.sssp(src)
        assert np.array_equal(mk.to_numpy_u32(d), od) and np.array_equal(mk.to_numpy_u32(p), op), k
        g.commit()
        assert g.last_error() == mk.MK_OK
    g.close()


@pytest.mark.parametrize("delta", [0, 40])
def test_frontier_staging_limits(cuda_lib, delta):
    """One round that improves every vertex: vertices with 1 to 20 lists (up
    to 8 are staged a warp, more are written by the whole warp), far more
    entries than the staging buffers hold, with and without far piles."""
    mk = _mk()
    rng = np.random.default_rng(31)
    V = 6000
    nb = rng.integers(1, 21, V).astype(np.uint32)
    nb[0] = 64
    g = mk.Graph(V, edge_capacity_hint=1 << 17, buckets=mk.to_device_u32(nb))
    g.set_sssp_delta(delta, delta)
    o = oracle.OracleGraph(V)
    s = np.concatenate([np.zeros(V - 1), rng.integers(0, V, 30000)]).astype(np.uint32)
    d = np.concatenate([np.arange(1, V), rng.integers(0, V, 30000)]).astype(np.uint32)
    w = rng.integers(1, 200, len(s)).astype(np.uint32)
    assert np.array_equal(g.insert(s, d, w).cpu().numpy(), o.insert(s, d, w))
    check_algos(g, o, [0])
    g.commit()
    g.delete(s[: V // 2], d[: V // 2])
    o.delete(s[: V // 2], d[: V // 2])
    check_algos(g, o, [0])
    g.close()


@pytest.mark.parametrize("store", ["map", "set"])
@pytest.mark.parametrize("V", [600, 20000, 1500000])  # no sample; bitmap in shared memory; in global memory
@pytest.mark.parametrize("shape", ["giant", "many", "path"])
def test_static_components(cuda_lib, store, V, shape):
    """Static components with one giant tree, with many small ones, and along
    a path, ids in no order, then after deletes."""
    mk = _mk()
    rng = np.random.default_rng(V + len(shape))
    name = rng.permutation(V).astype(np.uint32)
    if shape == "path":
        s, d = np.arange(V - 1), np.arange(1, V)
    else:
        n = V if shape == "giant" else V // 3
        s, d = rng.integers(0, V, n), rng.integers(0, V, n)
    s, d = name[s], name[d]
    o = oracle.OracleGraph(V)
    o.insert(s, d, np.ones(len(s), np.uint32))
    if store == "map":
        g = mk.Graph(V, edge_capacity_hint=2 * len(s), buckets=1)
        g.insert(s, d, np.ones(len(s), np.uint32))
    else:
        g = mk.SetGraph(V, edge_capacity_hint=2 * len(s), buckets=1)
        g.insert(s, d)
    assert np.array_equal(mk.to_numpy_u32(g.wcc()), o.wcc())
    cut = rng.permutation(len(s))[: len(s) // 4]
    g.delete(s[cut], d[cut])
    o.delete(s[cut], d[cut])
    assert np.array_equal(mk.to_numpy_u32(g.wcc()), o.wcc())
    assert g.last_error() == mk.MK_OK
    g.close()


@pytest.mark.parametrize("V", [33, 1638400, 1638401])  # the last with the bitmap in shared memory; the first without
def test_decremental_bitmap_limits(cuda_lib, V):
    """Distances after deletes that invalidate much of the tree, the last
    vertex included, with the invalidated set on each side of the scan."""
    mk = _mk()
    rng = np.random.default_rng(V)
    n = min(3 * V, 60000)
    name = np.unique(np.append(rng.integers(0, V, 20000), V - 1)).astype(np.uint32)  # the vertices in use
    s, d = rng.choice(name, n), rng.choice(name, n)
    s[:8], d[:8] = name[0], name[-8:]
    w = rng.integers(1, 100, n).astype(np.uint32)
    g, o = mk.Graph(V, edge_capacity_hint=2 * n, buckets=1), oracle.OracleGraph(V)
    g.insert(s, d, w)
    o.insert(s, d, w)
    src = int(name[0])
    for k in range(3):
        check_algos(g, o, [src], wcc=False)
        g.commit()
        cut = rng.permutation(n)[: n // 8]
        cut[:4] = range(4)  # tree edges of the root
        g.delete(s[cut], d[cut])
        o.delete(s[cut], d[cut])
    check_algos(g, o, [src], wcc=False)
    assert g.last_error() == mk.MK_OK
    g.close()


@pytest.mark.parametrize("store", ["map", "set"])
@pytest.mark.parametrize("degree", [3, 40, 400])  # less than a slab; a few; more than the sample reads
def test_static_components_after_churn(cuda_lib, store, degree):
    """Static components of lists that begin with deleted pairs: the oldest
    edges of every vertex gone, new ones behind them."""
    mk = _mk()
    V = 12000
    rng = np.random.default_rng(degree)
    src = np.arange(V, dtype=np.uint32)
    old = np.stack([(src + 1 + k) % V for k in range(degree)]).astype(np.uint32)
    new = np.stack([(src + 1 + 3 * V // 4) % V, rng.permutation(V)]).astype(np.uint32)
    o = oracle.OracleGraph(V)
    g = (mk.Graph if store == "map" else mk.SetGraph)(V, edge_capacity_hint=(degree + 4) * V, buckets=1)
    s = np.tile(src, degree)

    def insert(a, b):
        o.insert(a, b, np.ones(len(a), np.uint32))
        g.insert(a, b, np.ones(len(a), np.uint32)) if store == "map" else g.insert(a, b)

    insert(s, old.ravel())
    o.delete(s, old.ravel())
    g.delete(s, old.ravel())
    assert np.array_equal(mk.to_numpy_u32(g.wcc()), o.wcc())  # every vertex by itself
    insert(src[: V // 3], new[0][: V // 3])
    insert(src[::2], new[1][::2])
    assert np.array_equal(mk.to_numpy_u32(g.wcc()), o.wcc())
    assert g.last_error() == mk.MK_OK
    g.close()


def test_two_sizes_from_two_threads(cuda_lib):
    """Graphs of very different size worked on by two host threads, each on a
    stream of its own: kernels that size their shared memory by the graph."""
    import threading

    import torch

    mk = _mk()

    def build(V, n, seed):
        rng = np.random.default_rng(seed)
        s, d = rng.integers(0, V, n).astype(np.uint32), rng.integers(0, V, n).astype(np.uint32)
        o = oracle.OracleGraph(V)
        o.insert(s, d, np.ones(n, np.uint32))
        g = mk.Graph(V, edge_capacity_hint=2 * n, buckets=1)
        g.insert(s, d, np.ones(n, np.uint32))
        dist, _ = g.sssp(int(s[0]))
        g.commit()
        g.delete(s[: n // 8], d[: n // 8])
        o.delete(s[: n // 8], d[: n // 8])
        return g, int(s[0]), o

    work = [build(20000, 60000, 1), build(900000, 500000, 2)]
    torch.cuda.synchronize()
    out = [None, None]

    def run(k):
        g, src, _ = work[k]
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            d, p = g.sssp(src)
            for _ in range(20):
                lab = g.wcc()
                st.synchronize()
            r = g.pagerank(max_iter=8)[0]
            st.synchronize()
        out[k] = d, p, lab, r

    threads = [threading.Thread(target=run, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for k in range(2):
        g, src, o = work[k]
        assert out[k] is not None
        d, p, lab, r = out[k]
        od, op = o.sssp(src)
        assert np.array_equal(mk.to_numpy_u32(d), od) and np.array_equal(mk.to_numpy_u32(p), op)
        assert np.array_equal(mk.to_numpy_u32(lab), o.wcc())
        assert abs(float(r.sum().item()) - 1.0) < 1e-3
        assert g.last_error() == mk.MK_OK
        g.close()


@pytest.mark.parametrize("width", [16384, 16385, 262144, 262145])
def test_frontiers_of_constant_width(cuda_lib, width):
    """Layers of equal width, so that the frontier keeps its size (and, after
    deletes in one layer, does not), on each side of the sizes at which a
    round issues its minima without reading the nodes."""
    mk = _mk()
    rng = np.random.default_rng(width)
    layers = 4
    V = layers * width + 1
    at = 1 + np.arange(width)
    s, d = [np.zeros(width, np.int64)], [at]
    for k in range(layers - 1):
        for _ in range(2):
            s.append(k * width + at)
            d.append((k + 1) * width + rng.permutation(at))
    s, d = np.concatenate(s).astype(np.uint32), np.concatenate(d).astype(np.uint32)
    w = rng.integers(1, 50, len(s)).astype(np.uint32)
    nb = np.ones(V, np.uint32)
    nb[0] = 1 + width // 15
    g, o = mk.Graph(V, edge_capacity_hint=2 * len(s), buckets=mk.to_device_u32(nb)), oracle.OracleGraph(V)
    g.insert(s, d, w)
    o.insert(s, d, w)
    check_algos(g, o, [0], wcc=False)
    g.commit()
    cut = slice(width, width + width // 2)
    g.delete(s[cut], d[cut])
    o.delete(s[cut], d[cut])
    check_algos(g, o, [0], wcc=False)
    g.close()


@pytest.mark.parametrize("width", [193, 700, 2047, 2048])
@pytest.mark.parametrize("delta", [3, 60, 100000])
def test_ordered_rounds_while_the_pile_fills_and_empties(cuda_lib, width, delta):
    """Ordered rounds of the whole grid whose frontier is below the size at
    which the far pile is split: most of them meet an empty pile, and a few
    heavy edges fill it in the very round that the blocks decide about.  All
    have to take the same way, call after call."""
    mk = _mk()
    rng = np.random.default_rng(width + delta)
    layers = 40
    V = layers * width + 1
    at = 1 + np.arange(width)
    s, d = [np.zeros(width, np.int64)], [at]
    for k in range(layers - 1):
        for _ in range(2):
            s.append(k * width + at)
            d.append((k + 1) * width + rng.permutation(at))
    s, d = np.concatenate(s).astype(np.uint32), np.concatenate(d).astype(np.uint32)
    w = np.where(rng.random(len(s)) < 0.01, rng.integers(200, 5000, len(s)), rng.integers(1, 6, len(s))).astype(np.uint32)
    nb = np.ones(V, np.uint32)
    nb[0] = 1 + width // 15
    g, o = mk.Graph(V, edge_capacity_hint=4 * len(s), buckets=mk.to_device_u32(nb)), oracle.OracleGraph(V)
    g.set_sssp_delta(delta, delta)
    g.insert(s, d, w)
    o.insert(s, d, w)
    for _ in range(6):
        check_algos(g, o, [0], wcc=False)
        assert g.last_error() == mk.MK_OK
        g.commit()
        cut = rng.permutation(len(s))[: len(s) // 20]
        g.delete(s[cut], d[cut])
        o.delete(s[cut], d[cut])
        check_algos(g, o, [0], wcc=False)
        assert g.last_error() == mk.MK_OK
        g.insert(s[cut], d[cut], w[cut])
        o.insert(s[cut], d[cut], w[cut])
        g.commit()  # an epoch that the state has not followed: from scratch next
    g.close()
