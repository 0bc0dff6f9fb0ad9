"""Batches grouped by slab list, against the oracle: lists with just as many
edges of a batch as one 4-lane group applies (32), one fewer, one more and many
more; tails with room for some of them; repeats of a pair (the first one's
weight is stored); sparse and dense batches of one graph (fewer and more edges
than half its lists).  Everything is a whole number and has to be equal."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

PER_LIST = [1, 14, 15, 16, 30, 31, 32, 33, 47, 64, 200]


def _pairs(rng, V, per_list, repeat):
    """`n` edges of vertex 3 k for the k-th n of per_list, `repeat` of them again, shuffled."""
    src, dst = [], []
    for k, n in enumerate(per_list):
        d = rng.choice(V, n - min(repeat, n - 1), replace=False)
        d = np.concatenate([d, rng.choice(d, n - len(d))])
        src.append(np.full(n, 3 * k))
        dst.append(d)
    src, dst = np.concatenate(src), np.concatenate(dst)
    p = rng.permutation(len(src))
    return src[p].astype(np.uint32), dst[p].astype(np.uint32)


@pytest.mark.parametrize("store", ["map", "set"])
@pytest.mark.parametrize("repeat", [0, 3])
@pytest.mark.parametrize("V", [300, 5000])  # dense, sparse
@pytest.mark.parametrize("per_list", [PER_LIST, [n for n in PER_LIST if n <= 32]])
def test_edges_per_list(cuda_lib, store, repeat, V, per_list):
    import paper_2305_17813_gb300 as mk

    rng = np.random.default_rng(len(per_list) * 10 + repeat + V)
    make = mk.Graph if store == "map" else mk.SetGraph
    g, o = make(V, edge_capacity_hint=1 << 14, buckets=1), oracle.OracleGraph(V)
    live = []
    for step in range(4):
        s, d = _pairs(rng, V, per_list, repeat)
        w = rng.integers(1, 1000, len(s)).astype(np.uint32)
        f = g.insert(s, d, w) if store == "map" else g.insert(s, d)
        assert np.array_equal(f.cpu().numpy(), o.insert(s, d, w))
        live.append((s, d))
        s, d = live[rng.integers(len(live))]
        take = rng.permutation(np.arange(len(s)).repeat(1 + (repeat > 0)))[: len(s)]
        f = g.delete(s[take], d[take])
        assert np.array_equal(f.cpu().numpy(), o.delete(s[take], d[take]))
        s, d = (np.concatenate(x) for x in zip(*live))
        q, ow = o.query(s, d)
        if store == "map":
            bm, gw = g.query(s, d)
            assert np.array_equal(mk.to_numpy_u32(gw), ow)
            for a, b in zip(g.export(), o.export()):
                assert np.array_equal(mk.to_numpy_u32(a), b)
        else:
            bm = g.query(s, d)
        assert np.array_equal(mk.to_numpy_u32(bm), q)
    if store == "map":
        assert g.last_error() == mk.MK_OK
        dist, par = g.sssp(0)
        od, op = o.sssp(0)
        assert np.array_equal(mk.to_numpy_u32(dist), od) and np.array_equal(mk.to_numpy_u32(par), op)
    g.close()


def test_rejected_batch_leaves_the_grouping_clean(cuda_lib):
    """A batch with an invalid id changes nothing, and the batches after it
    find every list's count at zero again."""
    import paper_2305_17813_gb300 as mk

    rng = np.random.default_rng(5)
    V = 400
    g, o = mk.Graph(V, edge_capacity_hint=1 << 13, buckets=2), oracle.OracleGraph(V)
    for n in (40, 700):
        s, d = (rng.integers(0, V, n).astype(np.uint32) for _ in range(2))
        bad = d.copy()
        bad[n // 2] = V
        assert not g.insert(s, bad).any()
        assert g.last_error() == mk.MK_ERR_INVALID_ARG
        w = rng.integers(1, 50, n).astype(np.uint32)
        assert np.array_equal(g.insert(s, d, w).cpu().numpy(), o.insert(s, d, w))
        assert np.array_equal(g.delete(s[:9], d[:9]).cpu().numpy(), o.delete(s[:9], d[:9]))
        assert g.last_error() == mk.MK_OK
    for a, b in zip(g.export(), o.export()):
        assert np.array_equal(mk.to_numpy_u32(a), b)
    g.close()


def test_states_made_between_unlogged_and_logged_inserts(cuda_lib):
    """An insert is logged for the states that are current when it runs:
    states first computed in the middle of an epoch, after inserts that nobody
    logged, follow the later ones."""
    import paper_2305_17813_gb300 as mk

    rng = np.random.default_rng(6)
    V = 500
    g, o = mk.Graph(V, edge_capacity_hint=1 << 14, buckets=2), oracle.OracleGraph(V)

    def insert(n):
        s, d = (rng.integers(0, V, n).astype(np.uint32) for _ in range(2))
        w = rng.integers(1, 50, n).astype(np.uint32)
        assert np.array_equal(g.insert(s, d, w).cpu().numpy(), o.insert(s, d, w))

    def same(source):
        for (a, b), (x, y) in ((g.sssp(source), o.sssp(source)), (g.bfs(source), o.bfs(source))):
            assert np.array_equal(mk.to_numpy_u32(a), x) and np.array_equal(mk.to_numpy_u32(b), y)
        assert np.array_equal(mk.to_numpy_u32(g.wcc()), o.wcc())

    insert(300)            # no state yet: not logged
    same(0)                # from scratch
    same(0)                # nothing new
    insert(300)            # logged
    same(0)
    insert(300)
    same(1)                # a second source joins in the middle of the epoch
    same(0)
    g.commit()
    insert(300)
    same(0)
    g.commit()
    insert(300)            # an epoch that no state follows
    g.commit()
    insert(300)            # no state is current: not logged
    same(0)
    assert g.last_error() == mk.MK_OK
    g.close()


@pytest.mark.parametrize("store", ["map", "set"])
@pytest.mark.parametrize("part", [1, 100, 512])
def test_batches_in_parts(cuda_lib, store, part):
    """A batch beyond one grouping is applied in parts: pairs that repeat
    across parts, lists with many edges, the places of each part's flags and
    log entries, and an invalid edge of the last part, which rejects all of
    them."""
    import paper_2305_17813_gb300 as mk
    from paper_2305_17813_gb300._native import MK_DEBUG_PART_EDGES

    rng = np.random.default_rng(part)
    V, n = 300, 513 if part > 1 else 40
    make = mk.Graph if store == "map" else mk.SetGraph
    g, o = make(V, edge_capacity_hint=1 << 14, buckets=1), oracle.OracleGraph(V)
    name = "mk_debug_set" if store == "map" else "mk_set_debug_set"
    assert getattr(mk.load(), name)(g.handle, MK_DEBUG_PART_EDGES, part) == mk.MK_OK

    def same():
        if store == "map":
            assert np.array_equal(mk.to_numpy_u32(g.wcc()), o.wcc())
            for (a, b), (x, y) in ((g.sssp(0), o.sssp(0)), (g.bfs(3), o.bfs(3))):
                assert np.array_equal(mk.to_numpy_u32(a), x) and np.array_equal(mk.to_numpy_u32(b), y)
            for a, b in zip(g.export(), o.export()):
                assert np.array_equal(mk.to_numpy_u32(a), b)

    for step in range(4):
        s = (rng.integers(0, V, n) * rng.random(n) ** 4).astype(np.uint32)  # a few vertices with most of the edges
        d = rng.integers(0, 60, n).astype(np.uint32)
        w = rng.integers(1, 1000, n).astype(np.uint32)
        f = g.insert(s, d, w) if store == "map" else g.insert(s, d)
        assert np.array_equal(f.cpu().numpy(), o.insert(s, d, w))
        same()
        if store == "map" and step % 2:
            g.commit()
        take = rng.permutation(np.arange(n).repeat(2))[:n]
        assert np.array_equal(g.delete(s[take], d[take]).cpu().numpy(), o.delete(s[take], d[take]))
        same()
        if store == "map":
            g.commit()
        assert np.array_equal(mk.to_numpy_u32(g.query(s, d)[0] if store == "map" else g.query(s, d)), o.query(s, d)[0])
        bad = d.copy()
        bad[n - 1] = V
        assert not (g.insert(s, bad, w) if store == "map" else g.insert(s, bad)).any()
        assert g.last_error() == mk.MK_ERR_INVALID_ARG
        assert not g.delete(s, bad).any()
        assert g.last_error() == mk.MK_ERR_INVALID_ARG
    same()
    g.close()


@pytest.mark.parametrize("store", ["map", "set"])
@pytest.mark.parametrize("limit", [1, 1 << 30])  # every batch grouped; none of those that need not be
@pytest.mark.parametrize("V", [300, 5000])
def test_batches_grouped_and_not(cuda_lib, store, limit, V):
    """Batches grouped by list or by their hash set alone: one edge up to
    several tiles, a hub's lists, repeats, pairs that are absent or gone,
    invalid edges (the flags of a rejected batch are all zero), and trees that
    follow the inserts and the deletes."""
    import torch

    import paper_2305_17813_gb300 as mk
    from paper_2305_17813_gb300._native import MK_DEBUG_HASH_EDGES

    rng = np.random.default_rng(V)
    make = mk.Graph if store == "map" else mk.SetGraph
    g, o = make(V, edge_capacity_hint=1 << 15, buckets=2), oracle.OracleGraph(V)
    name = "mk_debug_set" if store == "map" else "mk_set_debug_set"
    assert getattr(mk.load(), name)(g.handle, MK_DEBUG_HASH_EDGES, limit) == mk.MK_OK
    live = [np.zeros(0, np.uint32)] * 2

    def same():
        for (a, b), (x, y) in ((g.sssp(0), o.sssp(0)), (g.bfs(0), o.bfs(0))):
            assert np.array_equal(mk.to_numpy_u32(a), x) and np.array_equal(mk.to_numpy_u32(b), y)
        assert np.array_equal(mk.to_numpy_u32(g.wcc()), o.wcc())

    for n in (1, 2, 255, 256, 257, 1000, 4099):
        s = (rng.integers(0, V, n) * rng.random(n) ** 3).astype(np.uint32)
        d = rng.integers(0, V, n).astype(np.uint32)
        again = rng.integers(0, n, n // 4)
        s, d = np.concatenate([s, s[again]]), np.concatenate([d, d[again]])
        w = rng.integers(1, 1000, len(s)).astype(np.uint32)
        f = g.insert(s, d, w) if store == "map" else g.insert(s, d)
        assert np.array_equal(f.cpu().numpy(), o.insert(s, d, w))
        live = [np.concatenate(x) for x in zip(live, (s, d))]
        if store == "map":
            same()
            g.commit()
        at = rng.integers(0, len(live[0]), n)
        s, d = live[0][at], live[1][at]
        s[: n // 8] = rng.integers(0, V, n // 8)
        bad = s.copy()
        bad[n // 2] = V
        flags = torch.full((n,), 7, dtype=torch.uint8, device="cuda")
        call = mk.load().mk_delete_batch if store == "map" else mk.load().mk_set_delete_batch
        bs, bd = mk.to_device_u32(bad), mk.to_device_u32(d)
        assert call(g.handle, bs.data_ptr(), bd.data_ptr(), n, flags.data_ptr(), None) == mk.MK_OK
        assert g.last_error() == mk.MK_ERR_INVALID_ARG and not flags.any()
        if store == "map":
            same()  # from scratch, and current again, so that they follow the delete
        assert np.array_equal(g.delete(s, d).cpu().numpy(), o.delete(s, d))
        if store == "map":
            same()
            g.commit()
            for a, b in zip(g.export(), o.export()):
                assert np.array_equal(mk.to_numpy_u32(a), b)
        q = g.query(*live)
        assert np.array_equal(mk.to_numpy_u32(q[0] if store == "map" else q), o.query(*live)[0])
    assert g.last_error() == mk.MK_OK
    g.close()


@pytest.mark.parametrize("n", [50, 5000, 300000])
def test_a_delete_as_large_as_an_insert_grows_nothing(cuda_lib, n):
    """The arrays that an insert grew hold a delete of as many edges, so that it
    neither allocates nor waits for its stream (the set store: it keeps no
    logs beside them)."""
    import paper_2305_17813_gb300 as mk

    rng = np.random.default_rng(n)
    g = mk.SetGraph(1 << 14, edge_capacity_hint=n, buckets=1)
    s, d = (rng.integers(0, 1 << 14, n).astype(np.uint32) for _ in range(2))
    stored = g.insert(s, d)
    held = g.stats()["device_bytes"]
    assert np.array_equal(g.delete(s, d).cpu().numpy(), stored.cpu().numpy())
    assert g.stats()["device_bytes"] == held
    assert g.last_error() == mk.MK_OK
    g.close()
