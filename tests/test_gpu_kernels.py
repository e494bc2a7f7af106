"""The sweeps' kernels at the sizes where their variants and their edges lie."""
import numpy as np
import pytest

import graphs as G
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nk():
    torch = pytest.importorskip("torch")
    assert torch.cuda.is_available()
    from paper_1403_3005_gb300 import nk as m
    m.lib()
    return m


def forest(n_arcs_vertices: int, isolated: int):
    """(n, u, v, score): disjoint paths of 2, 3 and 5 vertices and stars of 4 leaves, in turn,
    over n_arcs_vertices vertices (a last path takes the rest), ids interleaved with isolated
    vertices, and the exact betweenness: i (m - 1 - i) on a path of m, 6 at a star's centre."""
    u, v, score, at, i = [], [], [], 0, 0
    while at < n_arcs_vertices:
        m = (2, 3, 5, 5)[i % 4]
        left = n_arcs_vertices - at
        if left - m < 2:
            m = left
        if i % 4 == 3 and m == 5:
            u += [at] * 4
            v += [at + j for j in range(1, 5)]
            score += [6.0, 0.0, 0.0, 0.0, 0.0]
        else:
            u += [at + j for j in range(m - 1)]
            v += [at + j + 1 for j in range(m - 1)]
            score += [float(j * (m - 1 - j)) for j in range(m)]
        at += m
        i += 1
    n = n_arcs_vertices + isolated
    ids = np.sort(np.random.default_rng(1).choice(n, n_arcs_vertices, replace=False))
    full = np.zeros(n)
    full[ids] = score
    return n, ids[np.array(u)].astype(np.int32), ids[np.array(v)].astype(np.int32), full


@pytest.mark.parametrize("with_arcs", [64, 65, 129, 32768, 32769])
def test_sources_ordered_over_batches(nk, with_arcs):
    """Every vertex as a source, through as many batches as it takes: the sources are put in
    another order (segments of 32768), which changes no score."""
    n, u, v, score = forest(with_arcs, 37)
    g = nk.graph_from_edges(n, u, v)
    for batch in (64, 128):
        got = nk.betweenness_sources(g, np.arange(n, dtype=np.int32), 0.5, nk.run_opts(mode=nk.MODE_BATCHED, batch=batch))
        assert np.allclose(got, score, rtol=1e-9, atol=1e-12)


# rows of 31..33 and 64, 65 arcs (windows of 32), 255..257 and 512 (chunks of 256) among short ones
# and isolated vertices; a graph of under 32 vertices; one whose groups are full (32 vertices a warp)
GROUPS = {
    "rows": G.with_hubs(G.disjoint_union(G.complete(1), G.gnp(600, 0.01, 3)), [31, 32, 33, 64, 65, 255, 256, 257, 512], 5),
    "tiny": G.gnp(20, 0.3, 2),
    "many": G.gnp(30000, 0.0001, 7),
}


@pytest.mark.parametrize("name", list(GROUPS))
@pytest.mark.parametrize("batch", [64, 128, 256])
def test_groups_of_rows(nk, name, batch):
    """The batched sweep, which walks the concatenated rows of groups of vertices, in both
    directions and with small chunks, against the oracle."""
    n, u, v = GROUPS[name]
    g = nk.graph_from_edges(n, u, v)
    rp, col = oracle.csr_build(n, u, v)
    k = min(n, 150)
    ref = oracle.betweenness_sampled(rp, col, 3, k)
    far = oracle.closeness_sampled(rp, col, 3, k)
    edges = oracle.edge_betweenness_sampled(rp, col, 3, k)
    for kw in (dict(direction=1), dict(direction=2), dict(alpha=2.0, chunk=32)):
        o = nk.run_opts(mode=nk.MODE_BATCHED, batch=batch, **kw)
        assert np.allclose(nk.betweenness_sampled(g, 3, k, o), ref, rtol=1e-9, atol=1e-12)
        assert np.allclose(nk.edge_betweenness_sampled(g, 3, k, o), edges, rtol=1e-9, atol=1e-12)
        assert all(np.array_equal(x, y) for x, y in zip(nk.closeness_sampled(g, 3, k, o), far))


@pytest.mark.parametrize("batch", [0, 64, 128, 256])
def test_closeness_levels(nk, batch):
    """Closeness from level bitsets: a search far deeper than the levels kept at a time, and
    source counts at the edges of the batch widths, against sums in closed form."""
    n = 700
    i = np.arange(n)
    g = nk.graph_from_edges(*G.path(n))
    for k in (63, 64, 65, 128, 129, 256, 257, n):
        src = oracle.sample_sources(n, 8, k)
        for direction in (0, 1, 2):
            far, reach = nk.closeness_sampled(g, 8, k, nk.run_opts(mode=nk.MODE_BATCHED, batch=batch, direction=direction))
            assert np.array_equal(far, np.abs(i[:, None] - src).sum(1) * (n / k))
            assert np.array_equal(reach, (i[:, None] != src).sum(1) * (n / k))


@pytest.mark.parametrize("direction", [0, 1, 2])
def test_more_sources_than_vertices(nk, direction):
    """Pairs are drawn with repetitions: a batch of 256 of them on 40 vertices."""
    n, u, v = G.path(40)
    rp, col = oracle.csr_build(n, u, v)
    want, r, vd = oracle.betweenness_rk(rp, col, 0.1, 0.1, 7)
    g = nk.graph_from_edges(n, u, v)
    for batch in (64, 256):
        got, r1, vd1 = nk.betweenness_rk(g, 0.1, 0.1, 7, nk.run_opts(mode=nk.MODE_BATCHED, batch=batch, direction=direction))
        assert (r1, vd1) == (r, vd) and np.array_equal(got, want)


@pytest.mark.parametrize("k", [65, 128, 192, 300])
def test_batches_side_by_side(nk, k):
    """Several batches of a small graph run in one launch, by teams with their own state and sums:
    2, 2, 3 and 5 batches of 64, the last one full or not, for vertex and edge scores, drawn pairs
    and counts that need 64-bit rows in some of the batches."""
    n, u, v = G.disjoint_union(G.gnp(400, 0.02, 11), G.grid(24, 24), G.star(300))
    g = nk.graph_from_edges(n, u, v)
    rp, col = oracle.csr_build(n, u, v)
    o = nk.run_opts(mode=nk.MODE_BATCHED, batch=64)
    assert np.allclose(nk.betweenness_sampled(g, 3, k, o), oracle.betweenness_sampled(rp, col, 3, k), rtol=1e-9, atol=1e-12)
    assert np.allclose(nk.edge_betweenness_sampled(g, 3, k, o), oracle.edge_betweenness_sampled(rp, col, 3, k),
                       rtol=1e-9, atol=1e-12)
    assert nk.last_run_stats()["launches"] >= (k + 63) // 64
    want, r, _ = oracle.betweenness_rk(rp, col, 0.15, 0.1, 7)
    got, r1, _ = nk.betweenness_rk(g, 0.15, 0.1, 7, o)
    assert r1 == r and np.array_equal(got, want)


@pytest.mark.parametrize("k", [1, 5, 40])
def test_weighted_rows(nk, k):
    """Weighted sweeps over rows of 1 to 600 arcs (8 lanes up to 32 arcs, a warp, chunks of 256) and
    isolated vertices, by many and by few blocks per search, against the oracle."""
    n, u, v = GROUPS["rows"]
    g = nk.graph_from_edges(n, u, v)
    rp, col = oracle.csr_build(n, u, v)
    nk.random_weights(g, 4, 5)
    ref = oracle.betweenness_weighted_sampled(rp, col, oracle.edge_weights(rp, col, 4, 5), 9, k)
    for ctas in (0, 1, 7):
        got = nk.betweenness_weighted_sampled(g, 9, k, nk.run_opts(grid_ctas=ctas))
        assert np.allclose(got, ref, rtol=1e-9, atol=1e-12)


@pytest.mark.parametrize("name", ["rows", "tiny", "many", "path", "grid"])
@pytest.mark.parametrize("k", [1, 4, 8, 9, 15])
def test_few_sources(nk, name, k):
    """Below 16 sources: batches of 8, rows of up to 32 arcs by parts of a warp, longer ones and
    chunks by all of it, searches deeper than the first attempt's level slabs."""
    n, u, v = {"path": G.path(300), "grid": G.grid(30, 31)}.get(name) or GROUPS[name]
    g = nk.graph_from_edges(n, u, v)
    rp, col = oracle.csr_build(n, u, v)
    src = oracle.sample_sources(n, 5, k)
    ref = oracle.betweenness_sources(rp, col, src, 2.0)
    for kw in (dict(), dict(direction=1), dict(direction=2), dict(chunk=32, alpha=4.0)):
        got = nk.betweenness_sources(g, src, 2.0, nk.run_opts(**kw))
        assert np.allclose(got, ref, rtol=1e-9, atol=1e-12)


def test_few_sources_overflow(nk):
    g = nk.graph_from_edges(*G.grid(36, 36))
    with pytest.raises(nk.NkError) as e:
        nk.betweenness_sources(g, np.array([0, 1, 2, 3, 4], np.int32), 1.0)
    assert e.value.rc == nk.ERR_OVERFLOW


def test_csr_rows_at_the_sort_sizes(nk):
    """Raw rows (with duplicates and loops) around the sizes where the sort changes: 32, 64, 128 and
    256 (registers), 512 and 4096 (shared memory), and above (bitmap)."""
    sizes = [1, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 4095, 4096, 4097, 9000]
    rng = np.random.default_rng(3)
    n = len(sizes) + 12000
    u = np.concatenate([np.full(s, i) for i, s in enumerate(sizes)] + [[5, 7000]]).astype(np.int32)
    v = np.concatenate([rng.integers(len(sizes), n, s) for s in sizes] + [[5, 7000]]).astype(np.int32)
    v[rng.random(len(v)) < 0.1] = n - 1  # duplicates
    order = rng.permutation(len(u))
    g = nk.graph_from_edges(n, u[order], v[order])
    rp, col = oracle.csr_build(n, u, v)
    a, b = g.export_csr()
    assert np.array_equal(a, rp) and np.array_equal(b, col)


@pytest.mark.parametrize("flag", ["RUN_NO_RELABEL", "RUN_RELABEL"])
def test_captured_run_after_another_chunk_size(nk, flag):
    """A captured run reads the chunk table that its kernel nodes point to.  A call with another chunk
    size in between rebuilds that table (with chunks of 32 arcs a larger one, elsewhere in memory)."""
    import torch
    n, u, v = GROUPS["rows"]
    g = nk.graph_from_edges(n, u, v)
    rp, col = oracle.csr_build(n, u, v)
    ref = oracle.betweenness_sampled(rp, col, 3, 150)
    out, other = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2))
    flags = getattr(nk, flag)
    captured = nk.run_opts(mode=nk.MODE_BATCHED, batch=64, chunk=128, flags=flags | nk.RUN_CUDA_GRAPH)
    for chunk in (0, 32, 96, 128):
        if chunk:
            nk.betweenness_sampled(g, 3, 150, nk.run_opts(mode=nk.MODE_BATCHED, batch=64, chunk=chunk, flags=flags), out=other)
            assert np.allclose(other.cpu().numpy(), ref, rtol=1e-9, atol=1e-12)
        for _ in range(2):
            out.fill_(-1.0)
            nk.betweenness_sampled(g, 3, 150, captured, out=out)
            assert np.allclose(out.cpu().numpy(), ref, rtol=1e-9, atol=1e-12)


def test_captured_run_follows_the_wait_limit(nk):
    """The bound on device-side waits is part of a captured run: a later nk_set_wait_limit_ns holds for
    the same call too (a bound of 1 ns runs out at once, the default one does not)."""
    import torch
    g = nk.graph_generate("er", 3000, 4, avg_deg=8.0)
    out = torch.empty(3000, dtype=torch.float64, device="cuda")
    o = nk.run_opts(mode=nk.MODE_BATCHED, batch=64, flags=nk.RUN_CUDA_GRAPH)
    nk.betweenness_sampled(g, 3, 100, o, out=out)
    want = out.cpu().numpy().copy()
    try:
        nk.set_wait_limit_ns(1)
        with pytest.raises(nk.NkError) as e:
            nk.betweenness_sampled(g, 3, 100, o, out=out)
        assert e.value.rc == nk.ERR_TIMEOUT
    finally:
        nk.set_wait_limit_ns(10_000_000_000)  # the default
    nk.betweenness_sampled(g, 3, 100, o, out=out)
    assert np.array_equal(out.cpu().numpy(), want)


@pytest.mark.parametrize("avg_deg", [15.0, 22.0])
@pytest.mark.parametrize("k", [4, 6, 13])
def test_few_sources_are_as_exact_as_one_by_one(nk, avg_deg, k):
    """Scores of a few sources swept together are no further from the oracle's FP64 than those of the
    per-source form, a quarter allowed for the oracle's own rounding and the order of the sums."""
    g = nk.graph_generate("er", 5000, 3, avg_deg=avg_deg)
    n, rp, col = oracle.generate("er", 5000, 3, avg_deg=avg_deg)
    src = oracle.sample_sources(n, 5, k)
    ref = oracle.betweenness_sources(rp, col, src, 1.0)
    off = [np.linalg.norm(nk.betweenness_sources(g, src, 1.0, nk.run_opts(mode=m)) - ref) / np.linalg.norm(ref)
           for m in (nk.MODE_AUTO, nk.MODE_PER_SOURCE)]
    assert off[0] <= 1.25 * off[1], off


def test_launches_and_sweeps_are_told_apart(nk):
    """Stats: batches, sources or searches swept, and the launches that held them."""
    g = nk.graph_generate("er", 1500, 4, avg_deg=8.0)
    n, rp, col = oracle.generate("er", 1500, 4, avg_deg=8.0)
    with_arcs = lambda k: int((np.diff(rp)[oracle.sample_sources(n, 2, k)] > 0).sum())  # noqa: E731
    stats = lambda: tuple(nk.last_run_stats()[x] for x in ("launches", "kernel_launches"))  # noqa: E731
    for k in (300, 64):
        batches = (with_arcs(k) + 63) // 64
        for call in (nk.betweenness_sampled, nk.edge_betweenness_sampled):
            call(g, 2, k, nk.run_opts(mode=nk.MODE_BATCHED, batch=64))
            assert stats() == (batches, 1)  # one launch, side by side
        nk.closeness_sampled(g, 2, k, nk.run_opts(mode=nk.MODE_BATCHED, batch=64))
        assert stats() == (batches, batches)
        # a grid given by the caller holds one batch at a time
        nk.betweenness_sampled(g, 2, k, nk.run_opts(mode=nk.MODE_BATCHED, batch=64, grid_ctas=200))
        assert stats() == (batches, batches)
    nk.betweenness_sampled(g, 2, 15)
    assert stats() == ((with_arcs(15) + 7) // 8, 1)
    nk.betweenness_sampled(g, 2, 5, nk.run_opts(mode=nk.MODE_PER_SOURCE))
    assert stats() == (with_arcs(5), with_arcs(5))
    nk.random_weights(g, 1, 4)
    nk.betweenness_weighted_sampled(g, 2, 5)
    assert stats() == (1, 1)


@pytest.mark.parametrize("kind,n,params,k", [("er", 3000, dict(avg_deg=8.0), 2900), ("ba", 4000, dict(m0=6), 700)])
def test_scores_do_not_depend_on_how_many_batches_run_at_once(nk, kind, n, params, k):
    """The same request with room for many batches side by side and with room for one at a time, and
    the same call without a server: the sums are added in one order, so the scores are equal."""
    g = nk.graph_generate(kind, n, 6, **params)
    probe = nk.Server(max_inflight=1, pack=False)
    assert probe.wait(probe.submit(g, 1, 100)[0], 300.0) == nk.OK
    need = probe.stats()["peak_bytes"]
    got = []
    for budget in (0, 1.3 * need):
        srv = nk.Server(mem_budget_bytes=budget, max_inflight=1, pack=False, batch=128)
        rid, out = srv.submit(g, 1, k)
        assert srv.wait(rid, 300.0) == nk.OK
        got.append(out.copy())
        srv.close()
    probe.close()
    got.append(nk.betweenness_sampled(g, 1, k, nk.run_opts(mode=nk.MODE_BATCHED, batch=128)))
    assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])


def test_served_batches_side_by_side_within_a_slots_memory(nk):
    """Batches beside a request's first one take memory within the slot's part of the budget, and no
    more of them are counted than the sweep runs side by side on a graph of that size."""
    def peak(g, k, **kw):
        srv = nk.Server(pack=False, batch=128, **kw)
        assert srv.wait(srv.submit(g, 1, k)[0], 300.0) == nk.OK
        bytes_ = srv.stats()["peak_bytes"]
        srv.close()
        return bytes_

    g = nk.graph_generate("er", 3000, 6, avg_deg=8.0)
    one = peak(g, 100, max_inflight=1)
    assert peak(g, 1000, max_inflight=4, mem_budget_bytes=4.4 * one) < 1.1 * one
    assert 3.9 * one < peak(g, 1000, max_inflight=4, mem_budget_bytes=18 * one) <= 4.5 * one
    g = nk.graph_generate("er", 1 << 20, 6, avg_deg=4.0)
    assert peak(g, 1024, max_inflight=1) < 3.1 * peak(g, 100, max_inflight=1)


def test_rows_side_by_side(nk):
    """Path-count and psi rows of the batches that share a launch: 12 bytes a source and vertex, batches
    until they reach 3300 MB together.  2^20 vertices, 128 sources (1536 MB each): three batches."""
    g = nk.graph_generate("er", 1 << 20, 6, avg_deg=4.0)
    for k, batches, launches in ((700, 6, 2), (300, 3, 1)):
        nk.betweenness_sampled(g, 1, k, nk.run_opts(mode=nk.MODE_BATCHED, batch=128))
        st = nk.last_run_stats()
        assert (st["launches"], st["kernel_launches"]) == (batches, launches)


@pytest.mark.parametrize("kind,n,params,k", [("er", 2000, dict(avg_deg=8.0), 1), ("rmat", 18, dict(edge_factor=16), 2)])
def test_sources_swept_one_by_one_are_compacted_once(nk, kind, n, params, k):
    """A single source, and two on a large hub graph, take the per-source form from the library's own
    choice with the launches that the form takes when it is asked for."""
    g = nk.graph_generate(kind, n, 4, **params)
    src = np.argsort(-np.diff(g.export_csr()[0]))[5:5 + k].astype(np.int32)  # vertices with arcs
    launches, scores = [], []
    for mode in (nk.MODE_AUTO, nk.MODE_PER_SOURCE):
        before = nk.launch_count()
        scores.append(nk.betweenness_sources(g, src, 1.0, nk.run_opts(mode=mode)))
        launches.append(nk.launch_count() - before)
        assert nk.last_run_stats()["mode"] == nk.MODE_PER_SOURCE
    assert launches[0] == launches[1]
    assert np.allclose(scores[0], scores[1], rtol=1e-9, atol=1e-12)


def test_width_follows_the_sources_with_arcs(nk):
    """150 sources, 100 of them with arcs, without a width from the caller: the width of 100 sources."""
    rng = np.random.default_rng(5)
    n, u, v = 1500, rng.integers(0, 1000, 6000), rng.integers(0, 1000, 6000)
    g = nk.graph_from_edges(n, u.astype(np.int32), v.astype(np.int32))
    rp, col = oracle.csr_build(n, u.astype(np.int32), v.astype(np.int32))
    src = np.concatenate([np.arange(1000, 1050), np.flatnonzero(np.diff(rp) > 0)[:100]]).astype(np.int32)
    got = nk.betweenness_sources(g, src, 1.0)
    assert nk.last_run_stats()["batch"] == 64
    assert np.allclose(got, oracle.betweenness_sources(rp, col, src, 1.0), rtol=1e-9, atol=1e-12)
    seed = next(s for s in range(100) if (np.diff(rp)[oracle.sample_sources(n, s, 150)] > 0).sum() <= 128)
    far, reach = nk.closeness_sampled(g, seed, 150)
    assert nk.last_run_stats()["batch"] == 128
    ref = oracle.closeness_sampled(rp, col, seed, 150)
    assert np.array_equal(far, ref[0]) and np.array_equal(reach, ref[1])


def test_deep_searches_side_by_side_stay_within_their_memory(nk):
    """Two batches of 8 whose searches are 1000 levels deep (a thousand paths of a thousand vertices from
    one vertex): level slabs for both together within 8 GB, beside 84 bytes a vertex of rows and queues."""
    import torch
    n = 1_000_001
    v = torch.arange(1, n, device="cuda", dtype=torch.int32)
    g = nk.graph_from_edges(n, torch.where((v - 1) % 1000 == 0, 0, v - 1).int(), v)
    src = np.concatenate([[0], 1000 * np.arange(14) + 1 + 37 * np.arange(14)]).astype(np.int32)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    got = nk.betweenness_sources(g, src, 1.0)
    assert nk.last_run_stats()["launches"] == 4  # both batches, with 48 levels and again with more
    held = before - torch.cuda.mem_get_info()[0]
    assert held < (8 << 30) + 2 * 84 * n + (1 << 28), held
    # in a tree a vertex's dependency is the number of vertices that it separates from the source.  Path p
    # has the vertices 1000 p + 1 + j, j = 0 ... 999 outwards: 999 - j beyond one; on the source's own path,
    # between it and the root, j nearer the root, the root, and the other 999 paths
    want = np.zeros(n)
    j = np.arange(1000)
    for s in src:
        below = np.tile(999.0 - j, 1000)  # vertices further out, per path
        if s:
            p, i = divmod(int(s) - 1, 1000)
            want[0] += 999 * 1000
            below[1000 * p: 1000 * (p + 1)] = np.where(j > i, 999 - j, np.where(j < i, j + 1 + 999 * 1000, 0))
        want[1:] += below
    assert np.allclose(got, want, rtol=1e-9, atol=1e-12)


@pytest.mark.parametrize("kind,n,params", [("er", 1151, dict(avg_deg=8.0)), ("er", 1152, dict(avg_deg=8.0)), ("ba", 21888, dict(m0=3)),
                                           ("rmat", 10, dict(edge_factor=8))])
def test_weighted_small_graphs(nk, kind, n, params):
    """A search of a small graph gets no more CTAs than its vertices can use (3 to 57), and a few sources
    are swept as they come, without a compaction: sampler, sweep, sum, scale.  R-MAT: some without arcs."""
    g = nk.graph_generate(kind, n, 4, **params)
    n, rp, col = oracle.generate(kind, n, 4, **params)
    nk.random_weights(g, 5, 16)
    before = nk.launch_count()
    nk.sample_sources(n, 6, 4)
    sampler = nk.launch_count() - before
    for k in (1, 4, 40):
        before = nk.launch_count()
        got = nk.betweenness_weighted_sampled(g, 6, k)
        if k == 4:
            assert nk.launch_count() - before == sampler + 3
        assert nk.last_run_stats()["tpv"] <= max(3, min(57, n // 384))
        ref = oracle.betweenness_weighted_sampled(rp, col, nk.export_weights(g), 6, k)
        assert np.allclose(got, ref, rtol=1e-9, atol=1e-12)


@pytest.mark.parametrize("kind,params", [("er", dict(avg_deg=8.0)), ("rmat", dict(edge_factor=8))])
def test_dependencies_of_a_batch_are_summed_exactly(nk, kind, params):
    """The scores of 64 sources in one batch against those of the same sources one to a batch, summed in
    FP64: a source's dependencies are the same numbers either way.  What the batch may lose is one
    double-single addition per lane, 2^-49 each and independent over 32 lanes (2e-16 in the mean square), and
    the FP64 roundings (1e-16).  Joining the lanes in double-single too loses 1e-15."""
    import math
    g = nk.graph_generate(kind, 1000 if kind == "er" else 10, 4, **params)
    src = np.argsort(-np.diff(g.export_csr()[0]), kind="stable")[40:104].astype(np.int32)
    opts = nk.run_opts(mode=nk.MODE_BATCHED, batch=64)
    one = np.array([nk.betweenness_sources(g, src[i:i + 1], 1.0, opts) for i in range(len(src))])
    want = np.array([math.fsum(c) for c in one.T])
    got = nk.betweenness_sources(g, src, 1.0, opts)
    assert np.array_equal(got == 0.0, want == 0.0)
    nz = want > 0.0
    assert np.sqrt(np.mean(((got[nz] - want[nz]) / want[nz]) ** 2)) < 5e-16
