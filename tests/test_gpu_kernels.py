"""The sweeps' kernels at the sizes where their variants and their edges lie."""
import numpy as np
import pytest

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
