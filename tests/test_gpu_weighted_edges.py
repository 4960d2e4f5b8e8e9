"""The weighted engine (csrc/bc_weighted.cu) where its windows, long rows, state
tiers and level tables end; results equal the oracle's bit for bit."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def _bipartite(a, b):
    u, v = np.divmod(np.arange(a * b, dtype=np.int64), b)
    return gg.from_edges(a + b, u, a + v)


# (graph, shortest and longest length): 32-bit distances in shared memory while
# (n - 1) * longest < 2^32 and n <= ~51,000, else 64 bits in global memory
CASES = {
    "one vertex": (lambda: gg.from_edges(1, [], []), 1, 5),
    "rows of up to 33": (lambda: gg.erdos_renyi(400, 17, 5), 1, 3),
    "star, row above 2048": (lambda: _bipartite(1, 2500), 1, 9),
    "70 rows of 2100": (lambda: _bipartite(70, 2100), 1, 2),
    "more rounds than the shared table": (lambda: gg.from_edges(700, np.arange(699), np.arange(1, 700)), 1, 9),
    "lengths near 2^32": (lambda: gg.rmat(9, 8, 0.57, 0.19, 0.19, 7), 1, 2**32 - 1),
    "counts beyond 2^64": (lambda: gg.grid(38), 7, 7),
    "large CTAs": (lambda: gg.rmat(13, 8, 0.57, 0.19, 0.19, 8), 1, 4),
}


@pytest.mark.parametrize("name", list(CASES))
def test_equals_the_oracle(name):
    import paper_1608_04472_gb300 as pkg
    make, lo, hi = CASES[name]
    g = make()
    w = gg.edge_lengths(g, lo, hi, 11)
    src = sorted({0, g.n // 2, g.n - 1})
    with pkg.Context(0, batch_width=64) as ctx:
        h = ctx.load_graph(g.row_ptr, g.col, lengths=w)
        delta, dist, sigma, sm, se, tier = ctx.source_dependencies_weighted(h, src)
        for i, s in enumerate(src):
            d_o, dist_o, sig_o = oracle.dependencies_w(g, w, s)[:3]
            assert np.array_equal(dist[i], dist_o) and np.array_equal(sigma[i], sig_o)
            assert np.array_equal(delta[i], d_o)
        assert np.array_equal(ctx.uniform_sources(h, 20, 2, 3), oracle.uniform_sources_w(g, w, 20, 2, 3))


@pytest.mark.parametrize("n", [50_000, 53_000])
def test_state_tiers(n):
    import paper_1608_04472_gb300 as pkg
    g = gg.erdos_renyi(n, 6, 4, pairwise=False)
    w = gg.edge_lengths(g, 1, 60, 12)
    with pkg.Context(0, batch_width=64) as ctx:
        h = ctx.load_graph(g.row_ptr, g.col, lengths=w)
        delta, dist = ctx.source_dependencies_weighted(h, [1, n - 1])[:2]
    for i, s in enumerate([1, n - 1]):
        d_o, dist_o = oracle.dependencies_w(g, w, s)[:2]
        assert np.array_equal(dist[i], dist_o) and np.array_equal(delta[i], d_o)
