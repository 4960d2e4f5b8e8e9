"""One source per CTA (csrc/bc_solo.cuh): the sizes where its tiles, tiers and
tables end. Every sum is exact, so results equal the oracle's, and on graphs too
large for it the 64-lane engine's, bit for bit."""
import os

import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def _ctx(solo_n=None):
    import paper_1608_04472_gb300 as pkg
    old = os.environ.pop("BCG_SOLO_N", None)
    try:
        if solo_n is not None:
            os.environ["BCG_SOLO_N"] = str(solo_n)
        return pkg.Context(0, batch_width=64)
    finally:
        os.environ.pop("BCG_SOLO_N", None)
        if old is not None:
            os.environ["BCG_SOLO_N"] = old


def _regular(n, d):
    """Circulant graph: every row has exactly d entries (d even)."""
    i = np.arange(n, dtype=np.int64)
    eu = np.concatenate([i] * (d // 2))
    ev = np.concatenate([(i + k) % n for k in range(1, d // 2 + 1)])
    return gg.from_edges(n, eu, ev)


def _bipartite(a, b):
    u, v = np.divmod(np.arange(a * b, dtype=np.int64), b)
    return gg.from_edges(a + b, u, a + v)


SMALL = {
    "one vertex": lambda: gg.from_edges(1, [], []),
    "two vertices": lambda: gg.from_edges(2, [0], [1]),
    "no edges": lambda: gg.from_edges(70, [], []),
    "rows of 32": lambda: _regular(203, 32),
    "rows of 34": lambda: _regular(203, 34),
    "rows of 2 to 33": lambda: gg.erdos_renyi(333, 17, 5),
    "star, row above 2048": lambda: _bipartite(1, 2500),
    "70 rows of 2100": lambda: _bipartite(70, 2100),   # more longest rows than the CTA's list holds
    "levels beyond the shared table": lambda: gg.from_edges(600, np.arange(599), np.arange(1, 600)),
    "counts beyond 2^64": lambda: gg.grid(38),
    "hubs and isolated vertices": lambda: gg.rmat(11, 8, 0.57, 0.19, 0.19, 7),
}


@pytest.mark.parametrize("name", list(SMALL))
def test_small_graphs_equal_the_oracle(name):
    g = SMALL[name]()
    src = sorted({0, g.n // 2, g.n - 1})
    with _ctx() as ctx:
        h = ctx.load_graph(g.row_ptr, g.col)
        delta, dist, sm, se, tier = ctx.source_dependencies_ext(h, src)
        for i, s in enumerate(src):
            d_o, dist_o = oracle.dependencies(g, s)[:2]
            assert np.array_equal(dist[i], dist_o)
            assert np.array_equal(delta[i], d_o)
        assert np.array_equal(ctx.uniform_sources(h, 40, 3, 4), oracle.uniform_sources(g, 40, 3, 4))
        if g.n > 1:
            t = [0, g.n - 1]
            got, ref = ctx.adaptive_sources(h, t, 2.0, 90, 5, 6), oracle.adaptive_sources(g, t, 2.0, 90, 5, 6)
            assert np.array_equal(got["k"], ref["k"]) and np.array_equal(got["S"], ref["S"])


# (n, degree, directed): the last size with everything in shared memory lies near 18,900;
# 65,536 is the largest graph by rule; a directed graph's 16-bit codes end at 65,535
@pytest.mark.parametrize("n,degree,directed", [(18_800, 6, False), (19_200, 6, False), (65_536, 5, False),
                                               (65_535, 5, True), (65_536, 5, True)])
def test_tier_edges_equal_the_64_lane_engine(n, degree, directed):
    g = gg.directed_er(n, degree, 8) if directed else gg.erdos_renyi(n, degree, 8, pairwise=False)
    out = []
    for solo_n in (None, 0):
        with _ctx(solo_n) as ctx:
            h = ctx.load_graph(g.row_ptr, g.col, directed=directed)
            delta, dist, sigma = ctx.source_dependencies(h, [0, n - 1], want_dist=True, want_sigma=True)
            out.append((ctx.uniform_sources(h, 70, 9, 1), delta, dist, sigma))
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_more_levels_than_the_16_bit_codes():
    """A path of 70,000 vertices: from s, delta_s(v) is the number of vertices beyond v."""
    n = 70_000
    g = gg.from_edges(n, np.arange(n - 1), np.arange(1, n))
    targets = np.array([0, 1, 35_000, 69_998, 69_999], np.int32)
    with _ctx() as ctx:
        h = ctx.load_graph(g.row_ptr, g.col)
        got = ctx.target_dependencies(h, targets, 4, 4, 0, 2)
        src = ctx.draw_sources(4, 4, 0, 2, n)
    for i, s in enumerate(src.tolist()):
        want = [0.0 if v == s else float(n - 1 - v if v > s else v) for v in targets.tolist()]
        assert got[:, i].tolist() == want


def _layers(w, layers):
    i, j = np.divmod(np.arange(w * w), w)
    k = w * np.arange(layers - 1)[:, None]
    return gg.from_edges(w * layers, (i + k).ravel(), (j + w + k).ravel())


@pytest.mark.parametrize("name,make", [("counts in L2 above one source per SM", lambda: gg.grid(80)),
                                       ("long rows beyond 2^64", lambda: _layers(40, 36))])
@pytest.mark.parametrize("k", [100, 200])
def test_deep_graphs_equal_the_oracle(name, make, k):
    """Narrow levels, in tier 0 or 1 by the number of sources; in the extended form
    a level's counts are pulled by the pass that pushes from it."""
    g = make()
    with _ctx() as ctx:
        h = ctx.load_graph(g.row_ptr, g.col)
        got = ctx.uniform_sources(h, k, 3, 9)
        pairs = ctx.adaptive_pairs(h, [5, g.n // 2, g.n - 7], 1.0, 64, 2, 3)  # searches that stop at a level
    assert np.array_equal(got, oracle.uniform_sources(g, k, 3, 9))
    ref = oracle.adaptive_pairs(g, [5, g.n // 2, g.n - 7], 1.0, 64, 2, 3)
    assert np.array_equal(pairs["S"], ref["S"]) and np.array_equal(pairs["k"], ref["k"])


def test_many_deep_graphs_of_every_residency():
    """Square grids that fit an SM four times to once, in one call."""
    gs = [gg.grid(s) for s in (40, 75, 150, 180, 210, 245)]
    with _ctx() as ctx:
        hs = [ctx.load_graph(g.row_ptr, g.col) for g in gs]
        got = ctx.uniform_sources_multi(hs, [3] * 6, [7] * 6, list(range(6)))
        for q, (g, h, e) in enumerate(zip(gs, hs, got)):
            assert np.array_equal(e, ctx.uniform_sources(h, 3, 7, q))
            if g.n < 6000:
                assert np.array_equal(e, oracle.uniform_sources(g, 3, 7, q))


def _every_call(ctx, h, n):
    """One call of each kind with few draws, and the sampling calls with many."""
    t, out = [1, n // 3, n - 2], []
    for k in (3, 64, 200, 700):
        out.append(ctx.uniform_sources(h, k, 3, 4))
        r = ctx.adaptive_sources(h, t, 2.0, k, 5, 6)
        out += [r["S"], r["k"]]
    out += list(ctx.source_dependencies(h, [0, n // 2, n - 1], want_dist=True, want_sigma=True))
    r = ctx.adaptive_pairs(h, t, 1.0, 90, 2, 3)
    out += [r["S"], r["k"], ctx.target_dependencies(h, t, 5, 6, 10, 70)]
    q = ctx.submit(h, 1, targets=t, c=2.0, cap=150, seed=8, qid=9)  # BC_QUERY_SOURCES
    ctx.poll(q, -1)
    out += [q.outputs()["S"], q.outputs()["k"]]
    return out + list(ctx.uniform_sources_multi([h, h], [5, 90], [1, 2], [3, 4]))


@pytest.mark.parametrize("name", ["hubs", "dense", "sparse", "tier 1"])
def test_both_engines_and_the_choice_by_count_agree(name):
    g = {"hubs": lambda: gg.rmat(13, 16, 0.57, 0.19, 0.19, 3), "dense": lambda: gg.erdos_renyi(1500, 200, 5),
         "sparse": lambda: gg.erdos_renyi(6000, 3, 4), "tier 1": lambda: gg.erdos_renyi(30_000, 8, 6, pairwise=False)}[name]()
    got = []
    for solo_n in (None, 0, 65536):  # by the number of sources, never, always
        with _ctx(solo_n) as ctx:
            got.append(_every_call(ctx, ctx.load_graph(g.row_ptr, g.col), g.n))
    for a, b, c in zip(*got):
        assert np.array_equal(a, b) and np.array_equal(a, c)
    assert np.array_equal(got[0][0], oracle.uniform_sources(g, 3, 3, 4))


@pytest.mark.parametrize("name", list(SMALL))
def test_small_graphs_equal_the_oracle_whatever_the_count(name):
    """As test_small_graphs_equal_the_oracle, with every call on one source per CTA."""
    g = SMALL[name]()
    src = sorted({0, g.n // 2, g.n - 1})
    with _ctx(65536) as ctx:
        h = ctx.load_graph(g.row_ptr, g.col)
        delta, dist = ctx.source_dependencies_ext(h, src)[:2]
        for i, s in enumerate(src):
            d_o, dist_o = oracle.dependencies(g, s)[:2]
            assert np.array_equal(dist[i], dist_o) and np.array_equal(delta[i], d_o)
        assert np.array_equal(ctx.uniform_sources(h, 40, 3, 4), oracle.uniform_sources(g, 40, 3, 4))


# (launches of the 64-lane forward pass: "fwd"; of one source per CTA: "ext_fwd")
@pytest.mark.parametrize("graph,draws,family", [
    ("hubs", 16, "fwd"), ("hubs", 64, "fwd"), ("hubs", 1024, "fwd"),       # 1.6 ms a source and CTA
    ("tier 1", 16, "fwd"), ("tier 1", 64, "fwd"), ("tier 1", 1024, "ext_fwd"),
    ("small", 1, "ext_fwd"), ("small", 64, "ext_fwd"), ("small", 1024, "ext_fwd"),
    ("sparse", 16, "ext_fwd"), ("sparse", 1024, "ext_fwd")])               # many levels
def test_the_engine_follows_the_number_of_sources(graph, draws, family):
    g = {"hubs": lambda: gg.rmat(15, 16, 0.57, 0.19, 0.19, 3), "tier 1": lambda: gg.erdos_renyi(60_000, 8, 6, pairwise=False),
         "small": lambda: gg.erdos_renyi(2000, 8, 1), "sparse": lambda: gg.erdos_renyi(60_000, 3, 4, pairwise=False)}[graph]()
    other = {"fwd": "ext_fwd", "ext_fwd": "fwd"}[family]
    with _ctx() as ctx:
        h = ctx.load_graph(g.row_ptr, g.col)
        ctx.uniform_sources(h, 65, 1, 1)  # depth and key are made
        for call in ("uniform", "bader", "served"):
            if call == "served" and draws != 64:
                continue  # (64 at a time whatever the query's draws)
            ctx.reset_stats()
            if call == "uniform":
                ctx.uniform_sources(h, draws, 3, 4)
            elif call == "bader":
                ctx.adaptive_sources(h, [1, 2], 1e9, draws, 3, 4)
            else:
                ctx.poll(ctx.submit(h, 3, k=64, seed=3, qid=4), -1)  # BC_QUERY_UNIFORM
            ran = ctx.stats()["kernels"]
            assert ran[family]["launches"] > 0 and ran[other]["launches"] == 0, call


@pytest.mark.parametrize("n,rows,family", [(43_309, 1, "fwd"), (43_309, 20, "ext_fwd"), (5000, 1, "ext_fwd")])
def test_the_engine_of_per_source_rows_follows_their_number(n, rows, family):
    g = gg.erdos_renyi(n, 6, 5, pairwise=False)
    other = {"fwd": "ext_fwd", "ext_fwd": "fwd"}[family]
    with _ctx() as ctx:
        h = ctx.load_graph(g.row_ptr, g.col)
        ctx.source_dependencies(h, np.arange(rows, dtype=np.int32))  # the depth is known from here on
        ctx.reset_stats()
        ctx.source_dependencies(h, np.arange(rows, dtype=np.int32))
        ran = ctx.stats()["kernels"]
        assert ran[family]["launches"] > 0 and ran[other]["launches"] == 0


@pytest.mark.parametrize("lengths", [False, True])
def test_a_refused_call_leaves_its_outputs_as_they_were(lengths):
    """Outputs large enough to have their pages touched (4 MB)."""
    import ctypes

    from paper_1608_04472_gb300 import capi
    g = gg.erdos_renyi(20_000, 6, 3, pairwise=False)
    src = np.array([0] * 39 + [g.n], np.int32)
    delta = np.full((40, g.n), -7.0)
    dist = np.full((40, g.n), -7, np.int32)
    with _ctx() as ctx:
        h = ctx.load_graph(g.row_ptr, g.col, lengths=gg.edge_lengths(g, 1, 9, 2) if lengths else None)
        rc = capi._lib.bc_source_dependencies(ctx.ptr, h, src.ctypes.data_as(ctypes.POINTER(ctypes.c_int32)), 40,
                                              delta.ctypes.data_as(ctypes.POINTER(ctypes.c_double)),
                                              dist.ctypes.data_as(ctypes.POINTER(ctypes.c_int32)) if not lengths else None,
                                              None)
    assert rc == -1  # BC_E_INVALID
    assert (delta == -7.0).all() and (dist == -7).all()


@pytest.mark.parametrize("name", ["rows of 34", "star, row above 2048", "70 rows of 2100", "layers beyond 2^64",
                                  "hubs and isolated vertices"])
@pytest.mark.parametrize("solo_n", [65536, 0])
def test_run_statistics_count_edges_and_vertices_of_the_searches(name, solo_n):
    """bc_get_stats: shortest-path edges and reached vertices, as the distances give
    them, whichever engine ran the sources."""
    g = _layers(60, 13) if name == "layers beyond 2^64" else SMALL[name]()
    src = sorted({0, g.n // 2, g.n - 1})
    row = np.repeat(np.arange(g.n), np.diff(g.row_ptr))
    with _ctx(solo_n) as ctx:
        h = ctx.load_graph(g.row_ptr, g.col)
        ctx.source_dependencies(h, src)  # the depth is known from here on
        ctx.reset_stats()
        dist = ctx.source_dependencies(h, src, want_dist=True)[1]
        st = ctx.stats()
    assert st["reached"] == sum(int((d > 0).sum()) for d in dist)
    assert st["dag_edges"] == sum(int(((d[row] >= 0) & (d[g.col] == d[row] + 1)).sum()) for d in dist)
