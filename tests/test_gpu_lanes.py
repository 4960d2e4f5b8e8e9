"""The 64-lane engine (csrc/bc_batch.cu) where its entry lists, lane groups,
segments and tables end, on graphs small enough for the oracle (which run one
source per CTA by rule: BCG_SOLO_N=0 sends them here)."""
import os

import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_1608_04472_gb300 as pkg
    os.environ["BCG_SOLO_N"] = "0"
    try:
        c = pkg.Context(0, batch_width=64)
    finally:
        del os.environ["BCG_SOLO_N"]
    yield c
    c.close()


def _regular(n, d):
    i = np.arange(n, dtype=np.int64)
    return gg.from_edges(n, np.concatenate([i] * (d // 2)), np.concatenate([(i + k) % n for k in range(1, d // 2 + 1)]))


def _fans(widths):
    """For each a in widths: x - a vertices - y - z, so that a paths reach y and z
    (the table of reciprocals ends at 2048)."""
    eu, ev, n = [], [], 0
    for a in widths:
        mid = np.arange(n + 1, n + 1 + a)
        y = n + 1 + a
        eu += [np.full(a, n), mid, [y]]
        ev += [mid, np.full(a, y), [y + 1]]
        n = y + 2
    return gg.from_edges(n, np.concatenate(eu), np.concatenate(ev))


GRAPHS = {
    "rows of 64 (light) and 66 (heavy)": lambda: gg.from_edges(
        500, *np.concatenate([_regular(250, 64).edges(), _regular(250, 66).edges() + 250]).T),
    "hubs of several segments": lambda: gg.barabasi_albert(3000, 6, 9, m0=8),
    "rows of 1 to 16": lambda: gg.erdos_renyi(700, 7, 3),
    "skewed rows": lambda: gg.rmat(11, 12, 0.57, 0.19, 0.19, 4),
    "counts of 2047, 2048, 2049": lambda: _fans([2047, 2048, 2049]),
    "counts beyond the 96-bit window": lambda: gg.grid(25),
}


@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("lanes", [1, 4, 5, 17, 33, 64])
def test_rows_equal_the_oracle(ctx, name, lanes):
    g = GRAPHS[name]()
    src = np.unique(np.linspace(0, g.n - 1, lanes).astype(np.int32))
    h = ctx.load_graph(g.row_ptr, g.col)
    delta, dist, sigma = ctx.source_dependencies(h, src, want_dist=True, want_sigma=True)
    ctx.free_graph(h)
    for i in range(0, len(src), max(1, len(src) // 6)):
        d_o, dist_o, sig_o = oracle.dependencies(g, int(src[i]))[:3]
        assert np.array_equal(dist[i], dist_o) and np.array_equal(sigma[i], sig_o)
        assert np.array_equal(delta[i], d_o)


@pytest.mark.parametrize("heavy,segment", [(32, 32), (64, 256), (129, 64), (257, 300), (5000, 256)])
def test_splits_equal_the_oracle(ctx, heavy, segment):
    """Light rows at and above the lists' capacities (128 backward, 256 forward)."""
    g = gg.from_edges(900, *np.concatenate([gg.erdos_renyi(420, 128, 6).edges(), gg.erdos_renyi(420, 257, 7).edges() + 440,
                                            [[419, 440], [430, 431]]]).T)
    h = ctx.load_graph(g.row_ptr, g.col)
    ctx.set_tuning(h, dict(ctx.get_tuning(h), heavy_degree=heavy, segment=segment))
    got = ctx.uniform_sources(h, 130, 3, 8)
    ctx.free_graph(h)
    assert np.array_equal(got, oracle.uniform_sources(g, 130, 3, 8))


def test_directed_rows_without_successors(ctx):
    g = gg.directed_rmat(11, 6, 0.57, 0.19, 0.19, 5)
    h = ctx.load_graph(g.row_ptr, g.col, directed=True)
    got = ctx.uniform_sources(h, 100, 2, 3)
    res = ctx.adaptive_sources(h, [0, 1, 7], 2.0, 200, 4, 5)
    ctx.free_graph(h)
    assert np.array_equal(got, oracle.uniform_sources(g, 100, 2, 3))
    ref = oracle.adaptive_sources(g, [0, 1, 7], 2.0, 200, 4, 5)
    assert np.array_equal(res["S"], ref["S"]) and np.array_equal(res["k"], ref["k"])


def test_batches_in_flight_with_extended_lanes(ctx):
    """Thirteen layers of 60 vertices: from the end layers counts reach 60^12 > 2^64,
    from the middle ones they stay below; several batches in flight."""
    w, layers = 60, 13
    i, j = np.divmod(np.arange(w * w), w)
    g = gg.from_edges(w * layers, np.concatenate([i + w * k for k in range(layers - 1)]),
                      np.concatenate([j + w * (k + 1) for k in range(layers - 1)]))
    h = ctx.load_graph(g.row_ptr, g.col)
    got = [ctx.uniform_sources(h, 333, 6, 1) for _ in range(2)]  # the depth is known the second time
    res = ctx.adaptive_sources(h, [0, 300, 779], 2.0, 600, 7, 2)
    ctx.free_graph(h)
    want = oracle.uniform_sources(g, 333, 6, 1)
    assert np.array_equal(got[0], want) and np.array_equal(got[1], want)
    ref = oracle.adaptive_sources(g, [0, 300, 779], 2.0, 600, 7, 2)
    assert np.array_equal(res["S"], ref["S"]) and np.array_equal(res["k"], ref["k"])


@pytest.mark.parametrize("shape", ["edgeless", "matching", "star", "two_stars", "complete", "chain_into_hub"])
def test_source_key_where_landmarks_run_out(ctx, shape):
    """No landmark but the hub, none that reaches it, none of another distance;
    a directed chain of 150 arcs into the hub (deeper than the hub's own reach)."""
    i = np.arange(60)
    edges = {"edgeless": (i[:0], i[:0]), "matching": (i[0:40:2], i[1:40:2]), "star": (0 * i[1:], i[1:]),
             "two_stars": (np.repeat([0, 30], 29), np.delete(i, [0, 30])), "complete": np.triu_indices(60, 1)}
    if shape == "chain_into_hub":
        c = np.arange(150)
        g = gg.from_edges_directed(200, np.r_[c, np.full(49, 150)], np.r_[c + 1, np.arange(151, 200)])
    else:
        g = gg.from_edges(60, *edges[shape])
    h = ctx.load_graph(g.row_ptr, g.col, directed=shape == "chain_into_hub")
    got, exact = ctx.uniform_sources(h, 300, 4, 6), ctx.exact(h)
    ctx.free_graph(h)
    assert np.array_equal(got, oracle.uniform_sources(g, 300, 4, 6))
    assert np.array_equal(exact, oracle.exact_bc(g))


def test_source_key_beside_a_long_path(ctx):
    """A star and, in another component, a path of 30,000 levels: the landmarks'
    pass stays in the hub's component (a level mask for each level of the path would
    take 24 GB)."""
    import torch
    star, path = 70000, 30000
    i = np.arange(1, star)
    p = np.arange(star, star + path - 1)
    g = gg.from_edges(star + path, np.r_[0 * i, p], np.r_[i, p + 1])
    h = ctx.load_graph(g.row_ptr, g.col)
    free = torch.cuda.mem_get_info()[0]
    res = ctx.adaptive_pairs(h, [0, 5], 1.0, 6, 3, 1)
    used = free - torch.cuda.mem_get_info()[0]
    ctx.free_graph(h)
    ref = oracle.adaptive_pairs(g, [0, 5], 1.0, 6, 3, 1)
    assert np.array_equal(res["S"], ref["S"]) and np.array_equal(res["k"], ref["k"])
    assert used < 12 << 30  # the pair search's own arrays: 34 B a vertex and resident CTA


def test_direction_switch_tests_the_first_level_in_every_batch(monkeypatch):
    """A top-down level is two launches, a bottom-up one a single launch. With push_div
    = 20 the level after the sources' neighbours (64 rows of about 9 entries are
    more than 16,000 / 20) runs bottom-up, the last ones top-down; the same batch
    takes the same levels whether or not the graph's depth is known."""
    import paper_1608_04472_gb300 as pkg
    monkeypatch.setenv("BCG_SOLO_N", "0")
    g = gg.erdos_renyi(2000, 8, 3)
    src = np.arange(0, 1920, 30, dtype=np.int32)
    launches = []
    with pkg.Context(0, batch_width=64) as c:
        h = c.load_graph(g.row_ptr, g.col)
        c.set_tuning(h, dict(c.get_tuning(h), push_div=20))
        for _ in range(2):
            c.reset_stats()
            delta = c.source_dependencies(h, src)[0]
            launches.append(c.stats()["kernels"]["fwd"]["launches"])
            assert np.array_equal(delta[7], oracle.dependencies(g, int(src[7]))[0])
    assert launches[0] == launches[1]


def _path_and_star(path, leaves=50):
    """A path 0 - 1 - .. and, in another component, a star around vertex `path`."""
    p, i = np.arange(path - 1), np.arange(leaves)
    return gg.from_edges(path + 1 + leaves, np.r_[p, 0 * i + path], np.r_[p + 1, path + 1 + i])


@pytest.mark.parametrize("before", [None, 26])
@pytest.mark.parametrize("path", [12, 21, 30, 33])
def test_levels_launched_unasked_follow_the_graph_s_own_depth(monkeypatch, before, path):
    """Once a batch from the path's end has shown the depth, a batch from the star is
    launched that deep without asking (up to 29 levels), whatever graph the context
    ran before."""
    import paper_1608_04472_gb300 as pkg
    monkeypatch.setenv("BCG_SOLO_N", "0")
    g = _path_and_star(path)
    with pkg.Context(0, batch_width=64) as c:
        if before:
            d = _path_and_star(before)
            c.source_dependencies(c.load_graph(d.row_ptr, d.col), [0])
        h = c.load_graph(g.row_ptr, g.col)
        far = c.source_dependencies(h, [0])[0]
        c.reset_stats()
        near = c.source_dependencies(h, [path])[0]
        levels = c.stats()["kernels"]["fwd"]["launches"] - 1  # (level 1 is a kernel of its own)
        est = c.uniform_sources(h, 200, 3, 1)
    assert np.array_equal(far[0], oracle.dependencies(g, 0)[0]) and np.array_equal(near[0], oracle.dependencies(g, path)[0])
    assert np.array_equal(est, oracle.uniform_sources(g, 200, 3, 1))
    assert levels == (path - 1 if path - 1 <= 29 else 1)


@pytest.mark.parametrize("shape", ["star_and_path", "hub_to_all_and_chain"])
def test_landmarks_take_no_level_per_vertex_of_a_long_path(ctx, shape):
    """Draws that all miss a path of 3,000 vertices: another component's on the
    undirected graph, a chain of arcs among the vertices the hub points to on the
    directed one. The source key's pass takes a few levels of 12 B a vertex, not one
    per path vertex (3.6 GB and as much again while they grow)."""
    import torch
    n, path, k = 100_000, 3000, 100
    p = np.arange(n - path, n - 1)
    if shape == "star_and_path":
        i = np.arange(1, n - path)
        g = gg.from_edges(n, np.r_[0 * i, p], np.r_[i, p + 1])
    else:
        i = np.arange(1, n)
        g = gg.from_edges_directed(n, np.r_[0 * i, p], np.r_[i, p + 1])
    seed = next(s for s in range(1000) if ctx.draw_sources(s, 1, 0, k, n).max() < n - path)
    h = ctx.load_graph(g.row_ptr, g.col, directed=shape != "star_and_path")
    free = torch.cuda.mem_get_info()[0]
    got = ctx.uniform_sources(h, k, seed, 1)
    used = free - torch.cuda.mem_get_info()[0]
    ctx.free_graph(h)
    # leaves of the star have one shortest path to every other one, through 0
    s = ctx.draw_sources(seed, 1, 0, k, n)
    leaves = n - path - 1
    want = np.zeros(n)
    if shape == "star_and_path":
        want[0] = n * (float(np.sum(s != 0)) * (leaves - 1)) / k
    assert np.array_equal(got, want)
    assert used < 1 << 30  # the 64-lane state of 100,000 vertices: 2 KB each, twice


def _fill(torch, left):
    """Holds the device's memory but for about `left` bytes."""
    torch.cuda.empty_cache()
    held, size = [], torch.cuda.mem_get_info()[0]
    while size >= 2 << 20:
        size = max(0, min(size, torch.cuda.mem_get_info()[0] - left)) >> 21 << 21
        try:
            held.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
        except torch.OutOfMemoryError:
            size //= 2
    return held


def test_a_call_that_ran_out_of_memory_leaves_nothing_half_built(monkeypatch):
    """Calls of a fresh context with more and more of the memory they need: each gives
    the result or BC_E_NOMEM, and the ones after it are right."""
    import torch
    import paper_1608_04472_gb300 as pkg
    monkeypatch.setenv("BCG_SOLO_N", "0")
    i, j = np.divmod(np.arange(60 * 60), 60)
    g = gg.erdos_renyi(200_000, 6, 5, pairwise=False)
    wide = gg.from_edges(60 * 13, np.concatenate([i + 60 * k for k in range(12)]),
                         np.concatenate([j + 60 * (k + 1) for k in range(12)]))
    with pkg.Context(0, batch_width=64) as c:  # every kernel is loaded before memory runs short
        want = c.uniform_sources(c.load_graph(g.row_ptr, g.col), 150, 2, 2)
        c.uniform_sources(c.load_graph(wide.row_ptr, wide.col), 150, 2, 2)
    failed = 0
    with pkg.Context(0, batch_width=64) as c:
        h = c.load_graph(g.row_ptr, g.col)
        for left in (2, 8, 24, 64, 128, 256, 512):
            rest = _fill(torch, left << 20)
            try:
                assert np.array_equal(c.uniform_sources(h, 150, 2, 2), want)
            except pkg.BCError as e:
                assert e.code == -2  # BC_E_NOMEM
                failed += 1
            rest.clear()
            torch.cuda.empty_cache()
        assert np.array_equal(c.uniform_sources(h, 150, 2, 2), want)
    assert failed


@pytest.mark.parametrize("call", ["pairs", "served pairs", "load", "rows"])
def test_memory_held_for_speed_is_given_back(monkeypatch, call):
    """A context that holds two batches' state (about 1.2 KB a vertex each) and, beside
    it, 24 MB of the device's memory: calls that need 100 to 300 MB."""
    import torch
    import paper_1608_04472_gb300 as pkg
    monkeypatch.setenv("BCG_SOLO_N", "0")
    g, big = gg.erdos_renyi(200_000, 6, 5, pairwise=False), gg.erdos_renyi(1_000_000, 24, 6, pairwise=False)
    targets, src = np.arange(0, 200_000, 4000, dtype=np.int32), np.arange(64, dtype=np.int32)

    def run(c, h):
        if call == "pairs":
            return c.adaptive_pairs(h, targets, 1.0, 40, 2, 3)["S"]
        if call == "served pairs":
            t = c.submit(h, pkg.BC_QUERY_PAIRS, targets=targets, c=1.0, cap=40, seed=2, qid=3)
            c.poll(t, -1)
            return t.outputs()["S"]
        if call == "load":
            c.free_graph(c.load_graph(big.row_ptr, big.col))
            return np.zeros(1)
        return c.source_dependencies(h, src)[0]

    with pkg.Context(0, batch_width=64) as c:  # (every kernel loaded, before memory runs short)
        h = c.load_graph(g.row_ptr, g.col)
        want, sums = run(c, h), c.uniform_sources(h, 200, 4, 4)
    with pkg.Context(0, batch_width=64) as c:
        h = c.load_graph(g.row_ptr, g.col)
        assert np.array_equal(c.uniform_sources(h, 200, 4, 4), sums)
        rest = _fill(torch, 24 << 20)
        try:
            assert np.array_equal(run(c, h), want)
        finally:
            rest.clear()
            torch.cuda.empty_cache()
        assert np.array_equal(c.uniform_sources(h, 200, 4, 4), sums)
