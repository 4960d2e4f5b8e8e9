"""The work that programs give this library, as measurable cases.

A case names a graph family, its size and one call of the public Python API
(:class:`paper_1608_04472_gb300.Context`). ``listed()`` holds the fixed cases,
``draw(rng)`` gives more of the same ranges. ``prepare`` makes a random graph of
the family from the seed, loads it into a context and keeps the handle, as a
program does that asks many questions about one graph; ``run`` is one call.
``exact`` gives the same outputs in 64-bit torch arithmetic (sparse products
over the breadth-first levels, Bellman-Ford rounds for edge lengths).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1608_04472_gb300 as bc

RMAT = (0.57, 0.19, 0.19)  # quadrant probabilities a, b, c
LANES = 64                 # sources per dense block in exact()
MAX_LENGTH = 100           # edge lengths are uniform on 1..MAX_LENGTH


# --------------------------------------------------------------------- cases --

def listed():
    return [
        # One look at a few vertices of a small graph: the per-source step with all
        # of its outputs. Latency and launches are everything here.
        dict(name="deps_er2k", call="deps", family="er", n=2000, degree=8, count=4),
        # The paper's estimator on the same small graph (16 targets, c = 5).
        dict(name="bader_er2k", call="bader", family="er", n=2000, degree=8, T=16, c=5.0, cap=4000),
        # Exact betweenness of a small graph, the yardstick of accuracy studies.
        dict(name="exact_er2k", call="exact", family="er", n=2000, degree=8),
        # A sparse graph of odd size without hubs, an odd number of draws.
        dict(name="uniform_er100k", call="uniform", family="er", n=100003, degree=7, k=333),
        # Adaptive sampling on a mid-sized graph with hubs, draws beyond the last window.
        dict(name="bader_rmat16", call="bader", family="rmat", n=1 << 16, degree=16, T=64, c=5.0, cap=1500),
        # Per-source rows of a mid-sized graph handed back to the host (counts and distances too).
        dict(name="deps_ba50k", call="deps", family="ba", n=50001, degree=4, count=70),
        # The benchmark's graph: all-vertex estimate, a quarter of its draws.
        dict(name="uniform_rmat20", call="uniform", family="rmat", n=1 << 20, degree=16, k=1024),
        # The same step along directed edges.
        dict(name="uniform_rmat17_directed", call="uniform", family="rmat", n=1 << 17, degree=16, k=512,
             directed=True),
        # Edge lengths 1..100: shortest paths by length.
        dict(name="uniform_rmat15_lengths", call="uniform", family="rmat", n=1 << 15, degree=16, k=256,
             lengths=True),
        # A road-like lattice: hundreds of levels, path counts beyond 2^64.
        dict(name="bader_grid200", call="bader", family="grid", n=200 * 200, degree=4, T=8, c=5.0, cap=256),
        # Algorithm 1: pairs of vertices on a scale-free graph, threshold c n (every target runs to the cap).
        dict(name="pairs_ba300k", call="pairs", family="ba", n=300007, degree=4, T=64, c=1.0, cap=6000),
        # Many graphs of uneven size and depth in one call.
        dict(name="multi_uneven24", call="multi", family="uneven", n=60000, degree=8, G=24, k=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["deps", "bader", "exact", "uniform", "uniform", "uniform", "pairs", "multi"])
    if call == "multi":
        return dict(call=call, family="uneven", n=_log_int(rng, 6000, 60000), degree=rng.randint(4, 10),
                    G=rng.randint(3, 24), k=rng.randint(17, 256))
    if call == "pairs":
        return dict(call=call, family=rng.choice(["ba", "er", "rmat"]), n=_log_int(rng, 1500, 300000),
                    degree=rng.randint(3, 6), T=_log_int(rng, 1, 64), c=1.0, cap=_log_int(rng, 100, 6000))
    if call == "exact":
        return dict(call=call, family=rng.choice(["er", "ba", "rmat"]), n=_log_int(rng, 500, 6000),
                    degree=rng.randint(3, 8))
    if call == "deps":
        case = dict(call=call, family=rng.choice(["er", "ba", "rmat"]), n=_log_int(rng, 500, 50000),
                    degree=rng.randint(3, 12), count=_log_int(rng, 1, 70))
    else:
        family = rng.choice(["er", "ba", "rmat", "rmat", "grid"])
        case = dict(call=call, family=family, n=_log_int(rng, 2000, 1 << 20), degree=rng.randint(3, 16))
        if family == "grid":
            case.update(n=_log_int(rng, 30, 200) ** 2, degree=4)
    form = rng.choice(["plain", "plain", "directed", "lengths"])
    if case["family"] == "grid" or call == "deps":
        form = "plain"
    if form == "directed":
        case.update(directed=True, n=min(case["n"], 1 << 18))
    if form == "lengths":
        case.update(lengths=True, n=min(case["n"], 1 << 15))
    if call == "deps":
        return case
    # draws such that the whole call stays within the largest listed one
    most = 256 if case["family"] == "grid" or form == "lengths" else 1024
    if call == "uniform":
        case["k"] = _log_int(rng, 30, most)
    else:
        case.update(T=_log_int(rng, 1, 128), c=rng.choice([2.0, 5.0, 10.0]), cap=_log_int(rng, 64, most))
    return case


# -------------------------------------------------------------------- graphs --

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)
    return g


def _csr(n, u, v, directed):
    """CSR of an edge list on the device: loops and duplicates dropped, rows sorted."""
    keep = u != v
    u, v = u[keep], v[keep]
    if not directed:
        u, v = torch.cat([u, v]), torch.cat([v, u])
    key = torch.unique(u * n + v)
    row = torch.div(key, n, rounding_mode="floor")
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    return rp, key - row * n


def _rmat_edges(gen, n, m):
    """R-MAT over 2^ceil(log2 n) vertices; endpoints beyond n are folded back."""
    a, b, c = RMAT
    u = torch.zeros(m, dtype=torch.int64, device="cuda")
    v = torch.zeros_like(u)
    for _ in range(max(1, (n - 1).bit_length())):
        r = torch.rand(m, device="cuda", generator=gen)
        u = u * 2 + (r >= a + b)
        v = v * 2 + (((r >= a) & (r < a + b)) | (r >= a + b + c))
    return u % n, v % n


def _ba_edges(gen, n, m):
    """Preferential attachment: edge e of the list goes from vertex e // m to an
    earlier endpoint of the list, drawn uniformly (which is by degree)."""
    e = n * m
    tail = torch.arange(e, dtype=torch.int64, device="cuda") // m
    # position 2e holds the tail, 2e+1 a copy of a random earlier position
    src = (torch.rand(e, device="cuda", generator=gen, dtype=torch.float64)
           * (2 * torch.arange(e, device="cuda") + 1)).to(torch.int64)
    while True:
        odd = (src & 1) == 1
        if not bool(odd.any()):
            break
        src = torch.where(odd, src[torch.div(src, 2, rounding_mode="floor")], src)
    return tail, tail[torch.div(src, 2, rounding_mode="floor")]


def _grid_edges(n):
    side = math.isqrt(n)
    i = torch.arange(side * side, dtype=torch.int64, device="cuda")
    right, down = i[i % side + 1 < side], i[i + side < side * side]
    return torch.cat([right, down]), torch.cat([right + 1, down + side])


def _graph(family, n, degree, gen, directed=False):
    """(n, row_ptr, col) on the device."""
    if family == "er":
        m = n * degree // (1 if directed else 2)
        u = torch.randint(0, n, (m,), device="cuda", generator=gen)
        v = torch.randint(0, n, (m,), device="cuda", generator=gen)
    elif family == "rmat":
        u, v = _rmat_edges(gen, n, n * degree)
    elif family == "ba":
        u, v = _ba_edges(gen, n, degree)
        if directed:
            swap = torch.rand(u.shape[0], device="cuda", generator=gen) < 0.5
            u, v = torch.where(swap, v, u), torch.where(swap, u, v)
    else:
        u, v = _grid_edges(n)
        n = math.isqrt(n) ** 2
    rp, col = _csr(n, u, v, directed)
    return n, rp, col


def _lengths(n, rp, col, seed):
    """A length per CSR entry, the same in both rows of an edge."""
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), rp[1:] - rp[:-1])
    h = torch.minimum(row, col) * 2654435761 + torch.maximum(row, col) * 40503 + int(seed) * 977
    h = (h ^ (h >> 15)) * 2246822519 & 0xFFFFFFFF
    return (h ^ (h >> 13)) % MAX_LENGTH + 1


def _make(case, seed):
    """The call's graphs and arguments, from the seed alone."""
    gen = _gen(seed)
    directed = bool(case.get("directed", False))
    made = dict(seed=int(seed) % (1 << 31), qid=int(seed) % 1009)
    if case["call"] == "multi":
        made["graphs"] = []
        for i in range(case["G"]):
            family = ("er", "rmat", "grid")[i % 3]
            share = (0.5 + i * (math.sqrt(5) - 1) / 2) % 1.0  # spread evenly, the same for every seed
            n = int(2000 * (case["n"] / 2000) ** share)
            made["graphs"].append(_graph(family, n, case["degree"], gen))
        return made
    n, rp, col = _graph(case["family"], case["n"], case["degree"], gen, directed)
    made.update(n=n, rp=rp, col=col)
    if case.get("lengths", False):
        made["lengths"] = _lengths(n, rp, col, seed)
    if case["call"] == "deps":
        made["sources"] = torch.randint(0, n, (case["count"],), device="cuda", generator=gen)
    if case["call"] in ("bader", "pairs"):
        T = min(case["T"], n)
        if case["call"] == "pairs":  # targets by degree, as hubs are the ones asked about
            order = col[torch.randperm(col.shape[0], device="cuda", generator=gen)[:64 * T]].cpu().numpy()
            _, first = np.unique(order, return_index=True)
            t = torch.from_numpy(order[np.sort(first)][:T].copy()).cuda()
            if t.shape[0] < T:
                t = torch.randperm(n, device="cuda", generator=gen)[:T]
        else:
            t = torch.randperm(n, device="cuda", generator=gen)[:T]
        made["targets"] = t
    return made


def prepare(case, seed):
    made = _make(case, seed)
    ctx = bc.Context(0)
    state = dict(case=case, ctx=ctx, seed=made["seed"], qid=made["qid"])

    def host(x, dtype=np.int32):
        return x.cpu().numpy().astype(dtype)

    if case["call"] == "multi":
        state["graphs"] = [ctx.load_graph(host(rp), host(col)) for _, rp, col in made["graphs"]]
        G = len(state["graphs"])
        state["seeds"] = [made["seed"] + i for i in range(G)]
        state["qids"] = list(range(G))
        return state
    lengths = host(made["lengths"], np.uint32) if "lengths" in made else None
    state["graph"] = ctx.load_graph(host(made["rp"]), host(made["col"]), directed=bool(case.get("directed", False)),
                                    lengths=lengths)
    for name in ("sources", "targets"):
        if name in made:
            state[name] = host(made[name])
    return state


def run(state):
    case, ctx = state["case"], state["ctx"]
    call = case["call"]
    if call == "deps":
        delta, dist, sigma = ctx.source_dependencies(state["graph"], state["sources"], want_dist=True,
                                                     want_sigma=True)
        return dict(delta=delta, dist=dist, sigma=sigma.view(np.int64))
    if call == "exact":
        return dict(bc=ctx.exact(state["graph"]))
    if call == "uniform":
        return dict(est=ctx.uniform_sources(state["graph"], case["k"], state["seed"], state["qid"]))
    if call == "bader":
        return ctx.adaptive_sources(state["graph"], state["targets"], case["c"], case["cap"], state["seed"],
                                    state["qid"])
    if call == "pairs":
        return ctx.adaptive_pairs(state["graph"], state["targets"], case["c"], case["cap"], state["seed"],
                                  state["qid"])
    return dict(est=np.concatenate(ctx.uniform_sources_multi(state["graphs"], case["k"], state["seeds"],
                                                             state["qids"])))


def work(case):
    """Bytes: the graph read once, the results written once. Operations: a test and
    an addition per CSR entry, forward and backward, for every source."""
    n = case["n"]
    if case["family"] == "uneven":
        n = case["G"] * (n - 2000) / math.log(n / 2000)  # the mean of the log-uniform sizes
        nnz = n * case["degree"] * 4 / 3
    elif case["family"] == "er" or case.get("directed", False):
        nnz = n * case["degree"]
    else:
        nnz = n * case["degree"] * (1 if case["family"] == "grid" else 2)
    graph = 4 * (n + 1 + nnz) + (4 * nnz if case.get("lengths", False) else 0)
    call = case["call"]
    sources = {"deps": case.get("count"), "exact": n, "uniform": case.get("k"), "multi": case.get("k"),
               "bader": case.get("cap"), "pairs": case.get("T")}[call]
    out = {"deps": 20 * n * (sources or 0), "bader": 28 * case.get("T", 0), "pairs": 28 * case.get("T", 0)}.get(call,
                                                                                                             8 * n)
    return {"bytes": float(graph + out), "flops": 4.0 * nnz * sources}


# --------------------------------------------------------------------- exact --

def _philox(i, seed, qid):
    """Philox4x64-10, counter (i, 0, 0, 0), key (seed, qid): the first two words."""
    M = (1 << 64) - 1
    c, k0, k1 = [i & M, 0, 0, 0], seed & M, qid & M
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B97F4A7C15) & M, (k1 + 0xBB67AE8584CAA73B) & M
        p0, p1 = 0xD2E7470EE14C6C93 * c[0], 0xCA5A826395121157 * c[2]
        c = [(p1 >> 64) ^ c[1] ^ k0, p1 & M, (p0 >> 64) ^ c[3] ^ k1, p0 & M]
    return c[0], c[1]


def _source_draws(k, seed, qid, n):
    return [(_philox(i, seed, qid)[0] * n) >> 64 for i in range(k)]


def _pair_draws(k, seed, qid, n):
    out = []
    for i in range(k):
        x0, x1 = _philox(i, seed, qid)
        u, w = (x0 * n) >> 64, (x1 * (n - 1)) >> 64
        out.append((u, w + (1 if w >= u else 0)))
    return out


def _matrix(n, rp, col):
    return torch.sparse_csr_tensor(rp, col, torch.ones(col.shape[0], dtype=torch.float64, device="cuda"), (n, n))


def _transposed(n, rp, col):
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), rp[1:] - rp[:-1])
    key, _ = torch.sort(col * n + row)
    r = torch.div(key, n, rounding_mode="floor")
    rpt = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rpt[1:] = torch.cumsum(torch.bincount(r, minlength=n), 0)
    return rpt, key - r * n


class _Levels:
    """Distances, counts and dependencies of blocks of sources, in float64."""

    def __init__(self, n, rp, col, directed=False):
        self.n = n
        self.out = _matrix(n, rp, col)
        self.inn = _matrix(n, *_transposed(n, rp, col)) if directed else self.out

    def forward(self, sources):
        B = len(sources)
        lane = torch.arange(B, device="cuda")
        s = torch.as_tensor(sources, dtype=torch.int64, device="cuda")
        dist = torch.full((self.n, B), -1, dtype=torch.int32, device="cuda")
        sigma = torch.zeros((self.n, B), dtype=torch.float64, device="cuda")
        dist[s, lane] = 0
        sigma[s, lane] = 1.0
        front, level = sigma.clone(), 0
        while True:
            x = self.inn @ front
            new = (x > 0) & (dist < 0)
            if not bool(new.any()):
                return dist, sigma, level
            level += 1
            front = torch.where(new, x, 0.0)
            dist[new] = level
            sigma += front

    def delta(self, sources):
        dist, sigma, level = self.forward(sources)
        delta = torch.zeros_like(sigma)
        for l in range(level, 1, -1):
            coef = torch.where(dist == l, (1.0 + delta) / sigma, 0.0)
            delta += torch.where(dist == l - 1, sigma * (self.out @ coef), 0.0)
        return delta, dist, sigma


class _Lengths:
    """The same with edge lengths: Bellman-Ford rounds, then rounds of the
    counts and dependencies over the shortest-path edges."""

    def __init__(self, n, rp, col, lengths):
        self.n, self.col, self.w = n, col, lengths
        self.row = torch.repeat_interleave(torch.arange(n, device="cuda"), rp[1:] - rp[:-1])

    def delta(self, sources):
        n, B, far = self.n, len(sources), 1 << 60
        lane = torch.arange(B, device="cuda")
        s = torch.as_tensor(sources, dtype=torch.int64, device="cuda")
        dist = torch.full((n, B), far, dtype=torch.int64, device="cuda")
        dist[s, lane] = 0
        to = self.col[:, None].expand(-1, B)
        while True:
            new = dist.scatter_reduce(0, to, dist[self.row] + self.w[:, None], "amin")
            new.clamp_(max=far)
            if torch.equal(new, dist):
                break
            dist = new
        on = (dist[self.row] + self.w[:, None] == dist[self.col]) & (dist[self.row] < far)
        # the longest shortest path in edges: that many rounds settle counts and dependencies
        hops = torch.zeros((n, B), dtype=torch.int32, device="cuda")
        while True:
            new = hops.scatter_reduce(0, to, torch.where(on, hops[self.row] + 1, 0), "amax")
            if torch.equal(new, hops):
                break
            hops = new
        rounds = int(hops.max())
        root = torch.zeros((n, B), dtype=torch.float64, device="cuda")
        root[s, lane] = 1.0
        sigma = root
        for _ in range(rounds):
            sigma = root.index_add(0, self.col, torch.where(on, sigma[self.row], 0.0))
        delta = torch.zeros_like(sigma)
        for _ in range(rounds):
            coef = torch.where(sigma > 0, (1.0 + delta) / sigma.clamp(min=1.0), 0.0)
            delta = sigma * torch.zeros_like(sigma).index_add(0, self.row, torch.where(on, coef[self.col], 0.0))
        delta[s, lane] = 0.0
        return delta, None, sigma


def _blocks(sources, lanes):
    return [sources[i:i + lanes] for i in range(0, len(sources), lanes)]


def _stop(values, bound, cap):
    """Sum in draw order until it exceeds the bound; (S, draws used)."""
    S, k = 0.0, 0
    for x in values[:cap]:
        S += x
        k += 1
        if S > bound:
            break
    return S, k


def _uniform(n, engine, lanes, k, seed, qid):
    total = torch.zeros(n, dtype=torch.float64, device="cuda")
    for block in _blocks(_source_draws(k, seed, qid, n), lanes):
        total += engine.delta(block)[0].sum(1)
    return (n * total / k).cpu().numpy()


def exact(case, seed):
    call = case["call"]
    made = _make(case, seed)
    if call == "multi":
        out = []
        for i, (n, rp, col) in enumerate(made["graphs"]):
            out.append(_uniform(n, _Levels(n, rp, col), LANES * 4, case["k"], made["seed"] + i, i))
        return dict(est=np.concatenate(out))
    n, rp, col = made["n"], made["rp"], made["col"]
    if "lengths" in made:
        engine, lanes = _Lengths(n, rp, col, made["lengths"]), 16
    else:
        engine, lanes = _Levels(n, rp, col, bool(case.get("directed", False))), LANES
    if call == "deps":
        delta = [engine.delta(b)[0].T.cpu().numpy() for b in _blocks(made["sources"].tolist(), lanes)]
        return dict(delta=np.concatenate(delta), dist=None, sigma=None)
    if call == "exact":
        total = torch.zeros(n, dtype=torch.float64, device="cuda")
        for block in _blocks(list(range(n)), 256):
            total += engine.delta(block)[0].sum(1)
        return dict(bc=total.cpu().numpy())
    if call == "uniform":
        return dict(est=_uniform(n, engine, lanes, case["k"], made["seed"], made["qid"]))
    targets, T = made["targets"], made["targets"].shape[0]
    if call == "bader":
        draws = _source_draws(case["cap"], made["seed"], made["qid"], n)
        rows = torch.cat([engine.delta(b)[0][targets] for b in _blocks(draws, lanes)], 1).cpu().numpy()
        scale = float(n)
    else:
        tdist, tsig = [torch.cat(x, 1) for x in
                       zip(*[engine.forward(b)[:2] for b in _blocks(targets.tolist(), lanes)])]
        rows = []
        for block in _blocks(_pair_draws(case["cap"], made["seed"], made["qid"], n), lanes):
            s = torch.tensor([p[0] for p in block], device="cuda")
            t = torch.tensor([p[1] for p in block], device="cuda")
            dist, sigma, _ = engine.forward(s.tolist())
            at = torch.arange(len(block), device="cuda")
            d, sig = dist[t, at], sigma[t, at]
            on = (tdist[s] >= 0) & (tdist[t] >= 0) & (d >= 0)[:, None] & (tdist[s] + tdist[t] == d[:, None])
            on &= (targets[None, :] != s[:, None]) & (targets[None, :] != t[:, None])
            rows.append(torch.where(on, tsig[s] * tsig[t] / sig.clamp(min=1.0)[:, None], 0.0).T)
        rows = torch.cat(rows, 1).cpu().numpy()
        scale = float(n) * (n - 1)
    stops = [_stop(rows[j].tolist(), case["c"] * n, case["cap"]) for j in range(T)]
    S = np.array([x[0] for x in stops])
    return dict(est=scale * S / np.array([x[1] for x in stops]), k=None, S=S, status=None)
