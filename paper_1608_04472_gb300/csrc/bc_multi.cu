// bc_multi.cu -- one source per persistent CTA: the kernels and host side of
// the engine in bc_solo.cuh, and uniform k-source estimates (n/k times the
// summed dependencies of k drawn sources, the per-sample step of Sec. 3 without
// the adaptive stop) for many graphs of uneven size and depth in one call.
//
// CTAs take sources (or, for many graphs, items (graph, run of draws) in
// decreasing order of estimated cost) from one atomic counter and run each on
// their own; levels are separated by CTA barriers, not kernel launches, so a
// small graph costs no launches and a deep one (a grid) no host round trip per
// level. All-vertex sums go to exact per-CTA (per-item) partials that a second
// kernel adds per vertex; for many graphs the launches are replayed from a
// captured CUDA graph.
//
// Arithmetic per source is the library's: exact uint64 counts and exact
// successor sums (order-free); a source whose counts exceed 2^64-1 continues
// in the extended form (bc_xf.cuh; sums in CSR order of the vertex).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <tuple>
#include <vector>

#include "bc_internal.h"
#include "bc_solo.cuh"

namespace bcg {

struct MItem {
  int32_t g;
  int32_t pad;
  int64_t i0, i1;  // draws [i0, i1) of the graph's stream
  int64_t part;    // first Acc of the item's partial sums
};

extern __shared__ uint4 solo_shared[];

__device__ __forceinline__ void prefetch_acc(const Acc *a) {
  asm volatile("prefetch.global.L1 [%0];" ::"l"(a));
  asm volatile("prefetch.global.L1 [%0];" ::"l"(&a->w2));
}

// Sources [0, count) delivered to the sink (lane t = source t; all-vertex sums
// to per-CTA partials) and, where asked, to per-source rows.
template <int TIER, int T>
__global__ void __launch_bounds__(T, 1024 / T)
k_solo(MGraph G, SoloSources src, int count, unsigned *__restrict__ next, unsigned char *__restrict__ scratch,
       size_t stride, Acc *__restrict__ partials, Sink sink, SoloRows rows, unsigned *__restrict__ err,
       unsigned long long *__restrict__ cnt) {
  __shared__ SoloCtl c;
  const SoloMem<TIER> S =
      solo_mem<TIER>(reinterpret_cast<unsigned char *>(solo_shared), scratch + (size_t)blockIdx.x * stride, G.n, G.nnz);
  Acc *part = partials ? partials + (size_t)blockIdx.x * G.n : nullptr;
  if (part)
    for (int32_t v = threadIdx.x; v < G.n; v += T) part[v] = acc_zero();
  solo_init(c);
  int ph = 0;
  unsigned e = 0u;
  for (;;) {
    if (threadIdx.x == 0) c.item = (int)atomicAdd(next, 1u);
    __syncthreads();
    const int t = c.item;
    if (t >= count) break;
    const uint64_t i = src.base + (uint64_t)t;
    const int32_t s = src.list ? src.list[t] : (src.draw ? draw_source(src.seed, src.qid, i, G.n) : (int32_t)i);
    bool ext;
    uint64_t maxc;
    const int L = solo_forward<TIER, T>(G, s, -1, S, c, ph, &ext, &maxc);
    if (rows.dist || rows.sig || rows.sm || rows.tier) {
      // before Theorem 1: coefficients take the counts' place
      const size_t row = (size_t)t * G.n;
      for (int32_t v = threadIdx.x; v < G.n; v += T) {
        const bool r = S.dist[v] != solo_unset<TIER>();
        if (rows.dist) rows.dist[row + v] = r ? (int32_t)S.dist[v] : -1;
        if (rows.sig) rows.sig[row + v] = r ? (ext ? ~0ull : S.get(v)) : 0ull;
        if (rows.sm) {
          Xf x{0.0, 0};
          if (r) x = ext ? solo_xf<TIER>(S, v) : xf_of_u64(S.get(v));
          rows.sm[row + v] = x.m;
          rows.se[row + v] = x.e;
        }
        if (rows.delta) rows.delta[row + v] = 0.0;
      }
      if (TIER == 1 && L >= 65535 && rows.dist) {  // codes wrapped: distances from the level offsets
        __syncthreads();
        for (int l = 65535; l <= L; ++l)
          for (int q = solo_lo<TIER>(S, c, l) + (int)threadIdx.x; q < solo_lo<TIER>(S, c, l + 1); q += T)
            rows.dist[row + S.queue[q]] = l;
      }
      if (rows.tier && threadIdx.x == 0) rows.tier[t] = ext ? 1 : 0;
      __syncthreads();
    }
    solo_backward<TIER, T>(G, L, ext, maxc, S, c, ph, e, [&](int32_t v, double delta) {
      if (rows.delta) rows.delta[(size_t)t * G.n + v] = delta;
      if (sink.tslot) sink_targets(sink, v, t, delta);
      if (part) {
        Acc cur = part[v];
        acc_add(cur, delta, e);
        part[v] = cur;
      }
    }, [&](int32_t v) {
      if (part) prefetch_acc(part + v);
      if (sink.tslot) asm volatile("prefetch.global.L1 [%0];" ::"l"(sink.tslot + v));
    });
    __syncthreads();
  }
  if (e) atomicOr(err, e);
  solo_stats(c, cnt);
}

// Items of many graphs (all within the launch's nmax).
template <int TIER, int T>
__global__ void __launch_bounds__(T, 1024 / T)
k_multi(const MGraph *__restrict__ graphs, const MItem *__restrict__ items, int nitems, unsigned *__restrict__ next,
        unsigned char *__restrict__ scratch, size_t stride, Acc *__restrict__ partials, unsigned *__restrict__ err,
        unsigned long long *__restrict__ cnt) {
  __shared__ SoloCtl c;
  unsigned e = 0u;
  solo_init(c);
  int ph = 0;
  for (;;) {
    if (threadIdx.x == 0) c.item = (int)atomicAdd(next, 1u);
    __syncthreads();
    const int it = c.item;
    if (it >= nitems) break;
    const MItem item = items[it];
    const MGraph G = graphs[item.g];
    const SoloMem<TIER> S =
        solo_mem<TIER>(reinterpret_cast<unsigned char *>(solo_shared), scratch + (size_t)blockIdx.x * stride, G.n, G.nnz);
    Acc *part = partials + item.part;
    for (int32_t v = threadIdx.x; v < G.n; v += T) part[v] = acc_zero();
    for (int64_t i = item.i0; i < item.i1; ++i) {
      bool ext;
      uint64_t maxc;
      const int L = solo_forward<TIER, T>(G, draw_source(G.seed, G.qid, (uint64_t)i, G.n), -1, S, c, ph, &ext, &maxc);
      solo_backward<TIER, T>(G, L, ext, maxc, S, c, ph, e, [&](int32_t v, double delta) {
        Acc cur = part[v];
        acc_add(cur, delta, e);
        part[v] = cur;
      }, [&](int32_t v) { prefetch_acc(part + v); });
    }
    __syncthreads();  // c.item is rewritten only after every thread has used it
  }
  if (e) atomicOr(err, e);
  solo_stats(c, cnt);
}

// Pair sampling on a deep graph. Targets: the full BFS of each target into the
// [n][Tp] tables (counts in the extended form, with tx[j] = 1, when the BFS
// overflows), or its depth alone. Pair lanes: the BFS from sources[t] until dests[t]'s level;
// sigma_st in the extended form (bit t of *pxmask) when a count up to that
// level overflowed.
template <int TIER, int T>
__global__ void __launch_bounds__(T, 1024 / T)
k_solo_targets(MGraph G, const int32_t *__restrict__ targets, int count, int Tp, unsigned *__restrict__ next,
               unsigned char *__restrict__ scratch, size_t stride, int32_t *__restrict__ tdist,
               uint64_t *__restrict__ tsig, int32_t *__restrict__ texp, int32_t *__restrict__ tx,
               int32_t *__restrict__ depth, unsigned long long *__restrict__ cnt) {
  __shared__ SoloCtl c;
  const SoloMem<TIER> S =
      solo_mem<TIER>(reinterpret_cast<unsigned char *>(solo_shared), scratch + (size_t)blockIdx.x * stride, G.n, G.nnz);
  solo_init(c);
  int ph = 0;
  for (;;) {
    if (threadIdx.x == 0) c.item = (int)atomicAdd(next, 1u);
    __syncthreads();
    const int j = c.item;
    if (j >= count) break;
    bool ext;
    uint64_t maxc;
    const int L = solo_forward<TIER, T>(G, targets[j], -1, S, c, ph, &ext, &maxc);
    if (depth) {  // only the depth is wanted
      if (threadIdx.x == 0) depth[j] = L;
      continue;
    }
    for (int32_t v = threadIdx.x; v < G.n; v += T) {
      const size_t o = (size_t)v * Tp + j;
      const bool r = S.dist[v] != solo_unset<TIER>();
      tdist[o] = r ? (int32_t)S.dist[v] : -1;
      tsig[o] = r ? S.get(v) : 0ull;
      texp[o] = (ext && r) ? S.exp[v] : 0;
    }
    if (TIER == 1 && L >= 65535) {
      __syncthreads();
      for (int l = 65535; l <= L; ++l)
        for (int q = solo_lo<TIER>(S, c, l) + (int)threadIdx.x; q < solo_lo<TIER>(S, c, l + 1); q += T)
          tdist[(size_t)S.queue[q] * Tp + j] = l;
    }
    if (threadIdx.x == 0) tx[j] = ext ? 1 : 0;
    __syncthreads();
  }
  if (cnt) solo_stats(c, cnt);
}

template <int TIER, int T>
__global__ void __launch_bounds__(T, 1024 / T)
k_solo_pairs(MGraph G, const int32_t *__restrict__ sources, const int32_t *__restrict__ dests, int count,
             unsigned *__restrict__ next, unsigned char *__restrict__ scratch, size_t stride,
             int32_t *__restrict__ pair_d, uint64_t *__restrict__ pair_sig, int32_t *__restrict__ pair_exp,
             unsigned long long *__restrict__ pxmask, unsigned long long *__restrict__ cnt) {
  __shared__ SoloCtl c;
  const SoloMem<TIER> S =
      solo_mem<TIER>(reinterpret_cast<unsigned char *>(solo_shared), scratch + (size_t)blockIdx.x * stride, G.n, G.nnz);
  solo_init(c);
  int ph = 0;
  for (;;) {
    if (threadIdx.x == 0) c.item = (int)atomicAdd(next, 1u);
    __syncthreads();
    const int t = c.item;
    if (t >= count) break;
    const int32_t dst = dests[t];
    bool ext;
    uint64_t maxc;
    const int L = solo_forward<TIER, T>(G, sources[t], dst, S, c, ph, &ext, &maxc);
    if (threadIdx.x == 0) {
      const bool reached = S.dist[dst] != solo_unset<TIER>();
      pair_d[t] = reached ? L : -1;  // the search ends with dst's level
      pair_sig[t] = reached ? S.get(dst) : 0ull;
      pair_exp[t] = (reached && ext) ? S.exp[dst] : 0;
      if (reached && ext) atomicOr(pxmask, 1ull << t);
    }
    __syncthreads();
  }
  solo_stats(c, cnt);
}

// acc[v] += the CTAs' partial sums (exact): a block takes 32 vertices, its 32
// warps a 32nd of the parts each (one thread per vertex over all parts left
// small graphs with few threads in flight).
__global__ void __launch_bounds__(1024) k_solo_acc(int32_t n, int nparts, const Acc *__restrict__ partials,
                                                   Acc *__restrict__ acc) {
  __shared__ Acc sh[32][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int32_t v = blockIdx.x * 32 + lane;
  Acc a = acc_zero();
  if (v < n)
    for (int p = warp; p < nparts; p += 32) acc_add_acc(a, partials[(size_t)p * n + v]);
  sh[warp][lane] = a;
  __syncthreads();
  a = acc_warp_sum(sh[lane][warp]);  // warp w: vertex w of the block
  const int32_t vw = blockIdx.x * 32 + warp;
  if (lane == 0 && vw < n) {
    acc_add_acc(a, acc[vw]);
    acc[vw] = a;
  }
}

// est[off_g + v] = (n * RN(sum of the items' exact partial sums)) / k
__global__ void k_multi_reduce(const MGraph *__restrict__ graphs, const int32_t *__restrict__ gio,
                               const int32_t *__restrict__ gitems, const MItem *__restrict__ items,
                               const Acc *__restrict__ partials, const int64_t *__restrict__ est_off,
                               double *__restrict__ est) {
  const int g = blockIdx.y;
  const MGraph G = graphs[g];
  const int32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= G.n) return;
  Acc a = acc_zero();
#pragma unroll 4
  for (int q = gio[g]; q < gio[g + 1]; ++q) acc_add_acc(a, partials[items[gitems[q]].part + v]);
  est[est_off[g] + v] = __ddiv_rn(__dmul_rn((double)G.n, acc_round(a)), (double)G.k);
}

// ------------------------------------------------------------------ host --

// Shared memory a CTA can have for its state beside SoloCtl.
constexpr size_t SOLO_SMEM_MAX = (size_t)227 * 1024 - sizeof(SoloCtl) - 64;

// An SM's shared memory and what a CTA takes of it.
constexpr size_t SOLO_SM_SMEM = (size_t)228 * 1024;
static size_t solo_cta_smem(int tier, int32_t n) { return solo_smem(tier, n) + sizeof(SoloCtl) + 1024; }

struct SoloCfg {
  int tier = 2, threads = 256, ncta = 1;
  size_t smem = 0, stride = 0;
};

// The state tier a graph's sources run in. Tier 1's distance codes need an
// undirected graph or n <= 65535 (bc_solo.cuh).
static int solo_tier(const Graph &g) {
  if (solo_smem(0, g.n) <= SOLO_SMEM_MAX) return 0;
  if (solo_smem(1, g.n) <= SOLO_SMEM_MAX && (!g.directed || g.n <= 65535)) return 1;
  return 2;
}

// Shallow graphs can run one source per CTA up to 65,536 vertices and a million
// entries (beyond, the 64-lane engine was faster whatever the draws; us a source,
// 1024 uniform draws, here / there: ER n = 100,000 degree 8 29 / 17, where 152 CTAs'
// counts no longer fit L2; R-MAT s16 with 1.82M entries 12.6 / 12.0). Whether a call
// does: solo_pays.
bool solo_fits(bc_ctx *ctx, const Graph &g) {
  return !g.w && g.n <= ctx->solo_n && g.nnz <= ctx->solo_nnz && solo_tier(g) < 2;
}

static int solo_sms() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return std::max(1, sms);
}

// fn(tier, threads) as compile-time constants.
template <int A, int B> struct SoloForm {
  static constexpr int tier = A, threads = B;
};
template <class F> static auto solo_form(const SoloCfg &c, F fn) {
  if (c.tier == 0) return c.threads == 1024 ? fn(SoloForm<0, 1024>{}) : fn(SoloForm<0, 256>{});
  if (c.tier == 1) return c.threads == 1024 ? fn(SoloForm<1, 1024>{}) : fn(SoloForm<1, 256>{});
  return fn(SoloForm<2, 256>{});
}

template <class K> static int solo_resident(K kern, const SoloCfg &c) {
  int per = 0;
  // (the most any graph asks for, so that another graph's launch, in this plan or
  // on another thread, does not lower it)
  if (c.smem) BCG_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SOLO_SMEM_MAX));
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, c.threads, c.smem) != cudaSuccess || per < 1) {
    cudaGetLastError();
    per = 1;
  }
  return per;
}

// Launch settings for `count` sources of graphs of up to n vertices. Deep
// graphs take CTAs of 256 threads: their levels are narrow, so more CTAs per SM
// beat more threads per level (200x200 grid 14.2 us a source, 21.8 with 1024).
// Shallow ones do so while at least three fit an SM's shared memory (ER n =
// 5000 0.60 us a source, 0.69 with 1024; n = 10,000 1.97 and 1.08; n = 50,000
// 16.6 and 6.6), unless there are too few sources to fill the SMs with small
// CTAs.
static SoloCfg solo_cfg(bc_ctx *ctx, int tier, int32_t n, int64_t nnz, int64_t count, bool deep) {
  SoloCfg c;
  c.tier = tier;
  c.smem = solo_smem(tier, n);
  c.stride = solo_stride(tier, n, nnz);
  if (tier < 2 && !deep) {
    const bool few = count <= solo_sms() && n >= 4096;
    c.threads = (tier == 0 && 3 * solo_cta_smem(tier, n) <= SOLO_SM_SMEM && !few) ? 256 : 1024;
  }
  if (tier < 2 && ctx->solo_threads) c.threads = ctx->solo_threads;
  return c;
}

// Whether `count` sources of a fitting graph that is not deep run one per CTA
// rather than 64 to a traversal (beside: draws of other graphs in the same
// launch). One source per CTA reads
// every row once per source at one CTA's speed, so a launch takes as long as a
// source on a CTA times the rounds over the CTAs, however few the sources; the
// 64-lane engine takes a batch's time for every 64, mostly per level. Both
// estimates, in us, follow the times of uniform, adaptive and served calls of 1 to
// 1024 draws on 40 graphs of 1,500 to 65,536 vertices and 16,000 to a million
// entries (ER, BA, R-MAT, directed ones among them) with either engine; the 64-lane
// engine has to be an eighth faster by them (they are off by about that much). The
// choice costs 1.4 % over the better engine in the geometric mean, for sums at worst
// 1.21 times what always here and 1.05 what the engine before this one took. Here / there, us a call
// of 16 / 64 / 200 / 1024 draws: ER n = 2000 degree 8 133 / 137 / 149 / 291 and 311 / 342
// / 760 / 2799; ER n = 50,000 934 / 950 / 1978 / 7013 and 528 / 658 / 1737 / 7073; R-MAT
// s14 (430,000 entries) 770 / 777 / 797 / 3708 and 399 / 469 / 917 / 3385; s15 (890,000)
// 1617 / 1635 / 1722 / 7246 and 489 / 566 / 1061 / 3995; ER n = 60,000 degree 3 878 / 906 /
// 1905 / 6825 and 1170 / 1320 / 3580 / 16,700.
bool solo_pays(bc_ctx *ctx, const Graph &g, int64_t count, SoloCall call, int64_t beside) {
  if (ctx->solo_always) return true;
  const int tier = solo_tier(g);
  const bool adaptive = call == CALL_ADAPTIVE;
  const double n = (double)g.n, z = (double)g.nnz, depth = (double)graph_depth_hint(ctx, g);
  const int64_t sms = solo_sms();
  auto ctas = [&](int64_t c, bool *small) {
    *small = solo_cfg(ctx, tier, g.n, g.nnz, c, false).threads == 256;
    return sms * (*small ? std::min<int64_t>(4, (int64_t)(SOLO_SM_SMEM / solo_cta_smem(tier, g.n))) : 1);
  };
  bool small;
  const int64_t first = adaptive ? std::max<int64_t>(64, ctas((int64_t)1 << 30, &small)) : 0;
  // a source on a CTA of 1024 and of 256 threads (rows above 64 entries: uneven work)
  const double lat[2] = {10e-3 * n + (g.max_deg > 64 ? 1.2e-3 : 0.85e-3) * z + 2.5 * depth, 30e-3 * n + 2.6e-3 * z};
  const double level = 125.0 + 37.0 * depth, rows = n * (3.8e-3 + 0.38e-3 * depth);
  double solo = 90.0, lane = 50.0;
  auto window = [](int64_t i, int64_t lo, int64_t hi, int64_t left) {
    return std::min(left, std::min(hi, std::max(lo, i / 2)));
  };
  const int64_t draws = adaptive ? std::min<int64_t>(count, 4096) : count;  // (both are linear beyond)
  for (int64_t i = 0, w; i < draws; i += w) {
    w = adaptive ? window(i, first, 4096, draws - i) : draws;
    const int64_t s = ctas(w, &small), all = w + beside;
    const double rounds = 0.5 * std::max(1.0, (double)all / (double)s) + 0.5 * (double)((all + s - 1) / s);
    solo += lat[small] * rounds * ((double)w / (double)all);
  }
  // a window's batches overlap but for the first
  auto lanes = [&](int64_t w) {
    const double share = std::min(1.0, (double)w / 64.0);
    return (level * (0.8 + 0.2 * share) + rows * (0.5 + 0.5 * share)) * (double)((w + 63) / 64 + 1) / 2.0;
  };
  if (adaptive) {
    for (int64_t i = 0, w; i < draws; i += w) {
      w = window(i, 64, 1024, draws - i);
      lane += lanes(w);
    }
  } else {
    lane += (double)(draws / 1024) * lanes(1024) + (draws % 1024 ? lanes(draws % 1024) : 0.0);
  }
  // per-source rows are extracted and transposed there, through buffers of the call,
  // which starts to cost with a few of them (here / there, us, 1 / 3 / 20 rows: ER n =
  // 43,309 degree 6 663 / 704 / 1071 and 544 / 732 / 1373; R-MAT n = 20,000 degree 6
  // 620 / 750 / 936 and 408 / 443 / 967)
  if (call == CALL_ROWS) {
    const double q = std::sqrt(1e-3 * n * (double)count);
    lane += std::min(14.0 * q, 250.0 + 8.0 * q) - 70.0;
  }
  return 0.87 * solo <= lane;
}

// A deep graph's levels keep few of an SM's threads busy, so what counts is how
// many sources an SM has at once: where four CTAs' counts don't fit its shared
// memory (n > 4,700) they go to L2 (tier 1), unless there is no more than one
// source per SM. 4096 sources on square grids, ms, tier 0 / tier 1: n = 2500 3.2 /
// 3.9, 5000 5.9 / 5.7, 10,000 21.3 / 8.6, 18,000 31.8 / 13.2.
static SoloCfg solo_cfg(bc_ctx *ctx, const Graph &g, int64_t count) {
  const bool deep = graph_depth_hint(ctx, g) > ctx->deep_levels;
  int tier = solo_tier(g);
  if (tier == 0 && deep && count > solo_sms() && 4 * solo_cta_smem(0, g.n) > SOLO_SM_SMEM) tier = 1;
  return solo_cfg(ctx, tier, g.n, g.nnz, count, deep);
}

// Resident CTAs over all SMs (at most `cap` per SM when cap > 0, at most
// `count`), within the scratch budget at `per` bytes each.
template <class K> static void solo_ctas(SoloCfg &c, K kern, int64_t count, size_t per, int cap) {
  int r = solo_resident(kern, c);
  if (cap > 0) r = std::min(r, cap);
  int64_t m = std::min<int64_t>(count, (int64_t)solo_sms() * r);
  if ((size_t)m * per > ((size_t)1 << 30)) m = std::min<int64_t>(m, (int64_t)(cta_scratch_budget() / per));
  c.ncta = (int)std::max<int64_t>(1, m);
}

static MGraph mgraph_of(const Graph &g) {
  MGraph G{};
  G.rp = g.rp;
  G.col = g.col;
  G.rp_in = g.rp_in;
  G.col_in = g.col_in;
  G.n = g.n;
  G.long_rows = g.max_deg > 32;
  G.nnz = g.nnz;
  return G;
}
static MGraph mgraph_of(bc_ctx *ctx, const Graph &g) {  // with run statistics
  MGraph G = mgraph_of(g);
  G.stats = graph_depth_hint(ctx, g) <= ctx->deep_levels;
  return G;
}

// ---- many graphs ----

struct MultiGroup {
  SoloCfg cfg;
  int item0 = 0, nitems = 0;
  size_t scratch = 0;  // byte offset of the group's CTAs in the plan's scratch
};

struct MultiPlan {
  std::vector<bc_graph> handles;
  int cap_per_sm = 0;
  std::vector<int64_t> k;
  std::vector<uint64_t> seed, qid;
  int nitems = 0, G = 0;
  int32_t nmax = 0;
  int64_t total_n = 0;
  std::vector<MultiGroup> groups;
  std::vector<cudaStream_t> streams;  // one per group after the first (fork and join)
  std::vector<cudaEvent_t> events;
  DevBuf d_graphs, d_items, d_gio, d_gitems, d_estoff, d_next, partials, scratch, est;
  cudaGraphExec_t exec = nullptr;
  void release() {
    if (exec) cudaGraphExecDestroy(exec);
    exec = nullptr;
    nitems = 0;
    for (cudaEvent_t e : events) cudaEventDestroy(e);
    for (cudaStream_t s : streams) cudaStreamDestroy(s);
    events.clear();
    streams.clear();
    groups.clear();
    for (DevBuf *b : {&d_graphs, &d_items, &d_gio, &d_gitems, &d_estoff, &d_next, &partials, &scratch, &est})
      b->release();
  }
};

static std::map<bc_ctx *, MultiPlan> g_plans;  // one cached plan per context
static std::mutex g_plans_mu;

void forget_multi_plan(bc_ctx *ctx) {
  std::lock_guard<std::mutex> lk(g_plans_mu);
  auto it = g_plans.find(ctx);
  if (it == g_plans.end()) return;
  it->second.release();
  g_plans.erase(it);
}

bool multi_plan_uses_graph(bc_ctx *ctx, bc_graph g) {
  std::lock_guard<std::mutex> lk(g_plans_mu);
  auto it = g_plans.find(ctx);
  if (it == g_plans.end()) return false;
  for (bc_graph h : it->second.handles)
    if (h == g) return true;
  return false;
}

// Groups run beside one another (a group's CTAs start as the one before it
// leaves the SMs), each on its own branch of the captured graph.
static void enqueue_multi(bc_ctx *ctx, MultiPlan &P) {
  cudaStream_t st = ctx->stream;
  cudaMemsetAsync(P.d_next.p, 0, 16 * P.groups.size(), st);
  if (P.groups.size() > 1) cudaEventRecord(P.events[0], st);
  for (size_t i = 0; i < P.groups.size(); ++i) {
    const MultiGroup &m = P.groups[i];
    cudaStream_t gs = i == 0 ? st : P.streams[i - 1];
    if (i > 0) cudaStreamWaitEvent(gs, P.events[0], 0);
    solo_form(m.cfg, [&](auto f) {
      k_multi<decltype(f)::tier, decltype(f)::threads><<<m.cfg.ncta, m.cfg.threads, m.cfg.smem, gs>>>(
          P.d_graphs.as<MGraph>(), P.d_items.as<MItem>() + m.item0, m.nitems, P.d_next.as<unsigned>() + 4 * i,
          P.scratch.as<unsigned char>() + m.scratch, m.cfg.stride, P.partials.as<Acc>(), ctx->ws.err.as<unsigned>(),
          ctx->ws.cnt.as<unsigned long long>());
      return 0;
    });
    if (i > 0) {
      cudaEventRecord(P.events[i], gs);
      cudaStreamWaitEvent(st, P.events[i], 0);
    }
  }
  k_multi_reduce<<<dim3((unsigned)((P.nmax + 255) / 256), (unsigned)P.G), 256, 0, st>>>(
      P.d_graphs.as<MGraph>(), P.d_gio.as<int32_t>(), P.d_gitems.as<int32_t>(), P.d_items.as<MItem>(),
      P.partials.as<Acc>(), P.d_estoff.as<int64_t>(), P.est.as<double>());
}

// Items: each graph's draws are cut into runs of about equal cost (cost of a
// source ~ n + nnz), at least 4 runs per CTA overall. Graphs whose state has
// the same tier and CTA size and fits an SM as often (up to four times) form a
// group with its own launch, so that the largest graph's shared memory does not
// set the CTAs per SM for all; a group's runs are queued largest first so its
// CTAs finish close together.
static void build_plan(bc_ctx *ctx, MultiPlan &P, const std::vector<const Graph *> &gs) {
  const int G = (int)gs.size();
  P.G = G;
  P.nmax = 1;
  P.total_n = 0;
  std::map<std::tuple<int, int, int>, std::vector<int>> by;  // (tier, threads, 4 - CTAs per SM) -> graphs
  for (int g = 0; g < G; ++g) {
    const SoloCfg c = solo_cfg(ctx, *gs[g], (int64_t)1 << 30);
    const int per_sm = (int)std::min<size_t>(c.threads == 1024 ? 1 : 4, SOLO_SM_SMEM / solo_cta_smem(c.tier, gs[g]->n));
    by[{c.tier, c.threads, 4 - per_sm}].push_back(g);
    P.nmax = std::max(P.nmax, gs[g]->n);
    P.total_n += gs[g]->n;
  }
  std::vector<MItem> items;
  int64_t part = 0;
  size_t scratch = 0;
  for (auto it = by.rbegin(); it != by.rend(); ++it) {  // the largest state first
    MultiGroup m;
    int32_t nmax = 1;
    int64_t zmax = 0;
    double total = 0.0;
    for (int g : it->second) {
      nmax = std::max(nmax, gs[g]->n);
      zmax = std::max(zmax, gs[g]->nnz);
      total += (double)P.k[g] * (double)(gs[g]->n + gs[g]->nnz);
    }
    m.cfg = solo_cfg(ctx, std::get<0>(it->first), nmax, zmax, (int64_t)1 << 30, false);
    m.cfg.threads = std::get<1>(it->first);
    solo_form(m.cfg, [&](auto f) {
      solo_ctas(m.cfg, k_multi<decltype(f)::tier, decltype(f)::threads>, (int64_t)1 << 30, m.cfg.stride, P.cap_per_sm);
      return 0;
    });
    const double target = std::max(1.0, total / (4.0 * m.cfg.ncta));
    std::vector<MItem> mine;
    std::vector<double> cost;
    for (int g : it->second) {
      const double c = (double)(gs[g]->n + gs[g]->nnz);
      const int64_t chunk = std::max<int64_t>(1, std::min<int64_t>(P.k[g], (int64_t)(target / c)));
      for (int64_t i0 = 0; i0 < P.k[g]; i0 += chunk) {
        MItem x{};
        x.g = g;
        x.i0 = i0;
        x.i1 = std::min(P.k[g], i0 + chunk);
        mine.push_back(x);
        cost.push_back(c * (double)(x.i1 - x.i0));
      }
    }
    std::vector<int> order(mine.size());
    for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return cost[a] > cost[b]; });
    m.item0 = (int)items.size();
    m.nitems = (int)mine.size();
    for (int i : order) {
      items.push_back(mine[i]);
      items.back().part = part;
      part += gs[mine[i].g]->n;
    }
    m.cfg.ncta = std::min(m.cfg.ncta, m.nitems);
    m.scratch = scratch;
    scratch += m.cfg.stride * (size_t)m.cfg.ncta;
    P.groups.push_back(m);
  }
  P.nitems = (int)items.size();
  std::vector<int32_t> gio(G + 1, 0), gitems(items.size());
  for (const MItem &it : items) gio[it.g + 1]++;
  for (int g = 0; g < G; ++g) gio[g + 1] += gio[g];
  {
    std::vector<int32_t> fill(gio.begin(), gio.end() - 1);
    for (size_t i = 0; i < items.size(); ++i) gitems[fill[items[i].g]++] = (int32_t)i;
  }
  std::vector<MGraph> mg(G);
  std::vector<int64_t> estoff(G);
  int64_t off = 0;
  for (int g = 0; g < G; ++g) {
    mg[g] = mgraph_of(ctx, *gs[g]);
    mg[g].k = P.k[g];
    mg[g].seed = P.seed[g];
    mg[g].qid = P.qid[g];
    estoff[g] = off;
    off += gs[g]->n;
  }
  cudaStream_t st = ctx->stream;
  P.d_graphs.ensure(sizeof(MGraph) * G);
  P.d_items.ensure(sizeof(MItem) * items.size());
  P.d_gio.ensure(4 * (G + 1));
  P.d_gitems.ensure(4 * std::max<size_t>(1, items.size()));
  P.d_estoff.ensure(8 * G);
  P.d_next.ensure(16 * P.groups.size());
  P.partials.ensure(sizeof(Acc) * (size_t)std::max<int64_t>(1, part));
  P.scratch.ensure(std::max<size_t>(scratch, 16));
  P.est.ensure(8 * (size_t)P.total_n);
  BCG_CUDA(cudaMemcpyAsync(P.d_graphs.p, mg.data(), sizeof(MGraph) * G, cudaMemcpyHostToDevice, st));
  BCG_CUDA(cudaMemcpyAsync(P.d_items.p, items.data(), sizeof(MItem) * items.size(), cudaMemcpyHostToDevice, st));
  BCG_CUDA(cudaMemcpyAsync(P.d_gio.p, gio.data(), 4 * (G + 1), cudaMemcpyHostToDevice, st));
  BCG_CUDA(cudaMemcpyAsync(P.d_gitems.p, gitems.data(), 4 * items.size(), cudaMemcpyHostToDevice, st));
  BCG_CUDA(cudaMemcpyAsync(P.d_estoff.p, estoff.data(), 8 * G, cudaMemcpyHostToDevice, st));
  BCG_CUDA(cudaStreamSynchronize(st));
  P.events.assign(P.groups.size(), nullptr);
  P.streams.assign(P.groups.size() - 1, nullptr);
  for (cudaEvent_t &e : P.events) BCG_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
  for (cudaStream_t &s : P.streams) BCG_CUDA(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
  // the per-call launch sequence, captured once and replayed (a stream that
  // cannot be captured, such as the legacy default stream, launches directly)
  cudaGraph_t graph = nullptr;
  if (cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
    cudaGetLastError();
    return;
  }
  enqueue_multi(ctx, P);
  const cudaError_t ce = cudaStreamEndCapture(st, &graph);
  if (ce != cudaSuccess) {
    if (graph) cudaGraphDestroy(graph);
    cuda_check(ce, "cudaStreamEndCapture");
  }
  const cudaError_t ie = cudaGraphInstantiate(&P.exec, graph, 0);
  cudaGraphDestroy(graph);
  cuda_check(ie, "cudaGraphInstantiate");
}

// ---- one graph ----

// Per-context scratch (grown on demand).
struct LaneScratch {
  DevBuf scratch, partials, next;
};
static std::map<bc_ctx *, LaneScratch> g_lane;
static std::mutex g_lane_mu;  // apart from g_plans_mu: a plan being built asks for a graph's depth

void forget_lane_scratch(bc_ctx *ctx) {
  std::lock_guard<std::mutex> lk(g_lane_mu);
  auto it = g_lane.find(ctx);
  if (it == g_lane.end()) return;
  it->second.scratch.release();
  it->second.partials.release();
  it->second.next.release();
  g_lane.erase(it);
}

static LaneScratch &lane_scratch(bc_ctx *ctx) {
  std::lock_guard<std::mutex> lk(g_lane_mu);
  LaneScratch &L = g_lane[ctx];
  L.next.ensure(16);
  BCG_CUDA(cudaMemsetAsync(L.next.p, 0, 16, ctx->stream));
  return L;
}

int solo_slots(bc_ctx *ctx, const Graph &g) {
  SoloCfg c = solo_cfg(ctx, g, (int64_t)1 << 30);
  solo_form(c, [&](auto f) {
    solo_ctas(c, k_solo<decltype(f)::tier, decltype(f)::threads>, (int64_t)1 << 30, c.stride, 0);
    return 0;
  });
  return c.ncta;
}

void add_partials(bc_ctx *ctx, const Graph &g, int nparts, const Acc *partials, Acc *acc) {
  LaunchScope ls(ctx, F_XBWD);
  k_solo_acc<<<(g.n + 31) / 32, 1024, 0, ctx->stream>>>(g.n, nparts, partials, acc);
}

void solo_sources(bc_ctx *ctx, const Graph &g, const SoloSources &src, int count, const Sink &sink,
                  const SoloRows &rows) {
  if (count < 1) return;
  SoloCfg c = solo_cfg(ctx, g, count);  // (may run a BFS of its own: before the counter is cleared)
  LaneScratch &L = lane_scratch(ctx);
  const size_t per = c.stride + (sink.acc ? sizeof(Acc) * (size_t)g.n : 0);
  cudaStream_t st = ctx->stream;
  solo_form(c, [&](auto f) {
    auto kern = k_solo<decltype(f)::tier, decltype(f)::threads>;
    solo_ctas(c, kern, count, per, 0);
    L.scratch.ensure(c.stride * c.ncta);
    if (sink.acc) L.partials.ensure(sizeof(Acc) * (size_t)g.n * c.ncta);
    LaunchScope ls(ctx, F_XFWD);
    kern<<<c.ncta, c.threads, c.smem, st>>>(mgraph_of(ctx, g), src, count, L.next.as<unsigned>(),
                                            L.scratch.as<unsigned char>(), c.stride,
                                            sink.acc ? L.partials.as<Acc>() : nullptr, sink, rows,
                                            ctx->ws.err.as<unsigned>(), ctx->ws.cnt.as<unsigned long long>());
    return 0;
  });
  if (sink.acc) add_partials(ctx, g, c.ncta, L.partials.as<Acc>(), sink.acc);
  ctx->samples += count;
  ctx->batches += 1;
}

void lane_sink(bc_ctx *ctx, const Graph &g, const int32_t *d_sources, int count, const Sink &sink) {
  SoloSources src{};
  src.list = d_sources;
  solo_sources(ctx, g, src, count, sink, SoloRows{});
}

int solo_depth(bc_ctx *ctx, const Graph &g, int32_t v) {
  LaneScratch &L = lane_scratch(ctx);
  SoloCfg c = solo_cfg(ctx, solo_tier(g), g.n, g.nnz, 1, false);
  cudaStream_t st = ctx->stream;
  int32_t *word = L.next.as<int32_t>() + 2;  // the counter is word 0
  BCG_CUDA(cudaMemcpyAsync(word, &v, 4, cudaMemcpyHostToDevice, st));
  solo_form(c, [&](auto f) {
    auto kern = k_solo_targets<decltype(f)::tier, decltype(f)::threads>;
    solo_ctas(c, kern, 1, c.stride, 0);
    L.scratch.ensure(c.stride * c.ncta);
    LaunchScope ls(ctx, F_MISC);
    kern<<<1, c.threads, c.smem, st>>>(mgraph_of(g), word, 1, 1, L.next.as<unsigned>(), L.scratch.as<unsigned char>(),
                                       c.stride, nullptr, nullptr, nullptr, nullptr, word + 1, nullptr);
    return 0;
  });
  int32_t *h = static_cast<int32_t *>(ctx->ws.pinned);
  BCG_CUDA(cudaMemcpyAsync(h, word + 1, 4, cudaMemcpyDeviceToHost, st));
  BCG_CUDA(cudaStreamSynchronize(st));
  return *h;
}

void lane_targets(bc_ctx *ctx, const Graph &g, const int32_t *d_targets, int T, int Tp, int32_t *tdist,
                  uint64_t *tsig, int32_t *texp, int32_t *d_tx) {
  if (T < 1) return;
  SoloCfg c = solo_cfg(ctx, g, T);
  LaneScratch &L = lane_scratch(ctx);
  solo_form(c, [&](auto f) {
    auto kern = k_solo_targets<decltype(f)::tier, decltype(f)::threads>;
    solo_ctas(c, kern, T, c.stride, 0);
    L.scratch.ensure(c.stride * c.ncta);
    LaunchScope ls(ctx, F_XFWD);
    kern<<<c.ncta, c.threads, c.smem, ctx->stream>>>(mgraph_of(ctx, g), d_targets, T, Tp, L.next.as<unsigned>(),
                                                     L.scratch.as<unsigned char>(), c.stride, tdist, tsig, texp, d_tx, nullptr,
                                                     ctx->ws.cnt.as<unsigned long long>());
    return 0;
  });
}

uint64_t lane_pairs(bc_ctx *ctx, const Graph &g, int count) {
  if (count < 1) return 0ull;
  SoloCfg c = solo_cfg(ctx, g, count);
  LaneScratch &L = lane_scratch(ctx);
  Workspace &ws = ctx->ws;
  cudaStream_t st = ctx->stream;
  solo_form(c, [&](auto f) {
    auto kern = k_solo_pairs<decltype(f)::tier, decltype(f)::threads>;
    solo_ctas(c, kern, count, c.stride, 0);
    L.scratch.ensure(c.stride * c.ncta);
    LaunchScope ls(ctx, F_PAIR);
    kern<<<c.ncta, c.threads, c.smem, st>>>(mgraph_of(ctx, g), ws.sources.as<int32_t>(), ws.targets.as<int32_t>(), count,
                                            L.next.as<unsigned>(), L.scratch.as<unsigned char>(), c.stride,
                                            ws.pair_d.as<int32_t>(), ws.pair_sig.as<uint64_t>(),
                                            ws.pair_exp.as<int32_t>(), L.next.as<unsigned long long>() + 1,
                                            ws.cnt.as<unsigned long long>());
    return 0;
  });
  uint64_t *h = static_cast<uint64_t *>(ws.pinned);
  BCG_CUDA(cudaMemcpyAsync(h, L.next.as<unsigned long long>() + 1, 8, cudaMemcpyDeviceToHost, st));
  BCG_CUDA(cudaStreamSynchronize(st));
  ctx->samples += count;
  ctx->batches += 1;
  return h[0];
}

void do_uniform_multi(bc_ctx *ctx, const std::vector<bc_graph> &handles, const std::vector<const Graph *> &gs,
                      const int64_t *k, const uint64_t *seed, const uint64_t *qid, double *est_out) {
  const int G = (int)gs.size();
  std::vector<int64_t> off(G + 1, 0);
  for (int g = 0; g < G; ++g) off[g + 1] = off[g] + gs[g]->n;
  std::vector<int> deep, shallow;
  // deep graphs and ones whose state fits shared memory (where their share of the
  // launch pays) go to the persistent kernels; weighted graphs run per graph (the
  // weighted engine)
  int64_t fitting = 0;
  for (int g = 0; g < G; ++g)
    if (solo_fits(ctx, *gs[g])) fitting += k[g];
  for (int g = 0; g < G; ++g)
    (one_source_per_cta(ctx, *gs[g], k[g], CALL_SUMS, fitting - k[g]) && !gs[g]->w ? deep : shallow).push_back(g);
  std::lock_guard<std::mutex> lk(g_plans_mu);
  MultiPlan &P = g_plans[ctx];
  cudaEvent_t done = nullptr;
  if (!deep.empty()) {
    std::vector<bc_graph> dh;
    std::vector<const Graph *> dg;
    std::vector<int64_t> dk;
    std::vector<uint64_t> ds, dq;
    for (int g : deep) {
      dh.push_back(handles[g]);
      dg.push_back(gs[g]);
      dk.push_back(k[g]);
      ds.push_back(seed[g]);
      dq.push_back(qid[g]);
    }
    const int cap = shallow.empty() ? 0 : ctx->multi_cap;
    const bool same = P.nitems > 0 && P.handles == dh && P.k == dk && P.seed == ds && P.qid == dq &&
                      P.cap_per_sm == cap;
    if (!ctx->stream2) BCG_CUDA(cudaStreamCreateWithFlags(&ctx->stream2, cudaStreamNonBlocking));
    cudaStream_t main = ctx->stream;
    if (!same) {
      P.release();
      P.handles = dh;
      P.k = dk;
      P.seed = ds;
      P.qid = dq;
      P.cap_per_sm = cap;
      ctx->stream = ctx->stream2;  // the plan's sequence is captured on the second stream
      try {
        build_plan(ctx, P, dg);
      } catch (...) {
        ctx->stream = main;
        P.release();  // (a plan cut short, e.g. out of memory, must not pass for the same one next time)
        throw;
      }
      ctx->stream = main;
    }
    // the second stream starts after everything already queued on the main one
    cudaEvent_t ready = nullptr;
    BCG_CUDA(cudaEventCreateWithFlags(&ready, cudaEventDisableTiming));
    BCG_CUDA(cudaEventCreateWithFlags(&done, cudaEventDisableTiming));
    BCG_CUDA(cudaEventRecord(ready, main));
    BCG_CUDA(cudaStreamWaitEvent(ctx->stream2, ready, 0));
    cudaEventDestroy(ready);
    if (P.exec) {
      BCG_CUDA(cudaGraphLaunch(P.exec, ctx->stream2));
    } else {
      ctx->stream = ctx->stream2;
      enqueue_multi(ctx, P);
      ctx->stream = main;
    }
    BCG_CUDA(cudaGetLastError());
    BCG_CUDA(cudaEventRecord(done, ctx->stream2));
    ctx->launches += (int64_t)P.groups.size() + 1;
    ctx->batches += P.nitems;
    for (int g : deep) ctx->samples += k[g];
  }
  try {
    for (int g : shallow) uniform_one(ctx, *gs[g], k[g], seed[g], qid[g], est_out + off[g]);
  } catch (...) {
    if (done) {
      cudaEventSynchronize(done);
      cudaEventDestroy(done);
    }
    throw;
  }
  if (done) {
    BCG_CUDA(cudaStreamWaitEvent(ctx->stream, done, 0));
    cudaEventDestroy(done);
    int64_t poff = 0;
    for (size_t i = 0; i < deep.size(); ++i) {
      const int g = deep[i];
      BCG_CUDA(cudaMemcpyAsync(est_out + off[g], P.est.as<double>() + poff, 8 * (size_t)gs[g]->n,
                               cudaMemcpyDeviceToHost, ctx->stream));
      poff += gs[g]->n;
    }
    BCG_CUDA(cudaStreamSynchronize(ctx->stream));
  }
}

}  // namespace bcg
