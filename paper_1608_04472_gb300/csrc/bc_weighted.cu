// bc_weighted.cu -- the per-sample step on graphs with positive integer edge
// lengths (Sec. 3 step 1 computes shortest paths with Dijkstra; Def. 3's
// predecessor test becomes d(s,u) + w(u,v) = d(s,v); Theorem 1 unchanged).
//
// One source per persistent CTA, in phases separated by CTA barriers:
//  1. Distances by near-far label correcting (Davidson, Baxter, Garland, Owens,
//     "Work-efficient parallel GPU methods for single-source shortest paths",
//     IPDPS 2014): vertices whose distance dropped below a threshold T are
//     relaxed in rounds (atomicMin on exact integer distances); the others wait
//     in a far list until T advances past the smallest of them. The loop ends
//     when no edge can be relaxed, so the distances are exact whatever the
//     threshold schedule.
//  2. One pass over the reached vertices' out-edges keeps a bit per edge that is
//     on a shortest path and counts each vertex's predecessors. Then Kahn rounds
//     over those edges alone: round 0 is s, a vertex pushes its exact count
//     along its shortest-path edges and releases the successors whose last
//     predecessor it was. A carry out of 64 bits marks the sample, whose counts
//     are then pulled in the extended form in the same rounds, in CSR order.
//  3. Theorem 1 over the rounds in reverse (every successor of a vertex is in a
//     later round), along the kept edges (solo_backward, bc_solo.cuh).
// Unit lengths (w == nullptr) give the unweighted step; the results equal the
// other engines' bit for bit.
//
// What bounds it: dependent random reads of distances. With one edge in flight
// per thread, 64-bit distances in global memory and four passes over all edges
// after the distances, R-MAT s15 (lengths 1-100, 256 sources) took 25 ms at 7 %
// of the issue slots. Now rows are walked as flattened 32-edge windows, four in
// flight per warp, by 1024 threads (as in bc_solo.cuh), and distances are 32
// bits in shared memory (tier 0) where the graph's size and longest edge allow,
// else 64 bits in global memory (tier 1): 6.3 ms; R-MAT s18, 152 sources, 277 ->
// 32 ms; ER n = 20,000 7.3 -> 1.6; 100x100 grid 7.9 -> 2.4.
#include <algorithm>
#include <map>
#include <mutex>
#include <vector>

#include "bc_internal.h"
#include "bc_solo.cuh"

namespace bcg {

struct WGraph {
  MGraph g;
  const uint32_t *w, *w_in;  // lengths of the entries (nullptr: all 1)
  uint64_t step;             // near-far threshold increment
};

template <int TIER> struct WMem {
  using D = typename std::conditional<TIER == 0, uint32_t, unsigned long long>::type;
  static constexpr D INF = (D)~(D)0;
  D *dist;
  uint32_t *nearb, *farb;  // one bit per vertex: on the next near list, on the far list
  int32_t *pend;           // predecessors not yet processed
  uint32_t *vmask;         // shortest-path bits of short rows, by vertex
  int32_t *la, *lb, *fa, *fb, *rl;  // near lists, far lists, reached vertices
  SoloMem<1> S;            // counts, topological queue and edge bits by queue position (its dist is unused)
};

__host__ __device__ inline size_t wbits(int32_t n) { return ((size_t)n + 127) / 128 * 16; }
__host__ __device__ inline size_t w_smem(int tier, int32_t n) {
  return tier == 0 ? ((size_t)n * 4 + 15) / 16 * 16 + 2 * wbits(n) : 0;
}
__host__ __device__ inline size_t w_stride(int tier, int32_t n, int64_t nnz) {
  const size_t a4 = solo_al((size_t)n * 4 + 8), a8 = solo_al((size_t)n * 8);
  return 11 * a4 + a8 + solo_al((size_t)(nnz / 16 + 2) * 4) + (tier ? a8 + 2 * solo_al(wbits(n)) : 0);
}

template <int TIER>
__device__ __forceinline__ WMem<TIER> w_mem(unsigned char *sm, unsigned char *gm, int32_t n, int64_t nnz) {
  const size_t a4 = solo_al((size_t)n * 4 + 8), a8 = solo_al((size_t)n * 8);
  WMem<TIER> M{};
  int32_t **p[] = {&M.S.exp, &M.S.far, &M.S.queue, &M.pend, &M.la, &M.lb, &M.fa, &M.fb, &M.rl};
  for (int32_t **q : p) {
    *q = reinterpret_cast<int32_t *>(gm);
    gm += a4;
  }
  M.S.qmask = reinterpret_cast<uint32_t *>(gm);
  M.vmask = reinterpret_cast<uint32_t *>(gm + a4);
  gm += 2 * a4;
  M.S.val = reinterpret_cast<uint64_t *>(gm);
  gm += a8;
  M.S.lmask = reinterpret_cast<uint32_t *>(gm);
  gm += solo_al((size_t)(nnz / 16 + 2) * 4);
  using D = typename WMem<TIER>::D;
  if (TIER == 0) {
    M.dist = reinterpret_cast<D *>(sm);
    M.nearb = reinterpret_cast<uint32_t *>(sm + ((size_t)n * 4 + 15) / 16 * 16);
    M.farb = M.nearb + wbits(n) / 4;
  } else {
    M.dist = reinterpret_cast<D *>(gm);
    M.nearb = reinterpret_cast<uint32_t *>(gm + a8);
    M.farb = reinterpret_cast<uint32_t *>(gm + a8 + solo_al(wbits(n)));
  }
  return M;
}

__device__ __forceinline__ uint32_t wlen(const uint32_t *__restrict__ w, int j) { return w ? w[j] : 1u; }

struct WCtl {
  SoloCtl c;  // c.tail: the topological queue's
  int nnext, nfar, nfar2, nreached;
  unsigned long long minfar;
};

// Appends the warp's flagged vertices to a list.
__device__ __forceinline__ void w_append(bool on, int32_t v, int32_t *list, int *count) {
  const unsigned m = __ballot_sync(FULL, on);
  if (!m) return;
  const int lane = threadIdx.x & 31;
  int base = 0;
  if (lane == 0) base = atomicAdd(count, __popc(m));
  base = __shfl_sync(FULL, base, 0);
  if (on) list[base + __popc(m & ((1u << lane) - 1u))] = v;
}

// The out-edges of list entries [0, e), op by op: rows of up to 32 entries of a
// run of 32 vertices as one flattened list, longer rows by the warp, the longest
// by the CTA. load(v) gives a thread's vertex value, again(v) the same for a row of
// the CTA (without load's side effects); visit(w[], j[], on[],
// value[], bal[]) handles U windows and returns each window's edge bits;
// short_bits(v, mask) and the row's words in lmask get them (BITS).
template <int T, bool BITS, class V, class Load, class Again, class Visit, class Short>
__device__ __forceinline__ void w_rows_pass(const MGraph &G, uint32_t *lmask, SoloCtl &c, const int32_t *list, int e,
                                            int &ph, Load load, Again again, Visit visit, Short short_bits) {
  constexpr int U = SOLO_U;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u, le = lt | (1u << lane);
  uint8_t *own = c.own[warp];
  solo_begin(c, ph);
  for (int cb = solo_next(c, 0, e, ph); cb < e; cb = solo_next(c, 0, e, ph)) {
    const int idx = cb + lane;
    int beg = 0, d = 0;
    int32_t v = -1;
    if (idx < e) {
      v = list[idx];
      beg = G.rp[v];
      d = G.rp[v + 1] - beg;
    }
    const V x = load(v);
    const int ds = d <= 32 ? d : 0;
    int incl = ds;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int y = __shfl_up_sync(FULL, incl, off);
      if (lane >= off) incl += y;
    }
    const int E = __shfl_sync(FULL, incl, 31), start = incl - ds, first = beg - start;
    const unsigned rows = __ballot_sync(FULL, ds > 0);
    if (ds > 0) own[__popc(rows & lt)] = (uint8_t)lane;
    __syncwarp();
    uint32_t mask = 0u;
    int before = -1;
    for (int i0 = 0; i0 < E; i0 += 32 * U) {
      int32_t w[U];
      int j[U];
      V xv[U];
      unsigned bal[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int s = start - (i0 + 32 * u);
        const unsigned f = __reduce_or_sync(FULL, (ds > 0 && (unsigned)s < 32u) ? 1u << s : 0u);
        const int i = i0 + 32 * u + lane;
        const int o = i < E ? (int)own[before + __popc(f & le)] : 0;
        before += __popc(f);
        j[u] = i + __shfl_sync(FULL, first, o);
        xv[u] = __shfl_sync(FULL, x, o);
        w[u] = i < E ? G.col[j[u]] : -1;
      }
      visit(w, j, xv, bal);
      if constexpr (BITS) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int s = start - (i0 + 32 * u);
          if (s >= 0 && s < 32) mask |= bal[u] >> s;
          else if (s < 0 && s > -32) mask |= bal[u] << -s;
        }
      }
    }
    if constexpr (BITS) {
      if (v >= 0) short_bits(v, ds == 32 ? mask : mask & ((1u << ds) - 1u));
    }
    __syncwarp();
    for (unsigned bm = __ballot_sync(FULL, d > 32); bm; bm &= bm - 1u) {
      const int k = __ffs(bm) - 1;
      const int hb = __shfl_sync(FULL, beg, k), he = hb + __shfl_sync(FULL, d, k);
      if (he - hb > SOLO_HUGE_DEG) {
        int slot = 0;
        if (lane == 0) {
          slot = atomicAdd(&c.nhuge[ph % 3], 1);
          if (slot < SOLO_HUGE) c.huge[slot] = cb + k;
        }
        if (__shfl_sync(FULL, slot, 0) < SOLO_HUGE) continue;
      }
      const V hx = __shfl_sync(FULL, x, k);
      for (int j0 = hb; j0 < he; j0 += 32 * U) {
        int32_t w[U];
        int j[U];
        V xv[U];
        unsigned bal[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          j[u] = j0 + 32 * u + lane;
          xv[u] = hx;
          w[u] = j[u] < he ? G.col[j[u]] : -1;
        }
        visit(w, j, xv, bal);
        if (BITS && lane == 0) {
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (j0 + 32 * u < he) lmask[(hb >> 4) + ((j0 - hb) >> 5) + u] = bal[u];
        }
      }
    }
  }
  __syncthreads();
  const int nh = min(c.nhuge[ph % 3], SOLO_HUGE);
  ++ph;
  if (nh) {
    for (int k = 0; k < nh; ++k) {
      const int32_t v = list[c.huge[k]];
      const int hb = G.rp[v], he = G.rp[v + 1];
      const V hx = again(v);
      for (int j0 = hb + warp * 32 * U; j0 < he; j0 += T * U) {
        int32_t w[U];
        int j[U];
        V xv[U];
        unsigned bal[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          j[u] = j0 + 32 * u + lane;
          xv[u] = hx;
          w[u] = j[u] < he ? G.col[j[u]] : -1;
        }
        visit(w, j, xv, bal);
        if (BITS && lane == 0) {
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (j0 + 32 * u < he) lmask[(hb >> 4) + ((j0 - hb) >> 5) + u] = bal[u];
        }
      }
    }
    __syncthreads();
  }
}

// Extended counts of round r (queue entries [b, e)): in-neighbours on shortest
// paths in CSR order.
template <int TIER, int T>
__device__ __forceinline__ void w_xf_level(const WGraph &W, const WMem<TIER> &M, int b, int e) {
  const MGraph &G = W.g;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  using D = typename WMem<TIER>::D;
  auto pred = [&](int j, D dv, int32_t *u) {
    *u = G.col_in[j];
    const D du = M.dist[*u];
    return du != WMem<TIER>::INF && (unsigned long long)du + wlen(W.w_in, j) == (unsigned long long)dv;
  };
  for (int cb = b + warp * 32; cb < e; cb += T) {
    const int idx = cb + lane;
    int32_t v = -1;
    int beg = 0, d = 0;
    if (idx < e) {
      v = M.S.queue[idx];
      beg = G.rp_in[v];
      d = G.rp_in[v + 1] - beg;
    }
    Xf acc{0.0, 0};
    const D dv = v >= 0 ? M.dist[v] : 0;
    if (d <= 32)
      for (int j = beg; j < beg + d; ++j) {
        int32_t u;
        if (pred(j, dv, &u)) acc = xf_add(acc, solo_xf<1>(M.S, u));
      }
    __syncwarp();
    for (unsigned bm = __ballot_sync(FULL, d > 32); bm; bm &= bm - 1u) {
      const int k = __ffs(bm) - 1;
      const int hb = __shfl_sync(FULL, beg, k), he = hb + __shfl_sync(FULL, d, k);
      const D hd = __shfl_sync(FULL, dv, k);
      Xf tot{0.0, 0};
      for (int j0 = hb; j0 < he; j0 += 32) {
        int32_t u = 0;
        const bool ok = j0 + lane < he && pred(j0 + lane, hd, &u);
        solo_xf_warp(tot, ok, ok ? solo_xf<1>(M.S, u) : Xf{0.0, 0});
      }
      if (lane == k) acc = tot;
    }
    if (v >= 0) solo_xf_set<1>(M.S, v, acc);
  }
}

// One source on the whole CTA. deliver(v, delta) gets every reached v != s (one
// thread each); rows(ext) runs on every thread once the counts are known
// (before Theorem 1).
template <int TIER, int T, class F, class RowsFn>
__device__ __forceinline__ void w_source(const WGraph &W, int32_t s, const WMem<TIER> &M, WCtl &sh, int &ph,
                                         unsigned &err, F deliver, RowsFn rows) {
  constexpr int U = SOLO_U;
  using D = typename WMem<TIER>::D;
  const D INF = WMem<TIER>::INF;
  const MGraph &G = W.g;
  SoloCtl &c = sh.c;
  const int tid = threadIdx.x, lane = tid & 31;
  // ---- 1. distances (near-far) ----
  for (int32_t v = tid; v < G.n; v += T) {
    M.dist[v] = INF;
    M.S.val[v] = 0ull;
    M.pend[v] = 0;
  }
  for (int i = tid; i < (int)(wbits(G.n) / 4); i += T) M.nearb[i] = M.farb[i] = 0u;
  __syncthreads();
  if (tid == 0) {
    M.dist[s] = 0;
    M.la[0] = s;
    M.rl[0] = s;
    sh.nreached = 1;
    sh.nnext = 0;
    sh.nfar = 0;
  }
  __syncthreads();
  unsigned long long Tn = W.step;  // threshold
  int nn = 1;
  bool flip = false, fflip = false;
  for (;;) {
    while (nn > 0) {
      const int32_t *cur = flip ? M.lb : M.la;
      int32_t *nxt = flip ? M.la : M.lb;
      int32_t *far = fflip ? M.fb : M.fa;
      w_rows_pass<T, false, D>(
          G, nullptr, c, cur, nn, ph,
          [&](int32_t v) -> D {
            // leave the near list before reading the distance: an improvement
            // from here on puts the vertex on the next one
            if (v >= 0) atomicAnd(&M.nearb[v >> 5], ~(1u << (v & 31)));
            __threadfence_block();
            return v >= 0 ? *(volatile D *)&M.dist[v] : INF;
          },
          [&](int32_t v) -> D { return *(volatile D *)&M.dist[v]; },
          [&](const int32_t(&w)[U], const int(&j)[U], const D(&dv)[U], unsigned(&)[U]) {
            unsigned long long nd[U];
            bool better[U], fresh[U];
#pragma unroll
            for (int u = 0; u < U; ++u) nd[u] = (unsigned long long)dv[u] + (w[u] >= 0 ? wlen(W.w, j[u]) : 0u);
#pragma unroll
            for (int u = 0; u < U; ++u)
              better[u] = w[u] >= 0 && nd[u] < (unsigned long long)*(volatile D *)&M.dist[w[u]];
#pragma unroll
            for (int u = 0; u < U; ++u) {
              D old = 0;
              if (better[u]) old = atomicMin(&M.dist[w[u]], (D)nd[u]);
              better[u] = better[u] && nd[u] < (unsigned long long)old;
              fresh[u] = better[u] && old == INF;
            }
            // the improved distances come before the list bits: whoever clears a
            // near bit after it was seen set here (load, above) reads them
            __threadfence_block();
#pragma unroll
            for (int u = 0; u < U; ++u) {
              const bool near = better[u] && nd[u] < Tn;
              const uint32_t bit = 1u << (w[u] & 31);
              bool push = false;
              if (better[u]) push = (atomicOr((near ? M.nearb : M.farb) + (w[u] >> 5), bit) & bit) == 0u;
              if (__any_sync(FULL, fresh[u])) w_append(fresh[u], w[u], M.rl, &sh.nreached);
              if (__any_sync(FULL, push)) {
                w_append(push && near, w[u], nxt, &sh.nnext);
                w_append(push && !near, w[u], far, &sh.nfar);
              }
            }
          },
          [](int32_t, uint32_t) {});
      nn = sh.nnext;
      __syncthreads();
      if (tid == 0) sh.nnext = 0;
      flip = !flip;
      __syncthreads();
    }
    // advance the threshold past the smallest far distance, then split the far
    // list; entries that came below the old threshold have been relaxed since
    const int nf = sh.nfar;
    if (nf == 0) break;
    if (tid == 0) {
      sh.minfar = ~0ull;
      sh.nfar2 = 0;
    }
    __syncthreads();
    int32_t *far = fflip ? M.fb : M.fa, *far2 = fflip ? M.fa : M.fb;
    unsigned long long mine = ~0ull;
    for (int k = tid; k < nf; k += T) {
      const unsigned long long d = M.dist[far[k]];
      if (d >= Tn && d < mine) mine = d;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const unsigned long long o = __shfl_xor_sync(FULL, mine, off);
      mine = o < mine ? o : mine;
    }
    if (lane == 0 && mine != ~0ull) atomicMin(&sh.minfar, mine);
    __syncthreads();
    const unsigned long long mf = sh.minfar, To = Tn;
    if (mf == ~0ull) break;  // every far entry has been relaxed
    Tn = mf + W.step;
    int32_t *cur = flip ? M.lb : M.la;
    for (int kb = tid - lane; kb < nf; kb += T) {
      const int k = kb + lane;
      int32_t u = 0;
      unsigned long long d = 0ull;
      if (k < nf) {
        u = far[k];
        d = M.dist[u];
        if (d < Tn) atomicAnd(&M.farb[u >> 5], ~(1u << (u & 31)));
        if (d >= To && d < Tn) atomicOr(&M.nearb[u >> 5], 1u << (u & 31));
      }
      w_append(k < nf && d >= To && d < Tn, u, cur, &sh.nnext);
      w_append(k < nf && d >= Tn, u, far2, &sh.nfar2);
    }
    __syncthreads();
    nn = sh.nnext;
    const int rest = sh.nfar2;
    __syncthreads();
    if (tid == 0) {
      sh.nnext = 0;
      sh.nfar = rest;
    }
    fflip = !fflip;
    __syncthreads();
  }
  __syncthreads();
  const int nreached = sh.nreached;
  // ---- 2. shortest-path edges, then Kahn rounds with exact counts ----
  w_rows_pass<T, true, D>(
      G, M.S.lmask, c, M.rl, nreached, ph, [&](int32_t v) -> D { return v >= 0 ? M.dist[v] : INF; },
      [&](int32_t v) -> D { return M.dist[v]; },
      [&](const int32_t(&w)[U], const int(&j)[U], const D(&dv)[U], unsigned(&bal)[U]) {
        bool dag[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
          dag[u] = w[u] >= 0 && (unsigned long long)dv[u] + wlen(W.w, j[u]) == (unsigned long long)M.dist[w[u]];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (dag[u]) atomicAdd(&M.pend[w[u]], 1);
          bal[u] = __ballot_sync(FULL, dag[u]);
        }
      },
      [&](int32_t v, uint32_t mask) { M.vmask[v] = mask; });
  if (tid == 0) {
    M.S.queue[0] = s;
    M.S.val[s] = 1ull;
    c.near[0] = 0;
    c.near[1] = 1;
    c.tail = 1;
    c.ovf = 0;
    c.maxc = 1ull;
  }
  __syncthreads();
  int R = 0, b = 0, e = 1;
  uint64_t mymax = 1ull;
  for (;;) {
    bool ov = false;
    // pushes sv along the edge bits of one word to rows' endpoints
    auto push = [&](bool on, int j, uint64_t sv) {
      int32_t w = -1;
      bool free = false;
      if (on) {
        w = G.col[j];
        ov |= M.S.add(w, sv);
        free = atomicSub(&M.pend[w], 1) == 1;
      }
      w_append(free, w, M.S.queue, &c.tail);
    };
    solo_begin(c, ph);
    for (int cb = solo_next(c, b, e, ph); cb < e; cb = solo_next(c, b, e, ph)) {
      const int idx = cb + lane;
      int beg = 0, d = 0;
      uint32_t mask = 0u;
      uint64_t sv = 0ull;
      if (idx < e) {
        const int32_t v = M.S.queue[idx];
        beg = G.rp[v];
        d = G.rp[v + 1] - beg;
        sv = M.S.val[v];
        mask = d <= 32 ? M.vmask[v] : 0u;
        M.S.qmask[idx] = mask;
      }
      mymax = sv > mymax ? sv : mymax;
      while (__any_sync(FULL, mask != 0u)) {
        push(mask != 0u, beg + __ffs(mask) - 1, sv);
        mask &= mask - 1u;
      }
      for (unsigned bm = __ballot_sync(FULL, d > 32); bm; bm &= bm - 1u) {
        const int k = __ffs(bm) - 1;
        const int hb = __shfl_sync(FULL, beg, k), he = hb + __shfl_sync(FULL, d, k);
        const uint64_t hs = __shfl_sync(FULL, sv, k);
        const uint32_t *words = M.S.lmask + (hb >> 4);
        for (int q0 = 0; hb + 32 * q0 < he; q0 += 32) {
          // 32 words at a time; only the ones with bits are walked
          const uint32_t mw = hb + 32 * (q0 + lane) < he ? words[q0 + lane] : 0u;
          for (unsigned nz = __ballot_sync(FULL, mw != 0u); nz; nz &= nz - 1u) {
            const int o = __ffs(nz) - 1;
            const uint32_t word = __shfl_sync(FULL, mw, o);
            push((word >> lane) & 1u, hb + 32 * (q0 + o) + lane, hs);
          }
        }
      }
    }
    if (ov) c.ovf = 1;
    ++ph;
    __syncthreads();
    const int nt = c.tail;
    if (nt == e) break;
    if (tid == 0) {
      if (R + 2 < SOLO_NEAR) c.near[R + 2] = nt;
      else M.S.far[R + 2] = nt;
    }
    ++R;
    b = e;
    e = nt;
    __syncthreads();
  }
  for (int off = 16; off > 0; off >>= 1) {
    const uint64_t o = __shfl_xor_sync(FULL, mymax, off);
    mymax = o > mymax ? o : mymax;
  }
  if (lane == 0 && mymax > 1ull) atomicMax(&c.maxc, (unsigned long long)mymax);
  const bool ext = c.ovf != 0;
  __syncthreads();
  if (ext) {
    if (tid == 0) solo_xf_set<1>(M.S, s, Xf{1.0, 0});
    __syncthreads();
    for (int r = 1; r <= R; ++r) {
      w_xf_level<TIER, T>(W, M, solo_lo<1>(M.S, c, r), solo_lo<1>(M.S, c, r + 1));
      __syncthreads();
    }
  }
  rows(ext);
  __syncthreads();
  // ---- 3. Theorem 1, rounds in reverse ----
  solo_backward<1, T>(G, R, ext, c.maxc, M.S, c, ph, err, deliver);
  __syncthreads();
}

extern __shared__ uint4 w_shared[];

template <int TIER>
__device__ __forceinline__ WMem<TIER> w_begin(const WGraph &W, unsigned char *scratch, size_t stride, WCtl &sh) {
  solo_init(sh.c);
  return w_mem<TIER>(reinterpret_cast<unsigned char *>(w_shared), scratch + (size_t)blockIdx.x * stride, W.g.n,
                     W.g.nnz);
}

// Batch of sources for a sink: all-vertex sums into per-CTA exact partials.
template <int TIER, int T>
__global__ void __launch_bounds__(T, 1024 / T)
k_w_sink(WGraph W, const int32_t *__restrict__ sources, int count, unsigned *__restrict__ next,
         unsigned char *__restrict__ scratch, size_t stride, Acc *__restrict__ partials, Sink sink,
         unsigned *__restrict__ err) {
  __shared__ WCtl sh;
  const WMem<TIER> M = w_begin<TIER>(W, scratch, stride, sh);
  Acc *part = partials ? partials + (size_t)blockIdx.x * W.g.n : nullptr;
  if (part)
    for (int32_t v = threadIdx.x; v < W.g.n; v += T) part[v] = acc_zero();
  unsigned e = 0u;
  int ph = 0;
  for (;;) {
    if (threadIdx.x == 0) sh.c.item = (int)atomicAdd(next, 1u);
    __syncthreads();
    const int t = sh.c.item;
    if (t >= count) break;
    w_source<TIER, T>(
        W, sources[t], M, sh, ph, e,
        [&](int32_t v, double delta) {
          if (sink.tslot) sink_targets(sink, v, t, delta);
          if (part) {
            Acc cur = part[v];
            acc_add(cur, delta, e);
            part[v] = cur;
          }
        },
        [&](bool) {});
  }
  if (e) atomicOr(err, e);
}

// Per-source rows: delta[t][v], dist[t][v] (int64, -1 unreachable),
// sig[t][v] (UINT64_MAX at reached vertices of an extended sample), the counts
// as mantissa/exponent, tier[t]. delta rows must be zero on entry.
template <int TIER, int T>
__global__ void __launch_bounds__(T, 1024 / T)
k_w_rows(WGraph W, const int32_t *__restrict__ sources, int count, unsigned *__restrict__ next,
         unsigned char *__restrict__ scratch, size_t stride, double *__restrict__ delta, int64_t *__restrict__ dist,
         uint64_t *__restrict__ sig, double *__restrict__ sm, int32_t *__restrict__ se, int32_t *__restrict__ tier,
         unsigned *__restrict__ err) {
  __shared__ WCtl sh;
  const WMem<TIER> M = w_begin<TIER>(W, scratch, stride, sh);
  unsigned e = 0u;
  int ph = 0;
  for (;;) {
    if (threadIdx.x == 0) sh.c.item = (int)atomicAdd(next, 1u);
    __syncthreads();
    const int t = sh.c.item;
    if (t >= count) break;
    const size_t row = (size_t)t * W.g.n;
    w_source<TIER, T>(
        W, sources[t], M, sh, ph, e, [&](int32_t v, double d) { delta[row + v] = d; },
        [&](bool ext) {
          for (int32_t v = threadIdx.x; v < W.g.n; v += T) {
            const bool r = M.dist[v] != WMem<TIER>::INF;
            if (dist) dist[row + v] = r ? (int64_t)M.dist[v] : -1;
            if (sig) sig[row + v] = r ? (ext ? ~0ull : M.S.val[v]) : 0ull;
            if (sm || se) {
              Xf x{0.0, 0};
              if (r) x = ext ? solo_xf<1>(M.S, v) : xf_of_u64(M.S.val[v]);
              if (sm) sm[row + v] = x.m;
              if (se) se[row + v] = x.e;
            }
          }
          if (threadIdx.x == 0 && tier) tier[t] = ext ? 1 : 0;
        });
  }
  if (e) atomicOr(err, e);
}

// ------------------------------------------------------------------ host --

struct WState {
  DevBuf scratch, partials, next;
};
static std::map<bc_ctx *, WState> g_w;
static std::mutex g_w_mu;

void forget_weighted_scratch(bc_ctx *ctx) {
  std::lock_guard<std::mutex> lk(g_w_mu);
  auto it = g_w.find(ctx);
  if (it == g_w.end()) return;
  it->second.scratch.release();
  it->second.partials.release();
  it->second.next.release();
  g_w.erase(it);
}

static WState &w_state(bc_ctx *ctx) {
  std::lock_guard<std::mutex> lk(g_w_mu);
  WState &W = g_w[ctx];
  W.next.ensure(16);
  BCG_CUDA(cudaMemsetAsync(W.next.p, 0, 16, ctx->stream));
  return W;
}

static WGraph w_graph(const Graph &g) {
  WGraph G{};
  G.g.rp = g.rp;
  G.g.col = g.col;
  G.g.rp_in = g.rp_in;
  G.g.col_in = g.col_in;
  G.g.n = g.n;
  G.g.nnz = g.nnz;
  G.w = g.w;
  G.w_in = g.w_in;
  // unit lengths: one unbounded threshold (frontier rounds are the BFS levels)
  G.step = g.w ? (g.w_step ? g.w_step : 1ull) : (1ull << 60);
  return G;
}

constexpr size_t W_SMEM_MAX = (size_t)226 * 1024;  // state, control words and a margin

struct WCfg {
  int tier, threads, ncta;
  size_t smem, stride;
};
template <int A, int B> struct WForm {
  static constexpr int tier = A, threads = B;
};
template <class F> static auto w_form(const WCfg &c, F fn) {
  if (c.tier == 0) return c.threads == 1024 ? fn(WForm<0, 1024>{}) : fn(WForm<0, 256>{});
  return c.threads == 1024 ? fn(WForm<1, 1024>{}) : fn(WForm<1, 256>{});
}

// Tier 0 (distances of 32 bits in shared memory) where no path can be longer
// than 32 bits hold. Small CTAs for small graphs and lattice-like ones, whose
// near lists are short.
static WCfg w_cfg(const Graph &g) {
  WCfg c{};
  const uint64_t longest = g.w ? g.w_max : 1ull;
  const bool narrow = longest * (uint64_t)std::max(1, g.n - 1) < 0xFFFFFFFFull;
  c.tier = narrow && w_smem(0, g.n) + sizeof(WCtl) + 1024 <= W_SMEM_MAX ? 0 : 1;
  c.smem = w_smem(c.tier, g.n);
  c.stride = w_stride(c.tier, g.n, g.nnz);
  c.threads = (g.n < 4096 || g.nnz < 5 * (int64_t)g.n) ? 256 : 1024;
  return c;
}

template <class K> static void w_ctas(WCfg &c, K kern, int count, size_t per) {
  int dev = 0, sms = 0, occ = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // (the most any graph asks for: another thread's graph does not lower it)
  if (c.smem)
    BCG_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)(W_SMEM_MAX - sizeof(WCtl) - 1024)));
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, c.threads, c.smem) != cudaSuccess || occ < 1) {
    cudaGetLastError();
    occ = 1;
  }
  size_t m = std::min<size_t>((size_t)count, (size_t)sms * occ);
  if (m * per > ((size_t)1 << 30)) m = std::min(m, cta_scratch_budget() / per);
  c.ncta = (int)std::max<size_t>(1, m);
}

void wlane_sink(bc_ctx *ctx, const Graph &g, const int32_t *d_sources, int count, const Sink &sink) {
  if (count < 1) return;
  WState &W = w_state(ctx);
  WCfg c = w_cfg(g);
  cudaStream_t st = ctx->stream;
  w_form(c, [&](auto f) {
    auto kern = k_w_sink<decltype(f)::tier, decltype(f)::threads>;
    w_ctas(c, kern, count, c.stride + (sink.acc ? sizeof(Acc) * (size_t)g.n : 0));
    W.scratch.ensure(c.stride * c.ncta);
    if (sink.acc) W.partials.ensure(sizeof(Acc) * (size_t)g.n * c.ncta);
    LaunchScope ls(ctx, F_XFWD);
    kern<<<c.ncta, c.threads, c.smem, st>>>(w_graph(g), d_sources, count, W.next.as<unsigned>(),
                                            W.scratch.as<unsigned char>(), c.stride,
                                            sink.acc ? W.partials.as<Acc>() : nullptr, sink, ctx->ws.err.as<unsigned>());
    return 0;
  });
  if (sink.acc) add_partials(ctx, g, c.ncta, W.partials.as<Acc>(), sink.acc);
  ctx->samples += count;
  ctx->batches += 1;
}

void wlane_rows(bc_ctx *ctx, const Graph &g, const int32_t *d_sources, int count, double *delta, int64_t *dist,
                uint64_t *sig, double *sm, int32_t *se, int32_t *tier) {
  if (count < 1) return;
  WState &W = w_state(ctx);
  WCfg c = w_cfg(g);
  cudaStream_t st = ctx->stream;
  BCG_CUDA(cudaMemsetAsync(delta, 0, sizeof(double) * (size_t)g.n * count, st));
  w_form(c, [&](auto f) {
    auto kern = k_w_rows<decltype(f)::tier, decltype(f)::threads>;
    w_ctas(c, kern, count, c.stride);
    W.scratch.ensure(c.stride * c.ncta);
    LaunchScope ls(ctx, F_XFWD);
    kern<<<c.ncta, c.threads, c.smem, st>>>(w_graph(g), d_sources, count, W.next.as<unsigned>(),
                                            W.scratch.as<unsigned char>(), c.stride, delta, dist, sig, sm, se, tier,
                                            ctx->ws.err.as<unsigned>());
    return 0;
  });
  ctx->samples += count;
  ctx->batches += 1;
}

}  // namespace bcg
