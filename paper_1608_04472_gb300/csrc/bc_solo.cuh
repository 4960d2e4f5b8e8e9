// bc_solo.cuh -- the per-sample Brandes step with one source per CTA (device
// side; kernels and host in bc_multi.cu). Sec. 3 steps 1-2 for one source s:
// a queue BFS (levels contiguous in the queue) whose single pass over a
// level's out-edges finds the next level, pushes the path counts along the
// shortest-path edges (exact integer sums in any order) and keeps one bit per
// edge, set where the edge is on a shortest path; then Theorem 1 over the levels
// in decreasing distance, which visits only the edges with a bit set. Levels
// are separated by CTA barriers.
//
// What bounds it: instruction issue (an edge visit costs a column read, a look
// at the neighbour's distance and its share of finding the row it belongs to)
// and, on deep graphs, the latency of a level's chain of dependent loads. Two
// passes over all edges forward and one backward, a row per group of threads,
// took 190 instructions per edge visit on ER n = 2000 (issue 56 %, 0.50 us a
// source); hence the single flattened pass and the edge bits. On deep graphs a
// level is one round of a few warps, so its chain was shortened: a level's
// entries also in shared memory, one barrier a level forward, the next level's
// entries and row bounds loaded a level ahead in the backward pass, in the
// extended form one pass instead of a push and a pull, no FP64 multiplication by
// powers of two (256 sources on a 200x200 grid 3.21 -> 2.55 ms). The state tiers:
//   tier 0  distances, queue and counts in shared memory, 12 B per vertex
//           (n up to ~18,500);
//   tier 1  distances (2 B) in shared memory, queue and counts in global
//           memory, where 152 CTAs' arrays mostly fit L2 (n up to ~111,000);
//   tier 2  everything in global memory (any n).
// Where each is taken, with the times: solo_pays, solo_cfg (bc_multi.cu).
#pragma once

#include <type_traits>

#include "bc_internal.h"
#include "bc_xf.cuh"

namespace bcg {

struct MGraph {
  const int32_t *rp;     // out-neighbours
  const int32_t *col;
  const int32_t *rp_in;  // in-neighbours (the same arrays for an undirected graph): counts in
  const int32_t *col_in; // the extended form are summed over them in CSR order
  int32_t n;
  uint8_t long_rows;     // a row has more than 32 entries
  uint8_t stats;         // count run statistics (not on deep graphs: 3 % of a 200x200 grid's calls)
  int64_t nnz;
  int64_t k;
  uint64_t seed, qid;
};

constexpr int SOLO_NEAR = 512;  // level offsets kept in shared memory (the rest in global)
constexpr int SOLO_HUGE = 64;   // rows taken by the whole CTA per pass (more fall back to a warp)
constexpr int SOLO_HUGE_DEG = 2048;
constexpr int SOLO_U = 4;       // 32-edge windows a warp has in flight at once
constexpr int SOLO_RING = 512;  // tiers 1, 2: entries of a level kept in shared memory too

struct SoloCtl {
  int item, tail;
  int ovf;                      // a count left 64 bits (tail, ovf: the weighted engine's)
  int nhuge[3];                 // longest rows found by pass ph in slot ph % 3
  int found[3], over[3];        // vertices reached by pass ph; a count left 64 bits in it
  int l53;                      // first level with a count of 2^53 or more
  int grab[2];                  // next list position of the running and of the next pass
  unsigned long long maxc;      // largest count
  int huge[SOLO_HUGE];          // queue positions
  int near[SOLO_NEAR];
  unsigned long long red[32][3];
  uint8_t own[32][32];          // per warp: the threads that hold non-empty short rows
  // run statistics: shortest-path edges of the last source and of the ones
  // before, vertices at distance >= 1
  unsigned last_edges;
  unsigned long long edges, reached;
};

// The state of one source. Distances are codes: the level (tier 2), or the
// level mod 65535 in 16 bits with 65535 for "not reached". On an undirected
// graph neighbours differ by at most one level, so the code tells levels
// apart at any depth; a directed graph takes the 16-bit form only while
// n <= 65535. Edge bits: qmask[i] for the row of queue entry i (up to 32
// entries); a longer row's words start at lmask[beg / 16] (rows above 32
// entries never share a word there: they advance beg / 16 by at least
// ceil(length / 32)).
template <int TIER> struct SoloMem {
  using D = typename std::conditional<TIER == 2, int32_t, uint16_t>::type;
  using Q = typename std::conditional<TIER == 0, uint16_t, int32_t>::type;
  D *dist;
  Q *queue;
  int32_t *ring;       // tiers 1, 2: the first SOLO_RING entries of level l at (l & 1) * SOLO_RING
  uint64_t *val;       // tiers 1, 2: counts, then coefficients (double bits; mantissas in the extended form)
  uint32_t *lo, *hi;   // tier 0: the same in halves (shared memory adds 32 bits at once)
  int32_t *exp;        // exponents of the extended form
  int32_t *far;        // level offsets beyond SOLO_NEAR
  uint32_t *qmask, *lmask;
  __device__ __forceinline__ uint64_t get(int32_t v) const {
    if constexpr (TIER == 0) return ((uint64_t)hi[v] << 32) | lo[v];
    else return val[v];
  }
  __device__ __forceinline__ void set(int32_t v, uint64_t x) const {
    if constexpr (TIER == 0) {
      lo[v] = (uint32_t)x;
      hi[v] = (uint32_t)(x >> 32);
    } else {
      val[v] = x;
    }
  }
  // Adds x to v's count; true when the sum left 64 bits.
  __device__ __forceinline__ bool add(int32_t v, uint64_t x) const {
    if constexpr (TIER == 0) {
      const uint32_t xl = (uint32_t)x, old = atomicAdd(&lo[v], xl);
      const uint32_t carry = old + xl < xl ? 1u : 0u, h = (uint32_t)(x >> 32) + carry;
      bool ov = h < carry;
      if (h) ov |= atomicAdd(&hi[v], h) + h < h;
      return ov;
    } else {
      return atomicAdd(reinterpret_cast<unsigned long long *>(val) + v, (unsigned long long)x) + x < x;
    }
  }
};

__host__ __device__ inline size_t solo_al(size_t x) { return (x + 255) / 256 * 256; }

// Shared and global bytes of one CTA's state.
__host__ __device__ inline size_t solo_smem(int tier, int32_t n) {
  const size_t d = ((size_t)n * 2 + 15) / 16 * 16, w = ((size_t)n * 4 + 15) / 16 * 16;
  return tier == 0 ? 2 * d + 2 * w : (tier == 1 ? d : 0) + 8 * SOLO_RING;
}
__host__ __device__ inline size_t solo_stride(int tier, int32_t n, int64_t nnz) {
  const size_t a4 = solo_al((size_t)n * 4 + 8);
  return 3 * a4 + solo_al((size_t)(nnz / 16 + 2) * 4) + (tier >= 1 ? a4 + solo_al((size_t)n * 8) : 0) +
         (tier == 2 ? a4 : 0);
}

template <int TIER>
__device__ __forceinline__ SoloMem<TIER> solo_mem(unsigned char *sm, unsigned char *gm, int32_t n, int64_t nnz) {
  SoloMem<TIER> S{};
  const size_t a4 = solo_al((size_t)n * 4 + 8);
  const size_t d = ((size_t)n * 2 + 15) / 16 * 16, w = ((size_t)n * 4 + 15) / 16 * 16;
  S.exp = reinterpret_cast<int32_t *>(gm);
  S.far = reinterpret_cast<int32_t *>(gm + a4);
  S.qmask = reinterpret_cast<uint32_t *>(gm + 2 * a4);
  S.lmask = reinterpret_cast<uint32_t *>(gm + 3 * a4);
  gm += 3 * a4 + solo_al((size_t)(nnz / 16 + 2) * 4);
  if constexpr (TIER == 0) {
    S.dist = reinterpret_cast<uint16_t *>(sm);
    S.queue = reinterpret_cast<uint16_t *>(sm + d);
    S.lo = reinterpret_cast<uint32_t *>(sm + 2 * d);
    S.hi = reinterpret_cast<uint32_t *>(sm + 2 * d + w);
  } else {
    S.queue = reinterpret_cast<int32_t *>(gm);
    S.val = reinterpret_cast<uint64_t *>(gm + a4);
    S.ring = reinterpret_cast<int32_t *>(sm);
    if constexpr (TIER == 1) S.dist = reinterpret_cast<uint16_t *>(sm + 8 * SOLO_RING);
    else S.dist = reinterpret_cast<int32_t *>(gm + a4 + solo_al((size_t)n * 8));
  }
  return S;
}

template <int TIER> __device__ __forceinline__ typename SoloMem<TIER>::D solo_code(int level) {
  if constexpr (TIER == 2) return level;
  else return (uint16_t)(level < 65535 ? level : level % 65535);
}
template <int TIER> __device__ __forceinline__ typename SoloMem<TIER>::D solo_unset() {
  if constexpr (TIER == 2) return -1;
  else return (uint16_t)0xFFFFu;
}

// First thread to give w its level wins. 16-bit codes: an AND of the code into
// the word's half turns "not reached" (all ones) into the code and leaves the
// same code unchanged; the other half is ANDed with ones.
template <int TIER> __device__ __forceinline__ bool solo_claim(const SoloMem<TIER> &S, int32_t w, int level) {
  if constexpr (TIER == 2) {
    return atomicCAS(&S.dist[w], -1, level) == -1;
  } else {
    const int sh = (w & 1) << 4;
    const uint32_t keep = ~(0xFFFFu << sh) | ((uint32_t)solo_code<TIER>(level) << sh);
    const uint32_t old = atomicAnd(reinterpret_cast<uint32_t *>(S.dist) + (w >> 1), keep);
    return ((old >> sh) & 0xFFFFu) == 0xFFFFu;
  }
}

template <int TIER> __device__ __forceinline__ int solo_lo(const SoloMem<TIER> &S, const SoloCtl &c, int l) {
  return l < SOLO_NEAR ? c.near[l] : S.far[l];
}

// Queue entry idx of level l, which starts at position b. A level's entries go
// to shared memory as they are found, so a narrow level's next pass starts
// without a round trip to L2.
template <int TIER> __device__ __forceinline__ int32_t solo_entry(const SoloMem<TIER> &S, int l, int b, int idx) {
  if constexpr (TIER != 0)
    if (idx - b < SOLO_RING) return S.ring[(l & 1) * SOLO_RING + idx - b];
  return S.queue[idx];
}

__device__ __forceinline__ void solo_init(SoloCtl &c) {
  if (threadIdx.x < 3) c.nhuge[threadIdx.x] = c.found[threadIdx.x] = c.over[threadIdx.x] = 0;
  if (threadIdx.x < 2) c.grab[threadIdx.x] = 0;
  if (threadIdx.x == 0) {
    c.edges = c.reached = 0ull;
    c.last_edges = 0u;
  }
}
// Adds the CTA's run statistics to the library's, after its last source.
__device__ __forceinline__ void solo_stats(const SoloCtl &c, unsigned long long *__restrict__ cnt) {
  if (threadIdx.x == 0 && c.reached) {
    atomicAdd(cnt, c.edges + c.last_edges);
    atomicAdd(cnt + 1, c.reached);
  }
}

// A pass over list positions [b, e) in runs of 32 from a shared counter (uneven
// rows spread over the warps). Returns the warp's next run or e. ph counts the
// passes, the same in every thread. A pass clears the next one's counters: that
// pass's list position was last used one pass ago, what it finds was last read
// two passes ago, each before the barrier that ended the pass before this one.
__device__ __forceinline__ void solo_begin(SoloCtl &c, int ph) {
  if (threadIdx.x == 0) {
    c.grab[(ph + 1) & 1] = 0;
    c.nhuge[(ph + 1) % 3] = c.found[(ph + 1) % 3] = c.over[(ph + 1) % 3] = 0;
  }
}
__device__ __forceinline__ int solo_next(SoloCtl &c, int b, int e, int ph) {
  if (b >= e) return e;  // (the first run is the warp's by its number: a narrow level has no other)
  int k = 0;
  if ((threadIdx.x & 31) == 0) k = atomicAdd(&c.grab[ph & 1], 32);
  return min(e, b + __shfl_sync(FULL, k, 0));
}

// U edge visits per thread (w[u] < 0: none): finds the vertices not reached so
// far (they join `level` and the queue), adds sv[u] to the count of every
// endpoint at `level`, and returns the warp's shortest-path bits in bal[u]. The
// level starts at queue position e; slot: the pass's counters.
template <int TIER, int U, bool COUNT>
__device__ __forceinline__ void solo_visit(const SoloMem<TIER> &S, SoloCtl &c, int level, int e, int slot,
                                           const int32_t (&w)[U], const uint64_t (&sv)[U], unsigned (&bal)[U],
                                           const int32_t *rp) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const typename SoloMem<TIER>::D code = solo_code<TIER>(level);
  bool won[U], dag[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const typename SoloMem<TIER>::D d = w[u] >= 0 ? S.dist[w[u]] : (typename SoloMem<TIER>::D)0;
    won[u] = w[u] >= 0 && d == solo_unset<TIER>();
    dag[u] = won[u] || (w[u] >= 0 && d == code);
  }
#pragma unroll
  for (int u = 0; u < U; ++u)
    if (won[u]) won[u] = solo_claim<TIER>(S, w[u], level);
  int total = 0, at[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const unsigned m = __ballot_sync(FULL, won[u]);
    at[u] = total + __popc(m & lt);
    total += __popc(m);
    bal[u] = __ballot_sync(FULL, dag[u]);
  }
  if (total) {  // one queue reservation for the warp's finds
    int base = 0;
    if (lane == 0) base = atomicAdd(&c.found[slot], total);
    base = __shfl_sync(FULL, base, 0);
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (won[u]) {
        const int q = base + at[u];
        S.queue[e + q] = (typename SoloMem<TIER>::Q)w[u];
        if constexpr (TIER != 0)
          if (q < SOLO_RING) S.ring[(level & 1) * SOLO_RING + q] = w[u];
        asm volatile("prefetch.global.L1 [%0];" ::"l"(rp + w[u]));  // the next pass reads its row bounds
      }
  }
  if constexpr (COUNT) {
    bool ov = false;
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (dag[u]) ov |= S.add(w[u], sv[u]);
    if (ov) c.over[slot] = 1;
  }
}

// One level of the forward pass: the out-edges of queue entries [b, e) (at
// level - 1). Short rows (up to 32 entries) of a run of 32 entries are walked
// as one list of edges, 32 to a window: the threads whose rows start in a
// window mark their first positions, and a visit's row is the last mark at or
// before it. Long rows go to the whole warp, the longest to the CTA.
template <int TIER, int T, bool COUNT>
__device__ __forceinline__ void solo_push(const MGraph &G, const SoloMem<TIER> &S, SoloCtl &c, int level, int b, int e,
                                          int &ph, uint64_t &maxc) {
  constexpr int U = SOLO_U;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u, le = lt | (1u << lane);
  uint8_t *own = c.own[warp];
  const int slot = ph % 3;
  solo_begin(c, ph);
  for (int cb = b + warp * 32; cb < e; cb = solo_next(c, b + T, e, ph)) {
    const int idx = cb + lane;
    int beg = 0, d = 0;
    uint64_t sv = 0ull;
    if (idx < e) {
      const int32_t v = solo_entry<TIER>(S, level - 1, b, idx);
      beg = G.rp[v];
      d = G.rp[v + 1] - beg;
      if constexpr (COUNT) sv = S.get(v);
    }
    if constexpr (COUNT) maxc = sv > maxc ? sv : maxc;
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
    int before = -1;  // index of the last row that starts before the window
    for (int i0 = 0; i0 < E; i0 += 32 * U) {
      int32_t w[U];
      int o[U];
      uint64_t svu[U];
      unsigned bal[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int s = start - (i0 + 32 * u);
        const unsigned f = __reduce_or_sync(FULL, (ds > 0 && (unsigned)s < 32u) ? 1u << s : 0u);
        const int i = i0 + 32 * u + lane;
        o[u] = i < E ? (int)own[before + __popc(f & le)] : 0;
        before += __popc(f);
        const int j = i + __shfl_sync(FULL, first, o[u]);
        w[u] = i < E ? G.col[j] : -1;
      }
      if constexpr (COUNT) {  // (the counts may still be on their way when the columns are asked for)
#pragma unroll
        for (int u = 0; u < U; ++u) svu[u] = __shfl_sync(FULL, sv, o[u]);
      }
      solo_visit<TIER, U, COUNT>(S, c, level, e, slot, w, svu, bal, G.rp);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int s = start - (i0 + 32 * u);
        if (s >= 0 && s < 32) mask |= bal[u] >> s;
        else if (s < 0 && s > -32) mask |= bal[u] << -s;
      }
    }
    if (idx < e) S.qmask[idx] = ds == 32 ? mask : mask & ((1u << ds) - 1u);
    __syncwarp();
    for (unsigned bm = __ballot_sync(FULL, d > 32); bm; bm &= bm - 1u) {
      const int k = __ffs(bm) - 1;
      const int hb = __shfl_sync(FULL, beg, k), he = hb + __shfl_sync(FULL, d, k);
      if (he - hb > SOLO_HUGE_DEG) {
        int at = 0;
        if (lane == 0) {
          at = atomicAdd(&c.nhuge[slot], 1);
          if (at < SOLO_HUGE) c.huge[at] = cb + k;
        }
        if (__shfl_sync(FULL, at, 0) < SOLO_HUGE) continue;
      }
      uint32_t *words = S.lmask + (hb >> 4);
      uint64_t svu[U];
      svu[0] = __shfl_sync(FULL, sv, k);
#pragma unroll
      for (int u = 1; u < U; ++u) svu[u] = svu[0];
      for (int j0 = hb; j0 < he; j0 += 32 * U) {
        int32_t w[U];
        unsigned bal[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int j = j0 + 32 * u + lane;
          w[u] = j < he ? G.col[j] : -1;
        }
        solo_visit<TIER, U, COUNT>(S, c, level, e, slot, w, svu, bal, G.rp);
        if (lane == 0) {
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (j0 + 32 * u < he) words[((j0 - hb) >> 5) + u] = bal[u];
        }
      }
    }
  }
  __syncthreads();
  const int nh = min(c.nhuge[slot], SOLO_HUGE);
  ++ph;
  if (nh) {
    for (int k = 0; k < nh; ++k) {
      const int32_t v = S.queue[c.huge[k]];
      const int hb = G.rp[v], he = G.rp[v + 1];
      uint64_t svu[1] = {0ull};
      if constexpr (COUNT) svu[0] = S.get(v);
      for (int j0 = hb + warp * 32; j0 < he; j0 += T) {
        int32_t w[1];
        unsigned bal[1];
        w[0] = j0 + lane < he ? G.col[j0 + lane] : -1;
        solo_visit<TIER, 1, COUNT>(S, c, level, e, slot, w, svu, bal, G.rp);
        if (lane == 0) S.lmask[(hb >> 4) + ((j0 - hb) >> 5)] = bal[0];
      }
    }
    __syncthreads();
  }
}

// Theorem 1 for the vertices of one level (queue entries [b, e)): exact sums of
// the coefficients over the shortest-path edges the forward pass kept, then
// delta and the vertex's own coefficient in place of its count. deliver(v,
// delta) gets every vertex once.
template <bool NARROW> struct SoloAcc {
  using A = typename std::conditional<NARROW, Acc3, Acc>::type;
  static __device__ __forceinline__ A zero() {
    if constexpr (NARROW) return Acc3{0u, 0u, 0u};
    else return acc_zero();
  }
  static __device__ __forceinline__ void add(A &a, uint64_t bits, int bias, unsigned &err) {
    if constexpr (NARROW) acc3_add(a, bits, bias, err);
    else acc_add(a, __longlong_as_double((long long)bits), err);
  }
  static __device__ __forceinline__ A warp_sum(A a) {
    if constexpr (NARROW) {
#pragma unroll
      for (int off = 16; off > 0; off >>= 1)
        acc3_add3(a, __shfl_xor_sync(FULL, a.l0, off), __shfl_xor_sync(FULL, a.l1, off),
                  __shfl_xor_sync(FULL, a.l2, off));
      return a;
    } else {
      return acc_warp_sum(a);
    }
  }
  static __device__ __forceinline__ double round(const A &a, int unit) {
    if constexpr (NARROW) return acc_round(acc3_widen(a, unit));
    else return acc_round(a);
  }
  static __device__ __forceinline__ void put(unsigned long long *p, const A &a) {
    if constexpr (NARROW) {
      p[0] = a.l0;
      p[1] = a.l1;
      p[2] = a.l2;
    } else {
      p[0] = a.w0;
      p[1] = a.w1;
      p[2] = a.w2;
    }
  }
  static __device__ __forceinline__ A take(const unsigned long long *p) {
    if constexpr (NARROW) return Acc3{(uint32_t)p[0], (uint32_t)p[1], (uint32_t)p[2]};
    else return Acc{p[0], p[1], p[2]};
  }
};

// Adds the successors of words first, first + step, ... of a long row.
template <int TIER, bool NARROW>
__device__ __forceinline__ void solo_long_sum(const MGraph &G, const SoloMem<TIER> &S, int hb, int he, int first,
                                              int step, int bias, typename SoloAcc<NARROW>::A &a, unsigned &err) {
  const int lane = threadIdx.x & 31;
  const uint32_t *words = S.lmask + (hb >> 4);
  const int nw = (he - hb + 31) >> 5;
  for (int q = first; q < nw; q += 4 * step) {
    uint64_t x[4];
    int32_t w[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = q + u * step;
      w[u] = (i < nw && ((words[i] >> lane) & 1u)) ? G.col[hb + 32 * i + lane] : -1;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = w[u] >= 0 ? S.get(w[u]) : 0ull;  // (a coefficient is never 0)
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (x[u]) SoloAcc<NARROW>::add(a, x[u], bias, err);
  }
}

template <int TIER, bool NARROW, class F>
__device__ __forceinline__ void solo_finish(const SoloMem<TIER> &S, int32_t v, const typename SoloAcc<NARROW>::A &a,
                                            int unit, F &deliver) {
  const uint64_t sg = S.get(v);
  const double delta = delta_rn_fp(sg, SoloAcc<NARROW>::round(a, unit));
  S.set(v, (uint64_t)__double_as_longlong(coef_of_fp(delta, sg)));
  deliver(v, delta);
}

// A thread's entry in the first run of a level of the backward pass: its loads
// are issued a level ahead (they depend on nothing that the level between
// changes), so a narrow level's chain is the successors' coefficients and the
// arithmetic alone.
struct SoloAhead {
  int32_t v = -1;
  uint32_t mask = 0u;
  int beg = 0, d = 0;
};
template <int TIER> __device__ __forceinline__ SoloAhead solo_ahead(const SoloMem<TIER> &S, int b, int e) {
  SoloAhead p;
  const int idx = b + (int)threadIdx.x;
  if (idx < e) {
    p.v = S.queue[idx];
    p.mask = S.qmask[idx];
  }
  return p;
}
template <class H>
__device__ __forceinline__ void solo_ahead_row(const MGraph &G, SoloAhead &p, bool narrow_level, H &hint) {
  if (p.v < 0) return;
  p.beg = G.rp[p.v];
  p.d = G.rp[p.v + 1] - p.beg;
  if (!narrow_level) return;  // (a wide level has other runs to hide the loads behind)
  if (p.mask) asm volatile("prefetch.global.L1 [%0];" ::"l"(G.col + p.beg));
  hint(p.v);
}

// (p: this level's first run; [nb, b): the next level to come, loaded into p)
template <int TIER, int T, bool NARROW, class F, class H>
__device__ __forceinline__ void solo_back(const MGraph &G, const SoloMem<TIER> &S, SoloCtl &c, int nb, int b, int e,
                                          int unit, int &ph, unsigned &err, F &deliver, H &hint, SoloAhead &p) {
  using A = SoloAcc<NARROW>;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int bias = 1075 - unit;
  solo_begin(c, ph);
  int32_t v = p.v;
  int beg = p.beg, d = p.d;
  uint32_t mask = p.mask;
  p = solo_ahead<TIER>(S, nb, b);
  bool first = true;
  for (int cb = b + warp * 32; cb < e; cb = solo_next(c, b + T, e, ph)) {
    if (!first) {
      const int idx = cb + lane;
      v = -1;
      beg = d = 0;
      mask = 0u;
      if (idx < e) {
        v = S.queue[idx];
        mask = S.qmask[idx];
        beg = G.rp[v];
        d = G.rp[v + 1] - beg;
      }
    }
    first = false;
    typename A::A a = A::zero();
    while (mask) {  // up to four successors in flight per thread
      int32_t w[4];
      uint64_t x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        w[u] = mask ? G.col[beg + __ffs(mask) - 1] : -1;
        mask &= mask - 1u;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] = w[u] >= 0 ? S.get(w[u]) : 0ull;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (x[u]) A::add(a, x[u], bias, err);
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
        if (__shfl_sync(FULL, slot, 0) < SOLO_HUGE) {
          if (lane == k) v = -1;  // finished after the others
          continue;
        }
      }
      typename A::A x = A::zero();
      solo_long_sum<TIER, NARROW>(G, S, hb, he, 0, 1, bias, x, err);
      x = A::warp_sum(x);
      if (lane == k) a = x;
    }
    if (v >= 0) solo_finish<TIER, NARROW>(S, v, a, unit, deliver);
    __syncwarp();
  }
  solo_ahead_row(G, p, b - nb <= T, hint);
  __syncthreads();
  const int nh = min(c.nhuge[ph % 3], SOLO_HUGE);
  ++ph;
  if (nh) {
    for (int k = 0; k < nh; ++k) {
      const int32_t v = S.queue[c.huge[k]];
      typename A::A x = A::zero();
      solo_long_sum<TIER, NARROW>(G, S, G.rp[v], G.rp[v + 1], warp, T / 32, bias, x, err);
      x = A::warp_sum(x);
      if (lane == 0) A::put(c.red[warp], x);
      __syncthreads();
      if (warp == 0) {
        typename A::A y = A::zero();
        if (lane < T / 32) y = A::take(c.red[lane]);
        y = A::warp_sum(y);
        if (lane == 0) solo_finish<TIER, NARROW>(S, v, y, unit, deliver);
      }
      __syncthreads();
    }
  }
}

// ---- extended form (counts beyond 2^64-1; sums in CSR order of the vertex) --

template <int TIER> __device__ __forceinline__ Xf solo_xf(const SoloMem<TIER> &S, int32_t v) {
  return Xf{__longlong_as_double((long long)S.get(v)), S.exp[v]};
}
template <int TIER> __device__ __forceinline__ void solo_xf_set(const SoloMem<TIER> &S, int32_t v, Xf x) {
  S.set(v, (uint64_t)__double_as_longlong(x.m));
  S.exp[v] = x.e;
}

// Adds the warp's values x (threads with ok) to acc in thread order.
__device__ __forceinline__ void solo_xf_warp(Xf &acc, bool ok, Xf x) {
  for (unsigned b = __ballot_sync(FULL, ok); b; b &= b - 1u) {
    const int k = __ffs(b) - 1;
    acc = xf_add(acc, Xf{__shfl_sync(FULL, x.m, k), __shfl_sync(FULL, x.e, k)});
  }
}

// Extended counts of the vertices of level l (queue entries [b, e)), pulled
// over the in-neighbours in CSR order: a vertex per thread, rows above 32
// entries by the whole warp.
template <int TIER, int T>
__device__ __forceinline__ void solo_xf_level(const MGraph &G, const SoloMem<TIER> &S, int l, int b, int e) {
  const typename SoloMem<TIER>::D prev = solo_code<TIER>(l - 1);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int cb = b + warp * 32; cb < e; cb += T) {
    const int idx = cb + lane;
    int32_t v = -1;
    int beg = 0, d = 0;
    if (idx < e) {
      v = S.queue[idx];
      beg = G.rp_in[v];
      d = G.rp_in[v + 1] - beg;
    }
    Xf acc{0.0, 0};
    const int ds = d <= 32 ? d : 0;
    for (int j = 0; j < ds; j += 4) {
      int32_t u[4];
      Xf x[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) u[q] = j + q < ds ? G.col_in[beg + j + q] : -1;
#pragma unroll
      for (int q = 0; q < 4; ++q) x[q] = (u[q] >= 0 && S.dist[u[q]] == prev) ? solo_xf<TIER>(S, u[q]) : Xf{0.0, 0};
#pragma unroll
      for (int q = 0; q < 4; ++q) acc = xf_add(acc, x[q]);
    }
    __syncwarp();
    for (unsigned bm = __ballot_sync(FULL, d > 32); bm; bm &= bm - 1u) {
      const int k = __ffs(bm) - 1;
      const int hb = __shfl_sync(FULL, beg, k), he = hb + __shfl_sync(FULL, d, k);
      Xf tot{0.0, 0};
      for (int j0 = hb; j0 < he; j0 += 32) {
        bool ok = false;
        Xf x{0.0, 0};
        if (j0 + lane < he) {
          const int32_t u = G.col_in[j0 + lane];
          ok = S.dist[u] == prev;
          if (ok) x = solo_xf<TIER>(S, u);
        }
        solo_xf_warp(tot, ok, x);
      }
      if (lane == k) acc = tot;
    }
    if (v >= 0) solo_xf_set<TIER>(S, v, acc);
  }
}

// The same pull fused with the push from the same vertices (an undirected
// graph's rows are both): counts of level l = level - 1 from the neighbours a
// level below, the next level from those not reached yet, one pass and one
// barrier a level. Rows up to 32 entries by a thread in CSR order, four at a
// time; longer ones by the warp.
template <int TIER, int T>
__device__ __forceinline__ void solo_xf_push(const MGraph &G, const SoloMem<TIER> &S, SoloCtl &c, int level, int b,
                                             int e, int &ph) {
  const typename SoloMem<TIER>::D prev = solo_code<TIER>(level - 2 + (level < 2));
  const bool pull = level >= 2;  // the source's count stands
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int slot = ph % 3;
  const uint64_t none[4] = {0ull, 0ull, 0ull, 0ull};
  solo_begin(c, ph);
  for (int cb = b + warp * 32; cb < e; cb += T) {
    const int idx = cb + lane;
    int32_t v = -1;
    int beg = 0, d = 0;
    if (idx < e) {
      v = solo_entry<TIER>(S, level - 1, b, idx);
      beg = G.rp[v];
      d = G.rp[v + 1] - beg;
    }
    Xf acc{0.0, 0};
    uint32_t mask = 0u;
    const int ds = d <= 32 ? d : 0, most = __reduce_max_sync(FULL, ds);
    for (int j = 0; j < most; j += 4) {
      int32_t w[4];
      Xf x[4];
      unsigned bal[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) w[u] = j + u < ds ? G.col[beg + j + u] : -1;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        x[u] = (pull && w[u] >= 0 && S.dist[w[u]] == prev) ? solo_xf<TIER>(S, w[u]) : Xf{0.0, 0};
      solo_visit<TIER, 4, false>(S, c, level, e, slot, w, none, bal, G.rp);
#pragma unroll
      for (int u = 0; u < 4; ++u) mask |= ((bal[u] >> lane) & 1u) << ((j + u) & 31);
#pragma unroll
      for (int q = 0; q < 4; ++q) acc = xf_add(acc, x[q]);
    }
    __syncwarp();
    for (unsigned bm = __ballot_sync(FULL, d > 32); bm; bm &= bm - 1u) {
      const int k = __ffs(bm) - 1;
      const int hb = __shfl_sync(FULL, beg, k), he = hb + __shfl_sync(FULL, d, k);
      uint32_t *words = S.lmask + (hb >> 4);
      Xf tot{0.0, 0};
      for (int j0 = hb; j0 < he; j0 += 32) {
        int32_t w[1];
        const uint64_t zero[1] = {0ull};
        unsigned bal[1];
        w[0] = j0 + lane < he ? G.col[j0 + lane] : -1;
        const bool ok = pull && w[0] >= 0 && S.dist[w[0]] == prev;
        const Xf x = ok ? solo_xf<TIER>(S, w[0]) : Xf{0.0, 0};
        solo_visit<TIER, 1, false>(S, c, level, e, slot, w, zero, bal, G.rp);
        if (lane == 0) words[(j0 - hb) >> 5] = bal[0];
        solo_xf_warp(tot, ok, x);
      }
      if (lane == k) acc = tot;
    }
    if (v >= 0) {
      if (pull) solo_xf_set<TIER>(S, v, acc);
      S.qmask[idx] = mask;
    }
  }
  __syncthreads();
  ++ph;
}

// Theorem 1 for one level in the extended form (successors in CSR order).
template <int TIER, int T, class F, class H>
__device__ __forceinline__ void solo_xf_back(const MGraph &G, const SoloMem<TIER> &S, int nb, int b, int e, F &deliver,
                                             H &hint, SoloAhead &p) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int32_t v = p.v;
  int beg = p.beg, d = p.d;
  uint32_t mask = p.mask;
  p = solo_ahead<TIER>(S, nb, b);
  for (int cb = b + warp * 32; cb < e; cb += T) {
    if (cb >= b + T) {
      const int idx = cb + lane;
      v = -1;
      beg = d = 0;
      mask = 0u;
      if (idx < e) {
        v = S.queue[idx];
        mask = S.qmask[idx];
        beg = G.rp[v];
        d = G.rp[v + 1] - beg;
      }
    }
    Xf acc{0.0, 0};
    while (mask) {
      int32_t w[2];
      Xf x[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        w[u] = mask ? G.col[beg + __ffs(mask) - 1] : -1;
        mask &= mask - 1u;
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) x[u] = w[u] >= 0 ? solo_xf<TIER>(S, w[u]) : Xf{0.0, 0};
      acc = xf_add(xf_add(acc, x[0]), x[1]);
    }
    __syncwarp();
    for (unsigned bm = __ballot_sync(FULL, d > 32); bm; bm &= bm - 1u) {
      const int k = __ffs(bm) - 1;
      const int hb = __shfl_sync(FULL, beg, k), he = hb + __shfl_sync(FULL, d, k);
      const uint32_t *words = S.lmask + (hb >> 4);
      Xf tot{0.0, 0};
      for (int q = 0; hb + 32 * q < he; ++q) {
        const bool ok = (words[q] >> lane) & 1u;
        solo_xf_warp(tot, ok, ok ? solo_xf<TIER>(S, G.col[hb + 32 * q + lane]) : Xf{0.0, 0});
      }
      if (lane == k) acc = tot;
    }
    if (v >= 0) {
      const Xf sg = solo_xf<TIER>(S, v);
      const double delta = xf_mul_to_double(sg, acc);
      solo_xf_set<TIER>(S, v, xf_div(__dadd_rn(1.0, delta), sg));
      deliver(v, delta);
    }
  }
  solo_ahead_row(G, p, b - nb <= T, hint);
}

// The shortest-path edges of queue entries [0, e), from their bits. (A pass of its
// own: counted where the bits are made, the counter's register cost the passes
// 3-6 % on ER n = 2000.)
template <class Q, int T>
__device__ __forceinline__ void solo_count_edges(const int32_t *rp, const Q *queue, const uint32_t *qmask,
                                              const uint32_t *lmask, int e, bool long_rows, unsigned *total) {
  unsigned edges = 0u;
#pragma unroll 4
  for (int i = (int)threadIdx.x; i < e; i += T) edges += (unsigned)__popc(qmask[i]);
  if (long_rows)
    for (int i = (int)threadIdx.x; i < e; i += T) {
      const int hb = rp[queue[i]], d = rp[queue[i] + 1] - hb;
      if (d > 32)
        for (int q = 0; 32 * q < d; ++q) edges += (unsigned)__popc(lmask[(hb >> 4) + q]);
    }
  edges = __reduce_add_sync(FULL, edges);
  if ((threadIdx.x & 31) == 0 && edges) atomicAdd(total, edges);
}

// Forward pass of source s: distance codes, counts, level offsets and edge
// bits; with dest >= 0 it stops once dest's level is settled. Returns the
// deepest level; *ext: the counts are in the extended form (a count of the
// settled levels exceeded 2^64-1); *maxc: the largest count of the levels
// above the deepest and of the deepest too unless dest stopped the search
// (when not extended).
// Counts below 2^53 are exact in both forms, so a sample that overflows at
// level L is converted, not recomputed, up to its first level with a count of
// 2^53 or more, and goes on in the extended form from there.
template <int TIER, int T>
__device__ int solo_forward(const MGraph &G, int32_t s, int32_t dest, const SoloMem<TIER> &S, SoloCtl &c, int &ph,
                            bool *ext, uint64_t *maxc) {
  const int tid = threadIdx.x;
  if constexpr (TIER == 2) {
    for (int32_t v = tid; v < G.n; v += T) S.dist[v] = -1;
  } else {
    uint4 *d = reinterpret_cast<uint4 *>(S.dist);
    const int words = (int)(((size_t)G.n * 2 + 15) / 16);
    for (int i = tid; i < words; i += T) d[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
  }
  if constexpr (TIER == 0) {
    for (int32_t v = tid; v < G.n; v += T) S.lo[v] = S.hi[v] = 0u;
  } else {
    for (int32_t v = tid; v < G.n; v += T) S.val[v] = 0ull;
  }
  __syncthreads();
  if (tid == 0) {
    S.dist[s] = 0;
    S.set(s, 1ull);
    S.queue[0] = (typename SoloMem<TIER>::Q)s;
    if constexpr (TIER != 0) S.ring[0] = s;
    c.near[0] = 0;
    c.near[1] = 1;
    c.l53 = 0x7FFFFFFF;
    c.maxc = 1ull;
    c.edges += c.last_edges;
    c.last_edges = 0u;
  }
  __syncthreads();
  int L = 0, b = 0, e = 1;
  bool xf = false;
  const bool fused = G.rp_in == G.rp;  // (extended form) level L's counts come with the push from it
  uint64_t mymax = 1ull;
  bool pushed = true;  // the last level's edges have been looked at
  for (;;) {
    const int slot = ph % 3;
    if (xf && fused) {
      solo_xf_push<TIER, T>(G, S, c, L + 1, b, e, ph);
    } else if (xf) {
      uint64_t none = 0ull;
      solo_push<TIER, T, false>(G, S, c, L + 1, b, e, ph, none);
    } else {
      uint64_t lmax = 0ull;
      solo_push<TIER, T, true>(G, S, c, L + 1, b, e, ph, lmax);
      if (lmax >= (1ull << 53)) atomicMin(&c.l53, L);
      mymax = lmax > mymax ? lmax : mymax;
    }
    // (a pass's counters stand until the pass after the next one begins)
    const int nt = e + c.found[slot];
    if (nt == e) break;  // no vertex at distance L + 1
    if (xf && !fused) {
      solo_xf_level<TIER, T>(G, S, L + 1, e, nt);
      __syncthreads();
    }
    if (tid == 0) {
      if (L + 2 < SOLO_NEAR) c.near[L + 2] = nt;
      else S.far[L + 2] = nt;
    }
    ++L;
    b = e;
    e = nt;
    if (!xf && c.over[slot]) {
      // to the extended form: convert the exact levels, pull the rest
      __syncthreads();
      const int l53 = min(c.l53, L);
      const int conv = solo_lo<TIER>(S, c, l53);
      for (int i = tid; i < conv; i += T) {
        const int32_t v = S.queue[i];
        solo_xf_set<TIER>(S, v, xf_of_u64(S.get(v)));
      }
      __syncthreads();
      for (int l = l53; l <= L; ++l) {
        solo_xf_level<TIER, T>(G, S, l, solo_lo<TIER>(S, c, l), solo_lo<TIER>(S, c, l + 1));
        __syncthreads();
      }
      xf = true;
    }
    if (dest >= 0 && __syncthreads_or(S.dist[dest] != solo_unset<TIER>())) {  // dest settled at level L
      if (xf && fused) solo_xf_level<TIER, T>(G, S, L, b, e);
      pushed = false;
      break;
    }
  }
  if (!xf) {
    for (int off = 16; off > 0; off >>= 1) {
      const uint64_t o = __shfl_xor_sync(FULL, mymax, off);
      mymax = o > mymax ? o : mymax;
    }
    if ((tid & 31) == 0 && mymax > 1ull) atomicMax(&c.maxc, (unsigned long long)mymax);
  }
  if (G.stats) {
    solo_count_edges<typename SoloMem<TIER>::Q, T>(G.rp, S.queue, S.qmask, S.lmask, pushed ? e : b, G.long_rows != 0,
                                                   &c.last_edges);
    if (tid == 0) c.reached += (unsigned long long)(e - 1);
  }
  __syncthreads();
  *ext = xf;
  *maxc = c.maxc;
  return L;
}

struct SoloNoHint {
  __device__ void operator()(int32_t) const {}
};

// Theorem 1 for levels L..1 after solo_forward; deliver(v, delta) is called by
// one thread for every vertex at distance >= 1, hint(v) at least a level's
// barrier earlier for some of them (to prefetch what deliver reads).
template <int TIER, int T, class F, class H = SoloNoHint>
__device__ __forceinline__ void solo_backward(const MGraph &G, int L, bool ext, uint64_t maxc, const SoloMem<TIER> &S,
                                              SoloCtl &c, int &ph, unsigned &err, F deliver, H hint = H{}) {
  if (L < 1) return;
  int b = solo_lo<TIER>(S, c, L), e = solo_lo<TIER>(S, c, L + 1);
  SoloAhead p = solo_ahead<TIER>(S, b, e);
  solo_ahead_row(G, p, e - b <= T, hint);
  // ceil(log2) of the largest count and of n
  const int unit = 52 + (maxc <= 1ull ? 0 : 64 - __clzll((long long)(maxc - 1ull)));
  const int nlog = G.n <= 1 ? 0 : 32 - __clz(G.n - 1);
  const bool narrow = unit + nlog + 1 <= 96;
  for (int l = L; l >= 1; --l) {
    const int nb = l > 1 ? solo_lo<TIER>(S, c, l - 1) : b;  // (level 0, the source, has no part in it)
    if (ext) {
      solo_xf_back<TIER, T>(G, S, nb, b, e, deliver, hint, p);
      __syncthreads();
    } else if (narrow) {
      solo_back<TIER, T, true>(G, S, c, nb, b, e, unit, ph, err, deliver, hint, p);
    } else {
      solo_back<TIER, T, false>(G, S, c, nb, b, e, unit, ph, err, deliver, hint, p);
    }
    e = b;
    b = nb;
  }
}

}  // namespace bcg
