// bc_batch.cu -- lane-batched Brandes step: 64 sampled sources share one
// level-synchronous traversal of the CSR.
//
// Layout (n vertices, 64 lanes, lane t = one sampled source):
//   lm[l][v]    u64  bit t set iff d(s_t, v) = l            (level masks)
//   visited[v]  u64  OR of lm[0..l][v]
//   sigma[v][t] u64  sigma_{s_t v}. Lane-minor rows of 512 B, so one warp reads a
//                    neighbour's 32 lanes with one request.
//   coef[v][t]  coef = (1+delta)/sigma as a 96-bit fixed-point number (12 B),
//               written once v's level in lane t is done; where counts are too
//               large for that, its double bits in the slot of sigma[v][t].
//
// Forward level l (Sec. 3 step 1, predecessor sets of Def. 3): every vertex v
// with lanes still unvisited pulls from its CSR neighbours w:
//   new(v)       = OR_w lm[l-1][w] & ~visited[v]
//   sigma[v][t]  = sum over w with t in lm[l-1][w] of sigma[w][t]   (t in new)
// Backward level l (Sec. 3 step 2, Theorem 1): every vertex v with lanes at
// level l pulls coefficients from its successors (neighbours one level deeper
// in the same lane), summing them exactly:
//   delta[v][t] = RN(sigma[v][t] * RN(sum_w coef[w][t]))
//   coef[v][t]  = RN(RN(1 + delta[v][t]) / sigma[v][t]).
// Vertices of degree > HEAVY are split into SEG-long neighbour segments, each
// handled by one warp; partial results are combined exactly afterwards.
//
// R-MAT s20, uniform k = 1024 (16 batches): 56.3 ms with neighbours walked by
// warp shuffles and doubles converted at every add; 50.6 with entry lists and
// work lists, 46.8 with vertices above degree 64 (before: 256) split, 41.6 with
// coefficients kept in 96 bits, 39.5 with listed heavy segments. s16, Bader 1500
// draws: 21.0 -> 14.0.
#include <algorithm>
#include <cstdlib>
#include <memory>

#include "bc_internal.h"

namespace bcg {

constexpr int HEAVY_DEFAULT = 64;    // vertices above this degree are split into segments
constexpr int SEG_DEFAULT = 256;     // neighbours per heavy segment
constexpr int UNR = 3;               // neighbours gathered per unrolled step of a top-down level's pull
constexpr int FWD_THREADS = 256;
// Resident blocks per SM of the backward kernels (48 registers a thread); the
// forward kernels take four (64 registers).
constexpr int BWD_MIN_BLOCKS = 5;

__device__ __forceinline__ uint64_t warp_or64(uint64_t x) {
  const unsigned lo = __reduce_or_sync(FULL, (unsigned)x);
  const unsigned hi = __reduce_or_sync(FULL, (unsigned)(x >> 32));
  return ((uint64_t)hi << 32) | lo;
}

__device__ __forceinline__ uint64_t warp_max64(uint64_t x) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const uint64_t o = __shfl_xor_sync(FULL, x, off);
    x = o > x ? o : x;
  }
  return x;
}

__device__ __forceinline__ unsigned long long warp_sum64(unsigned long long x) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(FULL, x, off);
  return x;
}

__device__ __forceinline__ void block_or_to(uint64_t x, uint64_t *dst) {
  __shared__ unsigned long long s_or;
  if (threadIdx.x == 0) s_or = 0ull;
  __syncthreads();
  if ((threadIdx.x & 31) == 0 && x) atomicOr(&s_or, (unsigned long long)x);
  __syncthreads();
  if (threadIdx.x == 0 && s_or) atomicOr((unsigned long long *)dst, s_or);
}


// Dynamic work distribution: a warp takes `step` consecutive items per atomic
// (several light vertices; one heavy segment or heavy vertex, whose work is large).
__device__ __forceinline__ int grab(unsigned *wq, int step) {
  int base = 0;
  if ((threadIdx.x & 31) == 0) base = (int)atomicAdd(wq, (unsigned)step);
  return __shfl_sync(FULL, base, 0);
}

// Takes up to UNR neighbours with a non-empty lane mask from the warp ballot
// `bal` (lowest CSR positions first); every lane receives (mask, vertex).
__device__ __forceinline__ void take(unsigned &bal, uint64_t m, int32_t w, uint64_t (&mk)[UNR],
                                     int32_t (&wk)[UNR]) {
#pragma unroll
  for (int k = 0; k < UNR; ++k) {
    const int src = bal ? (__ffs(bal) - 1) : 0;
    const uint64_t mm = __shfl_sync(FULL, m, src);
    wk[k] = __shfl_sync(FULL, w, src);
    mk[k] = bal ? mm : 0ull;
    bal &= bal - 1u;
  }
}

// ------------------------------------------------------------------ init --
__global__ void k_batch_init(int count, const int32_t *__restrict__ sources,
                             uint64_t *__restrict__ lm0, uint64_t *__restrict__ visited,
                             uint64_t *__restrict__ sigma, uint64_t *__restrict__ active0,
                             uint64_t *__restrict__ enable, int32_t *__restrict__ pair_d,
                             uint64_t *__restrict__ pair_sig, const int32_t *__restrict__ rp,
                             int32_t *__restrict__ list0, unsigned *__restrict__ vcnt0,
                             unsigned long long *__restrict__ vedges0) {
  const int t = threadIdx.x;
  if (t < 64) {
    pair_d[t] = -1;
    pair_sig[t] = 0ull;
  }
  if (t == 0) {
    enable[0] = (count >= 64) ? ~0ull : ((1ull << count) - 1ull);
    enable[2] = 1ull;  // largest sigma of the batch (sources have sigma 1)
    enable[3] = 0ull;  // lanes whose path counts exceeded 2^64-1
  }
  __syncthreads();
  if (t < count) {
    const int32_t s = sources[t];
    const uint64_t bit = 1ull << t;
    const unsigned long long old = atomicOr((unsigned long long *)&lm0[s], (unsigned long long)bit);
    atomicOr((unsigned long long *)&visited[s], (unsigned long long)bit);
    sigma[(size_t)s * 64 + t] = 1ull;
    atomicOr((unsigned long long *)active0, (unsigned long long)bit);
    if (old == 0ull) {  // first lane with this source: it joins the level-0 list
      list0[atomicAdd(vcnt0, 1u)] = s;
      atomicAdd(vedges0, (unsigned long long)(rp[s + 1] - rp[s]));
    }
  }
}

// Appends the vertices of this warp flagged `first` to a level list (one
// atomic per warp) and adds their degrees to the level's edge count.
__device__ __forceinline__ void list_append(bool first, int32_t v, int deg, int32_t *__restrict__ list,
                                            unsigned *__restrict__ vcnt, unsigned long long *__restrict__ vedges) {
  const int lane = threadIdx.x & 31;
  const unsigned fb = __ballot_sync(FULL, first);
  if (!fb) return;
  unsigned pos0 = 0u;
  if (lane == 0) pos0 = atomicAdd(vcnt, (unsigned)__popc(fb));
  pos0 = __shfl_sync(FULL, pos0, 0);
  if (first) list[pos0 + __popc(fb & ((1u << lane) - 1u))] = v;
  unsigned long long ds = first ? (unsigned long long)deg : 0ull;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) ds += __shfl_xor_sync(FULL, ds, off);
  if (lane == 0) atomicAdd(vedges, ds);
}

// Zero sigma rows of heavy vertices (their lanes are filled with atomics).
__global__ void k_zero_heavy_rows(int nh, const int32_t *__restrict__ heavy, uint64_t *__restrict__ sigma) {
  const int h = blockIdx.x;
  if (h < nh && threadIdx.x < 64) sigma[(size_t)heavy[h] * 64 + threadIdx.x] = 0ull;
}

// Level 1 directly: the vertices at distance 1 from s_t are its neighbours, each
// with exactly one shortest path (sigma = 1). One block per lane.
__global__ void k_fwd_level1(int count, const int32_t *__restrict__ sources, const int32_t *__restrict__ rp,
                             const int32_t *__restrict__ col, uint64_t *__restrict__ lm1,
                             uint64_t *__restrict__ visited, uint64_t *__restrict__ sigma,
                             uint64_t *__restrict__ active1, unsigned long long *__restrict__ cnt,
                             int32_t *__restrict__ list1, unsigned *__restrict__ vcnt1,
                             unsigned long long *__restrict__ vedges1) {
  const int t = blockIdx.x;
  if (t >= count) return;
  const int32_t s = sources[t];
  const uint64_t bit = 1ull << t;
  const int beg = rp[s], end = rp[s + 1];
  for (int jb = beg; jb < end; jb += blockDim.x) {  // block-uniform trip count
    const int j = jb + (int)threadIdx.x;
    bool first = false;
    int32_t v = 0;
    int dv = 0;
    if (j < end) {
      v = col[j];
      sigma[(size_t)v * 64 + t] = 1ull;
      first = atomicOr((unsigned long long *)&lm1[v], (unsigned long long)bit) == 0ull;
      atomicOr((unsigned long long *)&visited[v], (unsigned long long)bit);
      if (first) dv = rp[v + 1] - rp[v];
    }
    list_append(first, v, dv, list1, vcnt1, vedges1);
  }
  if (threadIdx.x == 0 && end > beg) {
    atomicOr((unsigned long long *)active1, (unsigned long long)bit);
    atomicAdd(cnt, (unsigned long long)(end - beg));      // DAG edges s -> v
    atomicAdd(cnt + 1, (unsigned long long)(end - beg));  // reached at distance 1
  }
}

// ------------------------------------------------ neighbour entry lists --
// Both passes reduce, for a vertex and its lanes at a level, over the
// neighbours that share a lane with it (predecessors forward, successors
// backward). A warp first lists those neighbours, (mask, vertex) entries of 16
// bytes in shared memory, then sums their rows. Every kernel here is bound by
// instruction issue (62-76 % on R-MAT s20), so what counts is the instructions
// per entry: a broadcast read of the entry, a bit test, an address, a load and
// the add. Walking neighbours by warp shuffles with two lanes per thread took
// 30 (forward) to 60; from the list it is 8 to 20, with one lane per thread
// while at most 32 lanes are in play and several entries per step below 17.
//
// Rows of a whole run of vertices are listed as one flattened list of edges, 32
// to a window: the threads whose rows start in a window mark their first
// positions and a visit's row is the last mark at or before it, so short rows
// (7 of 32 threads on ER degree 7) cost no idle threads.
constexpr int ECAP_F = 256;  // entries per warp, forward
constexpr int ECAP_B = 128;  // ... and backward, where a ring shares the shared memory

// Lists the entries of the rows held by the warp's threads (thread k: entries
// [beg, beg + d) of col, wanted lanes `want`; d = 0: none; the sum of d at most
// the list's capacity). Returns the number of entries; a row's are contiguous
// from `first`. tri counts (edge, lane) pairs.
__device__ __forceinline__ int list_rows(const int32_t *__restrict__ col, const uint64_t *__restrict__ lm, int beg,
                                         int d, uint64_t want, uint4 *ent, uint8_t *own, int &first,
                                         unsigned long long &tri) {
  constexpr int U = 4;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u, le = lt | (1u << lane);
  int incl = d;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int y = __shfl_up_sync(FULL, incl, off);
    if (lane >= off) incl += y;
  }
  const int E = __shfl_sync(FULL, incl, 31), start = incl - d, shift = beg - start;
  const unsigned rows = __ballot_sync(FULL, d > 0);
  if (d > 0) own[__popc(rows & lt)] = (uint8_t)lane;
  __syncwarp();
  int before = -1, total = 0;
  first = 0;
  for (int i0 = 0; i0 < E; i0 += 32 * U) {
    int32_t w[U];
    uint64_t m[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int s = start - (i0 + 32 * u);
      const unsigned f = __reduce_or_sync(FULL, (d > 0 && (unsigned)s < 32u) ? 1u << s : 0u);
      const int i = i0 + 32 * u + lane;
      const int o = i < E ? (int)own[before + __popc(f & le)] : 0;
      before += __popc(f);
      const int j = i + __shfl_sync(FULL, shift, o);
      m[u] = __shfl_sync(FULL, want, o);
      w[u] = i < E ? col[j] : -1;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) m[u] = w[u] >= 0 ? lm[w[u]] & m[u] : 0ull;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const unsigned bal = __ballot_sync(FULL, m[u] != 0ull);
      const int s = start - (i0 + 32 * u);
      if (d > 0 && (unsigned)s < 32u) first = total + __popc(bal & ((1u << s) - 1u));
      if (m[u]) ent[total + __popc(bal & lt)] = make_uint4((uint32_t)m[u], (uint32_t)(m[u] >> 32), (uint32_t)w[u], 0u);
      tri += (unsigned long long)__popcll((long long)m[u]);
      total += __popc(bal);
    }
  }
  __syncwarp();
  return total;
}

// The same for one row's entries [beg, end) (at most the list's capacity).
__device__ __forceinline__ int list_row(const int32_t *__restrict__ col, const uint64_t *__restrict__ lm, int beg,
                                        int end, uint64_t want, uint4 *ent, unsigned long long &tri) {
  constexpr int U = 4;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  int total = 0;
  for (int j0 = beg; j0 < end; j0 += 32 * U) {
    int32_t w[U];
    uint64_t m[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int j = j0 + 32 * u + lane;
      w[u] = j < end ? col[j] : -1;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) m[u] = w[u] >= 0 ? lm[w[u]] & want : 0ull;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const unsigned bal = __ballot_sync(FULL, m[u] != 0ull);
      if (m[u]) ent[total + __popc(bal & lt)] = make_uint4((uint32_t)m[u], (uint32_t)(m[u] >> 32), (uint32_t)w[u], 0u);
      tri += (unsigned long long)__popcll((long long)m[u]);
      total += __popc(bal);
    }
  }
  __syncwarp();
  return total;
}

// OR of the masks of entries [f, e).
__device__ __forceinline__ uint64_t entries_or(const uint4 *ent, int f, int e) {
  uint64_t m = 0ull;
  for (int i = f + (int)(threadIdx.x & 31); i < e; i += 32) {
    const uint4 x = ent[i];
    m |= ((uint64_t)x.y << 32) | x.x;
  }
  return warp_or64(m);
}

// Lanes of a vertex packed over the warp: groups of 2^glog threads each take
// another entry per step; thread i of a group owns the i-th lane in increasing
// order (p0; -1: none), and the (i+32)-th when more than 32 are set (p1).
struct Packed {
  int glog;
  int p0, p1;
  bool two;
};

__device__ __forceinline__ Packed pack_lanes(uint64_t lanes, int8_t *tab) {
  const int lane = threadIdx.x & 31;
  const unsigned lo = (unsigned)lanes, hi = (unsigned)(lanes >> 32);
  const unsigned lt = (1u << lane) - 1u;
  const int nlo = __popc(lo), L = nlo + __popc(hi);
  if ((lo >> lane) & 1u) tab[__popc(lo & lt)] = (int8_t)lane;
  if ((hi >> lane) & 1u) tab[nlo + __popc(hi & lt)] = (int8_t)(lane + 32);
  __syncwarp();
  Packed pk;
  pk.glog = L > 16 ? 5 : (L > 8 ? 4 : (L > 4 ? 3 : 2));
  const int slot = lane & ((1 << pk.glog) - 1);
  pk.p0 = slot < L ? (int)tab[slot] : -1;
  pk.p1 = (pk.glog == 5 && lane + 32 < L) ? (int)tab[lane + 32] : -1;
  pk.two = L > 32;
  __syncwarp();
  return pk;
}

// acc0 / acc1 take the row values of entries [f, e) in the thread's lanes p0 /
// p1, four steps in flight (only the last four check the list's end). R reads
// a row's lane: R::V, R::zero(), R(w, lane).
template <class R, class F0, class F1>
__device__ __forceinline__ void entries_sum(const uint4 *ent, int f, int e, const Packed &pk, const R &rows, F0 acc0,
                                            F1 acc1) {
  const int lane = threadIdx.x & 31;
  const int NG = 32 >> pk.glog, g = lane >> pk.glog;
  const bool h0 = pk.p0 >= 32;
  const uint32_t b0 = pk.p0 >= 0 ? 1u << (pk.p0 & 31) : 0u;
  const int t0 = pk.p0 < 0 ? 0 : pk.p0;
  if (!pk.two) {
    int r = f;
    for (; r + 4 * NG <= e; r += 4 * NG) {
      typename R::V x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint4 n = ent[r + u * NG + g];
        x[u] = ((h0 ? n.y : n.x) & b0) ? rows(n.z, t0) : R::zero();
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) acc0(x[u]);
    }
    if (r < e) {
      typename R::V x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int q = r + u * NG + g;
        const uint4 n = ent[q < e ? q : f];
        x[u] = (q < e && ((h0 ? n.y : n.x) & b0)) ? rows(n.z, t0) : R::zero();
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) acc0(x[u]);
    }
  } else {  // (the 33rd lane and later: always 32 or above)
    const uint32_t b1 = pk.p1 >= 0 ? 1u << (pk.p1 & 31) : 0u;
    const int t1 = pk.p1 < 0 ? 0 : pk.p1;
    int i = f;
    for (; i + 2 <= e; i += 2) {
      typename R::V x[2], y[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const uint4 n = ent[i + u];
        x[u] = ((h0 ? n.y : n.x) & b0) ? rows(n.z, t0) : R::zero();
        y[u] = (n.y & b1) ? rows(n.z, t1) : R::zero();
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        acc0(x[u]);
        acc1(y[u]);
      }
    }
    if (i < e) {
      const uint4 n = ent[i];
      acc0(((h0 ? n.y : n.x) & b0) ? rows(n.z, t0) : R::zero());
      acc1((n.y & b1) ? rows(n.z, t1) : R::zero());
    }
  }
}

// Rows of 64 words of 64 bits.
struct WordRows {
  using V = uint64_t;
  const uint64_t *__restrict__ p;
  static __device__ __forceinline__ V zero() { return 0ull; }
  __device__ __forceinline__ V operator()(uint32_t w, int t) const { return p[(size_t)w * 64 + t]; }
};

// --------------------------------------------------------------- forward --
// Exact 64-bit counts. CHECK: note carries out of 64 bits (not needed while
// the largest count so far times n stays below 2^64).
template <bool CHECK> struct CountAcc {
  uint64_t s = 0ull;
  bool ov = false;
  __device__ __forceinline__ void add(uint64_t x) {
    s += x;
    if constexpr (CHECK) ov |= s < x;
  }
  __device__ __forceinline__ void group_sum(int glog) {  // over the groups: threads with the same slot
    for (int off = 1 << glog; off < 32; off <<= 1) {
      const uint64_t o = __shfl_xor_sync(FULL, s, off);
      add(o);
    }
  }
};

// Sums of the entries [f, e) in the packed lanes; the bits of lanes whose count
// left 64 bits go to ovf.
template <bool CHECK>
__device__ __forceinline__ void count_entries(const uint4 *ent, int f, int e, const Packed &pk,
                                              const uint64_t *__restrict__ sigma, uint64_t &s0, uint64_t &s1,
                                              uint64_t &ovf) {
  CountAcc<CHECK> a, b;
  entries_sum(ent, f, e, pk, WordRows{sigma}, [&](uint64_t x) { a.add(x); }, [&](uint64_t x) { b.add(x); });
  a.group_sum(pk.glog);
  a.add(s0);
  b.add(s1);
  s0 = a.s;
  s1 = b.s;
  if constexpr (CHECK) {
    if (a.ov && pk.p0 >= 0) ovf |= 1ull << pk.p0;
    if (b.ov && pk.p1 >= 0) ovf |= 1ull << pk.p1;
  }
}

__device__ __forceinline__ bool counts_fit(uint64_t largest, int32_t n) {
  return __umul64hi(largest, (uint64_t)n) == 0ull;
}

// Light vertices of a level (degree at most heavy_deg): the list `list_in`
// (*cnt_in of them) holds the ones with lanes still to reach; a warp takes gsz
// at a time. The vertices that stay unfinished go to list_out, the ones that
// got lanes at this level to the level's list. The next level's masks must be
// clear on entry.
__global__ void __launch_bounds__(FWD_THREADS, 4)
k_fwd_light(int32_t n, const int32_t *__restrict__ list_in, const unsigned *__restrict__ cnt_in,
            int32_t *__restrict__ list_out, unsigned *__restrict__ cnt_out, const int32_t *__restrict__ rp,
            const int32_t *__restrict__ col, const uint64_t *__restrict__ lm_prev, uint64_t *__restrict__ lm_cur,
            uint64_t *__restrict__ visited, uint64_t *__restrict__ sigma, const uint64_t *__restrict__ active_prev,
            uint64_t *__restrict__ enable, uint64_t *__restrict__ active_cur, unsigned long long *__restrict__ cnt,
            unsigned *__restrict__ wq, int32_t *__restrict__ list_next, unsigned *__restrict__ vcnt_next,
            unsigned long long *__restrict__ vedges_next, int gsz) {
  __shared__ uint4 ents[FWD_THREADS / 32][ECAP_F];
  __shared__ int8_t tabs[FWD_THREADS / 32][64];
  __shared__ uint8_t owns[FWD_THREADS / 32][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  uint4 *ent = ents[wid];
  int8_t *tab = tabs[wid];
  const uint64_t act = *active_prev & *enable;
  const int total = (int)*cnt_in;
  const bool fit = counts_fit(enable[2], n);  // (grows during the level: still a bound for the level before)
  uint64_t any_new = 0ull, smax = 0ull, ovf = 0ull;
  unsigned long long tri = 0ull, rch = 0ull;
  if (act)
    for (int base = grab(wq, gsz); base < total; base = grab(wq, gsz)) {
      int32_t v = -1;
      int hb = 0, d = 0;
      uint64_t vis = 0ull, pend = 0ull, mine = 0ull;
      if (lane < gsz && base + lane < total) {
        v = list_in[base + lane];
        hb = rp[v];
        d = rp[v + 1] - hb;
        vis = visited[v];
        pend = ~vis & act;
      }
      // one vertex's new lanes nm with counts s0 / s1 in the packed lanes
      auto store = [&](int k, int32_t u, uint64_t nm, const Packed &pk, uint64_t s0, uint64_t s1) {
        uint64_t *row = sigma + (size_t)u * 64;
        if ((lane >> pk.glog) == 0 && pk.p0 >= 0 && ((nm >> pk.p0) & 1ull)) {
          row[pk.p0] = s0;
          smax = s0 > smax ? s0 : smax;
        }
        if (pk.p1 >= 0 && ((nm >> pk.p1) & 1ull)) {
          row[pk.p1] = s1;
          smax = s1 > smax ? s1 : smax;
        }
        if (lane == k) mine = nm;
        any_new |= nm;
      };
      unsigned todo = __ballot_sync(FULL, pend != 0ull && d <= ECAP_F);
      while (todo) {
        const int dd = ((todo >> lane) & 1u) ? d : 0;
        int incl = dd;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const int y = __shfl_up_sync(FULL, incl, off);
          if (lane >= off) incl += y;
        }
        const unsigned sub = __ballot_sync(FULL, ((todo >> lane) & 1u) && incl <= ECAP_F);
        todo &= ~sub;
        int first;
        const int ne = list_rows(col, lm_prev, hb, ((sub >> lane) & 1u) ? d : 0, pend, ent, owns[wid], first, tri);
        for (unsigned r = sub; r;) {
          const int k = __ffs(r) - 1;
          r &= r - 1u;
          const int f = __shfl_sync(FULL, first, k), e = r ? __shfl_sync(FULL, first, __ffs(r) - 1) : ne;
          if (f == e) continue;
          const int32_t u = __shfl_sync(FULL, v, k);
          const uint64_t nm = entries_or(ent, f, e);
          const Packed pk = pack_lanes(nm, tab);
          uint64_t s0 = 0ull, s1 = 0ull;
          if (fit) count_entries<false>(ent, f, e, pk, sigma, s0, s1, ovf);
          else count_entries<true>(ent, f, e, pk, sigma, s0, s1, ovf);
          store(k, u, nm, pk, s0, s1);
        }
        __syncwarp();
      }
      for (unsigned r = __ballot_sync(FULL, pend != 0ull && d > ECAP_F); r; r &= r - 1u) {
        // (only with heavy_deg above the list's capacity) piece by piece
        const int k = __ffs(r) - 1;
        const int32_t u = __shfl_sync(FULL, v, k);
        const int b = __shfl_sync(FULL, hb, k), e = b + __shfl_sync(FULL, d, k);
        const uint64_t pl = __shfl_sync(FULL, pend, k);
        const Packed pk = pack_lanes(pl, tab);
        uint64_t s0 = 0ull, s1 = 0ull, nm = 0ull;
        for (int j = b; j < e; j += ECAP_F) {
          const int ne = list_row(col, lm_prev, j, min(e, j + ECAP_F), pl, ent, tri);
          nm |= entries_or(ent, 0, ne);
          count_entries<true>(ent, 0, ne, pk, sigma, s0, s1, ovf);
          __syncwarp();
        }
        if (nm) store(k, u, nm, pk, s0, s1);
      }
      if (mine) {
        lm_cur[v] = mine;
        visited[v] = vis | mine;
        rch += (unsigned long long)__popcll((long long)mine);
      }
      // unfinished vertices stay on the list; found ones join the level's
      const unsigned left = __ballot_sync(FULL, (pend & ~mine) != 0ull), found = __ballot_sync(FULL, mine != 0ull);
      unsigned p0 = 0u, p1 = 0u;
      if (lane == 0 && left) p0 = atomicAdd(cnt_out, (unsigned)__popc(left));
      if (lane == 1 && found) p1 = atomicAdd(vcnt_next, (unsigned)__popc(found));
      p0 = __shfl_sync(FULL, p0, 0);
      p1 = __shfl_sync(FULL, p1, 1);
      if ((left >> lane) & 1u) list_out[p0 + __popc(left & lt)] = v;
      if ((found >> lane) & 1u) list_next[p1 + __popc(found & lt)] = v;
      if (vedges_next && found) {
        const unsigned ds = __reduce_add_sync(FULL, mine ? (unsigned)d : 0u);
        if (lane == 0) atomicAdd(vedges_next, (unsigned long long)ds);
      }
    }
  ovf = warp_or64(ovf);
  if (lane == 0 && ovf) atomicOr((unsigned long long *)(enable + 3), (unsigned long long)ovf);
  tri = warp_sum64(tri);
  rch = warp_sum64(rch);
  if (lane == 0 && (tri | rch)) {
    atomicAdd(cnt, tri);
    atomicAdd(cnt + 1, rch);
  }
  smax = warp_max64(smax);
  if (lane == 0 && smax > 1ull) atomicMax((unsigned long long *)(enable + 2), (unsigned long long)smax);
  any_new = warp_or64(any_new);
  block_or_to(any_new, active_cur);
}

// One warp per listed segment (list null: every segment) of a heavy vertex; the
// segments' sums meet in the vertex's count row by 64-bit atomics, and the last
// of them sees the row's total, so the largest count is taken here.
__global__ void __launch_bounds__(FWD_THREADS, 4)
k_fwd_heavy(int32_t n, int nseg, const int32_t *__restrict__ list, const unsigned *__restrict__ nlist,
            const int32_t *__restrict__ seg_v, const int32_t *__restrict__ seg_b,
            const int32_t *__restrict__ seg_e, const int32_t *__restrict__ col, const uint64_t *__restrict__ lm_prev,
            uint64_t *__restrict__ lm_cur, const uint64_t *__restrict__ visited, uint64_t *__restrict__ sigma,
            const uint64_t *__restrict__ active_prev, uint64_t *__restrict__ enable,
            unsigned long long *__restrict__ cnt, unsigned *__restrict__ wq) {
  __shared__ uint4 ents[FWD_THREADS / 32][ECAP_F];
  __shared__ int8_t tabs[FWD_THREADS / 32][64];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint4 *ent = ents[wid];
  int8_t *tab = tabs[wid];
  const uint64_t act = *active_prev & *enable;
  const bool fit = counts_fit(enable[2], n);
  unsigned long long tri = 0ull;
  uint64_t ovf = 0ull, smax = 0ull;
  const int total = list ? (int)*nlist : nseg;
  if (act)
    for (int i = grab(wq, 1); i < total; i = grab(wq, 1)) {
      const int s = list ? list[i] : i;
      const int32_t v = seg_v[s];
      const int beg = seg_b[s], end = seg_e[s];
      const uint64_t pend = ~visited[v] & act;
      if (!pend) continue;
      for (int b = beg; b < end; b += ECAP_F) {
        const int ne = list_row(col, lm_prev, b, min(end, b + ECAP_F), pend, ent, tri);
        if (!ne) continue;
        const uint64_t nm = entries_or(ent, 0, ne);
        const Packed pk = pack_lanes(nm, tab);
        uint64_t s0 = 0ull, s1 = 0ull;
        if (fit) count_entries<false>(ent, 0, ne, pk, sigma, s0, s1, ovf);
        else count_entries<true>(ent, 0, ne, pk, sigma, s0, s1, ovf);
        unsigned long long *dst = (unsigned long long *)(sigma + (size_t)v * 64);
        if ((lane >> pk.glog) == 0 && pk.p0 >= 0) {
          const unsigned long long x = (unsigned long long)s0, old = atomicAdd(dst + pk.p0, x);
          if (old + x < x) ovf |= 1ull << pk.p0;
          smax = old + x > smax ? old + x : smax;
        }
        if (pk.p1 >= 0) {
          const unsigned long long x = (unsigned long long)s1, old = atomicAdd(dst + pk.p1, x);
          if (old + x < x) ovf |= 1ull << pk.p1;
          smax = old + x > smax ? old + x : smax;
        }
        if (lane == 0) atomicOr((unsigned long long *)&lm_cur[v], (unsigned long long)nm);
        __syncwarp();
      }
    }
  ovf = warp_or64(ovf);
  if (lane == 0 && ovf) atomicOr((unsigned long long *)(enable + 3), (unsigned long long)ovf);
  tri = warp_sum64(tri);
  if (lane == 0 && tri) atomicAdd(cnt, tri);
  smax = warp_max64(smax);
  if (lane == 0 && smax > 1ull) atomicMax((unsigned long long *)(enable + 2), (unsigned long long)smax);
}

// Appends the segments [first, first + k) of the warp's threads to a list.
__device__ __forceinline__ void append_segments(int first, int k, int32_t *__restrict__ list,
                                                unsigned *__restrict__ count) {
  const int lane = threadIdx.x & 31;
  int incl = k;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int y = __shfl_up_sync(FULL, incl, off);
    if (lane >= off) incl += y;
  }
  const int total = __shfl_sync(FULL, incl, 31);
  if (!total) return;
  unsigned base = 0u;
  if (lane == 0) base = atomicAdd(count, (unsigned)total);
  base = __shfl_sync(FULL, base, 0);
  int32_t *out = list + base + incl - k;
  if (k <= 8)
    for (int i = 0; i < k; ++i) out[i] = first + i;
  for (unsigned m = __ballot_sync(FULL, k > 8); m; m &= m - 1u) {  // a hub's: the whole warp
    const int o = __ffs(m) - 1;
    const int kk = __shfl_sync(FULL, k, o), ff = __shfl_sync(FULL, first, o), at = __shfl_sync(FULL, incl - k, o);
    for (int i = lane; i < kk; i += 32) list[base + at + i] = ff + i;
  }
}

// After the segments of a level: the heavy vertices' masks. Also records, for
// the host, whether any heavy vertex has lanes at this level (*hflag) and the
// lanes in which some heavy vertex is still unvisited (*hpend): levels without
// heavy work then skip the heavy kernels; and lists the segments of the
// vertices with lanes left for the next level (one atomic per segment taken is
// what a level without work costs otherwise: 130,000 of them on R-MAT s20, 0.1
// ms).
__global__ void k_fwd_heavy_fin(int nh, const int32_t *__restrict__ heavy, const int32_t *__restrict__ hseg0,
                                const uint64_t *__restrict__ lm_cur, uint64_t *__restrict__ visited,
                                uint64_t *__restrict__ active_cur, unsigned long long *__restrict__ cnt,
                                const uint64_t *__restrict__ enable, unsigned *__restrict__ hflag,
                                unsigned long long *__restrict__ hpend, const int32_t *__restrict__ rp,
                                int32_t *__restrict__ list_next, unsigned *__restrict__ vcnt_next,
                                unsigned long long *__restrict__ vedges_next, int32_t *__restrict__ seg_list,
                                unsigned *__restrict__ seg_cnt) {
  const int lane = threadIdx.x & 31;
  const int h = blockIdx.x * blockDim.x + threadIdx.x;
  const uint64_t en = *enable;
  uint64_t newm = 0ull, left = 0ull;
  int32_t v = 0;
  int first = 0, k = 0;
  if (h < nh) {
    v = heavy[h];
    newm = lm_cur[v];
    const uint64_t vis = visited[v];
    if (newm) visited[v] = vis | newm;
    left = ~(vis | newm) & en;
    first = hseg0[h];
    k = left ? hseg0[h + 1] - first : 0;
  }
  append_segments(first, k, seg_list, seg_cnt);
  const unsigned found = __ballot_sync(FULL, newm != 0ull);
  if (found) {
    unsigned pos = 0u;
    if (lane == 0) pos = atomicAdd(vcnt_next, (unsigned)__popc(found));
    pos = __shfl_sync(FULL, pos, 0);
    if (newm) list_next[pos + __popc(found & ((1u << lane) - 1u))] = v;
    if (vedges_next && newm) atomicAdd(vedges_next, (unsigned long long)(rp[v + 1] - rp[v]));
  }
  const unsigned long long rch = __reduce_add_sync(FULL, (unsigned)__popcll((long long)newm));
  newm = warp_or64(newm);
  left = warp_or64(left);
  if (lane == 0) {
    if (newm) {
      atomicAdd(cnt + 1, rch);
      atomicOr((unsigned long long *)active_cur, (unsigned long long)newm);
      atomicOr(hflag, 1u);
    }
    if (left) atomicOr(hpend, (unsigned long long)left);
  }
}

// ------------------------------------------------------- top-down levels --
// Sec. 3 step 1 batched over lanes, run top-down for a level whose vertices
// have few edges: each vertex w of level l pushes its lanes to the neighbours
// that are not visited in them, which join level l+1 in those lanes
// (lm_next must be zero before). Each newly reached vertex is listed once.
__global__ void __launch_bounds__(FWD_THREADS)
k_fwd_push(const int32_t *__restrict__ rp, const int32_t *__restrict__ col, const int32_t *__restrict__ list_cur,
           const unsigned *__restrict__ vcnt_cur, const uint64_t *__restrict__ lm_cur_lvl,
           uint64_t *__restrict__ lm_next, const uint64_t *__restrict__ visited,
           const uint64_t *__restrict__ active_cur, const uint64_t *__restrict__ enable,
           int32_t *__restrict__ list_next, unsigned *__restrict__ vcnt_next,
           unsigned long long *__restrict__ vedges_next, unsigned *__restrict__ wq) {
  const int lane = threadIdx.x & 31;
  const uint64_t act = *active_cur & *enable;
  const int cnt = (int)*vcnt_cur;
  for (int i = grab(wq, 1); i < cnt; i = grab(wq, 1)) {
    const int32_t w = list_cur[i];
    const uint64_t mw = lm_cur_lvl[w] & act;
    if (!mw) continue;
    const int beg = rp[w], end = rp[w + 1];
    for (int base = beg; base < end; base += 32) {
      const int j = base + lane;
      bool first = false;
      int32_t v = 0;
      int dv = 0;
      if (j < end) {
        v = col[j];
        const uint64_t nl = mw & ~visited[v];
        if (nl) {
          first = atomicOr((unsigned long long *)&lm_next[v], (unsigned long long)nl) == 0ull;
          if (first) dv = rp[v + 1] - rp[v];
        }
      }
      list_append(first, v, dv, list_next, vcnt_next, vedges_next);
    }
  }
}

// Path counts of the vertices a top-down level reached (their new lanes are
// lm_next[v], complete after k_fwd_push): pulled from the neighbours at level
// l in those lanes (Def. 3), then visited, the largest count, the overflowed
// lanes and the level's lane set are updated as by the bottom-up kernels.
// Counts are exact integer sums, so the direction does not change any value.
__global__ void __launch_bounds__(FWD_THREADS)
k_fwd_pull_list(const int32_t *__restrict__ rp, const int32_t *__restrict__ col,
                const int32_t *__restrict__ list_next, const unsigned *__restrict__ vcnt_next,
                const uint64_t *__restrict__ lm_cur_lvl, const uint64_t *__restrict__ lm_next,
                uint64_t *__restrict__ visited, uint64_t *__restrict__ sigma, uint64_t *__restrict__ enable,
                uint64_t *__restrict__ active_next, unsigned long long *__restrict__ cnt,
                unsigned *__restrict__ wq, int heavy_deg, unsigned *__restrict__ hflag) {
  const int lane = threadIdx.x & 31;
  uint64_t any_new = 0ull, smax = 0ull, ovf = 0ull;
  unsigned long long tri = 0ull, rch = 0ull;
  const int nv = (int)*vcnt_next;
  for (int i = grab(wq, 1); i < nv; i = grab(wq, 1)) {
    const int32_t v = list_next[i];
    const uint64_t newm = lm_next[v];
    const int beg = rp[v], end = rp[v + 1];
    if (lane == 0 && end - beg > heavy_deg) atomicOr(hflag, 1u);  // the backward's heavy kernels run here
    uint64_t s0 = 0ull, s1 = 0ull;
    for (int base = beg; base < end; base += 32) {
      const int j = base + lane;
      int32_t w = 0;
      uint64_t m = 0ull;
      if (j < end) {
        w = col[j];
        m = lm_cur_lvl[w] & newm;
      }
      tri += (unsigned long long)__popcll((long long)m);
      unsigned bal = __ballot_sync(FULL, m != 0ull);
      while (bal) {
        uint64_t mk[UNR];
        int32_t wk[UNR];
        take(bal, m, w, mk, wk);
        uint64_t x0[UNR], x1[UNR];
#pragma unroll
        for (int k = 0; k < UNR; ++k) {
          const uint64_t *row = sigma + (size_t)wk[k] * 64;
          x0[k] = ((mk[k] >> lane) & 1ull) ? row[lane] : 0ull;
          x1[k] = ((mk[k] >> (lane + 32)) & 1ull) ? row[lane + 32] : 0ull;
        }
#pragma unroll
        for (int k = 0; k < UNR; ++k) {
          const uint64_t t0 = s0 + x0[k];
          if (t0 < s0) ovf |= 1ull << lane;
          s0 = t0;
          const uint64_t t1 = s1 + x1[k];
          if (t1 < s1) ovf |= 1ull << (lane + 32);
          s1 = t1;
        }
      }
    }
    if ((newm >> lane) & 1ull) {
      sigma[(size_t)v * 64 + lane] = s0;
      smax = s0 > smax ? s0 : smax;
    }
    if ((newm >> (lane + 32)) & 1ull) {
      sigma[(size_t)v * 64 + 32 + lane] = s1;
      smax = s1 > smax ? s1 : smax;
    }
    if (lane == 0) visited[v] |= newm;
    rch += (unsigned long long)__popcll((long long)newm);
    any_new |= newm;
  }
  ovf = warp_or64(ovf);
  if (lane == 0 && ovf) atomicOr((unsigned long long *)(enable + 3), (unsigned long long)ovf);
  tri = warp_sum64(tri);
  if (lane == 0 && (tri | rch)) {
    atomicAdd(cnt, tri);
    atomicAdd(cnt + 1, rch);
  }
  smax = warp_max64(smax);
  if (lane == 0 && smax > 1ull) atomicMax((unsigned long long *)(enable + 2), (unsigned long long)smax);
  block_or_to(any_new, active_next);
}

// Pair lanes: lane i is finished once its destination appears at this level.
__global__ void k_pair_check(int count, int level, const int32_t *__restrict__ dest,
                             const uint64_t *__restrict__ lm_cur, const uint64_t *__restrict__ sigma,
                             uint64_t *__restrict__ enable, int32_t *__restrict__ pair_d,
                             uint64_t *__restrict__ pair_sig, const uint64_t *__restrict__ active_cur,
                             uint64_t *__restrict__ cont) {
  const int i = threadIdx.x;
  const uint64_t en = *enable;
  bool done = false;
  if (i < count && ((en >> i) & 1ull)) {
    const int32_t t = dest[i];
    if ((lm_cur[t] >> i) & 1ull) {
      pair_d[i] = level;
      pair_sig[i] = sigma[(size_t)t * 64 + i];
      done = true;
    }
  }
  const unsigned b0 = __ballot_sync(FULL, done);  // block = 2 full warps
  __shared__ unsigned long long s_done;
  if (i == 0) s_done = 0ull;
  __syncthreads();
  if ((i & 31) == 0) atomicOr(&s_done, ((unsigned long long)b0) << (i & 32));
  __syncthreads();
  if (i == 0) {
    const uint64_t en2 = en & ~(uint64_t)s_done;
    *enable = en2;
    *cont = *active_cur & en2;
  }
}

// -------------------------------------------------------------- backward --
// Exact sums of coefficients. Narrow: 96 bits in units of 2^-unit where the
// batch's largest count allows (bc_common.cuh), and the coefficients are kept
// in that form, 12 bytes (rows of 64 low words, then 64 high halves), so that
// adding one is three instructions: with doubles, converted at every add, the
// heavy segments of R-MAT s20's hub level kept the ALU pipe 87 % busy. Wide:
// doubles in the counts' slots and the 192-bit window.
struct NarrowAcc {
  using A = Acc3;
  static constexpr bool narrow = true;
  struct Rows {
    using V = Acc3;
    const uint64_t *__restrict__ p;
    static __device__ __forceinline__ V zero() { return V{0u, 0u, 0u}; }
    __device__ __forceinline__ V operator()(uint32_t w, int t) const {
      const uint64_t *row = p + (size_t)w * 96;
      const uint64_t lo = row[t];
      return V{(uint32_t)lo, (uint32_t)(lo >> 32), reinterpret_cast<const uint32_t *>(row + 64)[t]};
    }
  };
  static __device__ __forceinline__ A zero() { return A{0u, 0u, 0u}; }
  static __device__ __forceinline__ void add(A &a, const Acc3 &x, unsigned &) { add_acc(a, x); }
  static __device__ __forceinline__ void add_double(A &a, double x, int unit, unsigned &e) {
    if (x != 0.0) acc3_add(a, (uint64_t)__double_as_longlong(x), 1075 - unit, e);
  }
  static __device__ __forceinline__ void put(uint64_t *rows, int32_t v, int t, const A &a) {
    uint64_t *row = rows + (size_t)v * 96;
    row[t] = (uint64_t)a.l0 | ((uint64_t)a.l1 << 32);
    reinterpret_cast<uint32_t *>(row + 64)[t] = a.l2;
  }
  static __device__ __forceinline__ void put_double(uint64_t *rows, int32_t v, int t, double x, int unit, unsigned &e) {
    A a = zero();
    add_double(a, x, unit, e);
    put(rows, v, t, a);
  }
  static __device__ __forceinline__ void add_acc(A &a, const A &b) { acc3_add3(a, b.l0, b.l1, b.l2); }
  static __device__ __forceinline__ A shfl_xor(const A &a, int off) {
    return A{__shfl_xor_sync(FULL, a.l0, off), __shfl_xor_sync(FULL, a.l1, off), __shfl_xor_sync(FULL, a.l2, off)};
  }
  static __device__ __forceinline__ A shfl_up(const A &a, int off) {
    return A{__shfl_up_sync(FULL, a.l0, off), __shfl_up_sync(FULL, a.l1, off), __shfl_up_sync(FULL, a.l2, off)};
  }
  static __device__ __forceinline__ bool any(const A &a) { return (a.l0 | a.l1 | a.l2) != 0u; }
  static __device__ __forceinline__ Acc widen(const A &a, int unit) { return acc3_widen(a, unit); }
};
struct WideAcc {
  using A = Acc;
  static constexpr bool narrow = false;
  using Rows = WordRows;
  static __device__ __forceinline__ A zero() { return acc_zero(); }
  static __device__ __forceinline__ void add(A &a, uint64_t x, unsigned &e) {
    acc_add(a, __longlong_as_double((long long)x), e);  // (0 adds nothing)
  }
  static __device__ __forceinline__ void add_double(A &a, double x, int, unsigned &e) { acc_add(a, x, e); }
  static __device__ __forceinline__ void put_double(uint64_t *rows, int32_t v, int t, double x, int, unsigned &) {
    rows[(size_t)v * 64 + t] = (uint64_t)__double_as_longlong(x);
  }
  static __device__ __forceinline__ void add_acc(A &a, const A &b) { acc_add_acc(a, b); }
  static __device__ __forceinline__ A shfl_xor(const A &a, int off) {
    return A{__shfl_xor_sync(FULL, a.w0, off), __shfl_xor_sync(FULL, a.w1, off), __shfl_xor_sync(FULL, a.w2, off)};
  }
  static __device__ __forceinline__ A shfl_up(const A &a, int off) {
    return A{__shfl_up_sync(FULL, a.w0, off), __shfl_up_sync(FULL, a.w1, off), __shfl_up_sync(FULL, a.w2, off)};
  }
  static __device__ __forceinline__ bool any(const A &a) { return (a.w0 | a.w1 | a.w2) != 0ull; }
  static __device__ __forceinline__ Acc widen(const A &a, int) { return a; }
};

// A pair without successors has delta = 0 and coefficient RN(1 / sigma), and
// most pairs are such (the deepest level of each lane): for counts below
// RECIPS the coefficient comes from a table (made for the batch's unit), and
// the pair skips the ring. (No sink needs a zero delta: the rows and target
// blocks start cleared.)
constexpr int RECIPS = 2048;
__global__ void k_recips(int unit, Acc3 *__restrict__ out) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= RECIPS) return;
  Acc3 a{0u, 0u, 0u};
  unsigned e = 0u;
  if (s > 0) NarrowAcc::add_double(a, coef_of(0.0, (uint64_t)s), unit, e);
  out[s] = e ? Acc3{0u, 0u, 0u} : a;  // (a count above the batch's largest: never asked for)
}

// Finished (vertex, lane) pairs wait in a per-warp ring in shared memory until
// 32 of them fill one warp-wide round of the per-vertex arithmetic (rounding
// the sum, product, quotient), so its many instructions run with all threads.
constexpr int RING = 96;  // up to 31 left over + 64 of one vertex
template <class P> struct Ring {
  typename P::A sum[RING];
  uint64_t sig[RING];
  int32_t v[RING];
  uint8_t t[RING];
};

// delta = RN(RN(sigma) * sum); a power-of-two sigma scales exactly (integer
// exponent add), everything else is one rounded product (integer-only below 2^53).
__device__ __forceinline__ double delta_of(double sum, uint64_t sg) {
  if ((sg & (sg - 1ull)) == 0ull) {
    const uint64_t b = (uint64_t)__double_as_longlong(sum);
    if (b == 0ull) return 0.0;
    const int k = 63 - __clzll((long long)sg);
    return __longlong_as_double((long long)(b + ((uint64_t)k << 52)));
  }
  return delta_rn(sg, sum);
}

// One warp-wide round over `count` (<= 32) records from ring position head. The
// coefficient goes to its own 96-bit row, or in the wide form over sigma[v][t].
template <class P>
__device__ __forceinline__ void ring_round(Ring<P> &R, int head, int count, uint64_t *__restrict__ coef,
                                           const Sink &sink, int unit, unsigned &e) {
  const int lane = threadIdx.x & 31;
  int32_t v = -1;
  double d = 0.0;
  if (lane < count) {
    int pos = head + lane;
    pos -= pos >= RING ? RING : 0;
    v = R.v[pos];
    const int t = R.t[pos];
    const uint64_t sg = R.sig[pos];
    const typename P::A a = R.sum[pos];
    if (P::any(a)) d = delta_of(acc_round(P::widen(a, unit)), sg);  // no successor: delta = 0
    P::put_double(coef, v, t, coef_of(d, sg), unit, e);
    if (sink.delta_lm) sink.delta_lm[(size_t)v * 64 + t] = d;
    if (sink.tslot) sink_targets(sink, v, t, d);
  }
  if (sink.acc && __any_sync(FULL, d != 0.0)) {
    // records of one vertex are consecutive: segmented exact inclusive scan
    // (a dependency is at least 2^-ceil(log2 of the largest count), so it is a
    // whole number of units too)
    typename P::A a = P::zero();
    P::add_double(a, d, unit, e);
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const typename P::A o = P::shfl_up(a, off);
      const int32_t vo = __shfl_up_sync(FULL, v, off);
      if (lane >= off && vo == v) P::add_acc(a, o);
    }
    const int32_t vn = __shfl_down_sync(FULL, v, 1);
    if (v >= 0 && (lane == 31 || vn != v) && P::any(a)) {
      Acc cur = sink.acc[v];
      acc_add_acc(cur, P::widen(a, unit));
      sink.acc[v] = cur;
    }
  }
}

// The finished lanes of v (their sums in the threads of group 0; sg0 / sg1: the
// counts of the thread's lanes): a lane without successors gets its tabulated
// coefficient, the others go into the ring, with a round whenever 32 wait.
template <class P>
__device__ __forceinline__ void ring_put(Ring<P> &R, int &head, int &have, int32_t v, const Packed &pk,
                                         const typename P::A &a0, const typename P::A &a1, uint64_t sg0, uint64_t sg1,
                                         uint64_t *__restrict__ coef, const Acc3 *__restrict__ recips,
                                         const Sink &sink, int unit, unsigned &e) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    if (h && !pk.two) break;
    const int t = h ? pk.p1 : ((lane >> pk.glog) == 0 ? pk.p0 : -1);
    const typename P::A &a = h ? a1 : a0;
    const uint64_t sg = h ? sg1 : sg0;
    bool on = t >= 0;
    if constexpr (P::narrow) {
      if (on && sg < (uint64_t)RECIPS && !P::any(a)) {
        P::put(coef, v, t, recips[sg]);
        on = false;
      }
    }
    const unsigned m = __ballot_sync(FULL, on);
    if (on) {
      int pos = head + have + __popc(m & lt);
      pos -= pos >= RING ? RING : 0;
      R.v[pos] = v;
      R.t[pos] = (uint8_t)t;
      R.sum[pos] = a;
      R.sig[pos] = sg;
    }
    have += __popc(m);
  }
  __syncwarp();
  while (have >= 32) {
    ring_round<P>(R, head, 32, coef, sink, unit, e);
    head += 32;
    head -= head >= RING ? RING : 0;
    have -= 32;
    __syncwarp();
  }
}

// Exact sums over entries [f, e) in the packed lanes, totals in group 0.
template <class P>
__device__ __forceinline__ void coef_entries(const uint4 *ent, int f, int e, const Packed &pk,
                                             const uint64_t *__restrict__ coef, typename P::A &a0,
                                             typename P::A &a1, unsigned &err) {
  entries_sum(ent, f, e, pk, typename P::Rows{coef}, [&](const typename P::Rows::V &x) { P::add(a0, x, err); },
              [&](const typename P::Rows::V &x) { P::add(a1, x, err); });
}
template <class P> __device__ __forceinline__ void group_sum(typename P::A &a, int glog) {
  for (int off = 1 << glog; off < 32; off <<= 1) P::add_acc(a, P::shfl_xor(a, off));
}

// The light vertices of level l (listed by the forward pass), a warp taking gsz
// at a time.
template <class P>
__global__ void __launch_bounds__(FWD_THREADS, P::narrow ? BWD_MIN_BLOCKS : 3)
k_bwd_light(const int32_t *__restrict__ list_l, const unsigned *__restrict__ vcnt_l, const int32_t *__restrict__ rp,
            const int32_t *__restrict__ col, const uint64_t *__restrict__ lm_cur, const uint64_t *__restrict__ lm_next,
            const uint64_t *__restrict__ sigma, uint64_t *__restrict__ coef, const Acc3 *__restrict__ recips, Sink sink,
            unsigned *__restrict__ err, unsigned *__restrict__ wq, int heavy_deg, uint64_t keep, int gsz, int unit) {
  __shared__ Ring<P> rings[FWD_THREADS / 32];
  __shared__ uint4 ents[FWD_THREADS / 32][ECAP_B];
  __shared__ int8_t tabs[FWD_THREADS / 32][64];
  __shared__ uint8_t owns[FWD_THREADS / 32][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  Ring<P> &R = rings[wid];
  uint4 *ent = ents[wid];
  int8_t *tab = tabs[wid];
  int head = 0, have = 0;
  unsigned e = 0u;
  unsigned long long tri = 0ull;  // (counted by the forward pass)
  const int total = (int)*vcnt_l;
  for (int base = grab(wq, gsz); base < total; base = grab(wq, gsz)) {
    int32_t v = -1;
    int hb = 0, d = 0;
    uint64_t lanes = 0ull;
    if (lane < gsz && base + lane < total) {
      v = list_l[base + lane];
      lanes = lm_cur[v] & keep;
      hb = rp[v];
      d = rp[v + 1] - hb;
      if (d > heavy_deg) lanes = 0ull;  // heavy: its segments' kernels
    }
    // sums of one vertex (thread k holds it): entries [f, e), or for a row
    // above the list's capacity piece by piece
    auto finish = [&](int k, int f, int en, bool pieces) {
      const int32_t u = __shfl_sync(FULL, v, k);
      const uint64_t ul = __shfl_sync(FULL, lanes, k);
      const Packed pk = pack_lanes(ul, tab);
      const uint64_t *row = sigma + (size_t)u * 64;
      const uint64_t sg0 = ((lane >> pk.glog) == 0 && pk.p0 >= 0) ? row[pk.p0] : 0ull;
      const uint64_t sg1 = pk.p1 >= 0 ? row[pk.p1] : 0ull;
      typename P::A a0 = P::zero(), a1 = P::zero();
      if (pieces) {
        const int b = __shfl_sync(FULL, hb, k), end = b + __shfl_sync(FULL, d, k);
        for (int j = b; j < end; j += ECAP_B) {
          const int ne = list_row(col, lm_next, j, min(end, j + ECAP_B), ul, ent, tri);
          coef_entries<P>(ent, 0, ne, pk, coef, a0, a1, e);
          __syncwarp();
        }
        group_sum<P>(a0, pk.glog);
      } else if (f < en) {
        coef_entries<P>(ent, f, en, pk, coef, a0, a1, e);
        group_sum<P>(a0, pk.glog);
      }
      ring_put<P>(R, head, have, u, pk, a0, a1, sg0, sg1, coef, recips, sink, unit, e);
    };
    for (unsigned r = __ballot_sync(FULL, lanes != 0ull && d == 0); r; r &= r - 1u)
      finish(__ffs(r) - 1, 0, 0, false);  // (directed graphs: no out-neighbour)
    unsigned todo = __ballot_sync(FULL, lanes != 0ull && d > 0 && d <= ECAP_B);
    while (todo) {
      const int dd = ((todo >> lane) & 1u) ? d : 0;
      int incl = dd;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(FULL, incl, off);
        if (lane >= off) incl += y;
      }
      const unsigned sub = __ballot_sync(FULL, ((todo >> lane) & 1u) && incl <= ECAP_B);
      todo &= ~sub;
      int first;
      const int ne = list_rows(col, lm_next, hb, ((sub >> lane) & 1u) ? d : 0, lanes, ent, owns[wid], first, tri);
      for (unsigned r = sub; r;) {
        const int k = __ffs(r) - 1;
        r &= r - 1u;
        const int f = __shfl_sync(FULL, first, k), en = r ? __shfl_sync(FULL, first, __ffs(r) - 1) : ne;
        finish(k, f, en, false);
      }
      __syncwarp();
    }
    for (unsigned r = __ballot_sync(FULL, lanes != 0ull && d > ECAP_B); r; r &= r - 1u)
      finish(__ffs(r) - 1, 0, 0, true);
  }
  if (have) ring_round<P>(R, head, have, coef, sink, unit, e);
  if (e) atomicOr(err, e);
}

// The heavy vertices with lanes at a level: their segments, and the vertices
// with several.
__global__ void k_bwd_heavy_list(int nh, const int32_t *__restrict__ heavy, const int32_t *__restrict__ hseg0,
                                 const uint64_t *__restrict__ lm_cur, uint64_t keep, int32_t *__restrict__ seg_list,
                                 int32_t *__restrict__ multi, unsigned *__restrict__ counts) {
  const int lane = threadIdx.x & 31;
  const int h = blockIdx.x * blockDim.x + threadIdx.x;
  int first = 0, k = 0;
  if (h < nh && (lm_cur[heavy[h]] & keep)) {
    first = hseg0[h];
    k = hseg0[h + 1] - first;
  }
  append_segments(first, k, seg_list, counts);
  const unsigned m = __ballot_sync(FULL, k > 1);
  if (!m) return;
  unsigned pos = 0u;
  if (lane == 0) pos = atomicAdd(counts + 1, (unsigned)__popc(m));
  pos = __shfl_sync(FULL, pos, 0);
  if (k > 1) multi[pos + __popc(m & ((1u << lane) - 1u))] = h;
}

// Heavy vertices: one warp per listed segment (taken dynamically). A vertex of
// one segment is finished here; the others' partial sums go to part[s][lane].
template <class P>
__global__ void __launch_bounds__(FWD_THREADS, P::narrow ? BWD_MIN_BLOCKS : 3)
k_bwd_heavy_seg(const int32_t *__restrict__ list, const unsigned *__restrict__ nlist,
                const int32_t *__restrict__ seg_v, const int32_t *__restrict__ seg_b,
                const int32_t *__restrict__ seg_e, const int32_t *__restrict__ rp, const int32_t *__restrict__ col,
                const uint64_t *__restrict__ lm_cur, const uint64_t *__restrict__ lm_next,
                const uint64_t *__restrict__ sigma, uint64_t *__restrict__ coef, const Acc3 *__restrict__ recips,
                typename P::A *__restrict__ part, Sink sink, unsigned *__restrict__ wq, unsigned *__restrict__ err,
                uint64_t keep, int unit) {
  __shared__ Ring<P> rings[FWD_THREADS / 32];
  __shared__ uint4 ents[FWD_THREADS / 32][ECAP_B];
  __shared__ int8_t tabs[FWD_THREADS / 32][64];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  Ring<P> &R = rings[wid];
  uint4 *ent = ents[wid];
  int head = 0, have = 0;
  unsigned e = 0u;
  unsigned long long tri = 0ull;
  const int total = (int)*nlist;
  for (int i = grab(wq, 1); i < total; i = grab(wq, 1)) {
    const int s = list[i];
    const int32_t v = seg_v[s];
    const uint64_t lanes = lm_cur[v] & keep;
    const int beg = seg_b[s], end = seg_e[s];
    const bool whole = rp[v] == beg && rp[v + 1] == end;
    const Packed pk = pack_lanes(lanes, tabs[wid]);
    typename P::A a0 = P::zero(), a1 = P::zero();
    for (int j = beg; j < end; j += ECAP_B) {
      const int ne = list_row(col, lm_next, j, min(end, j + ECAP_B), lanes, ent, tri);
      coef_entries<P>(ent, 0, ne, pk, coef, a0, a1, e);
      __syncwarp();
    }
    group_sum<P>(a0, pk.glog);
    if (whole) {
      const uint64_t *row = sigma + (size_t)v * 64;
      const uint64_t sg0 = ((lane >> pk.glog) == 0 && pk.p0 >= 0) ? row[pk.p0] : 0ull;
      const uint64_t sg1 = pk.p1 >= 0 ? row[pk.p1] : 0ull;
      ring_put<P>(R, head, have, v, pk, a0, a1, sg0, sg1, coef, recips, sink, unit, e);
    } else {
      if ((lane >> pk.glog) == 0 && pk.p0 >= 0) part[(size_t)s * 64 + pk.p0] = a0;
      if (pk.p1 >= 0) part[(size_t)s * 64 + pk.p1] = a1;
    }
  }
  if (have) ring_round<P>(R, head, have, coef, sink, unit, e);
  if (e) atomicOr(err, e);
}

template <class P>
__global__ void __launch_bounds__(FWD_THREADS, 4)
k_bwd_heavy_fin(const int32_t *__restrict__ multi, const unsigned *__restrict__ nmulti,
                const int32_t *__restrict__ heavy, const int32_t *__restrict__ hseg0,
                const uint64_t *__restrict__ lm_cur, const uint64_t *__restrict__ sigma, uint64_t *__restrict__ coef,
                const Acc3 *__restrict__ recips, const typename P::A *__restrict__ part, Sink sink,
                unsigned *__restrict__ err,
                unsigned *__restrict__ wq, uint64_t keep, int unit) {
  __shared__ Ring<P> rings[FWD_THREADS / 32];
  __shared__ int8_t tabs[FWD_THREADS / 32][64];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  Ring<P> &R = rings[wid];
  int head = 0, have = 0;
  unsigned e = 0u;
  const int total = (int)*nmulti;
  for (int i = grab(wq, 1); i < total; i = grab(wq, 1)) {
    const int h = multi[i];
    const int32_t v = heavy[h];
    const uint64_t lanes = lm_cur[v] & keep;
    const Packed pk = pack_lanes(lanes, tabs[wid]);
    const uint64_t *row = sigma + (size_t)v * 64;
    const uint64_t sg0 = ((lane >> pk.glog) == 0 && pk.p0 >= 0) ? row[pk.p0] : 0ull;
    const uint64_t sg1 = pk.p1 >= 0 ? row[pk.p1] : 0ull;
    // the groups take different segments (a hub has hundreds)
    typename P::A a0 = P::zero(), a1 = P::zero();
    const int NG = 32 >> pk.glog;
    const int sb = hseg0[h], se = hseg0[h + 1];
    const typename P::A *q0 = part + (pk.p0 < 0 ? 0 : pk.p0), *q1 = part + (pk.p1 < 0 ? 0 : pk.p1);
#pragma unroll 4
    for (int s = sb + (lane >> pk.glog); s < se; s += NG) {
      if (pk.p0 >= 0) P::add_acc(a0, q0[(size_t)s * 64]);
      if (pk.p1 >= 0) P::add_acc(a1, q1[(size_t)s * 64]);
    }
    __syncwarp();
    group_sum<P>(a0, pk.glog);
    ring_put<P>(R, head, have, v, pk, a0, a1, sg0, sg1, coef, recips, sink, unit, e);
  }
  if (have) ring_round<P>(R, head, have, coef, sink, unit, e);
  if (e) atomicOr(err, e);
}

// Per-lane distance / sigma extraction after a forward pass.
__global__ void k_extract(int32_t n, int count, int maxlevel, const uint64_t *__restrict__ lm,
                          const uint64_t *__restrict__ sigma, int32_t *__restrict__ dist,
                          uint64_t *__restrict__ sig_out, int64_t row_stride, int64_t lane_stride) {
  const int32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  uint64_t seen = 0ull;
  for (int l = 0; l <= maxlevel; ++l) {
    uint64_t m = lm[(size_t)l * n + v];
    seen |= m;
    while (m) {
      const int t = __ffsll((long long)m) - 1;
      m &= m - 1ull;
      if (t < count) {
        if (dist) dist[(int64_t)t * lane_stride + (int64_t)v * row_stride] = l;
        if (sig_out) sig_out[(int64_t)t * lane_stride + (int64_t)v * row_stride] = sigma[(size_t)v * 64 + t];
      }
    }
  }
  for (int t = 0; t < count; ++t) {
    if (!((seen >> t) & 1ull)) {
      if (dist) dist[(int64_t)t * lane_stride + (int64_t)v * row_stride] = -1;
      if (sig_out) sig_out[(int64_t)t * lane_stride + (int64_t)v * row_stride] = 0ull;
    }
  }
}

// ------------------------------------------------------------------ host --
// Control words of one level, cleared together before a batch.
struct LevelCtl {
  unsigned long long active;  // lanes with a vertex at the level
  unsigned long long vedges;  // degree sum of the level's vertices (kept with the direction switch on)
  unsigned long long hpend;   // lanes some heavy vertex has not reached after the level
  unsigned q_light, q_heavy, q_bwd_light, q_bwd_seg, q_bwd_fin;  // work counters
  unsigned hflag;                 // a heavy vertex has lanes at the level
  unsigned vcnt;                  // vertices at the level (their list: vlist)
  unsigned todo;                  // light vertices unfinished before the level's successor
  unsigned fseg;                  // heavy segments listed for the level's successor
  unsigned bseg, bmulti;          // backward: listed segments, heavy vertices with several
  unsigned pad[15];
};
static_assert(sizeof(LevelCtl) == 128, "one line per level");
// Levels launched without asking the device: as many as the pinned staging
// holds control words of (two levels more than the depth, and 16 bytes before).
constexpr int BLIND_DEPTH = (int)((4096 - 16) / sizeof(LevelCtl)) - 2;

struct HeavyMeta {
  int nh = 0, nseg = 0, heavy_deg = 0, seg = 0;
  int depth = 0;  // the deepest level of the batches so far: levels launched without asking the device
  DevBuf heavy, hseg0, seg_v, seg_b, seg_e;
  DevBuf light;  // count (first word), then the light vertices with neighbours, in id order
  template <class F> void each(F f) {
    for (DevBuf *b : {&heavy, &hseg0, &seg_v, &seg_b, &seg_e, &light}) f(*b);
  }
};
static std::map<const int32_t *, HeavyMeta> g_heavy;  // keyed by the CSR's device row pointers
static std::mutex g_heavy_mu;

// The heavy-vertex split of the CSR the forward pulls over (in_csr: the
// in-neighbour CSR, which is the CSR itself on an undirected graph) or of the
// out-CSR the backward walks; each is kept per row-pointer array.
static HeavyMeta &heavy_meta(bc_ctx *ctx, const Graph &g, bool in_csr) {
  std::lock_guard<std::mutex> lk(g_heavy_mu);
  const int want_deg = ctx->heavy_deg > 0 ? ctx->heavy_deg : HEAVY_DEFAULT;
  const int want_seg = ctx->seg_len > 0 ? ctx->seg_len : SEG_DEFAULT;
  const int32_t *grp = in_csr ? g.rp_in : g.rp;
  auto it = g_heavy.find(grp);
  if (it != g_heavy.end()) {
    HeavyMeta &old = it->second;
    if (old.heavy_deg == want_deg && old.seg == want_seg) return old;
    // the graph's split changed (a new tuning): rebuild
    cudaStreamSynchronize(ctx->stream);
    old.each([](DevBuf &b) { b.release(); });
    g_heavy.erase(it);
  }
  HeavyMeta hm;
  std::vector<int32_t> rp(g.n + 1);
  BCG_CUDA(cudaMemcpy(rp.data(), grp, sizeof(int32_t) * (g.n + 1), cudaMemcpyDeviceToHost));
  std::vector<int32_t> heavy, hseg0, sv, sb, se, light(1, 0);
  hm.heavy_deg = want_deg;
  hm.seg = want_seg;
  const int seg = want_seg;
  for (int32_t v = 0; v < g.n; ++v) {
    const int d = rp[v + 1] - rp[v];
    if (d <= hm.heavy_deg) {
      if (d > 0) light.push_back(v);
      continue;
    }
    hseg0.push_back((int32_t)sv.size());
    heavy.push_back(v);
    for (int b = rp[v]; b < rp[v + 1]; b += seg) {
      sv.push_back(v);
      sb.push_back(b);
      se.push_back(std::min(b + seg, rp[v + 1]));
    }
  }
  hseg0.push_back((int32_t)sv.size());
  hm.nh = (int)heavy.size();
  hm.nseg = (int)sv.size();
  auto up = [&](DevBuf &b, const std::vector<int32_t> &x) {
    b.ensure(std::max<size_t>(x.size(), 1) * sizeof(int32_t));
    if (!x.empty()) BCG_CUDA(cudaMemcpy(b.p, x.data(), x.size() * sizeof(int32_t), cudaMemcpyHostToDevice));
  };
  try {
    up(hm.heavy, heavy);
    up(hm.hseg0, hseg0);
    up(hm.seg_v, sv);
    up(hm.seg_b, sb);
    up(hm.seg_e, se);
    if (grp == g.rp_in) {  // the forward's first list
      light[0] = (int32_t)light.size() - 1;
      up(hm.light, light);
    }
  } catch (...) {  // (a split cut short must not pass for the graph's next time)
    hm.each([](DevBuf &b) { b.release(); });
    throw;
  }
  return g_heavy[grp] = std::move(hm);
}

void forget_heavy_meta(const int32_t *rp) {
  std::lock_guard<std::mutex> lk(g_heavy_mu);
  auto it = g_heavy.find(rp);
  if (it == g_heavy.end()) return;
  HeavyMeta &hm = it->second;
  hm.each([](DevBuf &b) { b.release(); });
  g_heavy.erase(it);
}

static int g_num_sms = 0;
static int grid_blocks() {
  if (!g_num_sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev);
    if (g_num_sms <= 0) g_num_sms = 148;
  }
  return g_num_sms * 8;
}

// Vertices a warp of the light kernels takes at a time, by one atomic on a shared
// counter. Forward 16 (8 below 2^16 vertices, 4 below 2^14, for more warps to have
// some): with 4 below 2^18 the wide levels of sparse graphs waited for the counter
// and for windows filled by 4 short rows; ms for 1024 draws with 4 / 8 / 16 / 32: directed ER n = 200,000 degree 2 66.8 / 54.4 /
// 49.8 / 50.7, ER n = 100,003 degree 7 13.5 / 11.8 / 11.1 / 11.0, R-MAT s16 5.53 /
// 5.38 / 5.35 / 5.64, directed s17 10.27 / 9.70 / 9.51 / 9.80, s20 37.9 / 35.1 / 34.4 /
// 34.3; with 4 / 8 / 16: ER degree 8 n = 10,000 3.80 / 3.69 / 4.06, n = 30,000 5.74 /
// 5.33 / 5.43, n = 50,000 7.79 / 7.07 / 6.70. Backward 4 below 2^18 vertices and 8 above (a vertex's sums are more work, and
// more warps then have some): ER degree 7 13.5 / 13.4 / 14.1 / 15.2, s16 5.51 / 5.55 /
// 5.90 / 6.24, s20 35.7 / 35.2 / 35.2 / 35.3. BCG_FWD_GRAB / BCG_BWD_GRAB override.
static int env_grab(const char *name) {
  const char *e = std::getenv(name);
  const int v = e ? std::atoi(e) : 0;
  return (v == 1 || v == 2 || v == 4 || v == 8 || v == 16 || v == 32) ? v : 0;
}

static int bwd_grab(int32_t n) {
  static const int env = env_grab("BCG_BWD_GRAB");
  return env ? env : (n >= (1 << 18) ? 8 : 4);
}

static int fwd_grab(int32_t n) {
  static const int env = env_grab("BCG_FWD_GRAB");
  return env ? env : (n >= (1 << 16) ? 16 : n >= (1 << 14) ? 8 : 4);
}

// The context's side stream and its fork / join events, made on first use.
static void side_stream(bc_ctx *ctx) {
  if (ctx->side) return;
  BCG_CUDA(cudaStreamCreateWithFlags(&ctx->side, cudaStreamNonBlocking));
  BCG_CUDA(cudaEventCreateWithFlags(&ctx->ev_fork, cudaEventDisableTiming));
  BCG_CUDA(cudaEventCreateWithFlags(&ctx->ev_join, cudaEventDisableTiming));
}

void batch_ensure(bc_ctx *ctx, const Graph &g) {
  Workspace &ws = ctx->ws;
  const size_t n = (size_t)g.n;
  // as many levels as this graph's batches have had (and 16 for the first),
  // whatever graphs the buffers served before
  ws.lcap = std::max(16, heavy_meta(ctx, g, true).depth + 3);
  ws.lm.ensure((size_t)ws.lcap * n * 8);
  ws.visited.ensure(n * 8);
  ws.sigma.ensure(n * 64 * 8);
  ws.ctl.ensure((size_t)(ws.lcap + 2) * sizeof(LevelCtl));
  ws.vlist.ensure((size_t)ws.lcap * n * 4);
  ws.slist.ensure(2 * n * 4);
  for (bool in : {true, false}) {
    const HeavyMeta &hm = heavy_meta(ctx, g, in);
    ws.hlist.ensure(std::max<size_t>(hm.nseg, 1) * sizeof(int32_t));
    ws.hmulti.ensure(std::max<size_t>(hm.nh, 1) * sizeof(int32_t));
  }
}

// A forward pass whose levels are launched one at a time or, up to the depth of
// the graph's earlier batches, without asking the device in between (a host
// read per level left the GPU idle between levels: R-MAT s16 spent a third of a
// batch that way). Kernels of a level without lanes return at once.
struct Forward {
  bc_ctx *ctx;
  const Graph &g;
  Workspace &ws;
  HeavyMeta &hm;
  size_t n;
  cudaStream_t st;
  int count;
  bool pairs;
  OvfMode mode;
  int l = 0;
  bool heavy_done = false, listed = false, flip = false;
  const int32_t *todo = nullptr;  // light vertices with lanes still to reach
  int todo_level = -1;            // level whose control word counts them (-1: the graph's own list)
  uint64_t fedges = 0ull;         // degree sum of the vertices at level l (direction test)
  int limit = 0x7FFFFFFF;         // levels wanted: vertices farther away may stay unreached

  Forward(bc_ctx *c, const Graph &gr, int cnt, bool pr, OvfMode m)
      : ctx(c), g(gr), ws(c->ws), hm(heavy_meta(c, gr, true)), n((size_t)gr.n), st(c->stream), count(cnt), pairs(pr),
        mode(m) {}
  LevelCtl *ctl(int lev) { return ws.ctl.as<LevelCtl>() + lev; }
  int32_t *lst(int lev) { return ws.vlist.as<int32_t>() + (size_t)lev * n; }
  uint64_t *lm(int lev) { return ws.lm.as<uint64_t>() + (size_t)lev * n; }
  static uint64_t *u64(unsigned long long *p) { return reinterpret_cast<uint64_t *>(p); }
  uint64_t *pinned() { return static_cast<uint64_t *>(ws.pinned); }

  // Level 0, and level 1 straight from the sources' adjacency (heavy sigma rows
  // are cleared before and only receive stores there).
  void init() {
    BCG_CUDA(cudaMemsetAsync(ws.lm.p, 0, 2 * n * 8, st));  // levels 0 and 1
    BCG_CUDA(cudaMemsetAsync(ws.visited.p, 0, n * 8, st));
    BCG_CUDA(cudaMemsetAsync(ws.ctl.p, 0, (size_t)(ws.lcap + 2) * sizeof(LevelCtl), st));
    todo = hm.light.as<int32_t>() + 1;
    if (hm.nh) {
      LaunchScope ls(ctx, F_INIT);
      k_zero_heavy_rows<<<hm.nh, 64, 0, st>>>(hm.nh, hm.heavy.as<int32_t>(), ws.sigma.as<uint64_t>());
    }
    {
      LaunchScope ls(ctx, F_INIT);
      k_batch_init<<<1, 64, 0, st>>>(count, ws.sources.as<int32_t>(), lm(0), ws.visited.as<uint64_t>(),
                                     ws.sigma.as<uint64_t>(), u64(&ctl(0)->active), ws.enable.as<uint64_t>(),
                                     ws.pair_d.as<int32_t>(), ws.pair_sig.as<uint64_t>(), g.rp, lst(0), &ctl(0)->vcnt,
                                     &ctl(0)->vedges);
    }
    ctx->samples += count;
    ctx->batches += 1;
    {
      LaunchScope ls(ctx, F_FWD);
      k_fwd_level1<<<count, 128, 0, st>>>(count, ws.sources.as<int32_t>(), g.rp, g.col, lm(1),
                                          ws.visited.as<uint64_t>(), ws.sigma.as<uint64_t>(), u64(&ctl(1)->active),
                                          ws.cnt.as<unsigned long long>(), lst(1), &ctl(1)->vcnt, &ctl(1)->vedges);
    }
    if (pairs) pair_check(1);
    l = 1;
  }

  void pair_check(int lev) {
    LaunchScope ls(ctx, F_PAIR);
    k_pair_check<<<1, 64, 0, st>>>(count, lev, ws.targets.as<int32_t>(), lm(lev), ws.sigma.as<uint64_t>(),
                                   ws.enable.as<uint64_t>(), ws.pair_d.as<int32_t>(), ws.pair_sig.as<uint64_t>(),
                                   u64(&ctl(lev)->active), ws.enable.as<uint64_t>() + 1);
  }

  void grow() {
    const int ncap = ws.lcap * 2;
    ws.lm.grow_keep((size_t)ncap * n * 8, st);
    ws.vlist.grow_keep((size_t)ncap * n * 4, st);
    ws.ctl.grow_keep((size_t)(ncap + 2) * sizeof(LevelCtl), st);
    BCG_CUDA(cudaMemsetAsync(ctl(ws.lcap + 2), 0, (size_t)(ncap - ws.lcap) * sizeof(LevelCtl), st));
    ws.lcap = ncap;
  }

  // Launches level l -> l + 1; returns whether the heavy kernels ran.
  bool level() {
    if (l + 2 >= ws.lcap) grow();
    const int blocks = grid_blocks();
    const int32_t *prp = g.rp_in, *pcol = g.col_in;
    const bool directions = ctx->push_div > 0;
    // top-down when the level's vertices have few edges (Beamer's direction
    // switch, here on the level's degree sum against the graph's edges)
    const bool push = directions && fedges * (uint64_t)ctx->push_div <= (uint64_t)g.nnz;
    const bool heavy_now = !push && hm.nseg && !heavy_done;
    if (push) listed = false;  // (the list was made for the level after the last heavy one)
    // With heavy work at this level, the heavy vertices' kernels (segments,
    // finisher) run on the side stream beside the light kernel: the two write
    // disjoint rows and read only level l's masks and counts, and the level
    // ends with a join.
    const bool fov = heavy_now && ctx->fwd_overlap;
    if (fov) side_stream(ctx);
    const cudaStream_t hst = fov ? ctx->side : st;
    LevelCtl *cur = ctl(l), *next = ctl(l + 1);
    unsigned long long *ve = directions ? &next->vedges : nullptr;
    unsigned long long *cnt = ws.cnt.as<unsigned long long>();
    uint64_t *visited = ws.visited.as<uint64_t>(), *sigma = ws.sigma.as<uint64_t>(),
             *enable = ws.enable.as<uint64_t>();
    auto heavy_chain = [&] {
      {
        LaunchScope ls(ctx, F_FWD, hst, false);
        k_fwd_heavy<<<std::min(blocks, (hm.nseg + 7) / 8), FWD_THREADS, 0, hst>>>(
            g.n, hm.nseg, listed ? ws.hlist.as<int32_t>() : nullptr, &cur->fseg, hm.seg_v.as<int32_t>(),
            hm.seg_b.as<int32_t>(), hm.seg_e.as<int32_t>(), pcol, lm(l), lm(l + 1), visited, sigma,
            u64(&cur->active), enable, cnt, &cur->q_heavy);
      }
      LaunchScope ls(ctx, F_FWD, hst, false);
      k_fwd_heavy_fin<<<(hm.nh + 255) / 256, 256, 0, hst>>>(
          hm.nh, hm.heavy.as<int32_t>(), hm.hseg0.as<int32_t>(), lm(l + 1), visited, u64(&next->active), cnt, enable,
          &next->hflag, &next->hpend, g.rp, lst(l + 1), &next->vcnt, ve, ws.hlist.as<int32_t>(), &next->fseg);
      listed = true;
    };
    // the level's time on the main stream (after the join) is the family's time
    LaunchScope level_scope(ctx, F_FWD, st, true, false);
    BCG_CUDA(cudaMemsetAsync(lm(l + 1), 0, n * 8, st));
    if (fov) {
      BCG_CUDA(cudaEventRecord(ctx->ev_fork, st));
      BCG_CUDA(cudaStreamWaitEvent(hst, ctx->ev_fork, 0));
      heavy_chain();
    }
    if (push) {
      {
        LaunchScope ls(ctx, F_FWD, st, false);
        k_fwd_push<<<blocks, FWD_THREADS, 0, st>>>(g.rp, g.col, lst(l), &cur->vcnt, lm(l), lm(l + 1), visited,
                                                  u64(&cur->active), enable, lst(l + 1), &next->vcnt, &next->vedges,
                                                  &cur->q_light);
      }
      LaunchScope ls(ctx, F_FWD, st, false);
      k_fwd_pull_list<<<blocks, FWD_THREADS, 0, st>>>(prp, pcol, lst(l + 1), &next->vcnt, lm(l), lm(l + 1), visited,
                                                     sigma, enable, u64(&next->active), cnt, &cur->q_heavy,
                                                     hm.heavy_deg, &next->hflag);
    } else {
      LaunchScope ls(ctx, F_FWD, st, false);
      int32_t *left = ws.slist.as<int32_t>() + (flip ? n : 0);
      flip = !flip;  // (a top-down level in between leaves the list as it is)
      k_fwd_light<<<blocks, FWD_THREADS, 0, st>>>(
          g.n, todo, todo_level < 0 ? hm.light.as<unsigned>() : &ctl(todo_level)->todo, left, &next->todo, prp, pcol,
          lm(l), lm(l + 1), visited, sigma, u64(&cur->active), enable, u64(&next->active), cnt, &cur->q_light,
          lst(l + 1), &next->vcnt, ve, fwd_grab(g.n));
      todo = left;
      todo_level = l + 1;
    }
    if (heavy_now && !fov) heavy_chain();
    if (fov) {
      BCG_CUDA(cudaEventRecord(ctx->ev_join, hst));
      BCG_CUDA(cudaStreamWaitEvent(st, ctx->ev_join, 0));
    }
    return heavy_now;
  }

  // Levels up to the depth of earlier batches, then their control words and
  // the batch's words (largest count, overflowed lanes) on their way to the
  // host. False when the levels have to be asked for one at a time.
  bool blind() {
    if (pairs || ctx->push_div > 0 || hm.depth < 1 || hm.depth > BLIND_DEPTH || hm.depth + 3 > ws.lcap) return false;
    for (; l <= hm.depth; ++l) level();
    uint64_t *h = pinned();
    BCG_CUDA(cudaMemcpyAsync(h, ws.enable.as<uint64_t>() + 2, 16, cudaMemcpyDeviceToHost, st));
    BCG_CUDA(cudaMemcpyAsync(h + 2, ws.ctl.p, (size_t)(l + 1) * sizeof(LevelCtl), cudaMemcpyDeviceToHost, st));
    return true;
  }

  int finished(int last, uint64_t sigmax, uint64_t ovf, const LevelCtl *levels) {
    ws.last_sigmax = sigmax;
    ws.last_ovf = ovf;
    // per level: did any heavy vertex get lanes there (level 1 is filled
    // without the heavy kernels: assume yes; a directed graph's backward splits
    // by out-degree, so its heavy kernels run at every level)
    ws.hlev.assign((size_t)last + 2, 1);
    if (hm.nseg && !g.directed)
      for (int k = 2; k <= last + 1; ++k) ws.hlev[k] = levels[k].hflag != 0u;
    if (ovf && mode == OVF_ERROR) raise_err_bits(ctx, ERR_SIGMA_OVERFLOW);
    if (!pairs) hm.depth = std::max(hm.depth, last);
    return last;
  }

  // After blind(): the deepest level, going on level by level where the batch
  // is deeper than the ones before.
  int end_blind() {
    BCG_CUDA(cudaStreamSynchronize(st));
    const uint64_t *h = pinned();
    const LevelCtl *lv = reinterpret_cast<const LevelCtl *>(h + 2);
    if (lv[l].active == 0ull) {
      int last = l;
      while (last > 0 && lv[last].active == 0ull) --last;
      return finished(last, h[0], h[1], lv);
    }
    return run();
  }

  // Level by level from level l (whose lanes are on) to the end.
  int run() {
    uint64_t *h = pinned();
    for (;; ++l) {
      const bool heavy_now = level();
      // Deep traversals also watch the overflowed lanes every level: once every
      // lane has overflowed the integer pass has nothing left to give (and its
      // per-level masks would only grow).
      const bool watch = mode == OVF_EXTEND && l >= 24;
      if (pairs) pair_check(l + 1);
      BCG_CUDA(cudaMemcpyAsync(h, ws.enable.p, 32, cudaMemcpyDeviceToHost, st));
      BCG_CUDA(cudaMemcpyAsync(h + 4, ctl(l + 1), sizeof(LevelCtl), cudaMemcpyDeviceToHost, st));
      BCG_CUDA(cudaStreamSynchronize(st));
      const LevelCtl &next = *reinterpret_cast<const LevelCtl *>(h + 4);
      const uint64_t cont = pairs ? h[1] : next.active, ovf = watch ? h[3] : 0ull;
      fedges = next.vedges;
      // no heavy vertex is unvisited in a lane that goes on: the heavy kernels
      // have nothing left to do in this batch (the lanes going on only shrink)
      if (heavy_now && (next.hpend & cont) == 0ull) heavy_done = true;
      // stop once every lane still going has overflowed (finished lanes are complete)
      const bool all_ovf = watch && ovf != 0ull && (cont & ~ovf) == 0ull;
      if (!cont || all_ovf || l >= limit) {
        const uint64_t sigmax = h[2], ov = h[3];
        std::vector<LevelCtl> lv((size_t)l + 2);
        if (hm.nseg && !g.directed) {
          BCG_CUDA(cudaMemcpyAsync(lv.data(), ws.ctl.p, lv.size() * sizeof(LevelCtl), cudaMemcpyDeviceToHost, st));
          BCG_CUDA(cudaStreamSynchronize(st));
        }
        return finished(l, sigmax, ov, lv.data());
      }
    }
  }

  // The whole pass, level by level.
  int all() {
    init();
    uint64_t *h = pinned();
    BCG_CUDA(cudaMemcpyAsync(h, ws.enable.p, 16, cudaMemcpyDeviceToHost, st));
    BCG_CUDA(cudaMemcpyAsync(h + 2, ctl(1), sizeof(LevelCtl), cudaMemcpyDeviceToHost, st));
    BCG_CUDA(cudaStreamSynchronize(st));
    const LevelCtl &one = *reinterpret_cast<const LevelCtl *>(h + 2);
    fedges = one.vedges;
    ws.last_ovf = 0ull;
    if (!(pairs ? h[1] : one.active)) {  // no vertex at distance 1 (or, for pairs, every destination found)
      ws.last_sigmax = 1ull;
      ws.hlev.assign(3, 1);
      return pairs ? 1 : 0;
    }
    return run();
  }
};

int batch_forward(bc_ctx *ctx, const Graph &g, int count, bool pairs, OvfMode mode, int limit) {
  batch_ensure(ctx, g);
  Forward f(ctx, g, count, pairs, mode);
  f.limit = limit;
  // (the direction switch needs level 1's degree sum before the first level)
  if (pairs || f.hm.depth < 1 || ctx->push_div > 0) return f.all();
  f.init();
  return f.blind() ? f.end_blind() : f.run();
}

// Whether a heavy vertex has lanes at level l in the last forward pass.
static inline bool heavy_at(const Workspace &ws, int l) { return l >= (int)ws.hlev.size() || ws.hlev[l]; }

void batch_backward(bc_ctx *ctx, const Graph &g, int maxlevel, const Sink &sink, uint64_t keep) {
  Workspace &ws = ctx->ws;
  HeavyMeta &hm = heavy_meta(ctx, g, false);  // successors: the out-CSR
  const size_t n = (size_t)g.n;
  cudaStream_t st = ctx->stream;
  const int blocks = grid_blocks();
  uint64_t *lm = ws.lm.as<uint64_t>();
  // exact sums: 96 bits while the counts and the graph's size allow (a sum of
  // coefficients is delta / sigma < n up to rounding, the per-vertex sums in a
  // ring round at most 32 of them), else 192
  const uint64_t largest = ws.last_sigmax;
  int unit = 52, nlog = 0;
  while (unit < 115 && largest > (1ull << (unit - 52))) ++unit;  // 52 + ceil(log2 of the largest count)
  while (nlog < 31 && (int64_t)g.n > ((int64_t)1 << nlog)) ++nlog;
  bool narrow = unit + nlog + 6 <= 96;
  if (narrow && ws.coef.bytes < n * 768) {  // 768 B per vertex more than the wide form: only where there is room
    size_t fr = 0, tot = 0;
    if (cudaMemGetInfo(&fr, &tot) != cudaSuccess) cudaGetLastError();
    narrow = n * 768 < fr / 2;
  }
  // A level's heavy-segment kernel and its light kernel touch disjoint data
  // (segment partials vs the light vertices' slots; both read only level l+1's
  // coefficients), so the segments run on the side stream beside the light
  // kernel and the finisher joins them: each kernel's tail overlaps the other.
  const bool overlap = ctx->bwd_overlap && hm.nseg;
  if (overlap) side_stream(ctx);
  cudaStream_t sst = overlap ? ctx->side : st;
  // the family's time is the pass's time on the main stream (the side stream's
  // kernels are joined into it): the overlapping launches are counted, not timed
  LaunchScope pass(ctx, F_BWD, st, true, false);
  ws.hpart.ensure(std::max<size_t>(hm.nseg, 1) * 64 * (narrow ? sizeof(Acc3) : sizeof(Acc)));
  uint64_t *coef = ws.sigma.as<uint64_t>();  // wide: in the counts' slots
  Acc3 *recips = nullptr;
  if (narrow) {
    ws.coef.ensure(n * 768);
    ws.recips.ensure(RECIPS * sizeof(Acc3));
    coef = ws.coef.as<uint64_t>();
    recips = ws.recips.as<Acc3>();
    LaunchScope ls(ctx, F_BWD, st, false);
    k_recips<<<RECIPS / 256, 256, 0, st>>>(unit, recips);
  }
  auto run = [&](auto policy) {
    using P = decltype(policy);
    typename P::A *part = ws.hpart.as<typename P::A>();
    for (int l = maxlevel; l >= 1; --l) {
      const bool hv = hm.nseg && heavy_at(ws, l);
      const uint64_t *cur = lm + (size_t)l * n, *next = lm + (size_t)(l + 1) * n;
      LevelCtl *ctl = ws.ctl.as<LevelCtl>() + l;
      if (hv) {
        if (overlap) {
          BCG_CUDA(cudaEventRecord(ctx->ev_fork, st));
          BCG_CUDA(cudaStreamWaitEvent(sst, ctx->ev_fork, 0));
        }
        {
          LaunchScope ls(ctx, F_BWD, sst, false);
          k_bwd_heavy_list<<<(hm.nh + 255) / 256, 256, 0, sst>>>(hm.nh, hm.heavy.as<int32_t>(), hm.hseg0.as<int32_t>(),
                                                                 cur, keep, ws.hlist.as<int32_t>(),
                                                                 ws.hmulti.as<int32_t>(), &ctl->bseg);
        }
        LaunchScope ls(ctx, F_BWD, sst, false);
        k_bwd_heavy_seg<P><<<std::min(blocks, (hm.nseg + 7) / 8), FWD_THREADS, 0, sst>>>(
            ws.hlist.as<int32_t>(), &ctl->bseg, hm.seg_v.as<int32_t>(), hm.seg_b.as<int32_t>(),
            hm.seg_e.as<int32_t>(), g.rp, g.col, cur, next, ws.sigma.as<uint64_t>(), coef, recips, part, sink,
            &ctl->q_bwd_seg, ws.err.as<unsigned>(), keep, unit);
      }
      {
        LaunchScope ls(ctx, F_BWD, st, false);
        k_bwd_light<P><<<blocks, FWD_THREADS, 0, st>>>(
            ws.vlist.as<int32_t>() + (size_t)l * n, &ctl->vcnt, g.rp, g.col, cur, next, ws.sigma.as<uint64_t>(), coef,
            recips, sink, ws.err.as<unsigned>(), &ctl->q_bwd_light, hm.heavy_deg, keep, bwd_grab(g.n), unit);
      }
      if (hv) {
        if (overlap) {
          BCG_CUDA(cudaEventRecord(ctx->ev_join, sst));
          BCG_CUDA(cudaStreamWaitEvent(st, ctx->ev_join, 0));
        }
        LaunchScope ls(ctx, F_BWD, st, false);
        k_bwd_heavy_fin<P><<<std::min(blocks, (hm.nh + 7) / 8), FWD_THREADS, 0, st>>>(
            ws.hmulti.as<int32_t>(), &ctl->bmulti, hm.heavy.as<int32_t>(), hm.hseg0.as<int32_t>(), cur,
            ws.sigma.as<uint64_t>(), coef, recips, part, sink, ws.err.as<unsigned>(), &ctl->q_bwd_fin, keep, unit);
      }
    }
  };
  if (narrow) run(NarrowAcc{});
  else run(WideAcc{});
}

// ---- batches in flight ----

__global__ void k_add_acc(int32_t n, const Acc *__restrict__ from, Acc *__restrict__ to) {
  const int32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  Acc a = to[v];
  acc_add_acc(a, from[v]);
  to[v] = a;
}

// The context's batch state and streams exchanged for the second slot's while
// in scope.
struct SlotScope {
  bc_ctx *ctx;
  bool on;
  SlotScope(bc_ctx *c, bool second) : ctx(c), on(second) {
    if (on) swap();
  }
  ~SlotScope() {
    if (on) swap();
  }
  void swap() {
    std::swap(static_cast<BatchState &>(ctx->ws), ctx->slot2.state);
    std::swap(ctx->stream, ctx->slot2.stream);
    std::swap(ctx->side, ctx->slot2.side);
    std::swap(ctx->ev_fork, ctx->slot2.ev_fork);
    std::swap(ctx->ev_join, ctx->slot2.ev_join);
  }
  SlotScope(const SlotScope &) = delete;
  SlotScope &operator=(const SlotScope &) = delete;
};

// Makes the second slot's state for graph g; false when its memory (about 1.9
// KB per vertex) would take more than a quarter of what is free.
static bool second_slot(bc_ctx *ctx, const Graph &g, bool acc) {
  if (!ctx->batch_overlap) return false;
  BatchSlot &s = ctx->slot2;
  const size_t need = (size_t)g.n * (1900 + (acc ? sizeof(Acc) : 0));
  if (s.state.sigma.bytes < (size_t)g.n * 512) {
    size_t fr = 0, tot = 0;
    if (cudaMemGetInfo(&fr, &tot) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    if (need > fr / 4) return false;
  }
  // (each by itself: a failure here must not pass for a finished slot next time)
  if (!s.stream) BCG_CUDA(cudaStreamCreateWithFlags(&s.stream, cudaStreamNonBlocking));
  for (cudaEvent_t *e : {&s.ev_begin, &s.ev_end})
    if (!*e) BCG_CUDA(cudaEventCreateWithFlags(e, cudaEventDisableTiming));
  if (!s.state.pinned) BCG_CUDA(cudaMallocHost(&s.state.pinned, 4096));
  s.state.enable.ensure(64);
  s.state.sources.ensure(64 * 4);
  if (acc) s.acc.ensure((size_t)g.n * sizeof(Acc));
  return true;
}

// The sources src[0 .. count) (device) in batches of 64 on the lane engine, lane
// t of a batch at column pos[b + t] of the sink (pos may be null). Two batches
// are in flight, each with its own state and stream: while one's forward pass
// runs, the other's backward pass fills the SMs its narrow levels leave idle,
// and the host reads a batch's depth and largest count without the GPU waiting
// for it. The batches write different columns; all-vertex sums are kept per
// slot and added at the end (exact sums: any order).
// ms with one batch at a time and with two: ER n = 100,003 k = 333 5.02 / 3.96,
// R-MAT s16 Bader 1500 draws 13.8 / 11.1, directed s17 k = 512 6.46 / 4.93, s20 k =
// 1024 37.3 / 33.8.
void run_lane_batches(bc_ctx *ctx, const Graph &g, const int32_t *src, const int32_t *pos, int count,
                      const Sink &sink) {
  if (count < 1) return;
  cudaStream_t main = ctx->stream;
  auto batch_sink = [&](int b, bool second) {
    Sink s = sink;
    if (s.tslot && pos) s.lane_col = pos + b;
    if (s.acc && second) s.acc = ctx->slot2.acc.as<Acc>();
    return s;
  };
  auto backward = [&](int maxl, int cnt, const Sink &s) {
    const uint64_t all = lanes_of(cnt), ovf = ctx->ws.last_ovf & all;
    if (ovf != all) batch_backward(ctx, g, maxl, s, all & ~ovf);
    if (ovf) {
      // the extended form's state is not per slot: the other batch waits
      for (cudaStream_t other : {ctx->stream, ctx->slot2.stream})
        if (other) BCG_CUDA(cudaStreamSynchronize(other));
      ext_source_batch(ctx, g, ctx->ws.sources.as<int32_t>(), ovf, s);
      BCG_CUDA(cudaStreamSynchronize(ctx->stream));
    }
  };
  auto load = [&](int b, int cnt) {
    batch_ensure(ctx, g);
    BCG_CUDA(cudaMemcpyAsync(ctx->ws.sources.p, src + b, (size_t)cnt * 4, cudaMemcpyDeviceToDevice, ctx->stream));
  };
  // one batch at a time while the graph's depth is not known, where levels are
  // asked for one by one (a second batch would have nothing to run beside), or
  // where a second batch has no room
  batch_ensure(ctx, g);
  const HeavyMeta &hm = heavy_meta(ctx, g, true);
  auto single = [&](int b) {
    const int cnt = std::min(64, count - b);
    load(b, cnt);
    const int maxl = batch_forward(ctx, g, cnt, false, OVF_EXTEND);
    backward(maxl, cnt, batch_sink(b, false));
  };
  int b0 = 0;
  if (hm.depth < 1) {
    single(0);
    b0 = 64;
  }
  const bool two = count - b0 > 64 && ctx->push_div == 0 && hm.depth >= 1 && hm.depth <= BLIND_DEPTH &&
                   second_slot(ctx, g, sink.acc != nullptr);
  if (!two) {
    for (; b0 < count; b0 += 64) single(b0);
    return;
  }
  BatchSlot &s2 = ctx->slot2;
  BCG_CUDA(cudaEventRecord(s2.ev_begin, main));
  BCG_CUDA(cudaStreamWaitEvent(s2.stream, s2.ev_begin, 0));
  if (sink.acc) BCG_CUDA(cudaMemsetAsync(s2.acc.p, 0, (size_t)g.n * sizeof(Acc), s2.stream));
  struct Flight {
    int b = -1, cnt = 0, l = 0;
    bool asked = false;  // the levels were launched blindly: ask for the outcome
    std::unique_ptr<Forward> f;
  } fl[2];
  auto end = [&](bool second) {
    Flight &f = fl[second];
    if (f.b < 0) return;
    SlotScope sc(ctx, second);
    const int maxl = f.asked ? f.f->end_blind() : f.l;
    backward(maxl, f.cnt, batch_sink(f.b, second));
    f.b = -1;
  };
  try {
    bool second = false;
    for (int b = b0; b < count; b += 64, second = !second) {
      Flight &f = fl[second];
      f.cnt = std::min(64, count - b);
      {
        SlotScope sc(ctx, second);
        load(b, f.cnt);
        f.f.reset(new Forward(ctx, g, f.cnt, false, OVF_EXTEND));
        f.f->init();
        f.asked = f.f->blind();
        if (!f.asked) f.l = f.f->run();
        f.b = b;
      }
      end(!second);
    }
    end(second);
    end(!second);
    BCG_CUDA(cudaEventRecord(s2.ev_end, s2.stream));
    BCG_CUDA(cudaStreamWaitEvent(main, s2.ev_end, 0));
  } catch (...) {
    cudaStreamSynchronize(s2.stream);
    cudaStreamSynchronize(main);
    throw;
  }
  if (sink.acc) {
    LaunchScope ls(ctx, F_MISC);
    k_add_acc<<<(g.n + 255) / 256, 256, 0, main>>>(g.n, s2.acc.as<Acc>(), sink.acc);
  }
}

void batch_extract(bc_ctx *ctx, const Graph &g, int count, int maxlevel, int32_t *dist, uint64_t *sigma,
                   int64_t row_stride, int64_t lane_stride) {
  LaunchScope ls(ctx, F_MISC);
  k_extract<<<(g.n + 255) / 256, 256, 0, ctx->stream>>>(g.n, count, maxlevel, ctx->ws.lm.as<uint64_t>(),
                                                        ctx->ws.sigma.as<uint64_t>(), dist, sigma, row_stride,
                                                        lane_stride);
}

}  // namespace bcg
