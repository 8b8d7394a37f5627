// merge.cu -- the DZS de-refinement (paper Sec. 2.2, Fig. 2; Eq. 3;
// Sec. 2.2.1 geometric criterion with the l_max limit).
//
// GPU formulation of the top-down walk: every octree cell is a run of the
// Morton-sorted particles, and its mass and mass-weighted position are exact
// differences of uint64 prefix sums (masses are integer multiples of m0, so
// the sums are exact in any order).  Each particle walks its own root-to-leaf
// path from the coarsest candidate level j_min (side <= l_max), locating its
// cell by binary search inside the parent's range, and stops at the first
// cell with >= 2 particles that qualifies:
//     d_COM^2 > T_j^2,   T_j = R_lat + b_lat + ceil(l_j / theta_dzs),
// which is l_j / D_n < theta_dzs with D_n = d_COM - R_lc - b (Eq. 3).  Every
// member reaches the same decision, so the walk needs no synchronisation.
// The first member of a merged cell becomes the new particle (mass K, integer
// COM rounded half up, p = (sum k p) / K summed left to right in FP64,
// id = min id); the others are dropped by a stable compaction.
//
// Dynamical criterion (Sec. 2.2.1: Eq. 2 with d replaced by D_n of Eq. 3 and
// |a_old| by the smallest |a| of the particles not yet crossed): merge iff
//     D > 0  and  G M l_j^2 / D^4 < alpha a_min,
//     D = (sqrt(d_COM^2) - (R_lat + b_lat)) L / 2^32,
// every operation a correctly rounded FP64 intrinsic in that order, so the
// decision equals a plain IEEE evaluation bit for bit.  a_min^2 is reduced
// on the device just before the mark pass from the accelerations the state
// carries (the previous step's forces) and the crossing flags of this step.
//
// Steps where little can merge cost little: a level whose T_j is beyond the
// largest possible COM distance (the box corner) is never tested, and with
// the geometric criterion (members must lie beyond R_lat + b_lat) a first
// mark pass sums the few particles of each candidate cell directly; only when
// some candidate cell holds more than kDirect particles are the prefix sums
// built and those candidates marked again from them (same decisions: the sums
// are exact either way).  The compaction writes only from the first particle
// that changes, into the spare arrays, and copies that tail back: a step that
// merges nothing writes nothing.
#include <cmath>
#include <type_traits>

#include "common.cuh"

namespace dzs {
namespace {

constexpr int kChunk = 1024;
constexpr int kDirect = 64;              // largest cell the first mark pass sums directly
constexpr int32_t kDeferred = INT32_MIN;  // mend of a candidate left to the prefix pass

struct MergeParams {
  uint64_t thr[kMaxLevel + 1];  // T_j (UINT64_MAX: level never merges)
  uint64_t rb2;                 // (R_lat + b_lat)^2: members must lie beyond
  int jmin;
  int jstart;                   // first level that can merge (>= max(jmin, 1))
  int filter;                   // 1 when theta_dzs <= 1/sqrt(3) (geometric only)
  int criterion;                // DZS_CRIT_GEOMETRIC / DZS_CRIT_DYNAMICAL
  double rb;                    // R_lat + b_lat (dynamical)
  uint64_t rbl;                 // the same as an integer
  double scale;                 // L / 2^32
  double gm0;                   // G m0 = 1.5 Omega_m L^3 / (4 pi N0)
  double alpha;                 // alpha of Eq. 2
  double l2[kMaxLevel + 1];     // (L / 2^j)^2
  const uint64_t* amin2_slot;   // ~bits of a_min^2 (0: no particle inside)
};

// a_min^2 = min over particles not yet crossed of |g|^2, FP64 without
// contraction.  Non-negative doubles order like their bit patterns, so the
// minimum is an integer max over the complemented bits (slot zeroed before).
template <class R>
__global__ void k_amin2(const int32_t* __restrict__ d_n, int64_t cap, const R* __restrict__ g,
                        const uint8_t* __restrict__ fl, unsigned long long* __restrict__ slot) {
  const int64_t n = *d_n;
  unsigned long long best = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    if (fl[i] & kFlCrossed) continue;
    double gx = (double)g[i], gy = (double)g[cap + i], gz = (double)g[2 * cap + i];
    double a2 = __dadd_rn(__dadd_rn(__dmul_rn(gx, gx), __dmul_rn(gy, gy)), __dmul_rn(gz, gz));
    if (!(a2 == a2)) continue;  // NaN never wins the minimum
    unsigned long long c = ~(unsigned long long)__double_as_longlong(a2);
    best = c > best ? c : best;
  }
  for (int o = 16; o > 0; o >>= 1) {
    unsigned long long t = __shfl_down_sync(0xffffffffu, best, o);
    best = t > best ? t : best;
  }
  __shared__ unsigned long long wbest[32];
  if ((threadIdx.x & 31) == 0) wbest[threadIdx.x >> 5] = best;
  __syncthreads();
  if (threadIdx.x < 32) {
    best = threadIdx.x < (blockDim.x >> 5) ? wbest[threadIdx.x] : 0ull;
    for (int o = 16; o > 0; o >>= 1) {
      unsigned long long t = __shfl_down_sync(0xffffffffu, best, o);
      best = t > best ? t : best;
    }
    if (threadIdx.x == 0 && best) atomicMax(slot, best);  // one atomic per block
  }
}

__device__ __forceinline__ bool dynamical_merge(const MergeParams& mp, uint64_t d2, uint64_t K, int j,
                                                double rhs) {
  double D = __dmul_rn(__dsub_rn(__dsqrt_rn((double)d2), mp.rb), mp.scale);
  if (!(D > 0.0)) return false;
  double D2 = __dmul_rn(D, D);
  double lhs = __ddiv_rn(__dmul_rn(__dmul_rn(mp.gm0, (double)K), mp.l2[j]), __dmul_rn(D2, D2));
  return lhs < rhs;
}

// ---- 4-channel uint64 exclusive prefix sums: k, k ux, k uy, k uz
__global__ void k_prefix_totals(const int32_t* __restrict__ d_n, int64_t cap, const uint32_t* __restrict__ u,
                                const uint32_t* __restrict__ k, uint64_t* __restrict__ tot,
                                const unsigned* __restrict__ need) {
  if (need && !*need) return;
  const int64_t n = *d_n;
  int64_t base = (int64_t)blockIdx.x * kChunk;
  unsigned long long s[4] = {0, 0, 0, 0};
  for (int t = threadIdx.x; t < kChunk; t += blockDim.x) {
    int64_t i = base + t;
    if (i < n) {
      uint64_t kk = k[i];
      s[0] += kk;
      for (int ax = 0; ax < 3; ++ax) s[1 + ax] += kk * u[ax * cap + i];
    }
  }
  for (int q = 0; q < 4; ++q) {
    for (int o = 16; o > 0; o >>= 1) s[q] += __shfl_down_sync(0xffffffffu, s[q], o);
  }
  __shared__ unsigned long long ws[4][32];
  if ((threadIdx.x & 31) == 0)
    for (int q = 0; q < 4; ++q) ws[q][threadIdx.x >> 5] = s[q];
  __syncthreads();
  if (threadIdx.x < 4) {
    unsigned long long a = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) a += ws[threadIdx.x][w];
    tot[(int64_t)threadIdx.x * (gridDim.x + 1) + blockIdx.x] = a;
  }
}

// block c scans row c (channel c) of the chunk totals, 1024 at a time
__global__ void k_prefix_scan_totals(uint64_t* __restrict__ tot, int nchunks, const unsigned* __restrict__ need) {
  if (need && !*need) return;
  __shared__ unsigned long long woff[32];
  __shared__ unsigned long long carry, block_total;
  uint64_t* row = tot + (int64_t)blockIdx.x * (nchunks + 1);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int base = 0; base < nchunks; base += blockDim.x) {
    int i = base + threadIdx.x;
    unsigned long long v = i < nchunks ? row[i] : 0ull, inc = v;
    for (int o = 1; o < 32; o <<= 1) {
      unsigned long long t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    if (lane == 31) woff[w] = inc;
    __syncthreads();
    if (w == 0) {
      unsigned long long t = lane < nw ? woff[lane] : 0ull, ti = t;
      for (int o = 1; o < 32; o <<= 1) {
        unsigned long long q = __shfl_up_sync(0xffffffffu, ti, o);
        if (lane >= o) ti += q;
      }
      if (lane < nw) woff[lane] = ti - t;
      if (lane == nw - 1) block_total = ti;
    }
    __syncthreads();
    if (i < nchunks) row[i] = carry + woff[w] + inc - v;
    __syncthreads();
    if (threadIdx.x == 0) carry += block_total;
    __syncthreads();
  }
  if (threadIdx.x == 0) row[nchunks] = carry;
}

__global__ void k_prefix_apply(const int32_t* __restrict__ d_n, int64_t cap, const uint32_t* __restrict__ u,
                               const uint32_t* __restrict__ k, const uint64_t* __restrict__ tot, int nchunks,
                               uint64_t* __restrict__ pre, const unsigned* __restrict__ need) {
  if (need && !*need) return;
  const int64_t n = *d_n;
  int64_t base = (int64_t)blockIdx.x * kChunk;
  if (base > n) return;
  // thread t owns items base + 4t .. base + 4t + 3
  int64_t i0 = base + 4 * threadIdx.x;
  unsigned long long v[4][4], s[4] = {0, 0, 0, 0};
  for (int q = 0; q < 4; ++q) {
    int64_t i = i0 + q;
    uint64_t kk = (i < n) ? k[i] : 0;
    v[0][q] = kk;
    for (int ax = 0; ax < 3; ++ax) v[1 + ax][q] = (i < n) ? kk * u[ax * cap + i] : 0;
    for (int c = 0; c < 4; ++c) s[c] += v[c][q];
  }
  // block exclusive scan per channel (warp shuffles + warp totals)
  __shared__ unsigned long long wt[4][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  unsigned long long inc[4];
  for (int c = 0; c < 4; ++c) {
    inc[c] = s[c];
    for (int o = 1; o < 32; o <<= 1) {
      unsigned long long t = __shfl_up_sync(0xffffffffu, inc[c], o);
      if (lane >= o) inc[c] += t;
    }
    if (lane == 31) wt[c][w] = inc[c];
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    unsigned long long a = 0;
    for (int q = 0; q < nw; ++q) {
      unsigned long long t = wt[threadIdx.x][q];
      wt[threadIdx.x][q] = a;
      a += t;
    }
  }
  __syncthreads();
  for (int c = 0; c < 4; ++c) {
    unsigned long long run = tot[(int64_t)c * (nchunks + 1) + blockIdx.x] + wt[c][w] + inc[c] - s[c];
    for (int q = 0; q < 4; ++q) {
      int64_t i = i0 + q;
      if (i <= n) pre[(int64_t)c * (cap + 1) + i] = run;
      run += v[c][q];
    }
  }
}

__device__ __forceinline__ int64_t lower_bound_key(const uint64_t* __restrict__ key, int64_t lo, int64_t hi,
                                                   uint64_t x) {
  while (lo < hi) {
    int64_t mid = (lo + hi) >> 1;
    if (key[mid] < x)
      lo = mid + 1;
    else
      hi = mid;
  }
  return lo;
}

// mend[i]: end of the merged run if i leads one, -1 if i is merged away, 0 if kept
// first index s <= i with key[s] >= x, given key[i] >= x: exponential steps
// down from i, then a binary search of the last step (cost ~2 log2(i - s))
__device__ __forceinline__ int64_t gallop_down(const uint64_t* __restrict__ key, int64_t i, uint64_t x) {
  int64_t hi = i, lo = 0;
  for (int64_t step = 1;; step <<= 1) {
    const int64_t p = i - step;
    if (p < 0) break;
    if (key[p] < x) {
      lo = p + 1;
      break;
    }
    hi = p;
  }
  return lower_bound_key(key, lo, hi + 1, x);
}

// first index >= i1 with key >= x (or n), given key[i1 - 1] < x
__device__ __forceinline__ int64_t gallop_up(const uint64_t* __restrict__ key, int64_t i1, int64_t n, uint64_t x) {
  int64_t lo = i1, hi = n;
  for (int64_t step = 1;; step <<= 1) {
    const int64_t p = i1 - 1 + step;
    if (p >= n) break;
    if (key[p] >= x) {
      hi = p;
      break;
    }
    lo = p + 1;
  }
  return lower_bound_key(key, lo, hi, x);
}

// particles of one block of the mark and write kernels: consecutive, so that
// the blocks' survivor counts give every survivor its place
__device__ __forceinline__ int64_t block_share(int64_t n) {
  return ((n + gridDim.x - 1) / gridDim.x + kThreads - 1) / kThreads * kThreads;
}

// this block's survivors to kept[block]; the smallest index with a nonzero mark
// (as its complement: 0 when there is none) and whether any candidate was
// deferred, one atomic each per block
__device__ __forceinline__ void block_result(int64_t first, bool deferred, unsigned kept,
                                             int32_t* __restrict__ block_kept,
                                             unsigned long long* __restrict__ first_slot, unsigned* __restrict__ need) {
  __shared__ unsigned long long wmax[32];
  __shared__ int wdef[32];
  __shared__ unsigned wkept[32];
  unsigned long long f = ~(unsigned long long)first;  // none: INT64_MAX, the smallest complement
  if (first == INT64_MAX) f = 0;
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long t = __shfl_down_sync(0xffffffffu, f, o);
    f = t > f ? t : f;
    kept += __shfl_down_sync(0xffffffffu, kept, o);
  }
  const int d = __any_sync(0xffffffffu, deferred) ? 1 : 0;
  if ((threadIdx.x & 31) == 0) {
    wmax[threadIdx.x >> 5] = f;
    wdef[threadIdx.x >> 5] = d;
    wkept[threadIdx.x >> 5] = kept;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long m = 0;
    int any = 0;
    unsigned sum = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      m = wmax[w] > m ? wmax[w] : m;
      any |= wdef[w];
      sum += wkept[w];
    }
    block_kept[blockIdx.x] = (int32_t)sum;
    if (m) atomicMax(first_slot, m);
    if (any && need) atomicOr(need, 1u);
  }
}

// first changed particle, n when there is none
__device__ __forceinline__ int64_t first_of(const unsigned long long* __restrict__ slot, int64_t n) {
  const unsigned long long f = *slot;
  return f && (int64_t)~f < n ? (int64_t)~f : n;
}

// A level whose cells cannot qualify for particle i needs no bounds: the COM lies
// in i's cell, so d_COM <= d_i + sqrt(3) l_j, and while that is at most T_j
// (dynamical: R_lat + b_lat, and then for every finer level too) the cell does
// not merge.  FP32, rounded to the safe side: reach(j) overestimates d_COM by
// less than 2^-20, `most` underestimates the bound.
__device__ __forceinline__ bool cannot_reach(float di, int j, uint64_t bound) {
  const float side = __int_as_float((127 + 32 - j) << 23);  // 2^(32 - j)
  return (di + 1.7320509f * side) * (1.0f + 0x1p-20f) <= (float)bound * (1.0f - 0x1p-20f);
}

// kPrefix false: the first pass over every particle (geometric criterion with
// the member filter): candidates whose cells at the levels that can merge hold
// at most kDirect particles are decided from direct sums, the others deferred.
// kPrefix true (only when something was deferred, or without the filter):
// the deferred particles (every particle without the filter) are decided from
// the prefix sums.
template <bool kPrefix>
__global__ void k_merge_mark(const int32_t* __restrict__ d_n, int64_t cap, const uint64_t* __restrict__ key,
                             const uint32_t* __restrict__ u, const uint32_t* __restrict__ kk,
                             const uint64_t* __restrict__ pre, int32_t* __restrict__ mend,
                             int32_t* __restrict__ block_kept, MergeParams mp,
                             unsigned long long* __restrict__ first_slot, unsigned* __restrict__ need) {
  if (kPrefix && need && !*need) return;
  const int64_t n = *d_n;
  const uint64_t* PK = pre;
  const uint64_t* PS = pre + (cap + 1);
  double rhs = 0.0;  // alpha a_min (dynamical)
  if (mp.criterion == DZS_CRIT_DYNAMICAL) {
    uint64_t c = *mp.amin2_slot;
    double amin2 = c ? __longlong_as_double((long long)~c) : __longlong_as_double(0x7ff0000000000000ll);
    rhs = __dmul_rn(mp.alpha, __dsqrt_rn(amin2));
  }
  int64_t first = INT64_MAX;
  bool deferred_any = false;
  unsigned kept = 0;
  const int64_t share = block_share(n), b0 = blockIdx.x * share, b1 = b0 + share < n ? b0 + share : n;
  for (int64_t i = b0 + threadIdx.x; i < b1; i += kThreads) {
    if (kPrefix && mp.filter) {
      const int32_t m = mend[i];
      if (m != kDeferred) {
        kept += m >= 0 ? 1u : 0u;
        continue;
      }
    }
    int32_t res = 0;
    bool deferred = false;
    bool cand = true;
    const uint64_t d2i = dist2_obs(u[i], u[cap + i], u[2 * cap + i]);
    if (mp.filter) cand = d2i > mp.rb2;
    if (cand) {
      uint64_t ki = key[i];
      // from the first level that can qualify: bounds by galloping out from i
      // (the coarser cells only contain it), deeper ones inside the previous
      int j0 = mp.jstart;
      const float di = sqrtf((float)d2i);
      if (mp.criterion == DZS_CRIT_GEOMETRIC)
        while (j0 <= kMaxLevel && (mp.thr[j0] == ~0ull || cannot_reach(di, j0, mp.thr[j0]))) ++j0;
      int64_t lo = 0, hi = n;
      for (int j = j0; j <= kMaxLevel; ++j) {
        if (mp.criterion == DZS_CRIT_DYNAMICAL && cannot_reach(di, j, mp.rbl)) break;
        int sh = 3 * (kMaxLevel - j);
        uint64_t cell = (ki >> sh) << sh;
        int64_t s, e;
        if (j == j0) {
          s = gallop_down(key, i, cell);
          e = gallop_up(key, i + 1, n, cell + (1ull << sh));
        } else {
          s = lower_bound_key(key, lo, i + 1, cell);
          e = lower_bound_key(key, i + 1, hi, cell + (1ull << sh));
        }
        lo = s;
        hi = e;
        if (e - s < 2) break;  // no finer cell holds two particles
        if (mp.criterion == DZS_CRIT_GEOMETRIC && mp.thr[j] == ~0ull) continue;
        uint64_t K = 0, S[3] = {0, 0, 0};
        if (kPrefix) {
          K = PK[e] - PK[s];
          for (int ax = 0; ax < 3; ++ax)
            S[ax] = PS[(int64_t)ax * (cap + 1) + e] - PS[(int64_t)ax * (cap + 1) + s];
        } else {
          if (e - s > kDirect) {
            deferred = true;
            break;
          }
          for (int64_t t = s; t < e; ++t) {
            const uint64_t m = kk[t];
            K += m;
            for (int ax = 0; ax < 3; ++ax) S[ax] += m * u[ax * cap + t];
          }
        }
        uint64_t d2 = 0;
        for (int ax = 0; ax < 3; ++ax) {
          uint32_t com = (uint32_t)((2 * S[ax] + K) / (2 * K));
          int64_t off = (int32_t)(com - 0x80000000u);
          d2 += (uint64_t)(off * off);
        }
        bool merge;
        if (mp.criterion == DZS_CRIT_DYNAMICAL) {
          merge = dynamical_merge(mp, d2, K, j, rhs);
        } else {
          uint64_t T = mp.thr[j];
          merge = d2 > T * T;
        }
        if (merge) {
          res = (s == i) ? (int32_t)e : -1;
          break;
        }
      }
    }
    mend[i] = deferred ? kDeferred : res;
    kept += !deferred && res >= 0 ? 1u : 0u;
    if (res != 0 && i < first) first = i;
    deferred_any = deferred_any || deferred;
  }
  block_result(first, deferred_any, kept, block_kept, first_slot, need);
}

// the compacted state from the first changed particle on, into the spare
// arrays (place = survivors of the blocks before, then in the block); merged
// cells summed directly; *d_n_out = survivors
template <class R>
__global__ void __launch_bounds__(kThreads)
    k_merge_write(const int32_t* __restrict__ d_n, int64_t cap, const int32_t* __restrict__ mend,
                              const int32_t* __restrict__ block_kept, const uint64_t* __restrict__ key,
                              const uint32_t* __restrict__ u, const R* __restrict__ p,
                              const uint32_t* __restrict__ k, const uint32_t* __restrict__ id,
                              const uint8_t* __restrict__ fl, const unsigned long long* __restrict__ first_slot,
                              uint64_t* __restrict__ key2, uint32_t* __restrict__ u2, R* __restrict__ p2,
                              uint32_t* __restrict__ k2, uint32_t* __restrict__ id2, uint8_t* __restrict__ fl2,
                              int32_t* __restrict__ d_n_out) {
  __shared__ unsigned wsum[kThreads / 32];
  const int64_t n = *d_n;
  const int64_t first = first_of(first_slot, n);
  const int64_t share = block_share(n), b0 = blockIdx.x * share, b1 = b0 + share < n ? b0 + share : n;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const bool last = blockIdx.x == gridDim.x - 1;
  if (b1 <= first && !last) return;  // nothing of this block changes
  unsigned before = 0;
  for (int q = threadIdx.x; q < (int)blockIdx.x; q += kThreads) before += (unsigned)block_kept[q];
  for (int o = 16; o > 0; o >>= 1) before += __shfl_down_sync(0xffffffffu, before, o);
  if (lane == 0) wsum[w] = before;
  __syncthreads();
  before = 0;
  for (int q = 0; q < kThreads / 32; ++q) before += wsum[q];
  if (last && threadIdx.x == 0) *d_n_out = (int32_t)before + block_kept[blockIdx.x];
  if (b1 <= first) return;
  for (int64_t i0 = b0; i0 < b1; i0 += kThreads) {
    const int64_t i = i0 + threadIdx.x;
    const int32_t m = i < b1 ? mend[i] : -1;
    const unsigned bal = __ballot_sync(0xffffffffu, m >= 0);
    __syncthreads();
    if (lane == 0) wsum[w] = __popc(bal);
    __syncthreads();
    int64_t j = before + __popc(bal & ((1u << lane) - 1u));
    for (int q = 0; q < kThreads / 32; ++q) {
      if (q < w) j += wsum[q];
      before += wsum[q];
    }
    if (m < 0 || i < first) continue;
    if (m == 0) {
      for (int ax = 0; ax < 3; ++ax) {
        u2[ax * cap + j] = u[ax * cap + i];
        p2[ax * cap + j] = p[ax * cap + i];
      }
      key2[j] = key[i];
      k2[j] = k[i];
      id2[j] = id[i];
      fl2[j] = fl[i];
      continue;
    }
    // one pass, the loads of four members in flight: the kernel waits for the chain
    // of loads of its largest cell (merge stage of a late 128^3 state, a pass each
    // for mass, axes and id 152 us, now 141)
    const int64_t e = m;
    uint64_t K = 0, S[3] = {0, 0, 0};
    double acc[3] = {0.0, 0.0, 0.0};  // left-to-right FP64 sums, no contraction
    uint32_t idm = id[i];
#pragma unroll 4
    for (int64_t t = i; t < e; ++t) {
      const uint32_t kt = k[t];
      K += kt;
      idm = min(idm, id[t]);
      for (int ax = 0; ax < 3; ++ax) {
        S[ax] += (uint64_t)kt * u[ax * cap + t];
        acc[ax] = __dadd_rn(acc[ax], __dmul_rn((double)kt, (double)p[ax * cap + t]));
      }
    }
    uint32_t com[3];
    for (int ax = 0; ax < 3; ++ax) {
      com[ax] = (uint32_t)((2 * S[ax] + K) / (2 * K));
      u2[ax * cap + j] = com[ax];
      p2[ax * cap + j] = (R)(acc[ax] / (double)K);
    }
    key2[j] = morton_key(com[0], com[1], com[2]);
    k2[j] = (uint32_t)K;
    id2[j] = idm;
    fl2[j] = (uint8_t)(kFlMerged | kFlCrossed);
  }
}

// the changed tail [first, n_new) back into the state arrays; the block that
// finishes last (all have read the slots) sets the count and clears the slots
// for the next merge
template <class R>
__global__ void k_merge_copyback(int32_t* d_n, int64_t cap, unsigned long long* first_slot, unsigned* need,
                                 unsigned* done, const uint64_t* __restrict__ key2,
                                 const uint32_t* __restrict__ u2, const R* __restrict__ p2,
                                 const uint32_t* __restrict__ k2, const uint32_t* __restrict__ id2,
                                 const uint8_t* __restrict__ fl2, uint64_t* __restrict__ key, uint32_t* __restrict__ u,
                                 R* __restrict__ p, uint32_t* __restrict__ k, uint32_t* __restrict__ id,
                                 uint8_t* __restrict__ fl) {
  const int64_t n = d_n[1];
  const int64_t first = first_of(first_slot, n);
  for (int64_t i = first + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    for (int ax = 0; ax < 3; ++ax) {
      u[ax * cap + i] = u2[ax * cap + i];
      p[ax * cap + i] = p2[ax * cap + i];
    }
    key[i] = key2[i];
    k[i] = k2[i];
    id[i] = id2[i];
    fl[i] = fl2[i];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(done, 1u) == gridDim.x - 1) {
      d_n[0] = (int32_t)n;
      *first_slot = 0;
      *need = 0;
      *done = 0;
    }
  }
}

}  // namespace

void launch_mass_prefix(dzs_ctx* c) {
  c->launches += 3;
  Buffers& B = c->B;
  const int nchunks = (int)((c->cap + kChunk) / kChunk);
  uint64_t* tot = (uint64_t*)B.blocksum;
  k_prefix_totals<<<nchunks, 256, 0, c->stream>>>(B.n, c->cap, B.u, B.k, tot, nullptr);
  k_prefix_scan_totals<<<4, 1024, 0, c->stream>>>(tot, nchunks, nullptr);
  k_prefix_apply<<<nchunks, 256, 0, c->stream>>>(B.n, c->cap, B.u, B.k, tot, nchunks, B.prefix, nullptr);
}

void launch_amin2(dzs_ctx* c) {
  c->launches += 1;
  Buffers& B = c->B;
  unsigned long long* slot = (unsigned long long*)(B.counters + 14);
  cudaMemsetAsync(slot, 0, sizeof(uint64_t), c->stream);
  int grid = grid_for(c->N0);
  if (c->fp64)
    k_amin2<double><<<grid, kThreads, 0, c->stream>>>(B.n, c->cap, (const double*)B.g, B.fl, slot);
  else
    k_amin2<float><<<grid, kThreads, 0, c->stream>>>(B.n, c->cap, (const float*)B.g, B.fl, slot);
  c->amin2_ready = true;
}

// the dynamical criterion reads a_min^2 from counters[14] (launch_amin2 first)
void launch_merge(dzs_ctx* c, uint64_t rlat) {
  const bool dyn = c->P.dzs_criterion == DZS_CRIT_DYNAMICAL;
  Buffers& B = c->B;
  MergeParams mp;
  // a COM offset from the observer is below 2^31 per axis: d^2 <= 3 * 2^62,
  // so a level with T_j^2 >= 3 * 2^62 never merges
  const uint64_t d2max = 3ull << 62;
  for (int j = 0; j <= kMaxLevel; ++j) {
    uint64_t t = (c->merge_thr[j] == ~0ull) ? ~0ull : rlat + c->merge_thr[j];
    if (t != ~0ull && (t >= 4294967296ull || t * t >= d2max)) t = ~0ull;
    mp.thr[j] = t;
  }
  uint64_t rb = rlat + c->blat;
  mp.rb2 = (rb >= 4294967296ull) ? ~0ull : rb * rb;
  mp.jmin = c->jmin;
  mp.jstart = c->jmin > 1 ? c->jmin : 1;
  if (!dyn)
    while (mp.jstart <= kMaxLevel && mp.thr[mp.jstart] == ~0ull) ++mp.jstart;
  mp.filter = (!dyn && c->P.theta_dzs <= 0.5773502691896257) ? 1 : 0;
  mp.criterion = c->P.dzs_criterion;
  mp.rb = (double)rb;
  mp.rbl = rb;
  mp.scale = c->scale;
  mp.gm0 = c->gm0;
  mp.alpha = c->P.alpha_dyn;
  for (int j = 0; j <= kMaxLevel; ++j) {
    double l = std::ldexp(c->P.box, -j);
    mp.l2[j] = l * l;
  }
  uint64_t* slot = c->B.counters + 14;
  mp.amin2_slot = slot;
  // zero between merges (the last block of the copy-back clears them)
  unsigned long long* first = (unsigned long long*)(c->B.counters + 22);
  unsigned* need = (unsigned*)(c->B.counters + 23);
  unsigned* done = (unsigned*)(c->B.counters + 17);
  int nchunks = (int)((c->cap + kChunk) / kChunk);
  uint64_t* tot = (uint64_t*)B.blocksum;
  int32_t* kept = B.iscan;  // survivors of each block
  const int grid = grid_for(c->cap);
  c->launches += mp.filter ? 7 : 6;
  if (mp.filter)
    k_merge_mark<false><<<grid, kThreads, 0, c->stream>>>(B.n, c->cap, B.key, B.u, B.k, B.prefix, B.mend, kept, mp,
                                                          first, need);
  // prefix sums and the second mark pass: they return at once unless needed
  // (without the filter every particle takes them)
  unsigned* when = mp.filter ? need : nullptr;
  k_prefix_totals<<<nchunks, 256, 0, c->stream>>>(B.n, c->cap, B.u, B.k, tot, when);
  k_prefix_scan_totals<<<4, 1024, 0, c->stream>>>(tot, nchunks, when);
  k_prefix_apply<<<nchunks, 256, 0, c->stream>>>(B.n, c->cap, B.u, B.k, tot, nchunks, B.prefix, when);
  k_merge_mark<true><<<grid, kThreads, 0, c->stream>>>(B.n, c->cap, B.key, B.u, B.k, B.prefix, B.mend, kept, mp, first,
                                                       when);
  auto finish = [&](auto* p, auto* p2) {
    using R = std::remove_pointer_t<decltype(p)>;
    k_merge_write<R><<<grid, kThreads, 0, c->stream>>>(B.n, c->cap, B.mend, kept, B.key, B.u, p, B.k, B.id, B.fl, first,
                                                       B.key2, B.u2, p2, B.k2, B.id2, B.fl2, B.n + 1);
    k_merge_copyback<R><<<grid, kThreads, 0, c->stream>>>(B.n, c->cap, first, need, done, B.key2, B.u2, p2, B.k2, B.id2,
                                                          B.fl2, B.key, B.u, p, B.k, B.id, B.fl);
  };
  if (c->fp64)
    finish((double*)B.p, (double*)B.p2);
  else
    finish((float*)B.p, (float*)B.p2);
}

}  // namespace dzs
