// fof.cu -- friends-of-friends haloes on the GPU (paper Sec. 3.1.1: the
// lightcone halo mass function is built from FoF catalogues of frequent
// outputs, keeping the haloes entirely inside the lightcone).
//
// Friends: minimum-image lattice distance d^2 <= T, T = floor((link 2^32 /
// n1d)^2) (link in units of the initial mean spacing).  On the Morton-sorted
// particles, cells of a depth whose side is at least the linking length are
// contiguous runs (CSR table); each particle scans the 27 neighbour cells and
// unites itself with every later friend.  Union-find without locks: a root is
// only ever hooked under a smaller index (one compare-and-swap; a failed swap
// means another thread changed that root, so the union retries with the new
// roots), so every component ends with its smallest sorted index as root,
// whatever the schedule.  Three things keep unions rare, because a union costs
// two chains of dependent L2 reads that diverge across a warp: the particles
// of a cell whose diagonal is within the linking length start as one tree
// (all are friends), a pair whose later member already points at the scanning
// particle's root is passed over before its distance is formed, and a union
// leaves both members pointing at the root.  2.1M particles with haloes of up
// to 512, link 0.2: k_fof_link 8.66 -> 5.34 ms, and with a warp per particle
// (below) -> 0.94 ms.  Per component, exact integer sums: count, mass,
// mass-weighted offsets from the member with the smallest caller-order index
// (the halo's label), the largest squared distance from the observer.
#include <cmath>

#include "common.cuh"

namespace dzs {
namespace {

constexpr int kUnionTries = 1 << 20;  // a union gives up (error bit) after this many retries

__device__ __forceinline__ int32_t uf_find(const int32_t* par, int32_t x) {
  // parents only ever decrease, so the chain ends at the root
  int32_t p = ((volatile const int32_t*)par)[x];
  while (p != x) {
    x = p;
    p = ((volatile const int32_t*)par)[x];
  }
  return x;
}

// unites the trees of a and b and returns the root it left them under; the
// callers' entries are pointed at it (an entry that is no root never becomes
// one again, and parents only move to ancestors, so the stores need no order)
__device__ __forceinline__ int32_t uf_union(int32_t* par, int32_t a0, int32_t b0, uint32_t* err) {
  int32_t a = a0, b = b0;
  for (int t = 0; t < kUnionTries; ++t) {
    a = uf_find(par, a);
    b = uf_find(par, b);
    if (a > b) {
      const int32_t s = a;
      a = b;
      b = s;
    }
    if (a == b || atomicCAS(&par[b], b, a) == b) {
      if (a0 != a) par[a0] = a;
      if (b0 != a) par[b0] = a;
      return a;
    }
  }
  atomicOr(err, kErrGroups);
  return a;
}

// first particle of i's run of equal key >> sh: steps down doubling, then a
// binary search
__device__ __forceinline__ int64_t run_first(const uint64_t* __restrict__ key, int64_t i, int sh) {
  const uint64_t cell = key[i] >> sh;
  int64_t hi = i, lo = 0;  // key[hi] is in the run; the first is in [lo, hi]
  for (int64_t step = 1;; step <<= 1) {
    const int64_t p = i - step;
    if (p < 0) break;
    if ((key[p] >> sh) != cell) {
      lo = p + 1;
      break;
    }
    hi = p;
  }
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if ((key[mid] >> sh) == cell)
      hi = mid;
    else
      lo = mid + 1;
  }
  return lo;
}

// fine: key shift of the cells whose members are all friends (-1: none)
__global__ void k_fof_init(const int32_t* __restrict__ d_n, const uint64_t* __restrict__ key, int fine,
                           int32_t* __restrict__ par, int32_t* __restrict__ cnt,
                           unsigned long long* __restrict__ mass, unsigned long long* __restrict__ rmax2,
                           int32_t* __restrict__ first, const uint32_t* __restrict__ idx, int32_t* __restrict__ inv,
                           unsigned long long* __restrict__ S) {
  const int64_t n = *d_n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    par[i] = fine >= 0 ? (int32_t)run_first(key, i, fine) : (int32_t)i;
    cnt[i] = 0;
    mass[i] = 0;
    rmax2[i] = 0;
    first[i] = 0x7fffffff;
    inv[idx[i]] = (int32_t)i;  // caller order -> sorted position
    S[i] = S[n + i] = S[2 * n + i] = 0;
  }
}

// d^2 <= T: FP32 decides unless within 2^-20 of T (its error is below 2^-21)
__device__ __forceinline__ bool friends(uint32_t x, uint32_t y, uint32_t z, uint64_t T, float Tlo, float Thi) {
  const int32_t dx = (int32_t)x, dy = (int32_t)y, dz = (int32_t)z;
  const float fx = (float)dx, fy = (float)dy, fz = (float)dz;
  const float d2 = fmaf(fx, fx, fmaf(fy, fy, fz * fz));
  if (d2 <= Tlo) return true;
  if (d2 >= Thi) return false;
  return (uint64_t)((int64_t)dx * dx) + (uint64_t)((int64_t)dy * dy) + (uint64_t)((int64_t)dz * dz) <= T;
}

// a warp per particle: 27 lanes look the neighbour cells up at once, then the
// later particles of those cells are taken 32 at a time (a lane finds its
// candidate's cell in the scanned lengths).  A thread per particle ran three
// lanes of 32: beside an empty cell of one lane lies a halo of another.
__global__ void __launch_bounds__(kThreads) k_fof_link(const int32_t* __restrict__ d_n, int64_t cap,
                                                       const uint32_t* __restrict__ u,
                                                       const int32_t* __restrict__ start, int depth, uint64_t T,
                                                       float Tlo, float Thi, int32_t* par,
                                                       uint32_t* __restrict__ err) {
  const int32_t n = *d_n;
  const int sh = 32 - depth, lane = threadIdx.x & 31;
  const uint32_t mask = (1u << depth) - 1u;
  const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t wi = w0; wi < n; wi += nw) {
    const int32_t i = (int32_t)wi;
    const uint32_t xi = u[i], yi = u[cap + i], zi = u[2 * cap + i];
    int32_t s = 0, len = 0;
    if (lane < 27) {
      const uint32_t ax = ((xi >> sh) + (uint32_t)(lane / 9) - 1u) & mask,
                     ay = ((yi >> sh) + (uint32_t)((lane / 3) % 3) - 1u) & mask,
                     az = ((zi >> sh) + (uint32_t)(lane % 3) - 1u) & mask;
      const uint64_t c = (spread3(ax) << 2) | (spread3(ay) << 1) | spread3(az);
      s = max(start[c], i + 1);
      len = max(start[c + 1] - s, 0);
    }
    int32_t incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    const int32_t total = __shfl_sync(0xffffffffu, incl, 31);
    if (total == 0) continue;
    const int32_t base = s - (incl - len);  // candidate t of a cell is particle base + t
    int32_t root = lane == 0 ? uf_find(par, i) : 0;
    root = __shfl_sync(0xffffffffu, root, 0);
    for (int32_t t0 = 0; t0 < total; t0 += 32) {
      const int32_t t = t0 + lane;
      int src = 0;
#pragma unroll
      for (int step = 16; step >= 1; step >>= 1) {
        const int32_t v = __shfl_sync(0xffffffffu, incl, src + step - 1);
        if (v <= t) src += step;
      }
      const int32_t j = __shfl_sync(0xffffffffu, base, src) + t;
      int32_t mine = root;
      // a stale parent only costs the test
      if (t < total && par[j] != root &&
          friends(u[j] - xi, u[cap + j] - yi, u[2 * cap + j] - zi, T, Tlo, Thi))
        mine = uf_union(par, i, j, err);
      root = __reduce_min_sync(0xffffffffu, mine);  // parents only move to smaller indices
    }
  }
}

// roots, sizes, masses, the observer distance bound and the label (smallest
// caller-order index) of every component
__global__ void k_fof_roots(const int32_t* __restrict__ d_n, int64_t cap, const uint32_t* __restrict__ u,
                            const uint32_t* __restrict__ k, const uint32_t* __restrict__ idx,
                            int32_t* __restrict__ par, int32_t* __restrict__ cnt,
                            unsigned long long* __restrict__ mass, unsigned long long* __restrict__ rmax2,
                            int32_t* __restrict__ first) {
  const int64_t n = *d_n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t r = uf_find(par, (int32_t)i);
    atomicAdd(&cnt[r], 1);
    atomicAdd(&mass[r], (unsigned long long)k[i]);
    atomicMax(&rmax2[r], (unsigned long long)dist2_obs(u[i], u[cap + i], u[2 * cap + i]));
    atomicMin(&first[r], (int32_t)idx[i]);
  }
}

// label every particle with its root (full compression), then offsets from the
// labelling member
__global__ void k_fof_offsets(const int32_t* __restrict__ d_n, int64_t cap, const uint32_t* __restrict__ u,
                              const uint32_t* __restrict__ k, int32_t* __restrict__ par,
                              const int32_t* __restrict__ first, const int32_t* __restrict__ inv,
                              unsigned long long* __restrict__ S) {
  const int64_t n = *d_n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t r = uf_find(par, (int32_t)i);
    const int32_t f = inv[first[r]];  // sorted position of the labelling member
    const long long kk = (long long)k[i];
    atomicAdd(&S[r], (unsigned long long)(kk * (long long)(int32_t)(u[i] - u[f])));
    atomicAdd(&S[n + r], (unsigned long long)(kk * (long long)(int32_t)(u[cap + i] - u[cap + f])));
    atomicAdd(&S[2 * n + r], (unsigned long long)(kk * (long long)(int32_t)(u[2 * cap + i] - u[2 * cap + f])));
  }
}

__global__ void k_fof_flags(const int32_t* __restrict__ d_n, const int32_t* __restrict__ par,
                            const int32_t* __restrict__ cnt, int nmin, int32_t* __restrict__ flag) {
  const int64_t n = *d_n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    flag[i] = (par[i] == (int32_t)i && cnt[i] >= nmin) ? 1 : 0;
}

__global__ void k_fof_write(const int32_t* __restrict__ d_n, int64_t cap, const uint32_t* __restrict__ u,
                            const int32_t* __restrict__ par, const int32_t* __restrict__ cnt,
                            const unsigned long long* __restrict__ mass, const unsigned long long* __restrict__ rmax2,
                            const int32_t* __restrict__ first, const int32_t* __restrict__ inv,
                            const unsigned long long* __restrict__ S, const int32_t* __restrict__ rank, int nmin,
                            double scale, double box, dzs_halo* __restrict__ out, int32_t* __restrict__ nh) {
  const int64_t n = *d_n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    if (par[i] != (int32_t)i || cnt[i] < nmin) continue;
    dzs_halo h;
    h.first = first[i];
    h.count = cnt[i];
    h.mass = mass[i];
    h.rmax2 = rmax2[i];
    const int32_t f = inv[first[i]];
    const double K = (double)mass[i];
    for (int ax = 0; ax < 3; ++ax) {
      const double off = (double)(long long)S[ax * n + i];
      double x = __dmul_rn(__dadd_rn((double)u[ax * cap + f], __ddiv_rn(off, K)), scale);
      if (x < 0.0) x = __dadd_rn(x, box);
      if (x >= box) x = __dsub_rn(x, box);
      h.x[ax] = x;
    }
    out[rank[i]] = h;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *nh = rank[n];
}

__global__ void k_fof_labels(const int32_t* __restrict__ d_n, const int32_t* __restrict__ par,
                             const int32_t* __restrict__ cnt, const int32_t* __restrict__ first,
                             const uint32_t* __restrict__ idx, int nmin, int64_t* __restrict__ label) {
  const int64_t n = *d_n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t r = uf_find(par, (int32_t)i);
    label[idx[i]] = cnt[r] >= nmin ? (int64_t)first[r] : -1;
  }
}

}  // namespace

// FoF on the (sorted) state with B.idx = the caller-order index of each sorted
// particle; scratch: prefix (per-root records), convert (offset sums), cicw
// (halo records, nmin >= 2 keeps them within 32 bytes per particle), the PM
// cell table (cells of depth `depth`).  Leaves the halo count in n[2].
void launch_fof(dzs_ctx* c, int depth, uint64_t T, int nmin, int64_t* d_label, dzs_halo** d_halos) {
  c->launches += d_label ? 7 : 6;  // (the cell table and the scan count their own)
  Buffers& B = c->B;
  const int64_t cap = c->cap;
  char* pre = (char*)B.prefix;
  unsigned long long* mass = (unsigned long long*)pre;
  unsigned long long* rmax2 = mass + cap;
  int32_t* par = (int32_t*)(rmax2 + cap);
  int32_t* cnt = par + cap;
  int32_t* first = cnt + cap;
  int32_t* inv = first + cap;
  unsigned long long* S = (unsigned long long*)B.convert;
  dzs_halo* out = (dzs_halo*)B.cicw;
  const int grid = grid_for(c->N0);
  // the coarsest cells whose members are all friends: 3 (side - 1)^2 <= T
  int fine = -1;
  for (int d = 1; d <= kMaxLevel && fine < 0; ++d) {
    const uint64_t side = (uint64_t)1 << (32 - d);
    if (3 * (side - 1) * (side - 1) <= T) fine = 3 * (kMaxLevel - d);
  }
  launch_cells(c, depth);
  k_fof_init<<<grid, kThreads, 0, c->stream>>>(B.n, B.key, fine, par, cnt, mass, rmax2, first, B.idx, inv, S);
  const float Tlo = std::nextafter((float)((double)T * (1.0 - 0x1p-20)), 0.0f);
  const float Thi = std::nextafter((float)((double)T * (1.0 + 0x1p-20)), INFINITY);
  k_fof_link<<<grid_for(32 * c->N0), kThreads, 0, c->stream>>>(B.n, cap, B.u, B.cell_start, depth, T, Tlo, Thi, par,
                                                               B.err);
  k_fof_roots<<<grid, kThreads, 0, c->stream>>>(B.n, cap, B.u, B.k, B.idx, par, cnt, mass, rmax2, first);
  k_fof_offsets<<<grid, kThreads, 0, c->stream>>>(B.n, cap, B.u, B.k, par, first, inv, S);
  int32_t* flag = B.iscan + (cap + 1);
  int32_t* rank = B.iscan;
  k_fof_flags<<<grid, kThreads, 0, c->stream>>>(B.n, par, cnt, nmin, flag);
  exclusive_scan_i32(c, flag, rank, B.n, cap);
  k_fof_write<<<grid, kThreads, 0, c->stream>>>(B.n, cap, B.u, par, cnt, mass, rmax2, first, inv, S, rank, nmin,
                                                c->scale, c->P.box, out, B.n + 2);
  if (d_label)
    k_fof_labels<<<grid, kThreads, 0, c->stream>>>(B.n, par, cnt, first, B.idx, nmin, d_label);
  *d_halos = out;
}

}  // namespace dzs
