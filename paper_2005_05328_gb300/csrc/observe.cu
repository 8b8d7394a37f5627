// observe.cu -- lightcone observables on the GPU (paper Sec. 3.1.2: sky map
// of the lightcone mass and its angular power spectrum, Fig. 4; Sec. 3.1.3:
// the 3D lightcone, Fig. 5).
//
// Binning: each lightcone record adds its mass k to the RING pixel of its
// direction from the observer and to the NGP cell of its crossing position
// (integer atomics: the maps are exact and independent of the order).  The
// step's record kernel does this as it writes the record; k_observe_records
// does it for records supplied by the caller.
//
// Harmonic analysis of the sky map, a_lm = Omega sum_p map_p conj(Y_lm(p)),
// in the two factors the iso-latitude rings allow:
//   1. per ring r: F_r(m) = sum_j map_j e^{-i m phi_j}   (k_ring_dft)
//   2. per m:      a_lm = Omega sum_r lambda_lm(z_r) F_r(m)   (k_legendre)
// with lambda_lm the orthonormal associated Legendre functions (Condon-
// Shortley phase), advanced in l by the three-term recursion
//   lambda_mm     = prod_k=1..m -sqrt((2k+1)/(2k)) (1 - z^2)^(m/2) / sqrt(4 pi)
//   lambda_m+1,m  = z sqrt(2m+3) lambda_mm
//   lambda_lm     = A_lm z lambda_l-1,m - B_lm lambda_l-2,m,
//   A_lm = sqrt((4l^2 - 1) / (l^2 - m^2)),
//   B_lm = sqrt((2l+1)((l-1)^2 - m^2) / ((2l-3)(l^2 - m^2))).
// C_l = (|a_l0|^2 + 2 sum_m>0 |a_lm|^2) / (2l + 1).  Every sum runs in a fixed
// order, so the spectrum is deterministic.
#include <cmath>

#include "common.cuh"
#include "observe.cuh"

namespace dzs {
namespace {

__global__ void k_observe_records(const dzs_lc_record* __restrict__ rec, int64_t n, ObserveTarget o) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const dzs_lc_record r = rec[i];
    observe_record(o, r.k, r.a_cross, r.x);
  }
}

struct RingGeom {
  int64_t nphi, start;
  double z;
  int twof;  // 2 f: the centre of pixel j (0-based) sits at (j + 1 - f) 2 pi / nphi
};

// ring r = 1 .. 4 nside - 1, north to south
__device__ __forceinline__ RingGeom ring_geom(int64_t nside, int64_t r) {
  RingGeom g;
  const double n2 = 3.0 * (double)nside * (double)nside;
  if (r < nside) {
    g.nphi = 4 * r;
    g.start = 2 * r * (r - 1);
    g.z = 1.0 - (double)(r * r) / n2;
    g.twof = 1;
  } else if (r <= 3 * nside) {
    g.nphi = 4 * nside;
    g.start = 2 * nside * (nside - 1) + (r - nside) * 4 * nside;
    g.z = (double)(2 * nside - r) * 2.0 / (3.0 * (double)nside);
    g.twof = ((r + nside) & 1) ? 2 : 1;
  } else {
    const int64_t s = 4 * nside - r;
    g.nphi = 4 * s;
    g.start = 12 * nside * nside - 2 * s * (s + 1);
    g.z = -1.0 + (double)(s * s) / n2;
    g.twof = 1;
  }
  return g;
}

constexpr int kAnchor = 32;          // without a table the phasor is recomputed exactly every kAnchor pairs
constexpr int kDftThreads = 256;
constexpr int64_t kTableRing = 4096;  // longest ring whose phasors are tabulated (72 KB of shared memory)

// lanes step through the table 2 (2a + 1) entries apart: every eighth entry a
// gap, so that the 8 lanes of a 128-byte phase fall on distinct banks
__host__ __device__ constexpr int64_t tab_slot(int64_t q) { return q + (q >> 3); }
// pairs of a ring's quarter with r' pixels, first pixel centre on phi = 0 or not
__host__ __device__ constexpr int ring_pairs(int quarter, bool on_zero) { return on_zero ? quarter / 2 + 1 : (quarter + 1) / 2; }

// F[r-1][m] for m = 0..lmax; one block per ring.  Every ring has 4 r' pixels
// placed symmetrically, so the four pixels a, a + r', a + 2r', a + 3r' enter
// F(m) through one phasor and a combination that depends on m mod 4 alone:
// e = their sum (0), o = alternating sum (2), d -+ i f with d = v0 - v2,
// f = v1 - v3 (1, 3); and a pixel and its mirror image in the quarter (primed;
// phi' = pi/2 - phi) share a cosine and a sine:
//   m = 0 mod 4:  re += (e + e') cos,  im -= (e - e') sin
//   m = 2 mod 4:  re += (o - o') cos,  im -= (o + o') sin
//   m = 1, 3:     re += (d - f') cos -+ (f - d') sin,  im += -+ (f + d') cos - (d + f') sin
// (upper sign m = 1 mod 4): 2 or 4 FP64 multiply-adds for eight pixels.  The
// phasors exp(-i pi q / nphi) come from a table (kTable: half a turn, the other
// half negated), else from a recurrence.  A warp takes even or odd m only.
// FP64 is the bound (82% of the unit busy with 3.5 operations per four
// pixels).  Nside 256, lmax 512: 5.69 ms with 6 operations a pixel, now 0.75 ms.
template <bool kTable>
__global__ void __launch_bounds__(kDftThreads) k_ring_dft(const unsigned long long* __restrict__ map, int64_t nside,
                                                          int lmax, double2* __restrict__ F) {
  extern __shared__ double2 ring_sm[];
  const int64_t r = blockIdx.x + 1;
  const RingGeom g = ring_geom(nside, r);
  const int nphi = (int)g.nphi, quarter = nphi / 4;
  const bool on_zero = g.twof == 2;
  const int npair = ring_pairs(quarter, on_zero), stride = ring_pairs((int)nside, true);
  double2* tab = ring_sm;                                              // [tab_slot(nphi)] (kTable)
  double* c = (double*)(ring_sm + (kTable ? tab_slot(4 * nside) : 0));  // [8][stride]
  for (int a = threadIdx.x; a < npair; a += kDftThreads) {
    const int b = on_zero ? quarter - a : quarter - 1 - a;  // the mirror image; b = quarter: none (phi = 0)
    const unsigned long long* v = map + g.start;
    double q[2][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      q[0][k] = (double)v[a + k * quarter];
      q[1][k] = b < quarter ? (double)v[b + k * quarter] : 0.0;
    }
    const double wt = b == a ? 0.5 : 1.0;  // its own image: counted once
    const double e0 = (q[0][0] + q[0][2]) + (q[0][1] + q[0][3]), e1 = (q[1][0] + q[1][2]) + (q[1][1] + q[1][3]);
    const double o0 = (q[0][0] + q[0][2]) - (q[0][1] + q[0][3]), o1 = (q[1][0] + q[1][2]) - (q[1][1] + q[1][3]);
    const double d0 = q[0][0] - q[0][2], f0 = q[0][1] - q[0][3], d1 = q[1][0] - q[1][2], f1 = q[1][1] - q[1][3];
    c[a] = wt * (e0 + e1);
    c[stride + a] = wt * (e0 - e1);
    c[2 * stride + a] = wt * (o0 - o1);
    c[3 * stride + a] = wt * (o0 + o1);
    c[4 * stride + a] = wt * (d0 - f1);
    c[5 * stride + a] = wt * (f0 - d1);
    c[6 * stride + a] = wt * (f0 + d1);
    c[7 * stride + a] = wt * (d0 + f1);
  }
  if (kTable)
    for (int q = threadIdx.x; q < nphi; q += kDftThreads) {
      double sn, cs;
      sincospi((double)q / (double)nphi, &sn, &cs);
      tab[tab_slot(q)] = make_double2(cs, sn);
    }
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int per = 2 * nphi;  // angles are pi q / nphi with q taken mod 2 nphi
  const int half = (lmax / 2 + 32) / 32;  // warps of even m, and as many of odd
  for (int task = w; task < 2 * half; task += kDftThreads / 32) {
    const bool odd = task & 1;
    const int m = 2 * ((task >> 1) * 32 + lane) + (odd ? 1 : 0);
    const bool up = m & 2;
    const double* c0 = c + (odd ? 4 * stride : up ? 2 * stride : 0);
    const int step = (int)((2 * (int64_t)m) % per);
    int q = (int)(((int64_t)m * (2 - g.twof)) % per);
    double re = 0.0, im = 0.0, sst = 0.0, cst = 1.0, sn = 0.0, cs = 1.0;
    if (!kTable) sincospi((double)step / (double)nphi, &sst, &cst);
    for (int a = 0; a < npair; ++a) {
      if (kTable) {
        const bool neg = q >= nphi;
        const double2 t = tab[tab_slot(neg ? q - nphi : q)];
        cs = neg ? -t.x : t.x;
        sn = neg ? -t.y : t.y;
      } else if (a % kAnchor == 0) {
        sincospi((double)q / (double)nphi, &sn, &cs);
      }
      if (!odd) {
        re += c0[a] * cs;
        im -= c0[stride + a] * sn;
      } else {
        const double s1 = up ? sn : -sn, c1 = up ? cs : -cs;
        re += c0[a] * cs;
        im += c0[2 * stride + a] * c1;
        re += c0[stride + a] * s1;
        im -= c0[3 * stride + a] * sn;
      }
      q += step;
      if (q >= per) q -= per;
      if (!kTable) {
        const double c2 = cs * cst - sn * sst;
        sn = sn * cst + cs * sst;
        cs = c2;
      }
    }
    if (m <= lmax) F[(r - 1) * (lmax + 1) + m] = make_double2(re, im);
  }
}

constexpr int kLegThreads = 64;
constexpr int kLegWarps = kLegThreads / 32;
constexpr int kRingsPerThread = 8;
constexpr int kLTile = 64;

__host__ __device__ inline int64_t alm_index(int lmax, int l, int m) {
  return (int64_t)m * (2 * lmax + 1 - m) / 2 + l;
}

// x^m, m >= 0, by repeated squaring in two words: a squaring's rounding would be
// doubled by every one that follows it (x^256 off by up to 128 of them); a m-fold
// product, which this replaced, rounds m times
__device__ __forceinline__ double ipow(double x, int m) {
  double v = 1.0, vl = 0.0, xl = 0.0;
  for (;;) {
    if (m & 1) {
      const double p = v * x;
      vl = fma(v, xl, fma(vl, x, fma(v, x, -p)));
      v = p;
    }
    m >>= 1;
    if (m == 0) return v + vl;
    const double p = x * x;
    xl = fma(2.0 * x, xl, fma(x, x, -p));
    x = p;
  }
}

// sums over the warp of the 8 values v, one shuffle-add per value instead of
// five: each level halves the values a lane still carries.  Returns the sum of
// v[lane >> 2] in lanes with (lane & 3) == 0.
__device__ __forceinline__ double warp_sum8(const double (&v)[8], int lane) {
  double a[4], b[2];
  const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4;
#pragma unroll
  for (int i = 0; i < 4; ++i)
    a[i] = (h16 ? v[4 + i] : v[i]) + __shfl_xor_sync(0xffffffffu, h16 ? v[i] : v[4 + i], 16);
#pragma unroll
  for (int i = 0; i < 2; ++i)
    b[i] = (h8 ? a[2 + i] : a[i]) + __shfl_xor_sync(0xffffffffu, h8 ? a[i] : a[2 + i], 8);
  double s = (h4 ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, h4 ? b[0] : b[1], 4);
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  return s;
}

// one block per m: alm[l, m] += Omega sum over rings, ring chunks in order.
// Rings north and south of the equator share |lambda|: lambda_lm(-z) =
// (-1)^(l+m) lambda_lm(z), so one recursion serves F_N + F_S (l + m even) or
// F_N - F_S (odd).  FP64-bound: 5 operations per (l, m, ring pair), and a
// quarter of a shuffle-add with 8 pairs a thread (74% of the unit busy).  lambda_mm is the m-th power
// of the sine times a product the block forms once (it was a loop of m square
// roots and divisions in every thread: most of the kernel's time).  Nside 256,
// lmax 512: 8.64 ms, now 1.12 ms.
__global__ void __launch_bounds__(kLegThreads) k_legendre(const double2* __restrict__ F, int64_t nside, int lmax,
                                                          double omega, double2* __restrict__ alm) {
  extern __shared__ double sh[];
  double* A = sh;                                     // [lmax + 1 + 4]
  double* Bc = A + (lmax + 5);                        // [lmax + 1 + 4]
  double2* part = (double2*)(Bc + (lmax + 5));        // [kLegWarps][kLTile]
  __shared__ double lead_w[kLegWarps];
  const int m = blockIdx.x;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int l = m + 1 + threadIdx.x; l < lmax + 5; l += blockDim.x) {
    const double dl = l, dm = m, d = dl * dl - dm * dm;
    const bool in = l <= lmax;
    A[l] = !in ? 0.0 : l == m + 1 ? sqrt(2.0 * dm + 3.0) : sqrt((4.0 * dl * dl - 1.0) / d);
    Bc[l] = !in || l == m + 1
                ? 0.0
                : sqrt((2.0 * dl + 1.0) * ((dl - 1.0) * (dl - 1.0) - dm * dm) / ((2.0 * dl - 3.0) * d));
  }
  // product of -sqrt((2k + 1) / (2k)) over k = 1..m, times 1 / sqrt(4 pi)
  double lead = 1.0;
  for (int k = 1 + threadIdx.x; k <= m; k += blockDim.x) lead *= -sqrt((2.0 * k + 1.0) / (2.0 * k));
  for (int o = 16; o > 0; o >>= 1) lead *= __shfl_xor_sync(0xffffffffu, lead, o);
  if (lane == 0) lead_w[w] = lead;
  __syncthreads();
  lead = 0.28209479177387814;
  for (int q = 0; q < kLegWarps; ++q) lead *= lead_w[q];
  const int64_t nrings = 4 * nside - 1, north = 2 * nside;  // north: 0-based rings 0 .. 2 nside - 1, equator last
  const int64_t chunk = (int64_t)kLegThreads * kRingsPerThread;
  for (int64_t c0 = 0; c0 < north; c0 += chunk) {
    double z[kRingsPerThread], l1[kRingsPerThread], l2[kRingsPerThread];
    double2 fe[kRingsPerThread], fo[kRingsPerThread];
#pragma unroll
    for (int q = 0; q < kRingsPerThread; ++q) {
      const int64_t r = c0 + threadIdx.x + (int64_t)q * kLegThreads;
      z[q] = l1[q] = l2[q] = 0.0;
      fe[q] = fo[q] = make_double2(0.0, 0.0);
      if (r < north) {
        z[q] = ring_geom(nside, r + 1).z;
        const double2 fn = F[r * (lmax + 1) + m];
        const int64_t s = nrings - 1 - r;
        const double2 fs = s > r ? F[s * (lmax + 1) + m] : make_double2(0.0, 0.0);
        fe[q] = make_double2(fn.x + fs.x, fn.y + fs.y);
        fo[q] = make_double2(fn.x - fs.x, fn.y - fs.y);
        l1[q] = lead * ipow(sqrt((1.0 - z[q]) * (1.0 + z[q])), m);
      }
    }
    for (int lt = m; lt <= lmax; lt += kLTile) {
      for (int d = 0; d < kLTile && lt + d <= lmax; d += 4) {
        double v[8];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int l = lt + d + e;
          const bool lead_l = l == m;  // e == 0 of the first tile
          const double al = lead_l ? 0.0 : A[l], bl = lead_l ? 0.0 : Bc[l];
          double re = 0.0, im = 0.0;
#pragma unroll
          for (int q = 0; q < kRingsPerThread; ++q) {
            if (!lead_l) {
              const double lam = al * (z[q] * l1[q]) - bl * l2[q];
              l2[q] = l1[q];
              l1[q] = lam;
            }
            re += l1[q] * ((e & 1) ? fo[q].x : fe[q].x);
            im += l1[q] * ((e & 1) ? fo[q].y : fe[q].y);
          }
          v[2 * e] = re;
          v[2 * e + 1] = im;
        }
        const double s = warp_sum8(v, lane);
        if ((lane & 3) == 0) ((double*)(part + w * kLTile + d))[lane >> 2] = s;
      }
      __syncthreads();
      if (lt + (int)threadIdx.x <= lmax && threadIdx.x < kLTile) {
        double2 s = make_double2(0.0, 0.0);
        for (int q = 0; q < kLegWarps; ++q) {
          s.x += part[q * kLTile + threadIdx.x].x;
          s.y += part[q * kLTile + threadIdx.x].y;
        }
        double2* out = &alm[alm_index(lmax, lt + threadIdx.x, m)];
        double2 acc = c0 == 0 ? make_double2(0.0, 0.0) : *out;
        acc.x += omega * s.x;
        acc.y += omega * s.y;
        *out = acc;
      }
      __syncthreads();
    }
  }
}

// block l: lane-strided sums over m, then a fixed shuffle tree and the warps in
// order (one thread per l walked the m serially: 157 us at lmax 512)
constexpr int kClThreads = 128;
__global__ void __launch_bounds__(kClThreads) k_cl(const double2* __restrict__ alm, int lmax, double* __restrict__ cl) {
  __shared__ double sh[kClThreads / 32];
  const int l = blockIdx.x;
  double s = 0.0;
  for (int m = threadIdx.x; m <= l; m += kClThreads) {
    const double2 a = alm[alm_index(lmax, l, m)];
    const double p = a.x * a.x + a.y * a.y;
    s += m == 0 ? p : 2.0 * p;
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kClThreads / 32; ++w) s += sh[w];
    cl[l] = s / (2.0 * l + 1.0);
  }
}

}  // namespace

void launch_observe_records(dzs_ctx* c, const dzs_lc_record* d_rec, int64_t n) {
  if (n <= 0) return;
  c->launches += 1;
  k_observe_records<<<grid_for(n), kThreads, 0, c->stream>>>(d_rec, n, c->obs);
}

size_t sht_work_bytes(int64_t nside, int lmax) {
  const size_t nr = (size_t)(4 * nside - 1), nl = (size_t)lmax + 1;
  const size_t nalm = nl * (nl + 1) / 2;
  return 16 * nr * nl + 16 * nalm + 8 * nl + 256;
}

size_t sht_shared_bytes(int lmax) { return 16 * ((size_t)lmax + 5) + 16 * kLegWarps * kLTile; }

// a_lm (m-major, index m (2 lmax + 1 - m) / 2 + l, complex interleaved) and C_l
// of the context's sky map into work: [F | alm | cl]
void launch_sht(dzs_ctx* c, int lmax, void* work, double2** d_alm, double** d_cl) {
  const int64_t nside = c->obs.nside, nr = 4 * nside - 1;
  char* w = (char*)work;
  double2* F = (double2*)w;
  double2* alm = (double2*)(w + 16 * (size_t)nr * (lmax + 1));
  const size_t nalm = (size_t)(lmax + 1) * (lmax + 2) / 2;
  double* cl = (double*)((char*)alm + 16 * nalm);
  c->launches += 3;
  const bool table = 4 * nside <= kTableRing;
  // the pairs' eight combinations and, with a table, the phasors
  const size_t dft_sm = 64 * (size_t)ring_pairs((int)nside, true) + (table ? 16 * (size_t)tab_slot(4 * nside) : 0);
  auto dft = table ? k_ring_dft<true> : k_ring_dft<false>;
  cudaFuncSetAttribute(dft, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dft_sm);
  cudaFuncSetAttribute(k_legendre, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sht_shared_bytes(lmax));
  dft<<<(unsigned)nr, kDftThreads, dft_sm, c->stream>>>(c->obs.sky, nside, lmax, F);
  const double omega = 4.0 * M_PI / (double)(12 * nside * nside);
  k_legendre<<<lmax + 1, kLegThreads, sht_shared_bytes(lmax), c->stream>>>(F, nside, lmax, omega, alm);
  k_cl<<<lmax + 1, kClThreads, 0, c->stream>>>(alm, lmax, cl);
  *d_alm = alm;
  *d_cl = cl;
}

// ---- twin-particle displacements (paper Sec. 3.2, integration accuracy):
// particles inside the lightcone (not crossed) in both runs of a twin pair,
// matched by id, the minimum-image distance of their positions over
// h = L / N^(1/3) / 40, binned by the caller's edges.  FP64 with correctly
// rounded operations in a fixed order (the CPU check does the same), integer
// atomics for the counts: exact and independent of the order.

__global__ void k_twin_map(const int32_t* __restrict__ d_n, const uint32_t* __restrict__ id,
                           const uint8_t* __restrict__ fl, int32_t* __restrict__ map, int64_t n0) {
  const int64_t n = *d_n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    if (fl[i] & kFlCrossed) continue;
    const uint32_t q = id[i];
    if ((int64_t)q < n0) map[q] = (int32_t)i;
  }
}

__global__ void k_twin_disp(const int32_t* __restrict__ d_n, int64_t cap, const uint32_t* __restrict__ u,
                            const uint32_t* __restrict__ id, const uint8_t* __restrict__ fl,
                            const int32_t* __restrict__ map, int64_t capb, const uint32_t* __restrict__ ub,
                            const double* __restrict__ edges, int nbins, double scale, double h, int64_t n0,
                            unsigned long long* __restrict__ counts, unsigned long long* __restrict__ stats) {
  const int64_t n = *d_n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    if (fl[i] & kFlCrossed) continue;
    const uint32_t q = id[i];
    if ((int64_t)q >= n0) continue;
    const int32_t j = map[q];
    if (j < 0) continue;
    double s = 0.0;
    for (int ax = 0; ax < 3; ++ax) {
      const double d = __dmul_rn((double)(int32_t)(u[ax * cap + i] - ub[ax * capb + j]), scale);
      s = __dadd_rn(s, __dmul_rn(d, d));
    }
    const double ratio = __ddiv_rn(__dsqrt_rn(s), h);
    // bin k: edges[k] <= ratio < edges[k + 1]
    int lo = 0, hi = nbins + 1;  // first edge > ratio, in [lo, hi)
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (edges[mid] <= ratio)
        lo = mid + 1;
      else
        hi = mid;
    }
    const int k = lo - 1;
    if (k >= 0 && k < nbins) atomicAdd(&counts[k], 1ull);
    atomicAdd(&stats[0], 1ull);
    atomicMax(&stats[1], (unsigned long long)__double_as_longlong(ratio));  // ratio >= 0: bits order like values
  }
}

void launch_twin_displacement(dzs_ctx* a, dzs_ctx* b, int32_t* map, const double* edges, int nbins, double h,
                              unsigned long long* counts, unsigned long long* stats) {
  a->launches += 2;
  cudaMemsetAsync(map, 0xff, sizeof(int32_t) * a->N0, a->stream);
  k_twin_map<<<grid_for(b->cap), kThreads, 0, a->stream>>>(b->B.n, b->B.id, b->B.fl, map, a->N0);
  k_twin_disp<<<grid_for(a->cap), kThreads, 0, a->stream>>>(a->B.n, a->cap, a->B.u, a->B.id, a->B.fl, map, b->cap,
                                                             b->B.u, edges, nbins, a->scale, h, a->N0, counts,
                                                             stats);
}

}  // namespace dzs
