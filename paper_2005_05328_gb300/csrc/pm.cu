// pm.cu -- particle-mesh long-range force (paper Sec. 2.1): atomic-free CIC
// deposit, FFT Poisson solve with the Gaussian split (fft.cu), four-point
// gradient and CIC interpolation back to the particles.
//
// Deposit: the particles are Morton-sorted, so the particles of one mesh cell
// (for M = 2^m the depth-m Morton prefix) are one contiguous run.  A CSR-like
// table start[c] (Morton cell index) is written once per cell by the particle
// that opens each run (covering the empty cells before it), then every mesh
// node gathers k w from the 8 cells it touches.  No atomics: each node sums
// in a fixed order (cell offset, then particle order), so the mesh is
// deterministic.  Mesh node (ix, iy, iz) sits at (ix, iy, iz) L / M.
#include <cmath>
#include <vector>

#include "common.cuh"

namespace dzs {

template <class R>
void fft_r2c_zy(dzs_ctx* c, const R* in, cplx<R>* out, int n, const cplx<R>* tw);

namespace {

__global__ void k_cell_start(const int32_t* __restrict__ d_n, const uint64_t* __restrict__ key, int sh,
                             int64_t ncell, int32_t* __restrict__ start) {
  // particle i writes i into the cells after its predecessor's cell up to its
  // own (i = n: up to the end); a lane fills a short run itself, the warp
  // fills long runs (gaps of empty cells) together, coalesced
  const int64_t n = *d_n;
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t w0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; w0 <= n; w0 += stride) {
    const int64_t i = w0 + lane;
    int64_t lo = 0, hi = 0;  // cells [lo, hi) take the value i
    if (i <= n) {
      const int64_t ci = (i < n) ? (int64_t)(key[i] >> sh) : ncell;
      const int64_t cp = (i > 0) ? (int64_t)(key[i - 1] >> sh) : -1;
      lo = cp + 1;
      hi = ci + 1;
    }
    const bool longrun = hi - lo > 32;
    if (!longrun)
      for (int64_t q = lo; q < hi; ++q) start[q] = (int32_t)i;
    unsigned lm = __ballot_sync(0xffffffffu, longrun);
    while (lm) {
      const int src = __ffs(lm) - 1;
      lm &= lm - 1;
      const int64_t qlo = __shfl_sync(0xffffffffu, lo, src), qhi = __shfl_sync(0xffffffffu, hi, src);
      const int32_t v = (int32_t)__shfl_sync(0xffffffffu, i, src);
      for (int64_t q = qlo + lane; q < qhi; q += 32) start[q] = v;
    }
  }
}

__device__ __forceinline__ uint32_t morton_cell(uint32_t x, uint32_t y, uint32_t z) {
  return (uint32_t)((spread3(x) << 2) | (spread3(y) << 1) | spread3(z));
}

template <class R>
__device__ __forceinline__ R frac32(uint32_t lo) {
  return (R)lo * (R)2.3283064365386963e-10;  // 2^-32
}

// 16-byte vectors of R (aligned loads and stores of 8 weights or a phi row)
template <class R>
struct Vec16;
template <>
struct Vec16<float> {
  using T = float4;
  static constexpr int N = 4;
};
template <>
struct Vec16<double> {
  using T = double2;
  static constexpr int N = 2;
};

template <class R>
__device__ __forceinline__ void store8(R* __restrict__ dst, const R (&v)[8]) {
  using V = typename Vec16<R>::T;
  constexpr int N = Vec16<R>::N;
#pragma unroll
  for (int q = 0; q < 8 / N; ++q) {
    V x;
    R* xs = reinterpret_cast<R*>(&x);
#pragma unroll
    for (int r = 0; r < N; ++r) xs[r] = v[q * N + r];
    reinterpret_cast<V*>(dst)[q] = x;
  }
}

// corner weight sums of one cell: acc[o] = sum over the cell's particles, in
// order, of k w_o, w_o the CIC weight of the cell's corner node o = (ox, oy, oz)
template <class R>
__device__ __forceinline__ void add_corners(uint32_t ux, uint32_t uy, uint32_t uz, uint32_t k, int M, R (&acc)[8]) {
  const R fx = frac32<R>((uint32_t)((uint64_t)ux * (uint64_t)M)), fy = frac32<R>((uint32_t)((uint64_t)uy * (uint64_t)M)),
          fz = frac32<R>((uint32_t)((uint64_t)uz * (uint64_t)M));
  const R kk = (R)k;
#pragma unroll
  for (int o = 0; o < 8; ++o) {
    const int ox = (o >> 2) & 1, oy = (o >> 1) & 1, oz = o & 1;
    acc[o] += kk * ((ox ? fx : (R)1 - fx) * (oy ? fy : (R)1 - fy) * (oz ? fz : (R)1 - fz));
  }
}

// M = 2^m: density contrast of one 16^3 tile of nodes per block.  Mesh cells are
// Morton cells, so the tile's own particles are one contiguous run, those of its
// lower neighbours' 8^3 cells 19 more; start is the table of Morton cells (2^sh9 per 8^3 cells).  The particle that
// opens a cell sums the cell's corner weights in registers; the block then adds
// corner o = 0..7 in turn, one barrier apart: the cells of a batch differ, so no
// two threads add to a node at once and the order is fixed (deterministic).
// Bound by latency: a tile is a few rounds of dependent loads.  It replaces a
// pass that wrote each cell's sums to memory and a gather that read the bounds
// of 729 cells and 8 records a node for each 8^3 tile: 177 + 29 (a finer cell
// table) -> 145 us for 128^3 on mesh 256.
constexpr int kCicThreads = 512;
constexpr int kT = 16;  // nodes per side of a tile
template <class R>
__global__ void __launch_bounds__(kCicThreads) k_cic_tile(const int32_t* __restrict__ start, int sh9,
                                                          const int32_t* __restrict__ d_n, int64_t cap,
                                                          const uint64_t* __restrict__ key, int sh,
                                                          const uint32_t* __restrict__ u, const uint32_t* __restrict__ k,
                                                          int M, R* __restrict__ delta, R inv_nbar) {
  constexpr int S = kT / 8, E = S + 1, kRuns = E * E * E;  // 8^3 cells per axis with the lower neighbour
  __shared__ R acc[kT * kT * kT];
  __shared__ int32_t first[32], upto[32];  // runs of the neighbours' cells, running totals (0 for the own ones)
  const int T = M / kT, T8 = M >> 3, tile = blockIdx.x;
  const int tx = tile / (T * T), ty = (tile / T) % T, tz = tile % T;
  const int64_t n = *d_n;
  auto cell8 = [](uint32_t x, uint32_t y, uint32_t z) {
    return (int64_t)((spread3(x) << 2) | (spread3(y) << 1) | spread3(z));
  };
  const int64_t own8 = cell8((uint32_t)(tx * S), (uint32_t)(ty * S), (uint32_t)(tz * S));
  const int32_t p0 = start[own8 << sh9], p1 = start[(own8 + S * S * S) << sh9];
  if (threadIdx.x < 32) {
    const int o = threadIdx.x;  // (x, y, z) offset + 1 per axis
    const int ox = o / (E * E), oy = (o / E) % E, oz = o % E;
    int32_t s = 0, len = 0;
    if (o < kRuns && (ox == 0 || oy == 0 || oz == 0)) {
      const int64_t c = cell8((uint32_t)(tx * S + ox - 1 + T8) % (uint32_t)T8, (uint32_t)(ty * S + oy - 1 + T8) % (uint32_t)T8,
                              (uint32_t)(tz * S + oz - 1 + T8) % (uint32_t)T8);
      s = start[c << sh9];
      len = start[(c + 1) << sh9] - s;
    }
#pragma unroll
    for (int q = 1; q < 32; q <<= 1) {
      const int32_t v = __shfl_up_sync(0xffffffffu, len, q);
      if (o >= q) len += v;
    }
    first[o] = s;
    upto[o] = len;
  }
  for (int q = threadIdx.x; q < kT * kT * kT; q += kCicThreads) acc[q] = (R)0;
  __syncthreads();
  const int own = p1 - p0, total = own + upto[31];
  for (int t0 = 0; t0 < total; t0 += kCicThreads) {
    // the thread's cell: its lowest corner node in tile coordinates (-1: below)
    int x = 0, y = 0, z = 0;
    bool take = false;
    R w[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    const int t = t0 + (int)threadIdx.x;
    if (t < total) {
      int64_t i = (int64_t)p0 + t;
      int ox = 1, oy = 1, oz = 1;
      if (t >= own) {
        const int v = t - own;
        int o = 0;
#pragma unroll
        for (int step = 16; step >= 1; step >>= 1)
          if (upto[o + step - 1] <= v) o += step;
        i = (int64_t)first[o] + v - (o > 0 ? upto[o - 1] : 0);
        ox = o / (E * E);
        oy = (o / E) % E;
        oz = o % E;
      }
      const uint64_t c = key[i] >> sh;
      const bool opens = i == 0 || (key[i - 1] >> sh) != c;
      const int mo = (int)c & (kT * kT * kT - 1);
      x = ((mo >> 6) & 4) | ((mo >> 4) & 2) | ((mo >> 2) & 1);
      y = ((mo >> 5) & 4) | ((mo >> 3) & 2) | ((mo >> 1) & 1);
      z = ((mo >> 4) & 4) | ((mo >> 2) & 2) | (mo & 1);
      x |= (mo >> 8) & 8;
      y |= (mo >> 7) & 8;
      z |= (mo >> 6) & 8;
      // a lower neighbour's cell counts when it touches the tile: its last layer
      take = opens && (ox > 0 || (x & 7) == 7) && (oy > 0 || (y & 7) == 7) && (oz > 0 || (z & 7) == 7);
      if (ox == 0) x = -1;
      if (oy == 0) y = -1;
      if (oz == 0) z = -1;
      if (take)
        for (int64_t j = i; j < n && (j == i || (key[j] >> sh) == c); ++j)
          add_corners<R>(u[j], u[cap + j], u[2 * cap + j], k[j], M, w);
    }
#pragma unroll
    for (int o = 0; o < 8; ++o) {
      const int ax = x + (o >> 2), ay = y + ((o >> 1) & 1), az = z + (o & 1);
      if (take && (unsigned)ax < (unsigned)kT && (unsigned)ay < (unsigned)kT && (unsigned)az < (unsigned)kT)
        acc[(ax * kT + ay) * kT + az] += w[o];
      __syncthreads();
    }
  }
  for (int t = threadIdx.x; t < kT * kT * kT; t += kCicThreads) {
    const int a = t / (kT * kT), b = (t / kT) % kT, c = t % kT;
    delta[((int64_t)(tx * kT + a) * M + (ty * kT + b)) * M + (tz * kT + c)] = acc[t] * inv_nbar - (R)1;
  }
}

// W[8 i + o], i the first particle of a cell = sum over the cell's particles,
// in order, of k w_o, w_o the CIC weight of the cell's corner node
// o = (ox, oy, oz); the 8 sums of a cell are one aligned 8-value record.  For the
// meshes tile_mesh leaves out.
template <class R>
__global__ void k_cic_cellw(const int32_t* __restrict__ d_n, int64_t cap, const uint64_t* __restrict__ key, int sh,
                            const uint32_t* __restrict__ u, const uint32_t* __restrict__ k, int M,
                            R* __restrict__ W) {
  const int64_t n = *d_n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t c = key[i] >> sh;
    if (i > 0 && (key[i - 1] >> sh) == c) continue;  // not the first of its cell
    R acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int64_t j = i; j < n && (key[j] >> sh) == c; ++j)
      add_corners<R>(u[j], u[cap + j], u[2 * cap + j], k[j], M, acc);
    store8(W + 8 * i, acc);
  }
}

// the same for M = 3 2^a, at sorted positions t: particles visited in row-major cell order through the
// cell sort (sorted cell keys ck, original indices perm)
template <class R>
__global__ void k_cic_cellw_perm(const int32_t* __restrict__ d_n, int64_t cap, const uint64_t* __restrict__ ck,
                                 const uint32_t* __restrict__ perm, const uint32_t* __restrict__ u,
                                 const uint32_t* __restrict__ k, int M, R* __restrict__ W) {
  const int64_t n = *d_n;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t c = ck[t];
    if (t > 0 && ck[t - 1] == c) continue;
    R acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int64_t s = t; s < n && ck[s] == c; ++s) {
      const int64_t j = perm[s];
      add_corners<R>(u[j], u[cap + j], u[2 * cap + j], k[j], M, acc);
    }
    store8(W + 8 * t, acc);
  }
}

__global__ void k_mesh_keys(const int32_t* __restrict__ d_n, int64_t cap, const uint32_t* __restrict__ u, int M,
                            uint64_t* __restrict__ ck) {
  const int64_t n = *d_n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t cx = ((uint64_t)u[i] * (uint64_t)M) >> 32, cy = ((uint64_t)u[cap + i] * (uint64_t)M) >> 32,
                   cz = ((uint64_t)u[2 * cap + i] * (uint64_t)M) >> 32;
    ck[i] = (cx * (uint64_t)M + cy) * (uint64_t)M + cz;
  }
}

// rho[node] = sum over the 8 cells node - o, o in {0,1}^3, of the cell's
// corner-o weight sum; output delta.  One block per 8^3 tile of nodes:
//   1. the CSR bounds of the 9^3 cells the tile touches: for Morton-ordered
//      cells the tile's own 8^3 cells are one run of the table (513
//      consecutive entries, coalesced) and only the 217 cells of the three
//      lower halo planes are looked up one by one;
//   2. each node adds the corner weight sums of its 8 cells in the fixed
//      order o = 0..7, read from the cells' records in global memory (L2;
//      empty cells add +0), so the mesh is deterministic.
template <class R, bool kMorton>
__global__ void __launch_bounds__(256) k_cic_gather(const int32_t* __restrict__ start, const int32_t* __restrict__ d_n,
                                                    const R* __restrict__ W, int M, R* __restrict__ delta,
                                                    R inv_nbar) {
  extern __shared__ unsigned char cg_raw[];
  int32_t* first = reinterpret_cast<int32_t*>(cg_raw);  // [729] first particle, -1 empty
  int32_t* sb = first + 729;                               // [513] the tile's own bounds
  const int T = M >> 3;
  const int tile = blockIdx.x;
  const int tx = tile / (T * T), ty = (tile / T) % T, tz = tile % T;
  const int bx = tx * 8, by = ty * 8, bz = tz * 8;
  const int32_t n = *d_n;
  auto clampb = [n](int32_t v) { return v < 0 ? 0 : (v > n ? n : v); };
  auto cell_of = [&](int i, int j, int l) -> int64_t {  // 9^3 coordinates (offset -1)
    if (kMorton) {  // M = 2^m: periodic wrap by a mask
      const uint32_t mk = (uint32_t)M - 1u;
      return (int64_t)morton_cell((uint32_t)(bx + i - 1) & mk, (uint32_t)(by + j - 1) & mk, (uint32_t)(bz + l - 1) & mk);
    }
    const uint32_t gx = (uint32_t)((bx + i - 1 + M) % M), gy = (uint32_t)((by + j - 1 + M) % M),
                   gz = (uint32_t)((bz + l - 1 + M) % M);
    return ((int64_t)gx * M + gy) * M + gz;
  };
  if (kMorton) {
    const int64_t base =
        (int64_t)((spread3((uint32_t)tx) << 2) | (spread3((uint32_t)ty) << 1) | spread3((uint32_t)tz)) << 9;
    for (int mo = threadIdx.x; mo <= 512; mo += blockDim.x) sb[mo] = clampb(start[base + mo]);
    for (int h = threadIdx.x; h < 217; h += blockDim.x) {
      int i, j, l;
      if (h < 81) {
        i = 0, j = h / 9, l = h % 9;
      } else if (h < 153) {
        i = 1 + (h - 81) / 9, j = 0, l = (h - 81) % 9;
      } else {
        i = 1 + (h - 153) / 8, j = 1 + (h - 153) % 8, l = 0;
      }
      const int64_t mc = cell_of(i, j, l);
      const int32_t s0 = clampb(start[mc]), e0 = clampb(start[mc + 1]);
      first[(i * 9 + j) * 9 + l] = e0 > s0 ? s0 : -1;
    }
    __syncthreads();
    for (int mo = threadIdx.x; mo < 512; mo += blockDim.x) {
      const int i = ((mo >> 6) & 4) | ((mo >> 4) & 2) | ((mo >> 2) & 1);
      const int j = ((mo >> 5) & 4) | ((mo >> 3) & 2) | ((mo >> 1) & 1);
      const int l = ((mo >> 4) & 4) | ((mo >> 2) & 2) | (mo & 1);
      first[((i + 1) * 9 + (j + 1)) * 9 + (l + 1)] = sb[mo + 1] > sb[mo] ? sb[mo] : -1;
    }
  } else {
    for (int q = threadIdx.x; q < 729; q += blockDim.x) {
      const int64_t mc = cell_of(q / 81, (q / 9) % 9, q % 9);
      const int32_t s0 = clampb(start[mc]), e0 = clampb(start[mc + 1]);
      first[q] = e0 > s0 ? s0 : -1;
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < 512; t += blockDim.x) {
    const int a = t >> 6, b = (t >> 3) & 7, c = t & 7;
    const int q0 = (a + 1) * 81 + (b + 1) * 9 + (c + 1);
    R acc = 0;
#pragma unroll
    for (int o = 0; o < 8; ++o) {
      const int ox = (o >> 2) & 1, oy = (o >> 1) & 1, oz = o & 1;
      const int32_t f = first[q0 - ox * 81 - oy * 9 - oz];
      acc += f >= 0 ? W[8 * f + o] : (R)0;  // 8 f + o < 8 cap <= 2^30
    }
    delta[((int64_t)(bx + a) * M + (by + b)) * M + (bz + c)] = acc * inv_nbar - (R)1;
  }
}

template <class R>
constexpr size_t gather_smem() {
  return (729 + 513) * sizeof(int32_t);
}

// g = -grad phi at the particles for any mesh (used for M = 3 2^a): the
// four-point stencil at the 8 surrounding nodes, CIC weights, from global memory
template <class R>
__global__ void k_pm_interp(const int32_t* __restrict__ d_n, int64_t cap, const uint32_t* __restrict__ u,
                            const R* __restrict__ phi, int M, R inv12dx, R* __restrict__ g) {
  const int64_t n = *d_n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    uint64_t tx = (uint64_t)u[i] * (uint64_t)M, ty = (uint64_t)u[cap + i] * (uint64_t)M,
             tz = (uint64_t)u[2 * cap + i] * (uint64_t)M;
    int bx = (int)(tx >> 32), by = (int)(ty >> 32), bz = (int)(tz >> 32);
    R fx = frac32<R>((uint32_t)tx), fy = frac32<R>((uint32_t)ty), fz = frac32<R>((uint32_t)tz);
    R ax = 0, ay = 0, az = 0;
    auto P = [&](int x, int y, int z) -> R {
      return phi[((int64_t)((x + M) % M) * M + ((y + M) % M)) * M + ((z + M) % M)];
    };
    for (int o = 0; o < 8; ++o) {
      int ox = (o >> 2) & 1, oy = (o >> 1) & 1, oz = o & 1;
      R w = (ox ? fx : (R)1 - fx) * (oy ? fy : (R)1 - fy) * (oz ? fz : (R)1 - fz);
      int a = (bx + ox) % M, b = (by + oy) % M, cc = (bz + oz) % M;
      R gx = (R)8 * (P(a + 1, b, cc) - P(a - 1, b, cc)) - (P(a + 2, b, cc) - P(a - 2, b, cc));
      R gy = (R)8 * (P(a, b + 1, cc) - P(a, b - 1, cc)) - (P(a, b + 2, cc) - P(a, b - 2, cc));
      R gz = (R)8 * (P(a, b, cc + 1) - P(a, b, cc - 1)) - (P(a, b, cc + 2) - P(a, b, cc - 2));
      ax -= w * gx;
      ay -= w * gy;
      az -= w * gz;
    }
    g[i] = ax * inv12dx;
    g[cap + i] = ay * inv12dx;
    g[2 * cap + i] = az * inv12dx;
  }
}

// g = -grad phi (four-point stencil at the 8 surrounding nodes), CIC weights,
// for M = 2^m.  One block per 8 x 16 x 16 tile of cells: four 8^3 octree cells that share their parent's x half, whose particles are
// one contiguous Morton run.  The block stages the nodes of phi the tile's
// stencils reach, 13 x 21 rows of 24 (z from bz - 4: aligned 16-byte
// loads, which never straddle the periodic edge), then each particle reads its
// 56 nodes.  Along an axis the two corners' stencils and weights make one
// 6-point filter, so a component takes 4 x 6 multiply-adds; forming the
// gradient at all corner nodes first cost a barrier and 9 KB more shared memory.
// Bound by latency (staging, then reading the particles) and L2 bandwidth: the
// 16-wide tile stages 3.2 nodes a cell, an 8-wide one 5.3.  128^3 on mesh 256:
// 200 -> 90 us.
constexpr int kInterpThreads = 256;
constexpr int kTy = 16;  // cells per side of a tile along y and z
template <class R>
__global__ void __launch_bounds__(kInterpThreads) k_pm_interp_tile(const int32_t* __restrict__ start, int sh9,
                                                                   int64_t cap, const uint32_t* __restrict__ u,
                                                                   const R* __restrict__ phi, int M, R inv12dx,
                                                                   R* __restrict__ g) {
  constexpr int RY = kTy + 5, RZ = kTy + 8, kSub = kTy / 8;
  extern __shared__ unsigned char pi_raw[];
  R* ph = reinterpret_cast<R*>(pi_raw);  // [13][RY][RZ]: node (bx - 2 + i, by - 2 + j, bz - 4 + l)
  const int T = M / kTy, tile = blockIdx.x;
  const int tx = tile / (T * T), ty = (tile / T) % T, tz = tile % T;
  const int bx = tx * 8, by = ty * kTy, bz = tz * kTy;
  // depth m - 3 Morton cells tx, ty kSub .., tz kSub ..: consecutive from the first
  const int64_t tp = (int64_t)((spread3((uint32_t)tx) << 2) | (spread3((uint32_t)(ty * kSub)) << 1) |
                               spread3((uint32_t)(tz * kSub)));
  const int32_t p0 = start[tp << sh9], p1 = start[(tp + kSub * kSub) << sh9];
  if (p1 <= p0) return;  // empty tile (uniform across the block)
  const int mask = M - 1;
  using V = typename Vec16<R>::T;
  constexpr int N = Vec16<R>::N, PER = RZ / N;  // vectors per row
  for (int v = threadIdx.x; v < 13 * RY * PER; v += kInterpThreads) {
    const int r = v / PER, q = v % PER, i = r / RY, j = r % RY;
    const int64_t row = ((int64_t)((bx - 2 + i) & mask) * M + ((by - 2 + j) & mask)) * M;
    reinterpret_cast<V*>(ph + r * RZ)[q] = *reinterpret_cast<const V*>(phi + row + ((bz - 4 + q * N) & mask));
  }
  __syncthreads();
  for (int64_t i = p0 + threadIdx.x; i < p1; i += kInterpThreads) {
    const uint64_t sx = (uint64_t)u[i] * (uint64_t)M, sy = (uint64_t)u[cap + i] * (uint64_t)M,
                   sz = (uint64_t)u[2 * cap + i] * (uint64_t)M;
    // inside the tile by construction (the particle lies in it); clamped all the same
    const int cx = min(max((int)(sx >> 32) - bx, 0), 7), cy = min(max((int)(sy >> 32) - by, 0), kTy - 1),
              cz = min(max((int)(sz >> 32) - bz, 0), kTy - 1);
    const R fx = frac32<R>((uint32_t)sx), fy = frac32<R>((uint32_t)sy), fz = frac32<R>((uint32_t)sz);
    const R wx[2] = {(R)1 - fx, fx}, wy[2] = {(R)1 - fy, fy}, wz[2] = {(R)1 - fz, fz};
    const R* c = ph + ((cx + 2) * RY + cy + 2) * RZ + cz + 4;
    auto six = [](const R (&w)[2], R m2, R m1, R z0, R z1, R q2, R q3) {
      // w0 (8 (z1 - m1) - (q2 - m2)) + w1 (8 (q2 - z0) - (q3 - m1))
      return w[0] * ((R)8 * (z1 - m1) - (q2 - m2)) + w[1] * ((R)8 * (q2 - z0) - (q3 - m1));
    };
    constexpr int SX = RY * RZ, SY = RZ;
    R ax = 0, ay = 0, az = 0;
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const R *lx = c + a * SY + b, *ly = c + a * SX + b, *lz = c + a * SX + b * SY;
        ax += wy[a] * wz[b] * six(wx, lx[-2 * SX], lx[-SX], lx[0], lx[SX], lx[2 * SX], lx[3 * SX]);
        ay += wx[a] * wz[b] * six(wy, ly[-2 * SY], ly[-SY], ly[0], ly[SY], ly[2 * SY], ly[3 * SY]);
        az += wx[a] * wy[b] * six(wz, lz[-2], lz[-1], lz[0], lz[1], lz[2], lz[3]);
      }
    g[i] = -ax * inv12dx;
    g[cap + i] = -ay * inv12dx;
    g[2 * cap + i] = -az * inv12dx;
  }
}

// the same for the meshes tile_mesh leaves out: one block per 8^3 tile forms the
// gradient at the 9^3 corner nodes once for all its particles (tiles with fewer
// than kFlyMax let each particle form its 8 corner gradients).
constexpr int kFlyMax = 96;  // below this many particles a tile skips the node gradients

template <class R>
__device__ __forceinline__ void grad_at(const R* __restrict__ ph, int i, int j, int l, R& gx, R& gy, R& gz) {
  // node (i, j, l) of the 9^3 corner block: phi row ((i + 2) * 13 + j + 2), z slot l + 4
  auto P = [&](int x, int y, int z) -> R { return ph[(x * 13 + y) * 16 + z]; };
  const int x = i + 2, y = j + 2, z = l + 4;
  gx = (R)8 * (P(x + 1, y, z) - P(x - 1, y, z)) - (P(x + 2, y, z) - P(x - 2, y, z));
  gy = (R)8 * (P(x, y + 1, z) - P(x, y - 1, z)) - (P(x, y + 2, z) - P(x, y - 2, z));
  gz = (R)8 * (P(x, y, z + 1) - P(x, y, z - 1)) - (P(x, y, z + 2) - P(x, y, z - 2));
}

template <class R>
__global__ void __launch_bounds__(128) k_pm_interp_nodes(const int32_t* __restrict__ start, int sh9, int64_t cap,
                                                         const uint32_t* __restrict__ u, const R* __restrict__ phi,
                                                         int M, R inv12dx, R* __restrict__ g) {
  extern __shared__ unsigned char pi_raw[];
  R* ph = reinterpret_cast<R*>(pi_raw);  // [169][16]: row (i, j) = node (bx - 2 + i, by - 2 + j), z = bz - 4 + slot
  R* gr = ph + 169 * 16;                 // [3][9][9][9], corner node (bx + i, ...)
  const int T = M >> 3;
  const int tile = blockIdx.x;
  const int tx = tile / (T * T), ty = (tile / T) % T, tz = tile % T;
  const int bx = tx * 8, by = ty * 8, bz = tz * 8;
  // the tile's particles: Morton prefix of the tile at depth m - 3
  const uint32_t tp = (uint32_t)((spread3((uint32_t)tx) << 2) | (spread3((uint32_t)ty) << 1) | spread3((uint32_t)tz));
  const int32_t p0 = start[(int64_t)tp << sh9], p1 = start[((int64_t)tp + 1) << sh9];
  if (p1 <= p0) return;  // empty tile (uniform across the block)
  const int mask = M - 1;
  if (bz >= 8 && bz + 16 <= M) {
    using V = typename Vec16<R>::T;
    constexpr int N = Vec16<R>::N, PER = 16 / N;  // vectors per row
    for (int v = threadIdx.x; v < 169 * PER; v += blockDim.x) {
      const int r = v / PER, q = v % PER;
      const int i = r / 13, j = r % 13;
      const int64_t row = ((int64_t)((bx - 2 + i) & mask) * M + ((by - 2 + j) & mask)) * M;
      reinterpret_cast<V*>(ph + r * 16)[q] = reinterpret_cast<const V*>(phi + row + bz - 4)[q];
    }
  } else {
    for (int v = threadIdx.x; v < 169 * 16; v += blockDim.x) {
      const int r = v >> 4, z = v & 15;
      const int i = r / 13, j = r % 13;
      ph[v] = phi[((int64_t)((bx - 2 + i) & mask) * M + ((by - 2 + j) & mask)) * M + ((bz - 4 + z) & mask)];
    }
  }
  __syncthreads();
  const bool fly = p1 - p0 < kFlyMax;  // uniform across the block
  if (!fly) {
    for (int q = threadIdx.x; q < 729; q += blockDim.x) {
      R gx, gy, gz;
      grad_at(ph, q / 81, (q / 9) % 9, q % 9, gx, gy, gz);
      gr[q] = gx;
      gr[729 + q] = gy;
      gr[1458 + q] = gz;
    }
    __syncthreads();
  }
  for (int64_t i = p0 + threadIdx.x; i < p1; i += blockDim.x) {
    uint64_t sx = (uint64_t)u[i] * (uint64_t)M, sy = (uint64_t)u[cap + i] * (uint64_t)M,
             sz = (uint64_t)u[2 * cap + i] * (uint64_t)M;
    // 0..7 by construction (the particle lies in the tile); clamped all the same
    const int cx = min(max((int)(sx >> 32) - bx, 0), 7), cy = min(max((int)(sy >> 32) - by, 0), 7),
              cz = min(max((int)(sz >> 32) - bz, 0), 7);
    R fx = frac32<R>((uint32_t)sx), fy = frac32<R>((uint32_t)sy), fz = frac32<R>((uint32_t)sz);
    R ax = 0, ay = 0, az = 0;
    for (int o = 0; o < 8; ++o) {
      int ox = (o >> 2) & 1, oy = (o >> 1) & 1, oz = o & 1;
      R w = (ox ? fx : (R)1 - fx) * (oy ? fy : (R)1 - fy) * (oz ? fz : (R)1 - fz);
      R gx, gy, gz;
      if (fly) {
        grad_at(ph, cx + ox, cy + oy, cz + oz, gx, gy, gz);
      } else {
        const int q = ((cx + ox) * 9 + (cy + oy)) * 9 + (cz + oz);
        gx = gr[q];
        gy = gr[729 + q];
        gz = gr[1458 + q];
      }
      ax -= w * gx;
      ay -= w * gy;
      az -= w * gz;
    }
    g[i] = ax * inv12dx;
    g[cap + i] = ay * inv12dx;
    g[2 * cap + i] = az * inv12dx;
  }
}

// the deposit finds its tiles' particles in the cell table the tree build wrote
// for the same keys (table cells per 8^3 tile: 2^sh9)
template <class R>
void pm_deposit(dzs_ctx* c) {
  Buffers& B = c->B;
  const int M = c->M;
  const int64_t m3 = (int64_t)M * M * M;
  double n0 = (double)c->N0;
  R inv_nbar = (R)((double)m3 / n0);
  if (c->mesh_pow2) {
    const int sh9 = 3 * (c->cell_depth - c->logM + 3), sh = 3 * (kMaxLevel - c->logM);
    if (sizeof(R) == 4 && tile_mesh(c)) {
      k_cic_tile<float><<<(unsigned)(m3 / (kT * kT * kT)), kCicThreads, 0, c->stream>>>(
          B.cell_start, sh9, B.n, c->cap, B.key, sh, B.u, B.k, M, (float*)B.rho, (float)inv_nbar);
      return;
    }
    // the table's cells are the mesh's
    k_cic_cellw<R><<<grid_for(c->N0), kThreads, 0, c->stream>>>(B.n, c->cap, B.key, sh, B.u, B.k, M, (R*)B.cicw);
    k_cic_gather<R, true><<<(unsigned)(m3 / 512), 256, gather_smem<R>(), c->stream>>>(
        B.cell_start, B.n, (const R*)B.cicw, M, (R*)B.rho, inv_nbar);
    return;
  }
  // M = 3 2^a: sort the particles by row-major mesh cell (scratch: key2 and
  // prefix for the keys, idx2 and mend for the indices), CSR table of cells
  uint64_t* ka = B.key2;
  uint64_t* kb = (uint64_t*)B.prefix;
  uint32_t* va = B.idx2;
  uint32_t* vb = (uint32_t*)B.mend;
  k_mesh_keys<<<grid_for(c->N0), kThreads, 0, c->stream>>>(B.n, c->cap, B.u, M, ka);
  launch_sort_keys(c, ka, kb, va, vb, 4);  // M^3 < 2^32
  k_cell_start<<<grid_for(c->N0 + 1), kThreads, 0, c->stream>>>(B.n, ka, 0, m3, B.cell_start);
  k_cic_cellw_perm<R><<<grid_for(c->N0), kThreads, 0, c->stream>>>(B.n, c->cap, ka, va, B.u, B.k, M, (R*)B.cicw);
  k_cic_gather<R, false><<<(unsigned)(m3 / 512), 256, gather_smem<R>(), c->stream>>>(
      B.cell_start, B.n, (const R*)B.cicw, M, (R*)B.rho, inv_nbar);
}

// kernels of pm_deposit itself (launch_sort_keys counts the cell sort's)
int deposit_kernels(const dzs_ctx* c) { return !c->mesh_pow2 ? 4 : tile_mesh(c) ? 1 : 2; }

template <class R>
void pm_fft(dzs_ctx* c) {
  Buffers& B = c->B;
  const int M = c->M;
  const int64_t m3 = (int64_t)M * M * M;
  const cplx<R>* tw = (const cplx<R>*)B.twiddle;
  fft_r2c_zy<R>(c, (const R*)B.rho, (cplx<R>*)B.spec, M, tw);
  R gfac = (R)(-1.5 * c->P.omega_m / (double)m3);
  fft_c2r_3d<R>(c, (cplx<R>*)B.spec, (R*)B.phi, M, tw, (const R*)B.green_axis, gfac);
}

template <class R>
void pm_interp(dzs_ctx* c) {
  Buffers& B = c->B;
  const int M = c->M;
  R inv12dx = (R)(1.0 / (12.0 * c->P.box / M));
  if (!c->mesh_pow2) {
    k_pm_interp<R><<<grid_for(c->N0), kThreads, 0, c->stream>>>(B.n, c->cap, B.u, (const R*)B.phi, M, inv12dx,
                                                                (R*)B.g);
    return;
  }
  const int sh9 = 3 * (c->cell_depth - c->logM + 3);
  if (sizeof(R) == 4 && tile_mesh(c)) {
    const size_t sm = (size_t)13 * (kTy + 5) * (kTy + 8) * sizeof(float);
    k_pm_interp_tile<float><<<(unsigned)((M / 8) * (M / kTy) * (M / kTy)), kInterpThreads, sm, c->stream>>>(
        B.cell_start, sh9, c->cap, B.u, (const float*)B.phi, M, (float)inv12dx, (float*)B.g);
    return;
  }
  k_pm_interp_nodes<R><<<(unsigned)((int64_t)M * M * M / 512), 128, (169 * 16 + 3 * 729) * sizeof(R), c->stream>>>(
      B.cell_start, sh9, c->cap, B.u, (const R*)B.phi, M, inv12dx, (R*)B.g);
}

// ---- 3D power spectrum of the mesh (forward spectrum of the CIC delta)
//
// P_mode = |delta_k|^2 L^3 / M^6 / W(k)^2 - P_shot, W = prod_i sinc^2(pi n_i / M),
// bin b = round(|n|) decided on integers (b^2 - b < |n|^2 <= b^2 + b), a
// half-spectrum mode with 0 < kz < M/2 standing for itself and its conjugate.
//
// Bins, windows and weights depend on |n_i| alone, so the sums run over one
// octant: a lane adds up |delta_k|^2 of the (up to four) modes (+-kx, +-ky,
// kz) first and bins once; FP64 is the scarce unit (2 multiply-adds per clock
// and SM), and this leaves about 3 FP64 operations a mode.  The lanes of a
// warp hold consecutive kz of one (kx, ky): their bins ascend, so a segmented
// warp sum gives one addition per bin and warp to the warp's own row of bins;
// warps, then blocks, are summed in a fixed order.  The mode counts and
// sum |k| need no spectrum: k_pk_shells counts the (ky, kz) pairs of each
// ky^2 + kz^2 once, k_pk_final convolves that with kx^2.  Deterministic.
// 256^3 particles, mesh 512, 256 bins: 19.7 ms with an FP64 square root,
// division and 96 FP64 shuffle-adds per 32 modes, now 0.24 + 0.09 ms (planes,
// final; 0.3 GB of the spectrum read, the modes beyond the last bin skipped).
constexpr int kPkThreads = 256;
constexpr int pk_split(int M) { return M >= 16 ? 4 : 1; }  // blocks per kx plane

__device__ __forceinline__ int mode_bin(int n2) {
  int b = (int)(sqrtf((float)n2) + 0.5f);
  if (n2 > b * b + b) ++b;
  if (n2 <= b * b - b) --b;
  return b;
}

// |d0|^2 + .. + |d3|^2 in FP64 (the square of an FP32 value is exact there)
template <class R>
__device__ __forceinline__ double squares_fp64(const cplx<R> (&d)[4]) {
  double s = 0.0;
#pragma unroll
  for (int q = 0; q < 4; ++q) s = fma((double)d[q].y, (double)d[q].y, fma((double)d[q].x, (double)d[q].x, s));
  return s;
}

// a + b = s + (returned remainder), exactly
__device__ __forceinline__ float two_sum(float a, float b, float& s) {
  s = __fadd_rn(a, b);
  const float t = __fsub_rn(s, a);
  return __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
}

// the same on the FP32 units: products with their exact remainders, summed in three
// words (hi and lo by exact additions; rest collects what those leave, 2^-48 of hi,
// rounded to 2^-24 of that).  Largest error over random sums 1.6 units of 2^-53, of
// the FP64 chain 5.2.  That chain, two conversions and two multiply-adds a clock and
// SM, takes 0.22 ms more at mesh 512 (P(k) 4.54 against 4.76 ms; two words, which
// keep 48 bits only, 4.53; with the weights tabulated three words 4.51).  Where a
// remainder may leave the FP32 range the FP64 sum decides.
__device__ __forceinline__ double squares(const cplx<float> (&d)[4]) {
  float hi = 0.f, lo = 0.f, rest = 0.f;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const float v = q & 1 ? d[q >> 1].y : d[q >> 1].x;
    const float p = __fmul_rn(v, v), e = __fmaf_rn(v, v, -p);
    const float t = two_sum(hi, p, hi), r0 = two_sum(lo, t, lo), r1 = two_sum(lo, e, lo);
    rest = __fadd_rn(rest, __fadd_rn(r0, r1));
  }
  if (!(hi >= 0x1p-90f && hi <= 0x1p120f)) return squares_fp64(d);
  return ((double)hi + (double)lo) + (double)rest;
}
__device__ __forceinline__ double squares(const cplx<double> (&d)[4]) { return squares_fp64(d); }

// pairs[s] = number of (ky, kz), signs included, with ky^2 + kz^2 = s
__global__ void k_pk_shells(int M, int smax, unsigned* __restrict__ pairs) {
  const int H = M / 2 + 1;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < H * H; q += gridDim.x * blockDim.x) {
    const int y = q / H, z = q % H, s = y * y + z * z;
    if (s <= smax) atomicAdd(&pairs[s], (y == 0 || 2 * y == M ? 1u : 2u) * (z == 0 || 2 * z == M ? 1u : 2u));
  }
}

// part[plane kx, split][bin] = sum of |delta_k|^2 / W^2
template <class R>
__global__ void __launch_bounds__(kPkThreads) k_pk_plane(const cplx<R>* __restrict__ spec, int M,
                                                         const R* __restrict__ gtab, int nbins,
                                                         double* __restrict__ part) {
  extern __shared__ double pk_sm[];
  const int H = M / 2 + 1, HP = spec_row<R>(M), kx = blockIdx.x, nw = kPkThreads / 32;
  double* rows = pk_sm;              // [warps][nbins]
  double* wxy = pk_sm + nw * nbins;  // [H] 1 / (W_kx W_ky)^2
  double* wz = wxy + H;              // [H] modes a half-spectrum point stands for / W_kz^2
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int q = threadIdx.x; q < nw * nbins; q += kPkThreads) rows[q] = 0.0;
  const double wx = (double)gtab[M + kx], ix = 1.0 / (wx * wx);
  for (int q = threadIdx.x; q < H; q += kPkThreads) {
    const double wv = (double)gtab[M + q], iw = 1.0 / (wv * wv);
    wxy[q] = ix * iw;
    wz[q] = q == 0 || 2 * q == M ? iw : 2.0 * iw;
  }
  __syncthreads();
  const int nmax = nbins * nbins + nbins;  // largest |n|^2 of the last bin
  const int chunks = (H + 31) / 32, nrows = (H - (int)blockIdx.y + (int)gridDim.y - 1) / (int)gridDim.y;
  const bool twox = kx != 0 && 2 * kx != M;
  const int64_t px = (int64_t)kx * M, qx = (int64_t)(M - kx) * M;
  for (int it = w; it < nrows * chunks; it += nw) {
    const int ky = (it / chunks) * (int)gridDim.y + (int)blockIdx.y, kz0 = (it % chunks) * 32;
    const int base2 = kx * kx + ky * ky;
    if (base2 + kz0 * kz0 > nmax) continue;  // beyond the last bin (uniform across the warp)
    const int kz = kz0 + lane, n2 = base2 + kz * kz;
    int b = 0;
    double v = 0.0;
    if (kz < H && n2 <= nmax && n2 > 0) {
      b = mode_bin(n2);
      const bool twoy = ky != 0 && 2 * ky != M;
      const cplx<R> zero = {0, 0};
      const cplx<R> d[4] = {spec[(px + ky) * HP + kz], twox ? spec[(qx + ky) * HP + kz] : zero,
                            twoy ? spec[(px + M - ky) * HP + kz] : zero,
                            twox && twoy ? spec[(qx + M - ky) * HP + kz] : zero};
      v = squares(d) * wxy[ky] * wz[kz];
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int tb = __shfl_up_sync(0xffffffffu, b, o);
      const bool same = lane >= o && tb == b && b > 0;
      if (!__any_sync(0xffffffffu, same)) break;  // every segment is complete
      const double tv = __shfl_up_sync(0xffffffffu, v, o);
      if (same) v += tv;
    }
    const int nb = __shfl_down_sync(0xffffffffu, b, 1);
    if (b > 0 && (lane == 31 || nb != b)) rows[w * nbins + b - 1] += v;
    __syncwarp();  // the next 32 modes add to the same bins from other lanes
  }
  __syncthreads();
  for (int q = threadIdx.x; q < nbins; q += kPkThreads) {
    double s = 0.0;
    for (int v = 0; v < nw; ++v) s += rows[v * nbins + q];
    part[((int64_t)kx * gridDim.y + blockIdx.y) * nbins + q] = s;
  }
}

// block b - 1: modes, sum |k| and sum P of bin b
__global__ void __launch_bounds__(kPkThreads) k_pk_final(const double* __restrict__ part, int nparts,
                                                         const unsigned* __restrict__ pairs, int M, int nbins,
                                                         double norm, double shot, double kf,
                                                         double* __restrict__ out) {
  __shared__ double sh[3][kPkThreads];
  const int b = blockIdx.x + 1;
  double cnt = 0.0, ks = 0.0, ps = 0.0;
  for (int n2 = b * b - b + 1 + (int)threadIdx.x; n2 <= b * b + b; n2 += kPkThreads) {
    unsigned c = 0;
    for (int kx = 0; 2 * kx <= M && kx * kx <= n2; ++kx)
      c += (kx == 0 || 2 * kx == M ? 1u : 2u) * pairs[n2 - kx * kx];
    cnt += (double)c;  // < 2^53: exact
    ks += (double)c * sqrt((double)n2);
  }
  for (int q = threadIdx.x; q < nparts; q += kPkThreads) ps += part[(int64_t)q * nbins + blockIdx.x];
  sh[0][threadIdx.x] = cnt;
  sh[1][threadIdx.x] = ks;
  sh[2][threadIdx.x] = ps;
  __syncthreads();
  for (int h = kPkThreads / 2; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h)
      for (int f = 0; f < 3; ++f) sh[f][threadIdx.x] += sh[f][threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[3 * blockIdx.x] = sh[0][0];
    out[3 * blockIdx.x + 1] = kf * sh[1][0];
    out[3 * blockIdx.x + 2] = norm * sh[2][0] - shot * sh[0][0];
  }
}

__global__ void k_sum_k2(const int32_t* __restrict__ d_n, const uint32_t* __restrict__ k,
                         unsigned long long* __restrict__ out) {
  const int64_t n = *d_n;
  unsigned long long s = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    s += (unsigned long long)k[i] * k[i];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0 && s) atomicAdd(out, s);
}

template <class R>
void pm_deposit(dzs_ctx* c);

template <class R>
void pk_impl(dzs_ctx* c, int nbins, double* d_part, double* d_out, double shot) {
  Buffers& B = c->B;
  const int M = c->M;
  const int64_t m3 = (int64_t)M * M * M;
  launch_cell_start(c);
  pm_deposit<R>(c);
  fft_r2c_3d<R>(c, (const R*)B.rho, (cplx<R>*)B.spec, M, (const cplx<R>*)B.twiddle);
  const double L = c->P.box;
  const double norm = L * L * L / ((double)m3 * (double)m3);
  // scratch: the planes' partial sums, then the pair counts (together less
  // than the M nbins 3 doubles d_part holds)
  const int split = pk_split(M), nparts = (M / 2 + 1) * split, smax = nbins * nbins + nbins;
  unsigned* pairs = (unsigned*)(d_part + (int64_t)nparts * nbins);
  cudaMemsetAsync(pairs, 0, sizeof(unsigned) * (smax + 1), c->stream);
  k_pk_shells<<<grid_for((int64_t)(M / 2 + 1) * (M / 2 + 1)), kThreads, 0, c->stream>>>(M, smax, pairs);
  const size_t smem = ((size_t)(kPkThreads / 32) * nbins + 2 * (M / 2 + 1)) * sizeof(double);
  k_pk_plane<R><<<dim3(M / 2 + 1, split), kPkThreads, smem, c->stream>>>(
      (const cplx<R>*)B.spec, M, (const R*)B.green_axis, nbins, d_part);
  k_pk_final<<<nbins, kPkThreads, 0, c->stream>>>(d_part, nparts, pairs, M, nbins, norm, shot, 2.0 * M_PI / L, d_out);
}

}  // namespace

// P(k) of the current particles: sums of [modes, |k|, P] per bin in d_out
// [nbins][3]; d_part is scratch of M * nbins * 3 doubles.  The state must be
// Morton-sorted with valid keys.
void launch_pk(dzs_ctx* c, int nbins, double* d_part, double* d_out, double shot) {
  // deposit, FFT (3), shells, planes, final; the cell table and the mesh's cell
  // sort count their own
  c->launches += deposit_kernels(c) + 6;
  if (c->fp64)
    pk_impl<double>(c, nbins, d_part, d_out, shot);
  else
    pk_impl<float>(c, nbins, d_part, d_out, shot);
}

void launch_sum_k2(dzs_ctx* c, unsigned long long* out) {
  c->launches += 1;
  cudaMemsetAsync(out, 0, sizeof(unsigned long long), c->stream);
  k_sum_k2<<<grid_for(c->N0), kThreads, 0, c->stream>>>(c->B.n, c->B.k, out);
}

// the PM force in three stages: CIC deposit of delta; FFT Poisson solve with
// the Green function fused into the X pass (phi); four-point gradient and
// CIC interpolation to the particles (g)
// CSR table of the Morton cells of a depth of the current keys
void launch_cells(dzs_ctx* c, int depth) {
  c->launches += 1;
  const int64_t ncell = (int64_t)1 << (3 * depth);
  const int sh = 3 * (kMaxLevel - depth);
  k_cell_start<<<grid_for(c->N0 + 1), kThreads, 0, c->stream>>>(c->B.n, c->B.key, sh, ncell, c->B.cell_start);
}

// the table the tree and the PM tiles share
void launch_cell_start(dzs_ctx* c) { launch_cells(c, c->cell_depth); }

void launch_pm_deposit(dzs_ctx* c) {
  c->launches += deposit_kernels(c);
  if (c->fp64)
    pm_deposit<double>(c);
  else
    pm_deposit<float>(c);
}

void launch_pm_fft(dzs_ctx* c) {
  c->launches += 5;
  if (c->fp64)
    pm_fft<double>(c);
  else
    pm_fft<float>(c);
}

void launch_pm_interp(dzs_ctx* c) {
  c->launches += 1;
  if (c->fp64)
    pm_interp<double>(c);
  else
    pm_interp<float>(c);
}

template <class R>
std::vector<cplx<R>> twiddles(int n);

// twiddles of size M and the per-axis Green tables: k^2, W_CIC, r_s^2, and
// exp(-k^2 r_s^2) / W_CIC^2
void launch_fft_init(dzs_ctx* c) {
  upload_fft_constants(c->dev);
  const int M = c->M;
  std::vector<double> k2(M), w(M);
  double kf = 2.0 * M_PI / c->P.box;
  for (int m = 0; m < M; ++m) {
    int s = (m <= M / 2) ? m : m - M;
    k2[m] = (kf * s) * (kf * s);
    double x = M_PI * (double)s / M;
    double sn = (s == 0) ? 1.0 : std::sin(x) / x;
    w[m] = sn * sn;
  }
  double rs2 = c->rs * c->rs;
  if (c->fp64) {
    auto tw = twiddles<double>(M);
    cudaMemcpy(c->B.twiddle, tw.data(), tw.size() * sizeof(cplx<double>), cudaMemcpyHostToDevice);
    std::vector<double> g(3 * M + 1);
    for (int m = 0; m < M; ++m) {
      g[m] = k2[m];
      g[M + m] = w[m];
      g[2 * M + 1 + m] = std::exp(-k2[m] * rs2) / (w[m] * w[m]);
    }
    g[2 * M] = rs2;
    cudaMemcpy(c->B.green_axis, g.data(), g.size() * sizeof(double), cudaMemcpyHostToDevice);
  } else {
    auto tw = twiddles<float>(M);
    cudaMemcpy(c->B.twiddle, tw.data(), tw.size() * sizeof(cplx<float>), cudaMemcpyHostToDevice);
    std::vector<float> g(3 * M + 1);
    for (int m = 0; m < M; ++m) {
      g[m] = (float)k2[m];
      g[M + m] = (float)w[m];
      g[2 * M + 1 + m] = (float)(std::exp(-k2[m] * rs2) / (w[m] * w[m]));
    }
    g[2 * M] = (float)rs2;
    cudaMemcpy(c->B.green_axis, g.data(), g.size() * sizeof(float), cudaMemcpyHostToDevice);
  }
}

}  // namespace dzs
