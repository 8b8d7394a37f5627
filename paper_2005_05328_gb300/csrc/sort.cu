// sort.cu -- stable LSD radix sort of the 63-bit Morton keys (8-bit digits,
// 8 passes) carrying the particle index, then one gather pass that permutes
// the particle state into Morton order.
//
// The oct-tree of the paper (Sec. 2.1) becomes an implicit octree over the
// sorted keys: every octree cell is a contiguous run of the sorted array.
// One kernel counts the digits of all passes; then each pass is one kernel: a
// block ranks a tile of keys, learns how many keys of each digit the tiles
// before it hold by looking back over their published counts, and writes the
// tile.  Ties keep the previous order, so the result is deterministic.
#include <atomic>
#include <type_traits>

#include "common.cuh"

namespace dzs {
namespace {

constexpr int kSortThreads = 256;
constexpr int kDigits = 256;
constexpr int kPasses = 8;
// Tiles.  Capacity from 2^19 on: 512 threads with 2, 6 or 14 keys each (14: what the
// shared memory of two blocks an SM takes).  The grid holds the capacity in tiles of
// 14, 152 blocks (one an SM) at least; the count decides on the device, as DZS
// shrinks the set under a fixed capacity: the smallest tile of which one wave of the
// grid (two blocks an SM) holds all keys.  Tiles of 14 for every count left most SMs
// without one: sort stage of 66k / 140k / 300k / 541k / 885k keys in a 128^3 context
// 171, 191, 204, 210, 215 us, now 92, 104, 124, 143, 157; 2.1M 247, 249, 16.8M 1510,
// 1490.  A grid of two blocks an SM for 96^3 too, and so 6 keys at 885k, is faster
// alone (165 -> 155 us) but took 2% off eight mocks stepping together.  Below 2^19:
// 256 x 4.
constexpr int kLargeThreads = 512, kLargeItems = 14, kSmallThreads = 256, kSmallItems = 4;
constexpr int kStep1 = 2, kStep2 = 6;
constexpr int64_t kLargeFrom = 1 << 19, kSMs = 152;
__device__ __forceinline__ int tile_items(int n, int tiles) {
  const int wave = kLargeThreads * min(tiles, 2 * (int)kSMs);
  return n <= kStep1 * wave ? kStep1 : n <= kStep2 * wave ? kStep2 : kLargeItems;
}

// status word of a (tile, digit): count in the low 30 bits, and whether it is
// the tile's own count or already the sum over all tiles up to it
constexpr uint32_t kOwn = 1u << 30, kSum = 2u << 30, kCount = kOwn - 1u;
constexpr int kLook = 8;
// polls (about a second) before a look-back counts the earlier tiles' keys itself
constexpr int kLookLimit = 1 << 21;
std::atomic<int> g_look_limit{kLookLimit};

// scratch of a sort (words): digit counts of every pass, a ticket per pass, two
// tables of status words (a pass fills one and clears the other for the next)
constexpr int kOffTicket = kPasses * kDigits, kOffStatus = kOffTicket + 32;

// tiles (blocks) of a context: no count up to cap needs more
inline int64_t sort_tiles(int64_t cap) {
  const int64_t tile = cap >= kLargeFrom ? kLargeThreads * kLargeItems : kSmallThreads * kSmallItems;
  const int64_t full = (cap + tile - 1) / tile;
  return cap >= kLargeFrom && full < kSMs ? kSMs : full;
}
// shared memory of a pass: the tile's keys and values, the warps' counters
constexpr size_t pass_smem(int threads, int items) {
  return (size_t)threads * items * 12 + (size_t)(threads / 32) * kDigits * 2;
}

// counts[pass][digit] over all keys; clears the first status table
__global__ void __launch_bounds__(kSortThreads) k_digit_counts(const uint64_t* __restrict__ key,
                                                               const int32_t* __restrict__ d_n, int passes,
                                                               uint32_t* __restrict__ scratch, int64_t tiles) {
  __shared__ uint32_t cnt[kPasses][kDigits];
  for (int q = threadIdx.x; q < passes * kDigits; q += kSortThreads) (&cnt[0][0])[q] = 0;
  for (int64_t q = (int64_t)blockIdx.x * kSortThreads + threadIdx.x; q < tiles * kDigits;
       q += (int64_t)gridDim.x * kSortThreads)
    scratch[kOffStatus + q] = 0;
  __syncthreads();
  const int64_t n = *d_n;
  const int lane = threadIdx.x & 31;
  // whole warps run every iteration, so that the votes see all lanes
  for (int64_t i0 = (int64_t)blockIdx.x * kSortThreads; i0 < n; i0 += (int64_t)gridDim.x * kSortThreads) {
    const int64_t i = i0 + threadIdx.x;
    const bool valid = i < n;
    const uint64_t k = key[valid ? i : n - 1];
    // nearly sorted input: 32 consecutive keys mostly share their top 15 bits,
    // which would be 32 additions to one counter
    const uint64_t k0 = __shfl_sync(0xffffffffu, k, 0);
    const unsigned take = __ballot_sync(0xffffffffu, valid);
    const bool top = passes == kPasses && __all_sync(0xffffffffu, (k >> 48) == (k0 >> 48));
    if (top && lane < 2) atomicAdd(&cnt[6 + lane][(uint32_t)(k >> (48 + 8 * lane)) & 0xffu], (uint32_t)__popc(take));
    if (valid) {
      const int each = top ? kPasses - 2 : passes;
#pragma unroll
      for (int p = 0; p < kPasses; ++p)
        if (p < each) atomicAdd(&cnt[p][(uint32_t)(k >> (8 * p)) & 0xffu], 1u);
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < passes * kDigits; q += kSortThreads) {
    const uint32_t c = (&cnt[0][0])[q];
    if (c) atomicAdd(&scratch[q], c);
  }
}

// inclusive scan over the threads of a block (warp scans, then the warps' totals)
__device__ __forceinline__ uint32_t block_incl_scan(uint32_t v, uint32_t* wtot) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  if (lane == 31) wtot[w] = v;
  __syncthreads();
  uint32_t before = 0;
  for (int q = 0; q < w; ++q) before += wtot[q];
  return v + before;
}

// lanes holding the same digit (invalid lanes: none in particular), by one
// ballot per bit: a tenth of the time of the match instruction
__device__ __forceinline__ unsigned same_digit(unsigned d, bool valid) {
  unsigned peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    const bool one = (d >> b) & 1u;
    const unsigned v = __ballot_sync(0xffffffffu, one);
    peers &= one ? v : ~v;
  }
  return peers;
}

// One pass.  Tiles are taken by ticket, so every tile before a block's is
// already held by a running block and the look-back ends; should a tile not
// publish within kLookLimit polls, the waiting block counts the digits of the
// keys before it from the pass's input, which nobody writes: no wait is without
// an end and no result depends on one.  A warp ranks its
// own consecutive keys 32 at a time against counters of its own: no block
// barrier inside the ranking (the tile used to pass four per 256 keys).
// The tile is placed in shared memory before the look-back, which gives the
// tiles before it time to publish (8 words in flight; 16 or 32, or one block
// less per SM, were 5-25% slower: polling competes with the ranking).  Bound by
// latency at small n (a launch, one round of loads, the look-back), at large n
// by the look-back and the ranking's instructions (~170 per 32 keys).  Sort
// stage of 33k / 262k / 2.1M / 16.8M particles with three kernels a pass (digit
// counts per tile, row scans, scatter): 137, 154, 317, 1850 us; now 63, 103,
// 230, 1440.  The keys of a thread are passed over in the three groups of its
// possible counts, one uniform branch before each; a body per count spilled (16.8M
// keys 22% slower), a branch per key cost the overlap between keys (2.1M 3%).
template <int kThr, int kItems>
__global__ void __launch_bounds__(kThr, 1024 / kThr)
    k_sort_pass(const uint64_t* __restrict__ kin, const uint32_t* __restrict__ vin, uint64_t* __restrict__ kout,
                uint32_t* __restrict__ vout, const int32_t* __restrict__ d_n, int pass, uint32_t* __restrict__ scratch,
                int tiles, int look_limit) {
  constexpr int kTile = kThr * kItems, kW = kThr / 32;  // the largest tile
  constexpr bool kVar = kItems == kLargeItems;  // keys per thread by the count
  // at most 2^27 keys; 64 bits where registers allow (20011 keys 3% slower with 32)
  using I = std::conditional_t<kVar, int, int64_t>;
  extern __shared__ uint64_t sort_sm[];
  uint64_t* sk = sort_sm;                                           // [kTile] the tile, stably sorted by digit
  uint32_t* sv = reinterpret_cast<uint32_t*>(sk + kTile);           // [kTile]
  uint16_t(*wcnt)[kDigits] = reinterpret_cast<uint16_t(*)[kDigits]>(sv + kTile);  // [kW]
  __shared__ uint32_t gbase[kDigits];  // output position of the tile's first key of each digit
  __shared__ uint32_t lbase[kDigits];  // the same within the tile
  __shared__ uint32_t wtot[2][kW];
  __shared__ int s_tile;
  const I n = *d_n;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5, shift = 8 * pass;
  if (t == 0) s_tile = (int)atomicAdd(&scratch[kOffTicket + pass], 1u);
  for (int q = t; q < kW * kDigits / 2; q += kThr) reinterpret_cast<uint32_t*>(&wcnt[0][0])[q] = 0;
  __syncthreads();
  const int items = kVar ? tile_items((int)n, tiles) : kItems;
  const I tkeys = kThr * items;
  const I tile = s_tile, base = tile * tkeys;
  if (tile >= tiles) return;  // never, unless calls that share the static scratch overlap
  uint32_t* status = scratch + kOffStatus + (pass & 1 ? tiles * kDigits : 0);
  uint32_t* other = scratch + kOffStatus + (pass & 1 ? 0 : tiles * kDigits);
  if (t < kDigits) other[tile * kDigits + t] = 0;  // the next pass's table
  if (base >= n) return;
  const int tile_n = (int)min(n - base, tkeys);
  uint64_t kreg[kItems];
  uint32_t vreg[kItems];
  uint16_t rank[kItems];
  const I i0 = base + w * 32 * items + lane;  // the warp's keys are consecutive
#pragma unroll
  for (int s = 0; s < kItems; ++s) {
    if (kVar && (s == kStep1 || s == kStep2) && s >= items) break;
    const I i = i0 + s * 32;
    kreg[s] = i < n ? kin[i] : 0ull;
    vreg[s] = i < n ? (pass == 0 ? (uint32_t)i : vin[i]) : 0u;  // indices start as the identity
  }
  const uint32_t total = t < kDigits ? scratch[pass * kDigits + t] : 0u;
  const unsigned lt = (1u << lane) - 1u;
#pragma unroll
  for (int s = 0; s < kItems; ++s) {
    if (kVar && (s == kStep1 || s == kStep2) && s >= items) break;
    const bool valid = i0 + s * 32 < n;
    const unsigned d = (unsigned)(kreg[s] >> shift) & 0xffu;
    const unsigned peers = same_digit(d, valid);
    const uint32_t before = valid ? wcnt[w][d] : 0u;
    __syncwarp();
    if (valid && (peers & lt) == 0u) wcnt[w][d] = (uint16_t)(before + __popc(peers));
    __syncwarp();
    rank[s] = (uint16_t)(before + __popc(peers & lt));
  }
  __syncthreads();
  // thread t < 256 owns digit t: warps' counts to offsets, the tile's count
  uint32_t run = 0;
  volatile uint32_t* st = status + t;
  if (t < kDigits) {
#pragma unroll
    for (int q = 0; q < kW; ++q) {
      const uint32_t c = wcnt[q][t];
      wcnt[q][t] = (uint16_t)run;
      run += c;
    }
    st[tile * kDigits] = run | (tile == 0 ? kSum : kOwn);
  }
  const uint32_t local0 = block_incl_scan(run, wtot[0]) - run;
  const uint32_t digit0 = block_incl_scan(total, wtot[1]) - total;
  if (t < kDigits) lbase[t] = local0;
  __syncthreads();
  // place the tile while the tiles before it publish their counts
#pragma unroll
  for (int s = 0; s < kItems; ++s) {
    if (kVar && (s == kStep1 || s == kStep2) && s >= items) break;
    if (i0 + s * 32 < n) {
      const int d = (int)((kreg[s] >> shift) & 0xff);
      const uint32_t lp = lbase[d] + wcnt[w][d] + rank[s];
      sk[lp] = kreg[s];
      sv[lp] = vreg[s];
    }
  }
  // keys of digit t in the tiles before this one, kLook status words in flight
  // at a time (one by one, the ~700 tiles of a wave cost as many L2 latencies)
  if (t < kDigits) {
    uint32_t prev = 0;
    I back = tile - 1;
    for (int polls = 0; back >= 0;) {
      uint32_t v[kLook];
#pragma unroll
      for (int q = 0; q < kLook; ++q) v[q] = back - q >= 0 ? st[(back - q) * kDigits] : 0u;
      I next = back;
      bool open = true;
#pragma unroll
      for (int q = 0; q < kLook; ++q) {
        open = open && (v[q] & (kOwn | kSum)) != 0u;
        if (open) {
          prev += v[q] & kCount;
          next = (v[q] & kSum) ? -1 : next - 1;
          open = next >= 0;
        }
      }
      if (next == back) {
        if (++polls > look_limit) {
          for (I j = 0; j < (back + 1) * tkeys; ++j) prev += ((uint32_t)(kin[j] >> shift) & 0xffu) == (uint32_t)t;
          break;
        }
        __nanosleep(64);
      }
      back = next;
    }
    if (tile > 0) st[tile * kDigits] = (prev + run) | kSum;
    gbase[t] = digit0 + prev;
  }
  __syncthreads();
  // runs of one digit are contiguous in the tile and in the output: coalesced
  for (int q = t; q < tile_n; q += kThr) {
    const uint64_t kv = sk[q];
    const int d = (int)((kv >> shift) & 0xff);
    const uint32_t pos = gbase[d] + (uint32_t)q - lbase[d];
    if ((I)pos < n) {  // always, unless calls that share the static scratch overlap
      kout[pos] = kv;
      vout[pos] = sv[q];
    }
  }
}

// an even number of passes from bit 0; the result is in ka / va again
void sort_passes(uint64_t* ka, uint64_t* kb, uint32_t* va, uint32_t* vb, const int32_t* d_n, int64_t cap, int passes,
                 uint32_t* scratch, cudaStream_t st) {
  const int64_t tiles = sort_tiles(cap);
  const bool large = cap >= kLargeFrom;
  auto kern = large ? k_sort_pass<kLargeThreads, kLargeItems> : k_sort_pass<kSmallThreads, kSmallItems>;
  const int threads = large ? kLargeThreads : kSmallThreads;
  const size_t sm = pass_smem(threads, large ? kLargeItems : kSmallItems);
  if (large) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  cudaMemsetAsync(scratch, 0, sizeof(uint32_t) * kOffStatus, st);
  k_digit_counts<<<grid_for(cap, 2 * kSortThreads, 4), kSortThreads, 0, st>>>(ka, d_n, passes, scratch, tiles);
  uint64_t *kin = ka, *kout = kb;
  uint32_t *vin = va, *vout = vb;
  const int look = g_look_limit.load(std::memory_order_relaxed);
  for (int pass = 0; pass < passes; ++pass) {
    kern<<<(unsigned)tiles, threads, sm, st>>>(kin, vin, kout, vout, d_n, pass, scratch, (int)tiles, look);
    std::swap(kin, kout);
    std::swap(vin, vout);
  }
}

template <class R>
__global__ void k_permute(const int32_t* __restrict__ d_n, int64_t cap, const uint32_t* __restrict__ idx,
                          const uint32_t* __restrict__ u, const R* __restrict__ p,
                          const uint32_t* __restrict__ k, const uint32_t* __restrict__ id,
                          const uint8_t* __restrict__ fl, uint32_t* __restrict__ u2, R* __restrict__ p2,
                          uint32_t* __restrict__ k2, uint32_t* __restrict__ id2, uint8_t* __restrict__ fl2) {
  const int64_t n = *d_n;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    int64_t s = idx[t];
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
      u2[ax * cap + t] = u[ax * cap + s];
      p2[ax * cap + t] = p[ax * cap + s];
    }
    k2[t] = k[s];
    id2[t] = id[s];
    fl2[t] = fl[s];
  }
}

}  // namespace

// words of sort scratch for n keys
size_t sort_scratch_words(int64_t n) {
  return (size_t)kOffStatus + 2 * kDigits * (size_t)sort_tiles(n);
}

// stable LSD radix sort of n keys (an even number of 8-bit passes from bit 0)
// with their indices (identity on input); the result is in ka / va again
void launch_sort_keys(dzs_ctx* c, uint64_t* ka, uint64_t* kb, uint32_t* va, uint32_t* vb, int passes) {
  c->launches += passes + 1;
  sort_passes(ka, kb, va, vb, c->B.n, c->cap, passes, c->B.hist, c->stream);
}

void launch_sort(dzs_ctx* c) {
  c->launches += 1;
  Buffers& B = c->B;
  launch_sort_keys(c, B.key, B.key2, B.idx, B.idx2, kPasses);
  // 8 passes: sorted keys and indices are back in key / idx
  int grid = grid_for(c->N0);
  if (c->fp64)
    k_permute<double><<<grid, kThreads, 0, c->stream>>>(B.n, c->cap, B.idx, B.u, (const double*)B.p, B.k, B.id,
                                                        B.fl, B.u2, (double*)B.p2, B.k2, B.id2, B.fl2);
  else
    k_permute<float><<<grid, kThreads, 0, c->stream>>>(B.n, c->cap, B.idx, B.u, (const float*)B.p, B.k, B.id,
                                                       B.fl, B.u2, (float*)B.p2, B.k2, B.id2, B.fl2);
  std::swap(B.u, B.u2);
  std::swap(B.p, B.p2);
  std::swap(B.k, B.k2);
  std::swap(B.id, B.id2);
  std::swap(B.fl, B.fl2);
}

}  // namespace dzs

// ---- helpers used by the state-injection entry points

namespace dzs {
namespace {

__global__ void k_keys(const int32_t* __restrict__ d_n, int64_t cap, const uint32_t* __restrict__ u,
                       uint64_t* __restrict__ key) {
  const int64_t n = *d_n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    key[i] = morton_key(u[i], u[cap + i], u[2 * cap + i]);
}

// undo the last sort: sorted slot t goes back to idx[t]; g (sorted) is written
// as double in the original order with stride n
template <class R>
__global__ void k_unpermute(const int32_t* __restrict__ d_n, int64_t cap, const uint32_t* __restrict__ idx,
                            const uint32_t* __restrict__ u, const R* __restrict__ p, const R* __restrict__ g,
                            const uint32_t* __restrict__ k, const uint32_t* __restrict__ id,
                            const uint8_t* __restrict__ fl, uint32_t* __restrict__ u2, R* __restrict__ p2,
                            uint32_t* __restrict__ k2, uint32_t* __restrict__ id2, uint8_t* __restrict__ fl2,
                            double* __restrict__ gout) {
  const int64_t n = *d_n;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    int64_t o = idx[t];
    for (int ax = 0; ax < 3; ++ax) {
      u2[ax * cap + o] = u[ax * cap + t];
      p2[ax * cap + o] = p[ax * cap + t];
      gout[ax * n + o] = (double)g[ax * cap + t];
    }
    k2[o] = k[t];
    id2[o] = id[t];
    fl2[o] = fl[t];
  }
}

template <class R>
__global__ void k_close_kick(const int32_t* __restrict__ d_n, int64_t cap, R* __restrict__ p,
                             const R* __restrict__ g, R kick) {
  const int64_t n = *d_n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    for (int ax = 0; ax < 3; ++ax) p[ax * cap + i] += g[ax * cap + i] * kick;
}

}  // namespace

void launch_keys(dzs_ctx* c) {
  c->launches += 1;
  k_keys<<<grid_for(c->N0), kThreads, 0, c->stream>>>(c->B.n, c->cap, c->B.u, c->B.key);
}

void launch_unpermute(dzs_ctx* c, double* g_out) {
  c->launches += 1;
  Buffers& B = c->B;
  int grid = grid_for(c->N0);
  if (c->fp64)
    k_unpermute<double><<<grid, kThreads, 0, c->stream>>>(B.n, c->cap, B.idx, B.u, (const double*)B.p,
                                                          (const double*)B.g, B.k, B.id, B.fl, B.u2,
                                                          (double*)B.p2, B.k2, B.id2, B.fl2, g_out);
  else
    k_unpermute<float><<<grid, kThreads, 0, c->stream>>>(B.n, c->cap, B.idx, B.u, (const float*)B.p,
                                                         (const float*)B.g, B.k, B.id, B.fl, B.u2, (float*)B.p2,
                                                         B.k2, B.id2, B.fl2, g_out);
  std::swap(B.u, B.u2);
  std::swap(B.p, B.p2);
  std::swap(B.k, B.k2);
  std::swap(B.id, B.id2);
  std::swap(B.fl, B.fl2);
}

void launch_close_kick(dzs_ctx* c, int step) {
  c->launches += 1;
  if (c->fp64)
    k_close_kick<double><<<grid_for(c->N0), kThreads, 0, c->stream>>>(c->B.n, c->cap, (double*)c->B.p,
                                                                      (const double*)c->B.g, c->T.kick2[step]);
  else
    k_close_kick<float><<<grid_for(c->N0), kThreads, 0, c->stream>>>(c->B.n, c->cap, (float*)c->B.p,
                                                                     (const float*)c->B.g, (float)c->T.kick2[step]);
}

}  // namespace dzs

// ---- allocation-free Morton sort for callers that cannot allocate device memory
//
// Some callers may not call cudaMalloc at all: code running inside a host
// framework whose device memory is fully owned by its own allocator, plugins
// with a fixed memory budget, or code paths that must not synchronise the
// device (cudaMalloc/cudaFree can).  dzs_morton_sort_noalloc serves them: its
// scratch (keys and indices ping-pong buffers, digit histograms and the
// device-side count) lives in one file-scope static device array of fixed
// size, allocated when the library is loaded and kept until the process exits.
// The caller passes device inputs and outputs; nothing is allocated per call.

#include <mutex>

namespace dzs {
namespace {

constexpr size_t kNoallocMaxN = DZS_NOALLOC_SORT_MAX_N;
// layout: keyA, keyB (uint64), valA, valB (uint32), the passes' scratch (n below
// kLargeFrom: the small tiles), count slot
constexpr size_t kNoallocTiles = (kNoallocMaxN + kSmallThreads * kSmallItems - 1) / (kSmallThreads * kSmallItems);
static_assert(kNoallocMaxN < (size_t)kLargeFrom, "tile size of the allocation-free sort");
constexpr size_t kOffKeyB = 8 * kNoallocMaxN;
constexpr size_t kOffValA = 16 * kNoallocMaxN;
constexpr size_t kOffValB = 20 * kNoallocMaxN;
constexpr size_t kOffHist = 24 * kNoallocMaxN;
constexpr size_t kOffCount = kOffHist + 4 * (kOffStatus + 2 * kDigits * kNoallocTiles);
constexpr size_t kNoallocBytes = kOffCount + 256;

static __device__ __align__(256) unsigned char g_sort_scratch[kNoallocBytes];

std::mutex g_scratch_mu;
void* g_scratch_dev[256] = {nullptr};  // device address per device ordinal

__global__ void k_set_count(int32_t* slot, int32_t n) { *slot = n; }

}  // namespace
}  // namespace dzs

extern "C" dzs_status dzs_morton_sort_noalloc(const uint32_t* d_u, size_t n, uint32_t* d_perm, uint64_t* d_keys,
                                              void* cuda_stream) {
  using namespace dzs;
  if (n > kNoallocMaxN) return DZS_EINVAL;  // above the static scratch capacity
  if (n > 0 && (!d_u || !d_perm)) return DZS_EINVAL;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) return DZS_EDEVICE;
  void* base = nullptr;
  {
    // set-up, once per device, with that device current: the host-side name of
    // the array is not a device address, so ask the runtime for it
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    if (!g_scratch_dev[dev]) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_sort_scratch) != cudaSuccess || !p) return DZS_ECUDA;
      g_scratch_dev[dev] = p;
    }
    base = g_scratch_dev[dev];
  }
  if (n == 0) return DZS_OK;
  // an error left pending by earlier work on this thread is not ours to
  // report or to clear: refuse before launching anything
  if (cudaPeekAtLastError() != cudaSuccess) return DZS_ECUDA;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  char* b = (char*)base;
  uint64_t* keyA = (uint64_t*)b;
  uint64_t* keyB = (uint64_t*)(b + kOffKeyB);
  uint32_t* valA = (uint32_t*)(b + kOffValA);
  uint32_t* valB = (uint32_t*)(b + kOffValB);
  uint32_t* hist = (uint32_t*)(b + kOffHist);
  int32_t* count = (int32_t*)(b + kOffCount);
  // every scratch word read below is first written by this call: the count,
  // the keys, the digit counts and tickets (cleared), the status tables (the
  // first cleared by the counting kernel, each other by the pass before), so
  // nothing left over from a previous call is used
  // each launch is checked with cudaPeekAtLastError (a launch error is sticky
  // for this call's own launches only: nothing was pending before them)
  k_set_count<<<1, 1, 0, st>>>(count, (int32_t)n);
  if (cudaPeekAtLastError() != cudaSuccess) return DZS_ECUDA;
  k_keys<<<grid_for((int64_t)n), kThreads, 0, st>>>(count, (int64_t)n, d_u, keyA);
  if (cudaPeekAtLastError() != cudaSuccess) return DZS_ECUDA;
  sort_passes(keyA, keyB, valA, valB, count, (int64_t)n, kPasses, hist, st);
  if (cudaPeekAtLastError() != cudaSuccess) return DZS_ECUDA;
  if (cudaMemcpyAsync(d_perm, valA, 4 * n, cudaMemcpyDeviceToDevice, st) != cudaSuccess) return DZS_ECUDA;
  if (d_keys && cudaMemcpyAsync(d_keys, keyA, 8 * n, cudaMemcpyDeviceToDevice, st) != cudaSuccess) return DZS_ECUDA;
  return DZS_OK;
}

extern "C" void dzs_debug_sort_look(int32_t polls) {
  dzs::g_look_limit.store(polls < 0 ? dzs::kLookLimit : polls, std::memory_order_relaxed);
}
