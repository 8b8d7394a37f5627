// tree.cu -- oct-tree over the Morton-sorted particles (paper Sec. 2.1: root =
// box, nodes split into octants, nodes carry mass and centre of mass).
//
// The tree is the top-down one (a cell is split when it holds more than B
// particles and is above depth 21), built without a pass per depth.  Every
// node is a Morton cell and starts at a particle: the particle i that opens a
// cell at depth j (its key differs from key[i-1] within the first j octal
// digits, i.e. L_i < j with L_i the digits key[i-1] and key[i] share) owns
// that node exactly when the enclosing depth-(j-1) cell holds more than B
// particles -- when some run of B + 1 consecutive sorted keys around i shares
// j - 1 digits.  So particle i owns the depths L_i < j <= J_i, with
// J_i = min(21, 1 + max over a in [i-B, i] of lcp(key[a], key[a+B])), and its
// node at depth j is internal iff j < J_i.  Likewise (with G for B) the walk
// group of i's chain sits at depth min(J_i, 1 + max lcp over the G-runs).
//
// Nodes are numbered depth by depth, each depth in Morton order, so the
// children of a node are consecutive: a count pass per tile of particles, a
// scan of the per-tile counts of each depth, then a pass in which each owner
// writes its nodes.  A node's first child index is the number of depth-(j+1)
// nodes before its start; the child count is the difference to the next node
// of the same depth.  Node boundaries: down to the cell table's depth m the cell
// ends come from the CSR table of the depth-m Morton cells; deeper, a binary
// search of the keys inside the parent's range.  The numbering depends only
// on the keys (no atomics), so the tree is deterministic.
//
// Node sums in one pass, without a climb: a node's mass and mass-weighted
// position (uint64, exact) are differences of exclusive prefix sums over the
// sorted particles at its range ends (a leaf sums its <= B particles
// directly), giving the rounded integer COM; the largest member
// multiplicity (node softening) starts at 1 everywhere, and only a leaf
// holding a merged particle (k > 1) raises its ancestors' value with
// atomicMax, stopping where an ancestor already holds at least as much (the
// maximum is order-free, so the tree is deterministic).  Walk groups (node
// with <= G particles whose parent holds more, or a leaf) are listed in Morton
// order.
// The two tile kernels are bound by latency and shared-memory reads, not by bytes
// (95 B a particle: 30 us at 128^3): run maxima by doubling, a tile's keys in
// shared memory, first indices by warp scans instead of serial loops, three
// 16-byte stores a node.  Tree stage of the 128^3 set early 228 -> 219 us, late
// (a quarter of the tiles hold particles) 130 -> 107, 256^3 1665 -> 1605.
#include "common.cuh"

namespace dzs {
namespace {

constexpr int kTreeTile = 1024;          // particles per block (one per thread)
constexpr int kHalo = 64;                // largest G (walk_group <= 64)
constexpr int kCols = kMaxLevel + 2;     // node counts per depth 0..21, then walk groups
constexpr unsigned kFull = 0xffffffffu;

// octal digits shared by two keys (21 for equal keys); keys are < 2^63
__device__ __forceinline__ int lcp_digits(uint64_t a, uint64_t b) {
  const uint64_t x = a ^ b;
  return x == 0 ? kMaxLevel : (__clzll((long long)x) - 1) / 3;
}

__device__ __forceinline__ int64_t lb(const uint64_t* __restrict__ key, int64_t lo, int64_t hi, uint64_t x) {
  while (lo < hi) {
    int64_t mid = (lo + hi) >> 1;
    if (key[mid] < x)
      lo = mid + 1;
    else
      hi = mid;
  }
  return lo;
}

// per particle: L_i, J_i and the group depth g_i (packed into info[i]); per
// tile: the number of nodes of each depth and of walk groups its particles own
__global__ void __launch_bounds__(kTreeTile) k_tree_count(const int32_t* __restrict__ d_n,
                                                          const uint64_t* __restrict__ key, int B, int G,
                                                          int32_t* __restrict__ info, int32_t* __restrict__ tcount,
                                                          int64_t ntiles) {
  __shared__ uint64_t ks[kTreeTile + 2 * kHalo];  // keys t0 - kHalo .. t0 + kTreeTile + kHalo
  // 1 + shared digits of the B-run (low half) and the G-run (high half) starting
  // at t0 - kHalo + q, then their maxima over windows of 2, 4, ... runs
  __shared__ uint32_t win[2][kTreeTile + kHalo];
  __shared__ int32_t wcnt[kTreeTile / 32][kCols];
  const int64_t n = *d_n;
  const int64_t t0 = (int64_t)blockIdx.x * kTreeTile;
  if (t0 >= n) {  // no particles (DZS shrinks the set): no nodes
    if (threadIdx.x < kCols) tcount[(int64_t)threadIdx.x * ntiles + blockIdx.x] = 0;
    return;
  }
  for (int q = threadIdx.x; q < kTreeTile + 2 * kHalo; q += kTreeTile) {
    const int64_t a = t0 - kHalo + q;
    ks[q] = (a >= 0 && a < n) ? key[a] : 0ull;
  }
  for (int q = threadIdx.x; q < (kTreeTile / 32) * kCols; q += kTreeTile) (&wcnt[0][0])[q] = 0;
  __syncthreads();
  for (int q = threadIdx.x; q < kTreeTile + kHalo; q += kTreeTile) {
    const int64_t a = t0 - kHalo + q;
    const uint32_t rb = a >= 0 && a + B < n ? lcp_digits(ks[q], ks[q + B]) + 1 : 0;
    const uint32_t rg = a >= 0 && a + G < n ? lcp_digits(ks[q], ks[q + G]) + 1 : 0;
    win[0][q] = rb | (rg << 16);
  }
  __syncthreads();
  const int64_t i = t0 + threadIdx.x;
  const int q = threadIdx.x + kHalo;
  // maxima over the B + 1 and G + 1 runs up to q by doubling (6 shared reads and
  // barriers instead of B + G + 2 reads): two windows of 2^s <= B + 1 cover B + 1
  uint32_t run_b = 0, run_g = 0;
  for (int s = 0, src = 0; (1 << s) <= G + 1; ++s, src ^= 1) {
    if ((2 << s) > B + 1 && (1 << s) <= B + 1) run_b = __vmaxu2(win[src][q], win[src][q - (B + 1 - (1 << s))]) & 0xffffu;
    if ((2 << s) > G + 1) {
      run_g = __vmaxu2(win[src][q], win[src][q - (G + 1 - (1 << s))]) >> 16;
      break;
    }
    for (int e = threadIdx.x; e < kTreeTile + kHalo; e += kTreeTile)
      win[src ^ 1][e] = __vmaxu2(win[src][e], win[src][max(e - (1 << s), 0)]);
    __syncthreads();
  }
  const bool valid = i < n;
  int L = 0, J = -1, g = -1;
  if (valid) {
    L = i > 0 ? lcp_digits(ks[q - 1], ks[q]) : -1;
    J = min(kMaxLevel, (int)run_b);
    g = min(J, (int)run_g);
    info[i] = (L + 1) | (J << 8) | (g << 16);
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const bool owner = valid && L < J;
  const int jlo = __reduce_min_sync(kFull, owner ? L + 1 : kMaxLevel + 1);
  const int jhi = __reduce_max_sync(kFull, owner ? J : -1);
  for (int j = jlo; j <= jhi; ++j) {
    const unsigned b = __ballot_sync(kFull, owner && L < j && j <= J);
    if (lane == 0) wcnt[w][j] = __popc(b);
  }
  const unsigned bg = __ballot_sync(kFull, valid && L < g);
  if (lane == 0) wcnt[w][kCols - 1] = __popc(bg);
  __syncthreads();
  if (threadIdx.x < kCols) {
    int s = 0;
    for (int ww = 0; ww < kTreeTile / 32; ++ww) s += wcnt[ww][threadIdx.x];
    tcount[(int64_t)threadIdx.x * ntiles + blockIdx.x] = s;
  }
}

// block c: exclusive scan of column c of the tile counts, column total to
// lvl[c].  The block that finishes last turns the totals into the node and group
// counts (a tree above the node capacity is not built: error bit, zero nodes and
// groups) and clears what the walk accumulates into.
__global__ void k_tree_scan(int32_t* __restrict__ tcount, int64_t ntiles, int32_t* lvl, int64_t node_cap,
                            uint64_t* counters, uint32_t* __restrict__ err) {
  __shared__ int32_t warp_tot[32];
  __shared__ int32_t carry;
  int32_t* col = tcount + (int64_t)blockIdx.x * ntiles;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int64_t b0 = 0; b0 < ntiles; b0 += blockDim.x) {
    const int64_t b = b0 + threadIdx.x;
    const int32_t v = b < ntiles ? col[b] : 0;
    int32_t inc = v;
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t t = __shfl_up_sync(kFull, inc, o);
      if (lane >= o) inc += t;
    }
    if (lane == 31) warp_tot[w] = inc;
    __syncthreads();
    if (w == 0) {
      const int32_t t = lane < (int)(blockDim.x >> 5) ? warp_tot[lane] : 0;
      int32_t ti = t;
      for (int o = 1; o < 32; o <<= 1) {
        const int32_t u = __shfl_up_sync(kFull, ti, o);
        if (lane >= o) ti += u;
      }
      warp_tot[lane] = ti - t;
    }
    __syncthreads();
    const int32_t ex = inc - v + warp_tot[w] + carry;
    if (b < ntiles) col[b] = ex;
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry = ex + v;
    __syncthreads();
  }
  if (threadIdx.x != 0) return;
  volatile int32_t* tot = lvl;
  tot[blockIdx.x] = carry;
  __threadfence();
  if (atomicAdd((unsigned*)(counters + 16), 1u) != gridDim.x - 1) return;
  __threadfence();
  int64_t total = 0;
  for (int j = 0; j <= kMaxLevel; ++j) total += tot[j];
  if (total > node_cap) {
    atomicOr(err, kErrNodes);
    for (int j = 0; j < kCols; ++j) tot[j] = 0;
    total = 0;
  }
  counters[2] = (uint64_t)tot[kCols - 1];
  counters[3] = (uint64_t)total;
  counters[6] = 0;   // the walk's work counter
  counters[24] = 0;  // its largest spline radius
  *(unsigned*)(counters + 16) = 0u;  // blocks done, for the next tree
}

// every owner writes its nodes: index = (nodes of shallower depths) + (nodes of
// the same depth starting before it); first-child index to cfirst
__global__ void __launch_bounds__(kTreeTile) k_tree_nodes(
    const int32_t* __restrict__ d_n, int64_t cap, const uint64_t* __restrict__ key, const uint32_t* __restrict__ u,
    const int32_t* __restrict__ info, const int32_t* __restrict__ tcount, int64_t ntiles,
    const int32_t* __restrict__ lvl, const int32_t* __restrict__ cstart, int depth_m, int B, Node* __restrict__ nodes,
    int32_t* __restrict__ cfirst, int32_t* __restrict__ parent,
    int32_t* __restrict__ groups) {
  __shared__ int32_t wcnt[kTreeTile / 32][kCols];
  __shared__ int32_t base[kCols];
  __shared__ uint64_t ks[kTreeTile + kHalo];  // keys t0 .. t0 + kTreeTile + kHalo
  const int64_t n = *d_n;
  const int64_t t0 = (int64_t)blockIdx.x * kTreeTile;
  if (t0 >= n) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (w == 0) {
    const int32_t t = lane < kCols ? tcount[(int64_t)lane * ntiles + blockIdx.x] : 0;
    const int32_t v = lane <= kMaxLevel ? lvl[lane] : 0;
    int32_t inc = v;
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t up = __shfl_up_sync(kFull, inc, o);
      if (lane >= o) inc += up;
    }
    // nodes of the shallower depths; groups have a numbering of their own; -1:
    // no tree (over capacity).  One lane writes each slot: the guard below keeps
    // every block off the node array and must not hang on the order of two stores
    const bool none = __shfl_sync(kFull, inc, 31) == 0;
    if (lane < kCols) base[lane] = none ? -1 : t + (lane <= kMaxLevel ? inc - v : 0);
  }
  for (int q = threadIdx.x; q < kTreeTile + kHalo; q += kTreeTile) ks[q] = t0 + q < n ? key[t0 + q] : ~0ull;
  for (int q = threadIdx.x; q < (kTreeTile / 32) * kCols; q += kTreeTile) (&wcnt[0][0])[q] = 0;
  __syncthreads();
  if (base[0] < 0) return;
  const int64_t i = t0 + threadIdx.x;
  const bool valid = i < n;
  int L = 0, J = -1, g = -1;
  if (valid) {
    const int32_t v = info[i];
    L = (v & 0xff) - 1;
    J = (v >> 8) & 0xff;
    g = (v >> 16) & 0xff;
  }
  const unsigned lt = (1u << lane) - 1u;
  const bool owner = valid && L < J;
  // depths whose ranks this warp needs: its nodes' depths and one below
  const int jlo = __reduce_min_sync(kFull, owner ? L + 1 : kMaxLevel + 1);
  const int jhi = min(kMaxLevel, __reduce_max_sync(kFull, owner ? J + 1 : -1));
  for (int j = jlo; j <= jhi; ++j) {
    const unsigned b = __ballot_sync(kFull, owner && L < j && j <= J);
    if (lane == 0) wcnt[w][j] = __popc(b);
  }
  const unsigned bg = __ballot_sync(kFull, valid && L < g);
  if (lane == 0) wcnt[w][kCols - 1] = __popc(bg);
  __syncthreads();
  // warp c turns the counts of column c into each warp's first index
  if (w < kCols) {
    const int32_t v = wcnt[lane][w];
    int32_t inc = v;
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t up = __shfl_up_sync(kFull, inc, o);
      if (lane >= o) inc += up;
    }
    wcnt[lane][w] = base[w] + inc - v;
  }
  __syncthreads();
  const int32_t wbase = lane < kCols ? wcnt[w][lane] : 0;  // lane c: column c
  const uint64_t k = ks[threadIdx.x];
  const uint32_t ux = valid ? u[i] : 0u, uy = valid ? u[cap + i] : 0u, uz = valid ? u[2 * cap + i] : 0u;
  int32_t prev = -1;      // index of this particle's node one depth up
  int64_t prev_end = 0;   // its end
  int32_t gnode = -1;
  for (int j = jlo; j <= jhi; ++j) {
    const bool mine = owner && L < j && j <= J;
    const unsigned b = __ballot_sync(kFull, mine);
    const int32_t rank = __shfl_sync(kFull, wbase, j) + __popc(b & lt);
    if (prev >= 0) cfirst[prev] = rank;  // depth-j nodes before this particle
    if (!mine) {
      prev = -1;
      continue;
    }
    const int sh = 3 * (kMaxLevel - j);
    const uint64_t pref = k >> sh;
    int64_t end;
    if (j <= depth_m) {
      end = cstart[(pref + 1) << (3 * (depth_m - j))];
    } else {
      int64_t hi = prev >= 0 ? prev_end : (int64_t)cstart[(k >> (3 * (kMaxLevel - depth_m))) + 1];
      if (j == J && J < kMaxLevel) hi = min(hi, i + B + 1);  // a leaf above depth 21 holds <= B
      const uint64_t x = (pref + 1) << sh;
      // (a leaf above depth 21 ends within the halo: B < kHalo)
      end = hi <= t0 + kTreeTile + kHalo ? t0 + lb(ks, threadIdx.x + 1, hi - t0, x) : lb(key, i + 1, hi, x);
    }
    const uint32_t half = 1u << (31 - j);
    const uint32_t mask = j == 0 ? 0u : ~((half << 1) - 1u);
    // COM and mass follow from the sums; every member has k >= 1 (raised by the
    // leaves that hold merged particles); an internal node is linked later
    int4* const nd = reinterpret_cast<int4*>(nodes + rank);
    nd[0] = make_int4(0, 0, 0, 0);
    nd[1] = make_int4((int)i, (int)(end - i), j < J ? 0 : -1, j);
    nd[2] = make_int4((int)((ux & mask) | half), (int)((uy & mask) | half), (int)((uz & mask) | half), 1);
    if (j == 0) parent[rank] = -1;
    if (j == g) gnode = rank;
    prev = rank;
    prev_end = end;
  }
  if (prev >= 0) cfirst[prev] = 0;  // depth 21: no children
  const int32_t gbase = __shfl_sync(kFull, wbase, kCols - 1);  // all lanes take part
  if (valid && L < g) groups[gbase + __popc(bg & lt)] = gnode;
}

// internal nodes: first child and child count (to the next node of the same
// depth, or to the end of the next depth), parent links of the children
__global__ void k_tree_link(const int32_t* __restrict__ lvl, Node* __restrict__ nodes,
                            const int32_t* __restrict__ cfirst, int32_t* __restrict__ parent) {
  __shared__ int32_t lb_[kMaxLevel + 3];
  if (threadIdx.x == 0) {
    int32_t s = 0;
    for (int j = 0; j <= kMaxLevel; ++j) {
      lb_[j] = s;
      s += lvl[j];
    }
    lb_[kMaxLevel + 1] = s;
    lb_[kMaxLevel + 2] = s;
  }
  __syncthreads();
  const int64_t total = lb_[kMaxLevel + 1];
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    if (nodes[t].child < 0) continue;
    const int j = (int)(nodes[t].meta & 0xff);
    const int32_t c0 = cfirst[t];
    const int32_t c1 = (t + 1 < lb_[j + 1]) ? cfirst[t + 1] : lb_[j + 2];
    nodes[t].child = c0;
    nodes[t].meta = (uint32_t)j | ((uint32_t)(c1 - c0) << 8);
    for (int32_t q = c0; q < c1; ++q) parent[q] = (int32_t)t;
  }
}

__device__ __forceinline__ void write_mass_com(Node* __restrict__ nodes, int64_t ni, uint64_t K,
                                               const uint64_t (&S)[3]) {
  nodes[ni].mass = (uint32_t)K;
  if (K > 0) {
    nodes[ni].comx = (uint32_t)((2 * S[0] + K) / (2 * K));
    nodes[ni].comy = (uint32_t)((2 * S[1] + K) / (2 * K));
    nodes[ni].comz = (uint32_t)((2 * S[2] + K) / (2 * K));
  }
}

// every node: leaves sum their particles (four loads in flight at a time) and
// raise their ancestors' largest multiplicity when it exceeds 1; internal
// nodes take prefix-sum differences (pre: exclusive [4][cap + 1])
__global__ void k_tree_sums(const int32_t* __restrict__ lvl, int64_t cap, const uint32_t* __restrict__ u,
                            const uint32_t* __restrict__ k, const uint64_t* __restrict__ pre,
                            Node* __restrict__ nodes, const int32_t* __restrict__ parent) {
  int64_t total = 0;
  for (int j = 0; j <= kMaxLevel; ++j) total += lvl[j];
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int32_t s0 = nodes[t].start, cnt = nodes[t].count, child = nodes[t].child;
    uint64_t K = 0, S[3] = {0, 0, 0};
    if (child >= 0) {
      const int64_t e = (int64_t)s0 + cnt;
      K = pre[e] - pre[s0];
      for (int ax = 0; ax < 3; ++ax) S[ax] = pre[(int64_t)(1 + ax) * (cap + 1) + e] - pre[(int64_t)(1 + ax) * (cap + 1) + s0];
      write_mass_com(nodes, t, K, S);
      continue;
    }
    uint32_t kmax = 0;
    const int64_t i1 = (int64_t)s0 + cnt;
    for (int64_t i0 = s0; i0 < i1; i0 += 4) {
      uint32_t kk[4], ux[4], uy[4], uz[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const bool in = i0 + q < i1;
        const int64_t i = in ? i0 + q : i0;
        kk[q] = in ? k[i] : 0u;
        ux[q] = u[i];
        uy[q] = u[cap + i];
        uz[q] = u[2 * cap + i];
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        K += kk[q];
        kmax = max(kmax, kk[q]);
        S[0] += (uint64_t)kk[q] * ux[q];
        S[1] += (uint64_t)kk[q] * uy[q];
        S[2] += (uint64_t)kk[q] * uz[q];
      }
    }
    write_mass_com(nodes, t, K, S);
    nodes[t].kmax = kmax;
    if (kmax > 1)
      for (int32_t a = parent[t]; a >= 0; a = parent[a])
        if (atomicMax(&nodes[a].kmax, kmax) >= kmax) break;  // the rest is raised already (or being raised)
  }
}

}  // namespace

void launch_tree(dzs_ctx* c) {
  c->launches += 5;
  Buffers& B = c->B;
  // the Morton cell table (also the PM tiles')
  launch_cell_start(c);
  const int64_t ntiles = (c->cap + kTreeTile - 1) / kTreeTile;
  int32_t* info = B.group_head;       // [cap] per-particle L, J, g
  int32_t* tcount = B.iscan;          // [kCols][ntiles] tile counts, then offsets
  int32_t* cfirst = B.cfirst;         // [node_cap]
  k_tree_count<<<(unsigned)ntiles, kTreeTile, 0, c->stream>>>(B.n, B.key, c->P.leaf_bucket, c->P.walk_group, info,
                                                              tcount, ntiles);
  k_tree_scan<<<kCols, 1024, 0, c->stream>>>(tcount, ntiles, B.lvl_count, c->node_cap, B.counters, B.err);
  k_tree_nodes<<<(unsigned)ntiles, kTreeTile, 0, c->stream>>>(B.n, c->cap, B.key, B.u, info, tcount, ntiles,
                                                              B.lvl_count, B.cell_start, c->cell_depth, c->P.leaf_bucket,
                                                              B.nodes, cfirst, B.parent, B.groups);
  k_tree_link<<<grid_for(c->node_cap, kThreads, 8), kThreads, 0, c->stream>>>(B.lvl_count, B.nodes, cfirst,
                                                                                     B.parent);
  launch_mass_prefix(c);
  k_tree_sums<<<grid_for(c->node_cap, kThreads, 8), kThreads, 0, c->stream>>>(B.lvl_count, c->cap, B.u, B.k,
                                                                               B.prefix, B.nodes, B.parent);
}

}  // namespace dzs
