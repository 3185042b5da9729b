// Tree stage (Sec. 2.2): canonical Morton-prefix octree, all levels at once
// from the sorted keys (node ranges stay on the device, no host round trip),
// per-node per-species monopoles reduced in double precision (every leaf in
// one launch, then the internal nodes bottom-up), and the walk
// groups.
//
// Canonical tree: nodes are the non-empty Morton cells reachable from the
// root; a cell is a leaf iff it holds <= leaf_size bodies or is at level 20;
// children are the non-empty octants in octant order; nodes are numbered
// level by level, and within a level in key order. Builds inside captured
// steps stop at a level cap two below the deepest level seen by the step
// before the capture (their sort then orders fewer key bits); a cell at the
// cap is then a leaf whatever it holds, and SF_DEPTH says so.
#include "ng_internal.cuh"

namespace ng {

struct Levels {
  uint32_t* start;   // [kMaxLevel + 2]: first node of each level, then end
  uint32_t* count;   // [kMaxLevel + 1]: nodes per level
};

__device__ __forceinline__ Levels levels_of(uint32_t* status) {
  return Levels{status + ST_LEVELS, status + ST_LEVELS + kMaxLevel + 2};
}

// The tree from the sorted keys in one pass over the bodies, all levels at
// once. With common(a, b) the number of octal digits two Morton keys share:
//   delta(i)  = common(key[i - 1], key[i]) (-1 for the first body): body i is
//               the first body of its cells of level delta(i) + 1 and deeper;
//   lambda(i) = 1 + the deepest level whose cell around i holds more than
//               leaf_size bodies (0 if none does), at most lmax. That level is
//               the largest common(key[j], key[j + leaf_size]) over the windows
//               j in [i - leaf_size, i], which are the runs of leaf_size + 1
//               consecutive bodies around i.
// A cell is a node iff its parent holds more than leaf_size bodies, so the
// nodes that start at body i are exactly those of levels delta(i) + 1 ..
// lambda(i); the last of them is a leaf, and the first child of each other
// one is the next. Nodes are numbered level by level, in key order within a
// level: the number of a node is the exclusive scan of the per-level start
// flags laid out level-major, which k_tree_count sums per tile, one device
// scan turns into offsets, and k_tree_emit completes inside the tile.
//
// Bound by reading the keys twice (8 B a body each) and by the launches: three
// to five for any size, where one launch triple per level took 81 (131k
// bodies: about 340 -> 33 us of kernels; 3 M: 560 -> 95 us), and a cluster of
// eight blocks walking the levels of a small tree 92 us at 4096 bodies (now 26).
constexpr int kTreeThreads = 256;
constexpr int kTreeItems = 4;
constexpr int kTreeTile = kTreeThreads * kTreeItems;   // bodies per block
constexpr int kTreeChunks = kTreeTile / 32;            // warp-wide runs of bodies per tile
constexpr int kMaxLeaf = 64;
static_assert(kTreeChunks == 32, "the chunk scan takes one chunk per lane");

// Octal digits that the Morton parts of two keys share (20: the same cell).
__device__ __forceinline__ int common_levels(uint64_t a, uint64_t b) {
  const uint64_t x = (a ^ b) >> 3;
  return x ? 19 - (63 - __clzll((long long)x)) / 3 : kMaxLevel;
}

struct TreeTile {
  uint64_t key[kTreeTile + 2 * kMaxLeaf];
  int8_t w[2][kTreeTile + kMaxLeaf];
};

// The tile's keys into shared memory and delta, lambda of the thread's bodies
// (body it: t0 + it * kTreeThreads + threadIdx.x). Returns the keys' offset:
// body i is sm.key[i - (t0 - leaf)].
__device__ __forceinline__ void tree_tile(TreeTile& sm, const uint64_t* __restrict__ keys, int64_t n,
                                          int64_t t0, int leaf, int lmax, int delta[kTreeItems],
                                          int lambda[kTreeItems]) {
  const int64_t base = t0 - leaf;
  for (int j = threadIdx.x; j < kTreeTile + 2 * leaf; j += kTreeThreads) {
    const int64_t i = base + j;
    sm.key[j] = i >= 0 && i < n ? keys[i] : 0ull;
  }
  __syncthreads();
  const int nw = kTreeTile + leaf;
  for (int j = threadIdx.x; j < nw; j += kTreeThreads) {
    const int64_t i = base + j;
    sm.w[0][j] = i >= 0 && i + leaf < n ? (int8_t)common_levels(sm.key[j], sm.key[j + leaf])
                                        : (int8_t)-1;
  }
  // maximum over windows of `span` entries, doubled while it fits leaf + 1
  int cur = 0, span = 1;
  for (; 2 * span <= leaf + 1; span *= 2) {
    __syncthreads();
    for (int j = threadIdx.x; j < nw; j += kTreeThreads) {
      const int8_t v = sm.w[cur][j];
      sm.w[cur ^ 1][j] = j + span < nw ? max(v, sm.w[cur][j + span]) : v;
    }
    cur ^= 1;
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < kTreeItems; ++it) {
    const int ii = it * kTreeThreads + threadIdx.x;
    const int64_t i = t0 + ii;
    delta[it] = kMaxLevel;
    lambda[it] = -1;   // no node starts here
    if (i < n) {
      delta[it] = i == 0 ? -1 : common_levels(sm.key[ii + leaf - 1], sm.key[ii + leaf]);
      lambda[it] = min(lmax, 1 + max(sm.w[cur][ii], sm.w[cur][ii + leaf + 1 - span]));
    }
  }
}

// cnt[l * gridDim.x + block]: nodes of level l that start in the block's tile.
__global__ void __launch_bounds__(kTreeThreads)
k_tree_count(const uint64_t* __restrict__ keys, int64_t n, int leaf, int lmax,
             uint32_t* __restrict__ cnt) {
  __shared__ TreeTile sm;
  __shared__ uint32_t total[kMaxLevel + 1];
  if (threadIdx.x <= kMaxLevel) total[threadIdx.x] = 0;
  int delta[kTreeItems], lambda[kTreeItems];
  tree_tile(sm, keys, n, (int64_t)blockIdx.x * kTreeTile, leaf, lmax, delta, lambda);
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int it = 0; it < kTreeItems; ++it) {
    const bool has = lambda[it] > delta[it];
    const int lo = __reduce_min_sync(0xffffffffu, has ? delta[it] + 1 : kMaxLevel + 1);
    const int hi = __reduce_max_sync(0xffffffffu, has ? lambda[it] : -1);
    for (int l = lo; l <= hi; ++l) {
      const uint32_t m = __ballot_sync(0xffffffffu, has && delta[it] < l && l <= lambda[it]);
      if (lane == 0 && m) atomicAdd(&total[l], (uint32_t)__popc(m));
    }
  }
  __syncthreads();
  if (threadIdx.x <= lmax) cnt[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = total[threadIdx.x];
}

// Level, prefix, first body and first child of every node (child: for a leaf
// the number the next child of its level would have, so that the child
// counts are differences of neighbours). off: the scanned cnt, with the node
// total in status[ST_NODES_NEEDED]; with SUM, cnt itself, which every block
// then adds up for itself. Block 0 writes the level table and raises
// SF_NODE_OVERFLOW if the nodes exceed the capacity. Clears the group stage's
// sizes and look-back state (its tiles are kGroupPer of these).
constexpr int kGroupThreads = 512, kGroupItems = 8, kGroupTile = kGroupThreads * kGroupItems;
constexpr int kGroupPer = kGroupTile / kTreeTile;

template <bool SUM>
__global__ void __launch_bounds__(kTreeThreads)
k_tree_emit(const uint64_t* __restrict__ keys, int64_t n, int leaf, int lmax,
            const uint32_t* __restrict__ off, uint32_t* status, int64_t cap,
            uint8_t* __restrict__ level, uint64_t* __restrict__ prefix,
            uint32_t* __restrict__ first, uint32_t* __restrict__ child, uint32_t* words,
            uint32_t* __restrict__ gsize, uint64_t* __restrict__ group_lb) {
  __shared__ TreeTile sm;
  __shared__ uint32_t start[kMaxLevel + 2], before[kMaxLevel + 1];   // per level: first node, nodes of earlier tiles
  __shared__ uint32_t pos[kTreeChunks][kMaxLevel + 2];   // per chunk and level: count, then number
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tiles = (int)gridDim.x, tile = (int)blockIdx.x;
  if (SUM) {
    // nodes of each level, and of its tiles before this one
    for (int l = warp; l <= lmax; l += kTreeThreads / 32) {
      uint32_t all = 0, pre = 0;
      for (int t = lane; t < tiles; t += 32) {
        const uint32_t v = off[(size_t)l * tiles + t];
        all += v;
        pre += t < tile ? v : 0u;
      }
      all = __reduce_add_sync(0xffffffffu, all);
      pre = __reduce_add_sync(0xffffffffu, pre);
      if (lane == 0) {
        start[l] = all;
        before[l] = pre;
      }
    }
    __syncthreads();
    if (warp == 0) {
      const uint32_t v = lane <= lmax ? start[lane] : 0u;
      uint32_t inc = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
      }
      __syncwarp();
      if (lane <= kMaxLevel + 1) start[lane] = inc - v;   // past lmax: the total
    }
  } else if (tid <= kMaxLevel + 1) {
    start[tid] = tid <= lmax ? off[(size_t)tid * tiles] : status[ST_NODES_NEEDED];
    if (tid <= lmax) before[tid] = off[(size_t)tid * tiles + tile] - start[tid];
  }
  __syncthreads();
  const uint32_t total = start[kMaxLevel + 1];
  if (tile == 0 && tid < kMonoWords) words[tid] = 0;   // the counters of the next stages
  if (tile == 0 && tid <= kMaxLevel + 1) {
    Levels lv = levels_of(status);
    lv.start[tid] = start[tid];
    if (tid <= kMaxLevel) lv.count[tid] = start[tid + 1] - start[tid];
    if (tid == 0) {
      status[ST_NODES_NEEDED] = total;
      status[ST_NGROUPS] = 0;
      if ((int64_t)total > cap) atomicOr(&status[ST_FLAGS], (uint32_t)SF_NODE_OVERFLOW);
    }
  }
  if (tile % kGroupPer == 0 && tid == 0) group_lb[tile / kGroupPer] = 0;
  for (int64_t i = (int64_t)tile * kTreeTile + tid; i < n && i < (int64_t)(tile + 1) * kTreeTile; i += kTreeThreads)
    gsize[i] = 0;
  for (int j = tid; j < kTreeChunks * (kMaxLevel + 2); j += kTreeThreads) (&pos[0][0])[j] = 0;
  const int64_t t0 = (int64_t)blockIdx.x * kTreeTile;
  int delta[kTreeItems], lambda[kTreeItems], lo[kTreeItems], hi[kTreeItems];
  tree_tile(sm, keys, n, t0, leaf, lmax, delta, lambda);
#pragma unroll
  for (int it = 0; it < kTreeItems; ++it) {
    const bool has = lambda[it] > delta[it];
    lo[it] = __reduce_min_sync(0xffffffffu, has ? delta[it] + 1 : kMaxLevel + 1);
    hi[it] = __reduce_max_sync(0xffffffffu, has ? lambda[it] : -1);
    for (int l = lo[it]; l <= hi[it]; ++l) {
      const uint32_t m = __ballot_sync(0xffffffffu, has && delta[it] < l && l <= lambda[it]);
      if (lane == 0) pos[it * (kTreeThreads / 32) + warp][l] = (uint32_t)__popc(m);
    }
  }
  __syncthreads();
  for (int l = warp; l <= lmax; l += kTreeThreads / 32) {
    const uint32_t v = pos[lane][l];
    uint32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    pos[lane][l] = start[l] + before[l] + inc - v;
  }
  __syncthreads();
  const uint32_t below = (1u << lane) - 1u;
#pragma unroll
  for (int it = 0; it < kTreeItems; ++it) {
    const int chunk = it * (kTreeThreads / 32) + warp;
    const int ii = it * kTreeThreads + tid;
    const bool has = lambda[it] > delta[it];
    const uint64_t key = sm.key[ii + leaf];
    bool prev = false;
    uint32_t id = 0;
    for (int l = lo[it]; l <= hi[it] + 1; ++l) {
      const bool starts = has && delta[it] < l && l <= lambda[it];
      const uint32_t m = __ballot_sync(0xffffffffu, starts);
      const uint32_t r = l <= lmax ? pos[chunk][l] + (uint32_t)__popc(m & below) : total;
      if (prev) child[id] = r;
      prev = starts && (int64_t)r < cap;
      if (prev) {
        id = r;
        level[r] = (uint8_t)l;
        prefix[r] = key >> (3 + 3 * (kMaxLevel - l));
        first[r] = (uint32_t)(t0 + ii);
      }
    }
  }
}

// Body and child counts of every node, each leaf's number at its bodies and
// each child's parent (in its link, for the monopoles' lists). Children are numbered in node order,
// so a node's child count is the difference of its first child and the next
// node's. The next node of the level ends a node with the same parent; the
// last child of a parent finds its end in the keys (doubling steps, then
// bisection). Nodes of level lmax above the leaf size raise SF_DEPTH (lmax
// below kMaxLevel).
__global__ void k_tree_nodes(uint32_t* status, int64_t cap, const uint64_t* __restrict__ keys,
                             int64_t n, int leaf, int lmax, const uint8_t* __restrict__ level,
                             const uint64_t* __restrict__ prefix,
                             const uint32_t* __restrict__ first, const uint32_t* __restrict__ child,
                             uint32_t* __restrict__ count, uint8_t* __restrict__ nchild,
                             uint32_t* __restrict__ bleaf, int4* __restrict__ link) {
  if (status[ST_FLAGS] & SF_NODE_OVERFLOW) return;
  Levels lv = levels_of(status);
  const uint32_t total = lv.start[kMaxLevel + 1];
  for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < total; k += gridDim.x * blockDim.x) {
    const int l = level[k];
    const bool more = k + 1 < lv.start[l + 1];
    const uint64_t pre = prefix[k];
    const uint32_t f = first[k];
    uint32_t end = more ? first[k + 1] : (uint32_t)n;
    if (l > 0 && !(more && (prefix[k + 1] >> 3) == (pre >> 3))) {
      const int shift = 3 + 3 * (kMaxLevel - l);
      uint32_t lo = f, step = 1;   // keys[lo] is in the cell
      while (step < end - lo && (keys[lo + step] >> shift) == pre) {
        lo += step;
        step <<= 1;
      }
      uint32_t hi = step < end - lo ? lo + step : end;   // keys[hi] is not (or hi is the bound)
      while (hi - lo > 1) {
        const uint32_t mid = lo + ((hi - lo) >> 1);
        if ((keys[mid] >> shift) == pre) lo = mid; else hi = mid;
      }
      end = hi;
    }
    count[k] = end - f;
    const uint32_t nch = l < lmax ? (more ? child[k + 1] : lv.start[l + 2]) - child[k] : 0u;
    nchild[k] = (uint8_t)nch;
    if (nch == 0) {
      for (uint32_t b = f; b < end; ++b) bleaf[b] = k;
    } else {
      const uint32_t c0 = child[k];
      for (uint32_t j = 0; j < nch; ++j) link[c0 + j].w = (int)k;   // until its monopoles are formed
    }
    if (l == lmax && lmax < kMaxLevel && end - f > (uint32_t)leaf)
      atomicOr(&status[ST_FLAGS], (uint32_t)SF_DEPTH);
  }
}

size_t tree_scratch_bytes(int64_t n) {   // node counts per level and tile
  return (size_t)((n + kTreeTile - 1) / kTreeTile) * (kMaxLevel + 1) * sizeof(uint32_t);
}

size_t group_lookback_bytes(int64_t n) {
  return (size_t)((n + kGroupTile - 1) / kGroupTile) * sizeof(uint64_t);
}

constexpr int kSumTiles = 256;

int build_octree(ng_ctx* c) {
  const int64_t n = c->n;
  const int64_t cap = c->cap_nodes;
  uint32_t* st = as<uint32_t>(c->status);
  const uint64_t* keys = as<uint64_t>(c->keys_a);
  uint32_t* cnt = as<uint32_t>(c->tree_cnt);
  const int leaf = c->p.leaf_size;
  const int lmax = std::min(std::max(c->level_cap, 0), kMaxLevel);
  const int tiles = (int)((n + kTreeTile - 1) / kTreeTile);
  stage_mark(c, NG_STAGE_OCTREE);
  k_tree_count<<<tiles, kTreeThreads, 0, c->stream>>>(keys, n, leaf, lmax, cnt);
  // up to kSumTiles tiles, adding their counts up again in every block costs
  // less than a scan's launch (4096 bodies: 3.6 us; 131k: 5.5 us)
  const bool sum = tiles <= kSumTiles;
  if (!sum) NG_TRY(scan_u32(c, cnt, cnt, (int64_t)tiles * (lmax + 1), st + ST_NODES_NEEDED));
  (sum ? k_tree_emit<true> : k_tree_emit<false>)<<<tiles, kTreeThreads, 0, c->stream>>>(
      keys, n, leaf, lmax, cnt, st, cap, as<uint8_t>(c->n_level), as<uint64_t>(c->n_prefix),
      as<uint32_t>(c->n_first), as<uint32_t>(c->n_child),
      as<uint32_t>(c->mono_words), as<uint32_t>(c->gsize), as<uint64_t>(c->group_lb));
  k_tree_nodes<<<work_grid(c, std::min<int64_t>(cap, 2 * n + 64), 8), 256, 0, c->stream>>>(
      st, cap, keys, n, leaf, lmax, as<uint8_t>(c->n_level), as<uint64_t>(c->n_prefix),
      as<uint32_t>(c->n_first), as<uint32_t>(c->n_child), as<uint32_t>(c->n_count),
      as<uint8_t>(c->n_nchild), as<uint32_t>(c->bleaf), as<int4>(c->n_link));
  c->launches += 3;   // count, emit, nodes (the scan counts itself)
  NG_CUDA(c, cudaGetLastError());
  return NG_OK;
}

// --------------------------------------------------------- monopoles


struct MonoArgs {
  const uint8_t* level;
  const uint64_t* prefix;
  const uint32_t* first;
  const uint32_t* count;
  const uint8_t* nchild;
  const uint32_t* child;
  const double* spos;      // [3][n] physical
  const float* smass;
  const uint8_t* stype;
  double* m64;             // [node][D][4]: mass, sum m x, sum m y, sum m z (box units)
  uint32_t* cnt;           // [node][D]
  float4* geo;
  float4* com;
  int4* link;
  float4* mono;            // [node][D]
  float4* body;            // [sorted body]
  uint32_t* bleaf;         // [sorted body] leaf index
  uint32_t* status;
  int64_t n;
  double invL, L;
  bool unit;               // L == 1: physical and box units are the same
};

// Below kBinnedMonoBodies bodies, and for small leaves, leaves are summed from tiles of consecutive
// bodies in shared memory: the body arrays are read once, coalesced, and every
// body's record (offset from its leaf's centre, subtracted in FP64 in physical
// units, scaled to box units in FP32) is written coalesced. A leaf is then summed by one thread
// (FP64 is ~1/64 of the FP32 rate here, so every FP64 operation counts): it
// adds each body to its own species, 4 FP64 operations per body, in
// shared-memory slots chosen by the species. A warp instruction costs the
// same with idle lanes, so the tile's leaves are taken in the order of their
// body counts: the threads of a warp then have about equal loop counts. An
// internal node is summed by one lane per species and component over its <= 8
// children, in child order. The FP32 walk records need no FP64 division: the mass-weighted
// offset sum(m x) - M c is formed with one FP64 FMA and divided by M in FP32.
constexpr int kMonoThreads = 128;

// The walk record {com - centre, mass} of FP64 sums about centre cen.
__device__ __forceinline__ float4 mono_record(double m, double x, double y, double z,
                                              const double cen[3]) {
  if (!(m > 0.0)) return make_float4(0.f, 0.f, 0.f, 0.f);
  const float mf = (float)m, im = 1.0f / mf;
  return make_float4((float)fma(-m, cen[0], x) * im, (float)fma(-m, cen[1], y) * im,
                     (float)fma(-m, cen[2], z) * im, mf);
}

// Lanes of an internal node's team: 4 components {m, m x, m y, m z} for each
// of walk_tab_pad(D) species. The children's records are contiguous, so a
// team reads whole lines, and a warp issues an FP64 instruction per child
// rather than four.
template <int D>
constexpr int kTeam = 4 * walk_tab_pad(D);

// An internal node as its team needs it, loaded ahead of the children's sums.
struct MonoNode {
  uint32_t k, nch, c0;   // nch = 0: no node
  uint32_t parent;
  int level;
  uint64_t prefix;
};
__device__ __forceinline__ MonoNode mono_load(bool valid, uint32_t k, const MonoArgs& a) {
  MonoNode v{k, 0u, 0u, 0u, 0, 0ull};
  if (valid) {
    v.nch = a.nchild[k];
    v.c0 = a.child[k];
    v.parent = (uint32_t)a.link[k].w;   // left there by k_tree_nodes
    v.level = a.level[k];
    v.prefix = a.prefix[k];
  }
  return v;
}

// geo of a node, {centre, half side} in box units: exact in FP32 (a centre
// is an odd number below 2^22 over a power of two).
__device__ __forceinline__ float4 mono_geo(int level, uint64_t prefix) {
  const float h = __int_as_float((127 - (level + 1)) << 23);   // 2^-(level + 1)
  return make_float4((float)(2u * morton_compact3(prefix >> 2) + 1u) * h,
                     (float)(2u * morton_compact3(prefix >> 1) + 1u) * h,
                     (float)(2u * morton_compact3(prefix) + 1u) * h, h);
}

// Sum of internal node v over its children by the kTeam<D> lanes of its team:
// the lane's component of its species, stored for the parent. All lanes of the
// warp call it together. The additions form a tree (FP64 results come tens of
// cycles apart, and a path to the root makes them at each of its levels).
template <int D>
__device__ __forceinline__ double mono_sum(const MonoNode& v, const MonoArgs& a) {
  constexpr int P = walk_tab_pad(D);
  const int lane = threadIdx.x & 31, e = lane & 3, q = (lane >> 2) & (P - 1);
  const bool mine = v.nch > 0 && q < D;
  double c[8];
  uint32_t cn = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    c[j] = 0.0;
    if (mine && j < (int)v.nch) {
      const size_t r = (size_t)(v.c0 + j) * D + q;
      c[j] = __ldcg(a.m64 + r * 4 + e);   // of any SM: past this one's L1
      if (e == 0) cn += __ldcg(a.cnt + r);
    }
  }
  // no further than the longest list of the warp
  double sum = c[0] + c[1];
  const int most = (int)__reduce_max_sync(0xffffffffu, v.nch);
  if (most > 2) sum += c[2] + c[3];
  if (most > 4) sum += (c[4] + c[5]) + (c[6] + c[7]);
  if (mine) {
    const size_t r = (size_t)v.k * D + q;
    a.m64[r * 4 + e] = sum;
    if (e == 0) a.cnt[r] = cn;
  }
  return sum;
}

// The walk's records of node v from the lanes' sums.
template <int D>
__device__ __forceinline__ void mono_node_records(const MonoNode& v, double sum, const MonoArgs& a) {
  constexpr int P = walk_tab_pad(D);
  const int lane = threadIdx.x & 31, e = lane & 3, q = (lane >> 2) & (P - 1);
  // over the species (zero in idle lanes), for the node's own centre of mass
  double all = sum;
#pragma unroll
  for (int o = 4; o < kTeam<D>; o <<= 1) all += __shfl_xor_sync(0xffffffffu, all, o);
  const double m = __shfl_sync(0xffffffffu, sum, 0, 4), mt = __shfl_sync(0xffffffffu, all, 0, 4);
  if (v.nch == 0 || q >= D) return;
  double cen[3], side;
  node_centre(v.level, v.prefix, cen, &side);
  const double ce = e == 1 ? cen[0] : e == 2 ? cen[1] : cen[2];
  // records {com - centre, mass}: component e - 1, or the mass for e = 0
  const size_t r = (size_t)v.k * D + q;
  const int at = (e + 3) & 3;
  const float mf = (float)m, f = e == 0 ? mf : (float)fma(-m, ce, sum) * (1.0f / mf);
  reinterpret_cast<float*>(a.mono)[r * 4 + at] = m > 0.0 ? f : 0.f;
  if (q == 0) {
    const float tf = (float)mt, g = e == 0 ? tf : (float)fma(-mt, ce, all) * (1.0f / tf);
    reinterpret_cast<float*>(a.com)[(size_t)v.k * 4 + at] = mt > 0.0 ? g : 0.f;
    if (e == 0) a.geo[v.k] = mono_geo(v.level, v.prefix);
    if (e == 1) a.link[v.k] = make_int4((int)v.c0, (int)v.nch, (int)a.first[v.k], (int)a.count[v.k]);
  }
}

// The same sums by the calling lane alone, all species: an FP64 instruction
// then serves 32 nodes, against 32 / kTeam<D> in teams, for four times as many
// of them in a row.
template <int D>
__device__ __forceinline__ void mono_internal_lane(const MonoNode& v, const MonoArgs& a) {
  if (v.nch == 0) return;
  double sm[D], sx[D], sy[D], sz[D];
  uint32_t sc[D];
#pragma unroll
  for (int q = 0; q < D; ++q) { sm[q] = sx[q] = sy[q] = sz[q] = 0.0; sc[q] = 0; }
  for (uint32_t j = 0; j < v.nch; ++j) {
    const size_t r = (size_t)(v.c0 + j) * D;
#pragma unroll
    for (int q = 0; q < D; ++q) {
      const double4_32a c = *reinterpret_cast<const double4_32a*>(a.m64 + (r + q) * 4);
      sm[q] += c.x;
      sx[q] += c.y;
      sy[q] += c.z;
      sz[q] += c.w;
      sc[q] += a.cnt[r + q];
    }
  }
  double cen[3], side;
  node_centre(v.level, v.prefix, cen, &side);
  double mt = 0, xt = 0, yt = 0, zt = 0;
#pragma unroll
  for (int q = 0; q < D; ++q) {
    const size_t r = (size_t)v.k * D + q;
    *reinterpret_cast<double4_32a*>(a.m64 + r * 4) = make_double4_32a(sm[q], sx[q], sy[q], sz[q]);
    a.cnt[r] = sc[q];
    a.mono[r] = mono_record(sm[q], sx[q], sy[q], sz[q], cen);
    mt += sm[q];
    xt += sx[q];
    yt += sy[q];
    zt += sz[q];
  }
  a.geo[v.k] = mono_geo(v.level, v.prefix);
  a.com[v.k] = mono_record(mt, xt, yt, zt, cen);
  a.link[v.k] = make_int4((int)v.c0, (int)v.nch, (int)a.first[v.k], (int)a.count[v.k]);
}

// Internal nodes are summed bottom-up without waiting: a node's link holds, until
// it is formed, its parent (w, from k_tree_nodes) and how many of its internal
// children are not formed yet (x). Who forms a node takes one off its parent's
// count, and who takes the last one forms the parent next. The nodes without
// internal children are ready at the start.
// Which sum a node takes, pairwise in a team (mono_sum) or child by child in a
// lane (mono_internal_lane: the nodes without internal children of trees of
// kBinnedMonoBodies bodies or more), is set by the tree, so results repeat.
// Bound by latency: a level of a path costs two dependent loads, the additions
// and one counter. Subtrees of 256 bodies by one block each, level by level
// with barriers, and a cluster of eight blocks for the nodes above took 88 us at
// 131k bodies and three species, 175 us at 300k and six; this 48 and 59 us. (A
// 131k-body force 687 -> 651 us, a 300k-body tree force 981 -> 894 us, a
// 200k-body step 713 -> 660 us, all with the tiles' loads below.)
//
// Counters (c->mono_words, zeroed by k_tree_emit): ready nodes (trees whose
// leaves go by tiles; listed in n_tmp), nodes listed by k_mono_ready, and the
// tiles of the group list.
constexpr int kMlReady = 0, kMlNext = 1, kGroupTicket = 2;
static_assert(kGroupTicket + 1 == kMonoWords && kMonoWords <= kTreeThreads, "counters");

// Internal children of node k
__device__ __forceinline__ int mono_pending(uint32_t k, uint32_t nch, const MonoArgs& a) {
  const uint32_t c0 = nch ? a.child[k] : 0u;
  int need = 0;
  for (uint32_t j = 0; j < nch; ++j) need += a.nchild[c0 + j] != 0;
  return need;
}

// One internal child of the node with this count is formed: the count before.
// What this thread (and, past a warp barrier, its warp) has written is seen by
// whoever finds the count at one, past its own.
__device__ __forceinline__ int mono_done(int* pending) {
  int v;
  asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], -1;" : "=r"(v) : "l"(pending) : "memory");
  return v;
}

// Tile: bodies whose leaves start in a block's turn (small, so that a small
// tree's leaves reach many SMs); a leaf may reach kMaxLeaf bodies into the next.
constexpr int kLeafThreads = 64, kLeafTile = 256, kLeafLoad = kLeafTile + kMaxLeaf;
template <int D>
struct LeafSmem {
  double x[3][kLeafLoad];
  float m[kLeafLoad];
  double acc[D][4][kLeafThreads];        // {m, m x, m y, m z} per species, physical units
  uint32_t start[kLeafTile];             // per leaf of the tile: local start | count class << 16
  uint32_t leaf[kLeafTile];              // and its node
  uint32_t order[kLeafTile];             // leaves in count order
  uint32_t heads[kLeafTile / 32];        // bodies that start a leaf
  uint32_t bins[kMaxLeaf + 2];
  uint8_t t[kLeafLoad];
};

// Every leaf and body record, one tile of bodies per block and turn; the
// counts of the internal nodes, and the list of those that are ready.
template <int D>
__global__ void __launch_bounds__(kLeafThreads) k_mono_tiles(MonoArgs a, uint32_t* words, uint32_t* ready) {
  __shared__ LeafSmem<D> sm;
  if (a.status[ST_FLAGS] & SF_NODE_OVERFLOW) return;   // truncated tree: do not read it
  const int tid = threadIdx.x;
  const uint32_t total = levels_of(a.status).start[kMaxLevel + 1];
  for (uint32_t k0 = blockIdx.x * blockDim.x + (tid & ~31); k0 < total; k0 += gridDim.x * blockDim.x) {
    // warps step together
    const uint32_t k = k0 + (tid & 31), nch = k < total ? a.nchild[k] : 0u;
    const int need = mono_pending(k, nch, a);
    if (nch) a.link[k].x = need;
    const uint32_t list = __ballot_sync(0xffffffffu, nch != 0 && need == 0);
    uint32_t at = 0;
    if ((tid & 31) == 0 && list) at = atomicAdd(&words[kMlReady], (uint32_t)__popc(list));
    at = __shfl_sync(0xffffffffu, at, 0) + __popc(list & ((1u << (tid & 31)) - 1u));
    if (nch != 0 && need == 0) ready[at] = k;
  }
  const float invLf = (float)a.invL;
  for (int64_t t0 = (int64_t)blockIdx.x * kLeafTile; t0 < a.n; t0 += (int64_t)gridDim.x * kLeafTile) {
    __syncthreads();   // the previous tile's readers are done
    const int held = (int)min((int64_t)kLeafLoad, a.n - t0), own = min(held, kLeafTile);
    for (int j = tid; j < kMaxLeaf + 2; j += kLeafThreads) sm.bins[j] = 0;
    constexpr int kRounds = kLeafLoad / kLeafThreads, kOwnRounds = kLeafTile / kLeafThreads;
    constexpr int kLeafWarps = kLeafThreads / 32;
    uint32_t leaf[kOwnRounds];
    bool head[kOwnRounds];
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
      // no barrier between the rounds: their loads overlap
      const int j = r * kLeafThreads + tid;
      const int64_t b = t0 + j;
      double xp = 0, yp = 0, zp = 0;
      float m = 0.f;
      if (j < held) {
        xp = a.spos[b];
        yp = a.spos[a.n + b];
        zp = a.spos[2 * a.n + b];
        m = a.smass[b];
        sm.x[0][j] = xp;
        sm.x[1][j] = yp;
        sm.x[2][j] = zp;
        sm.m[j] = m;
        sm.t[j] = a.stype[b];
      }
      if (r < kOwnRounds) {
        head[r] = false;
        leaf[r] = 0;
        if (j < own) {
          const uint32_t k = leaf[r] = a.bleaf[b];
          head[r] = b == 0 || a.bleaf[b - 1] != k;
          double cen[3], side;
          node_centre(a.level[k], a.prefix[k], cen, &side);
          if (!a.unit) {
            cen[0] *= a.L;
            cen[1] *= a.L;
            cen[2] *= a.L;
          }
          a.body[b] = make_float4((float)(xp - cen[0]) * invLf, (float)(yp - cen[1]) * invLf,
                                  (float)(zp - cen[2]) * invLf, m);
        }
        const uint32_t heads = __ballot_sync(0xffffffffu, head[r]);
        if ((tid & 31) == 0) sm.heads[r * kLeafWarps + (tid >> 5)] = heads;
      }
    }
    __syncthreads();
    uint32_t nleaf = 0;   // leaves that start in the tile (the same in every thread)
#pragma unroll
    for (int w = 0; w < kLeafTile / 32; ++w) {
      const uint32_t heads = sm.heads[w];
      if (w % kLeafWarps == (tid >> 5) && head[w / kLeafWarps]) {
        const uint32_t at = nleaf + __popc(heads & ((1u << (tid & 31)) - 1u));
        sm.start[at] = (uint32_t)(w / kLeafWarps * kLeafThreads + tid);
        sm.leaf[at] = leaf[w / kLeafWarps];
      }
      nleaf += __popc(heads);
    }
    __syncthreads();
    // the leaves by body count (one class for those above kMaxLeaf)
    for (uint32_t i = tid; i < nleaf; i += kLeafThreads) {
      const uint32_t cls = min(a.count[sm.leaf[i]], (uint32_t)(kMaxLeaf + 1));
      sm.start[i] |= cls << 16;
      atomicAdd(&sm.bins[cls], 1u);
    }
    __syncthreads();
    if (tid < 32) {
      uint32_t run = 0;
      for (int c = kMaxLeaf + 1; c >= 0; c -= 32) {   // longest first
        const int j = c - tid;
        const uint32_t v = j >= 0 ? sm.bins[j] : 0u;
        uint32_t inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t x = __shfl_up_sync(0xffffffffu, inc, o);
          if (tid >= o) inc += x;
        }
        if (j >= 0) sm.bins[j] = run + inc - v;
        run += __shfl_sync(0xffffffffu, inc, 31);
      }
    }
    __syncthreads();
    for (uint32_t i = tid; i < nleaf; i += kLeafThreads)
      sm.order[atomicAdd(&sm.bins[sm.start[i] >> 16], 1u)] = i;
    __syncthreads();
    for (uint32_t i = tid; i < nleaf; i += kLeafThreads) {
      const uint32_t at = sm.order[i], k = sm.leaf[at], cls = sm.start[at] >> 16;
      const uint32_t c = cls <= (uint32_t)kMaxLeaf ? cls : a.count[k];
      const int j0 = (int)(sm.start[at] & 0xffffu);
      uint32_t sc[D];
#pragma unroll
      for (int q = 0; q < D; ++q) {
        sc[q] = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) sm.acc[q][e][tid] = 0.0;
      }
      for (uint32_t h = 0; h < c; ++h) {
        const int j = j0 + (int)h;
        double xp, yp, zp, md;
        int t;
        if (j < held) {
          xp = sm.x[0][j];
          yp = sm.x[1][j];
          zp = sm.x[2][j];
          md = (double)sm.m[j];
          t = sm.t[j];
        } else {   // a leaf above kMaxLeaf bodies (a tree stopped at a level cap)
          const int64_t b = t0 + j;
          xp = a.spos[b];
          yp = a.spos[a.n + b];
          zp = a.spos[2 * a.n + b];
          md = (double)a.smass[b];
          t = a.stype[b];
        }
        sm.acc[t][0][tid] += md;
        sm.acc[t][1][tid] = fma(md, xp, sm.acc[t][1][tid]);
        sm.acc[t][2][tid] = fma(md, yp, sm.acc[t][2][tid]);
        sm.acc[t][3][tid] = fma(md, zp, sm.acc[t][3][tid]);
#pragma unroll
        for (int q = 0; q < D; ++q) sc[q] += t == q ? 1u : 0u;
      }
      double cen[3], side;
      node_centre(a.level[k], a.prefix[k], cen, &side);
      double mt = 0, xt = 0, yt = 0, zt = 0;
#pragma unroll
      for (int q = 0; q < D; ++q) {
        // to box units (exact when the box is a power of two)
        const double m = sm.acc[q][0][tid];
        double x = sm.acc[q][1][tid], y = sm.acc[q][2][tid], z = sm.acc[q][3][tid];
        if (!a.unit) {
          x *= a.invL;
          y *= a.invL;
          z *= a.invL;
        }
        // 32-byte records from a cudaMalloc base: one aligned 32-byte access each
        *reinterpret_cast<double4_32a*>(a.m64 + ((size_t)k * D + q) * 4) = make_double4_32a(m, x, y, z);
        a.cnt[(size_t)k * D + q] = sc[q];
        a.mono[(size_t)k * D + q] = mono_record(m, x, y, z, cen);
        mt += m;
        xt += x;
        yt += y;
        zt += z;
      }
      a.geo[k] = mono_geo(a.level[k], a.prefix[k]);
      a.com[k] = mono_record(mt, xt, yt, zt, cen);
      a.link[k] = make_int4(-1, 0, (int)(t0 + j0), (int)c);
    }
  }
}

// The listed nodes and all above them: a team takes a listed node, forms it,
// and goes on with the parent where that was the last child it waited for, else
// with its next listed node. Nothing waits: a path from a leaf to the root
// costs its loads and one counter per level.
template <int D>
__global__ void __launch_bounds__(kMonoThreads) k_mono_up(MonoArgs a, const uint32_t* __restrict__ list,
                                                          const uint32_t* __restrict__ skip,
                                                          const uint32_t* __restrict__ listed) {
  if (a.status[ST_FLAGS] & SF_NODE_OVERFLOW) return;
  const int lane = threadIdx.x & 31;
  if (skip) list += *skip;
  const uint32_t n = *listed, teams = gridDim.x * blockDim.x / kTeam<D>;
  uint32_t i = (blockIdx.x * blockDim.x + threadIdx.x) / kTeam<D>;
  MonoNode v = mono_load(i < n, i < n ? list[i] : 0u, a);
  while (__any_sync(0xffffffffu, v.nch > 0)) {
    const bool has = v.nch > 0, up = has && v.k != 0;
    // the parent is read while the children's sums are added
    const MonoNode p = mono_load(up, up ? v.parent : 0u, a);
    const double sum = mono_sum<D>(v, a);
    __syncwarp();   // the team's sums, before its count
    int left = 0;
    if (up && lane % kTeam<D> == 0) left = mono_done(&a.link[v.parent].x);
    mono_node_records<D>(v, sum, a);   // not waited for by the parent
    left = __shfl_sync(0xffffffffu, left, lane - lane % kTeam<D>);
    __syncwarp();   // the siblings' sums, after the count
    if (up && left == 1) {
      v = p;
    } else if (has) {
      i += teams;
      v = mono_load(i < n, i < n ? list[i] : 0u, a);
    }
  }
}

// Other trees of kBinnedMonoBodies bodies or more: the leaves one thread each, all
// in one launch, then the ready internal nodes one thread each, both in an
// order binned by the node's work. A leaf loops
// over its bodies and an internal node over its children, so a warp runs as
// long as its longest loop; FP64 issues at 1/64 of the FP32 rate here and a
// warp instruction costs the same with idle lanes. In Morton order the
// leaves of a warp hold 1 to leaf_size bodies and a warp ran 2.5 times the
// iterations its bodies need (2^24 clustered bodies, leaf 32); binned, the
// threads of a warp have equal loop counts. Each leaf is still summed by one
// thread in its own order, so the results do not depend on the binning.
// Tiles take no order first and read the bodies coalesced; this order keeps the
// FP64 pipe's lanes full, which a tile's few leaves do not when leaves are
// large (leaf sizes 9 to 31 from kBinnedMonoBodies bodies were not timed). Passes with tiles / in this order: a force on 131k bodies 664 / 676 us,
// a 200k-body step 668 / 698 us, a build of 3 M bodies in leaves of 8 1053 /
// 1114 us, two steps of 2^24 bodies in leaves of 32 145.5 / 144.3 ms: tiles
// below kBinnedMonoBodies bodies and for leaves up to kTileLeaf.
// From kBinnedMonoBodies bodies the ready nodes are taken one per lane (an FP64
// instruction serves 32 of them), and what is above them goes to teams. A
// launch per level (20 of them, most nearly empty, 10 to 20 us each for the
// lower ones) took 221 us at 3 M bodies and three species; this takes 140 us.
constexpr int kTileLeaf = 8;
static_assert(kMonoBins <= 256, "the bin scan takes one bin per thread of a 256-thread block");

// bin of node k, -1 for an internal node that is not ready (need > 0)
__device__ __forceinline__ int mono_bin(uint32_t nch, int need, uint32_t cnt) {
  return nch == 0 ? (int)min(cnt, (uint32_t)(kLeafBins - 1)) : need == 0 ? kLeafBins + (int)nch - 1 : -1;
}

// bins[0, kMonoBins): nodes per bin (zeroed before the launch)
__global__ void __launch_bounds__(256) k_mono_hist(MonoArgs a, uint32_t* bins) {
  __shared__ uint32_t h[kMonoBins];
  if (a.status[ST_FLAGS] & SF_NODE_OVERFLOW) return;   // truncated tree: do not read it
  for (int i = threadIdx.x; i < kMonoBins; i += blockDim.x) h[i] = 0;
  __syncthreads();
  const uint32_t total = levels_of(a.status).start[kMaxLevel + 1];
  for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < total; k += gridDim.x * blockDim.x)
  {
    const uint32_t nch = a.nchild[k];
    const int need = mono_pending(k, nch, a), bin = mono_bin(nch, need, a.count[k]);
    if (nch) a.link[k].x = need;
    if (bin >= 0) atomicAdd(&h[bin], 1u);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kMonoBins; i += blockDim.x)
    if (h[i]) atomicAdd(&bins[i], h[i]);
}

// order[]: node indices grouped by bin. bins[kMonoBins, 2 kMonoBins): cursors
// (zeroed before the launch); block 0 writes the bin starts to
// bins[2 kMonoBins, 3 kMonoBins] (the last entry: all nodes). Each block
// places one contiguous chunk of nodes, reserving its share of every bin with
// one atomic per bin. Launched with 256 threads.
__global__ void __launch_bounds__(256) k_mono_order(MonoArgs a, uint32_t* bins, uint32_t* order) {
  __shared__ uint32_t lh[kMonoBins];
  __shared__ uint32_t base[kMonoBins];
  __shared__ uint32_t warp_tot[8];
  __shared__ uint32_t all;
  if (a.status[ST_FLAGS] & SF_NODE_OVERFLOW) return;
  const int tid = threadIdx.x;
  // bin starts: exclusive scan of the bin counts
  const uint32_t v = tid < kMonoBins ? bins[tid] : 0u;
  const uint32_t inc = block_inclusive_scan<256>(v, warp_tot, &all);
  if (tid < kMonoBins) {
    base[tid] = inc - v;
    lh[tid] = 0;
    if (blockIdx.x == 0) bins[2 * kMonoBins + tid] = inc - v;
  }
  if (blockIdx.x == 0 && tid == 0) bins[3 * kMonoBins] = all;
  __syncthreads();
  const uint32_t total = levels_of(a.status).start[kMaxLevel + 1];
  const uint32_t chunk = (total + gridDim.x - 1) / gridDim.x;
  const uint32_t k0 = min(total, blockIdx.x * chunk), k1 = min(total, k0 + chunk);
  auto bin_of = [&](uint32_t k) {
    const uint32_t nch = a.nchild[k];
    return mono_bin(nch, mono_pending(k, nch, a), a.count[k]);
  };
  for (uint32_t k = k0 + tid; k < k1; k += blockDim.x) {
    const int bin = bin_of(k);
    if (bin >= 0) atomicAdd(&lh[bin], 1u);
  }
  __syncthreads();
  if (tid < kMonoBins && lh[tid]) base[tid] += atomicAdd(&bins[kMonoBins + tid], lh[tid]);
  __syncthreads();
  for (uint32_t k = k0 + tid; k < k1; k += blockDim.x) {
    const int bin = bin_of(k);
    if (bin >= 0) order[atomicAdd(&base[bin], 1u)] = k;
  }
}

// Sums of leaf k: its bodies into the node's FP64 monopoles and FP32 walk
// records. lacc: the calling thread's per-species sums {m, m x, m y, m z}
// (physical units), addressed by the body's species: no FP64 instruction is
// spent on the species a body does not have (predicated per-species sums
// would issue D times as many).
template <int D>
__device__ __forceinline__ void mono_leaf(uint32_t k, const MonoArgs& a,
                                          double (*lacc)[4][kMonoThreads], int tid) {
  double cen[3], side;
  node_centre(a.level[k], a.prefix[k], cen, &side);
  uint32_t sc[D];
#pragma unroll
  for (int q = 0; q < D; ++q) {
    sc[q] = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) lacc[q][j][tid] = 0.0;
  }
  const uint32_t f = a.first[k], c = a.count[k];
  // leaf centre in physical units; body records are offsets from it in box units
  const double cxL = cen[0] * a.L, cyL = cen[1] * a.L, czL = cen[2] * a.L;
  const float invLf = (float)a.invL;
  for (uint32_t b = f; b < f + c; ++b) {
    const double xp = a.spos[b], yp = a.spos[a.n + b], zp = a.spos[2 * a.n + b];
    const float m = a.smass[b];
    const int t = a.stype[b];
    a.body[b] = make_float4((float)(xp - cxL) * invLf, (float)(yp - cyL) * invLf,
                            (float)(zp - czL) * invLf, m);
    const double md = (double)m;
    lacc[t][0][tid] += md;
    lacc[t][1][tid] = fma(md, xp, lacc[t][1][tid]);
    lacc[t][2][tid] = fma(md, yp, lacc[t][2][tid]);
    lacc[t][3][tid] = fma(md, zp, lacc[t][3][tid]);
#pragma unroll
    for (int q = 0; q < D; ++q) sc[q] += t == q ? 1u : 0u;
  }
  double mt = 0, xt = 0, yt = 0, zt = 0;
#pragma unroll
  for (int q = 0; q < D; ++q) {
    // to box units (exact when the box is a power of two)
    const double m = lacc[q][0][tid], x = lacc[q][1][tid] * a.invL, y = lacc[q][2][tid] * a.invL,
                 z = lacc[q][3][tid] * a.invL;
    // 32-byte records from a cudaMalloc base: one aligned 32-byte access each
    *reinterpret_cast<double4_32a*>(a.m64 + ((size_t)k * D + q) * 4) = make_double4_32a(m, x, y, z);
    a.cnt[(size_t)k * D + q] = sc[q];
    a.mono[(size_t)k * D + q] = mono_record(m, x, y, z, cen);
    mt += m;
    xt += x;
    yt += y;
    zt += z;
  }
  a.geo[k] = mono_geo(a.level[k], a.prefix[k]);
  a.com[k] = mono_record(mt, xt, yt, zt, cen);
  a.link[k] = make_int4(-1, 0, (int)f, (int)c);
}

// Every leaf of the tree: order[0, start of the first internal bin).
template <int D>
__global__ void __launch_bounds__(kMonoThreads) k_mono_leaves(MonoArgs a, const uint32_t* __restrict__ bins,
                                                              const uint32_t* __restrict__ order) {
  __shared__ double lacc[D][4][kMonoThreads];
  if (a.status[ST_FLAGS] & SF_NODE_OVERFLOW) return;
  const uint32_t e = bins[2 * kMonoBins + kLeafBins];
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < e; i += gridDim.x * blockDim.x)
    mono_leaf<D>(order[i], a, lacc, threadIdx.x);
}

// The ready nodes order[*skip, *end), one per lane; the parents they complete
// are listed behind them for k_mono_up.
template <int D>
__global__ void __launch_bounds__(kMonoThreads) k_mono_ready(MonoArgs a, uint32_t* order,
                                                             const uint32_t* __restrict__ skip,
                                                             const uint32_t* __restrict__ end,
                                                             uint32_t* words) {
  if (a.status[ST_FLAGS] & SF_NODE_OVERFLOW) return;
  const uint32_t s = skip ? *skip : 0u, e = *end;
  const int lane = threadIdx.x & 31;
  for (uint32_t i0 = s + blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < e; i0 += gridDim.x * blockDim.x) {
    const bool has = i0 + lane < e;
    const MonoNode v = mono_load(has, has ? order[i0 + lane] : 0u, a);
    mono_internal_lane<D>(v, a);
    const bool last = has && v.k != 0 && mono_done(&a.link[v.parent].x) == 1;
    const uint32_t m = __ballot_sync(0xffffffffu, last);
    uint32_t at = 0;
    if (lane == 0 && m) at = atomicAdd(&words[kMlNext], (uint32_t)__popc(m));
    at = e + __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
    if (last) order[at] = v.parent;
  }
}

template <int D>
static int launch_monopoles(ng_ctx* c, const MonoArgs& a) {
  uint32_t* words = as<uint32_t>(c->mono_words);
  uint32_t* order = as<uint32_t>(c->n_tmp);
  const int64_t cap = std::min<int64_t>(c->cap_nodes, 2 * c->n + 64);
  const int grid = (int)std::min<int64_t>((int64_t)c->nsm * 16, (cap + kMonoThreads - 1) / kMonoThreads);
  const bool large = c->n >= kBinnedMonoBodies;
  if (!large || c->p.leaf_size <= kTileLeaf) {
    const int64_t tiles = (c->n + kLeafTile - 1) / kLeafTile;
    k_mono_tiles<D><<<(int)std::min<int64_t>((int64_t)c->nsm * 64, tiles), kLeafThreads, 0, c->stream>>>(a, words, order);
    c->launches += 1;
    if (large) {
      k_mono_ready<D><<<grid, kMonoThreads, 0, c->stream>>>(a, order, nullptr, words + kMlReady, words);
      k_mono_up<D><<<grid, kMonoThreads, 0, c->stream>>>(a, order, words + kMlReady, words + kMlNext);
      c->launches += 2;
    } else if (c->n > c->p.leaf_size) {   // else the root is a leaf
      // a ready node holds more than leaf_size bodies
      const int64_t teams = c->n / (c->p.leaf_size + 1);
      const int64_t blocks = (teams * kTeam<D> + kMonoThreads - 1) / kMonoThreads;
      k_mono_up<D><<<(int)std::min<int64_t>((int64_t)c->nsm * 16, blocks), kMonoThreads, 0, c->stream>>>(
          a, order, nullptr, words + kMlReady);
      c->launches += 1;
    }
    NG_CUDA(c, cudaGetLastError());
    return NG_OK;
  }
  uint32_t* bins = words + kMonoWords;
  NG_CUDA(c, cudaMemsetAsync(bins, 0, 2 * kMonoBins * sizeof(uint32_t), c->stream));
  const int sgrid = work_grid(c, cap, 4);
  k_mono_hist<<<sgrid, 256, 0, c->stream>>>(a, bins);
  k_mono_order<<<sgrid, 256, 0, c->stream>>>(a, bins, order);
  k_mono_leaves<D><<<grid, kMonoThreads, 0, c->stream>>>(a, bins, order);
  k_mono_ready<D><<<grid, kMonoThreads, 0, c->stream>>>(a, order, bins + 2 * kMonoBins + kLeafBins,
                                                          bins + 3 * kMonoBins, words);
  k_mono_up<D><<<grid, kMonoThreads, 0, c->stream>>>(a, order, bins + 3 * kMonoBins, words + kMlNext);
  c->launches += 5;
  NG_CUDA(c, cudaGetLastError());
  return NG_OK;
}

int reduce_monopoles(ng_ctx* c) {
  MonoArgs a;
  a.level = as<uint8_t>(c->n_level);
  a.prefix = as<uint64_t>(c->n_prefix);
  a.first = as<uint32_t>(c->n_first);
  a.count = as<uint32_t>(c->n_count);
  a.nchild = as<uint8_t>(c->n_nchild);
  a.child = as<uint32_t>(c->n_child);
  a.spos = as<double>(c->spos);
  a.smass = as<float>(c->smass);
  a.stype = as<uint8_t>(c->stype);
  a.m64 = as<double>(c->n_m64);
  a.cnt = as<uint32_t>(c->n_cnt);
  a.geo = as<float4>(c->n_geo);
  a.com = as<float4>(c->n_com);
  a.link = as<int4>(c->n_link);
  a.mono = as<float4>(c->n_mono);
  a.body = as<float4>(c->body);
  a.bleaf = as<uint32_t>(c->bleaf);
  a.status = as<uint32_t>(c->status);
  a.n = c->n;
  a.invL = 1.0 / c->L;
  a.L = c->L;
  a.unit = c->L == 1.0;
  stage_mark(c, NG_STAGE_MONOPOLES);
  switch (c->p.D) {
    case 1: return launch_monopoles<1>(c, a);
    case 2: return launch_monopoles<2>(c, a);
    case 3: return launch_monopoles<3>(c, a);
    case 4: return launch_monopoles<4>(c, a);
    case 5: return launch_monopoles<5>(c, a);
    default: return launch_monopoles<6>(c, a);
  }
}

// ------------------------------------------------------------- groups

// Walk groups: runs of consecutive sibling cells holding <= S bodies each
// (and <= S together) whose parent holds more than S, each run cut into
// ceil(c / G) contiguous chunks of balanced size; leaves with more than S
// bodies are cut the same way. Every body lands in exactly one group, so a
// group is named by its first body: gsize[first] = body count (zero
// elsewhere). A flag scan then numbers the groups in body (Morton) order,
// so that warps taking consecutive groups walk neighbouring regions and
// share the nodes they fetch in L2.
__global__ void k_groups(uint32_t* status, int64_t cap, int G, int S,
                         const uint32_t* __restrict__ first,
                         const uint32_t* __restrict__ count, const uint8_t* __restrict__ nchild,
                         const uint32_t* __restrict__ child, uint32_t* gsize) {
  if (status[ST_FLAGS] & SF_NODE_OVERFLOW) return;
  Levels lv = levels_of(status);
  uint32_t total = lv.start[kMaxLevel + 1];
  if (total > cap) total = (uint32_t)cap;
  auto emit = [&](uint32_t f, uint32_t c) { gsize[f] = c; };
  auto emit_chunks = [&](uint32_t f, uint32_t c) {
    const uint32_t k = (c + G - 1) / G, base = c / k, rem = c % k;
    for (uint32_t j = 0, o = 0; j < k; ++j) {
      const uint32_t len = base + (j < rem ? 1u : 0u);
      emit(f + o, len);
      o += len;
    }
  };
  const uint32_t SS = (uint32_t)S;
  for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < total;
       k += gridDim.x * blockDim.x) {
    const uint32_t c = count[k];
    if (k == 0 && c <= SS) { emit_chunks(first[0], c); continue; }
    if (c <= SS) continue;
    const uint32_t nch = nchild[k];
    if (nch == 0) {
      if (k == 0) emit_chunks(first[0], c);
      continue;
    }
    uint32_t bf = 0, bc = 0;
    for (uint32_t j = 0; j < nch; ++j) {
      const uint32_t ch = child[k] + j;
      const uint32_t cc = count[ch];
      if (cc > SS) {
        if (bc) { emit_chunks(bf, bc); bc = 0; }
        if (nchild[ch] == 0) emit_chunks(first[ch], cc);
        continue;
      }
      if (bc + cc > SS) { emit_chunks(bf, bc); bc = 0; }
      if (bc == 0) bf = first[ch];
      bc += cc;
    }
    if (bc) emit_chunks(bf, bc);
  }
}

// The groups (b, gsize[b]) in the order of their first bodies, and their number.
// One launch: a block takes the next tile, ranks its group starts by ballots and
// adds up the tiles before by look-back. A clear, a two-launch scan into a rank
// per body and a compaction took 17 us at 131k bodies, 33 at 3 M.
__global__ void __launch_bounds__(kGroupThreads)
k_group_list(int64_t n, const uint32_t* __restrict__ gsize, uint32_t* words, uint64_t* lb,
             uint32_t* status, int2* __restrict__ groups) {
  constexpr int kChunks = kGroupTile / 32, kPer = kChunks / 32;
  __shared__ uint32_t cnt[kChunks];   // per chunk: group starts, then place in the list
  __shared__ uint32_t tile_s;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (tid == 0) tile_s = atomicAdd(&words[kGroupTicket], 1u);
  __syncthreads();
  const int64_t tile = tile_s, t0 = tile * kGroupTile;
  const uint32_t lt = (1u << lane) - 1u;
  uint32_t size[kGroupItems], rank[kGroupItems];
#pragma unroll
  for (int it = 0; it < kGroupItems; ++it) {
    const int64_t i = t0 + it * kGroupThreads + tid;
    size[it] = i < n ? gsize[i] : 0u;
  }
#pragma unroll
  for (int it = 0; it < kGroupItems; ++it) {
    const uint32_t m = __ballot_sync(0xffffffffu, size[it] != 0);
    rank[it] = __popc(m & lt);
    if (lane == 0) cnt[it * (kGroupThreads / 32) + w] = __popc(m);
  }
  __syncthreads();
  if (w == 0) {
    uint32_t v[kPer], sum = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      v[j] = cnt[lane * kPer + j];
      sum += v[j];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += x;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    if (lane == 0) lb_store(&lb[tile], (tile == 0 ? kLbPrefix : kLbAggregate) | total);
    const uint64_t before = lb_before(lb, 1, tile, [&] {
      uint64_t c = 0;
      for (int64_t i = lane; i < t0; i += 32) c += gsize[i] != 0;
      return c;
    });
    if (lane == 0 && tile > 0) lb_store(&lb[tile], kLbPrefix | (before + total));
    if (lane == 0 && tile == gridDim.x - 1) status[ST_NGROUPS] = (uint32_t)before + total;
    uint32_t run = (uint32_t)before + incl - sum;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      cnt[lane * kPer + j] = run;
      run += v[j];
    }
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < kGroupItems; ++it)
    if (size[it])
      groups[cnt[it * (kGroupThreads / 32) + w] + rank[it]] =
          make_int2((int)(t0 + it * kGroupThreads + tid), (int)size[it]);
}

int build_groups(ng_ctx* c) {
  const int64_t n = c->n;
  uint32_t* gsize = as<uint32_t>(c->gsize);
  stage_mark(c, NG_STAGE_GROUPS);
  k_groups<<<work_grid(c, std::min<int64_t>(c->cap_nodes, 2 * n + 64), 4), 256, 0, c->stream>>>(
      as<uint32_t>(c->status), c->cap_nodes, c->p.group_size, c->p.group_cell,
      as<uint32_t>(c->n_first),
      as<uint32_t>(c->n_count), as<uint8_t>(c->n_nchild), as<uint32_t>(c->n_child), gsize);
  k_group_list<<<(int)((n + kGroupTile - 1) / kGroupTile), kGroupThreads, 0, c->stream>>>(
      n, gsize, as<uint32_t>(c->mono_words), as<uint64_t>(c->group_lb), as<uint32_t>(c->status),
      as<int2>(c->groups));
  c->launches += 2;
  NG_CUDA(c, cudaGetLastError());
  return NG_OK;
}

}  // namespace ng
