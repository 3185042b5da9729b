// Sort stage (Sec. 2.4): periodic wrap, 63-bit Morton+type keys, stable LSD
// radix sort, one gather of the particle data into sorted order, and the
// type-major order (bodies grouped by type, each type in key order).
#include <cmath>
#include <cstdarg>
#include <cstdio>

#include "ng_internal.cuh"

namespace ng {

constexpr int kScanThreads = 1024;
constexpr int kScanBlocks = 256;

__global__ void __launch_bounds__(kScanThreads)
k_scan_partial(const uint32_t* __restrict__ in, int64_t len, uint32_t* part) {
  const int64_t chunk = (len + gridDim.x - 1) / gridDim.x;
  const int64_t b0 = (int64_t)blockIdx.x * chunk;
  const int64_t b1 = b0 + chunk < len ? b0 + chunk : len;
  uint32_t s = 0;
  for (int64_t i = b0 + threadIdx.x; i < b1; i += blockDim.x) s += in[i];
#pragma unroll
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  __shared__ uint32_t ws[32];
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    s = threadIdx.x < blockDim.x / 32 ? ws[threadIdx.x] : 0;
#pragma unroll
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
  }
}

__global__ void __launch_bounds__(kScanThreads)
k_scan_final(const uint32_t* in, uint32_t* out, int64_t len, const uint32_t* __restrict__ part,
             uint32_t* d_total) {
  __shared__ uint32_t warp_tot[32];
  __shared__ uint32_t tile_total;
  __shared__ uint32_t off;
  const int64_t chunk = (len + gridDim.x - 1) / gridDim.x;
  const int64_t b0 = (int64_t)blockIdx.x * chunk;
  const int64_t b1 = b0 + chunk < len ? b0 + chunk : len;
  if (threadIdx.x < 32) {
    uint32_t s = 0;
    for (int j = threadIdx.x; j < (int)blockIdx.x; j += 32) s += part[j];
#pragma unroll
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) off = s;
  }
  __syncthreads();
  uint32_t carry = off;
  for (int64_t base = b0; base < b1; base += kScanThreads) {
    const int64_t i = base + threadIdx.x;
    const uint32_t v = i < b1 ? in[i] : 0u;
    const uint32_t inc = block_inclusive_scan<kScanThreads>(v, warp_tot, &tile_total);
    if (i < b1) out[i] = carry + inc - v;
    __syncthreads();
    carry += tile_total;
    __syncthreads();
  }
  if (d_total && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *d_total = carry;
}

static int scan_blocks(int64_t len) {
  return (int)std::max<int64_t>(
      1, std::min<int64_t>(kScanBlocks, (len + 4 * kScanThreads - 1) / (4 * kScanThreads)));
}

int scan_u32(ng_ctx* c, const uint32_t* in, uint32_t* out, int64_t len, uint32_t* d_total) {
  NG_TRY(ensure(c, c->scan_part, kScanBlocks * sizeof(uint32_t)));
  uint32_t* part = as<uint32_t>(c->scan_part);
  // blocks for at most 4 tiles each; both kernels split the range by gridDim
  const int blocks = scan_blocks(len);
  // one block needs no partial sums (its offset is zero)
  if (blocks > 1) k_scan_partial<<<blocks, kScanThreads, 0, c->stream>>>(in, len, part);
  k_scan_final<<<blocks, kScanThreads, 0, c->stream>>>(in, out, len, part, d_total);
  c->launches += blocks > 1 ? 2 : 1;
  NG_CUDA(c, cudaGetLastError());
  return NG_OK;
}

// --------------------------------------------------------------- keys

struct KeyArgs {
  int64_t n;
  const double* pos;
  const uint8_t* type;
  double L, invL;
  bool pow2;
  int ebox, D;
  const float* mass;
  double4_32a* rec;   // packed bodies in caller order (nullptr: not packed)
};

// Packed bodies: the gather into sorted order reads a body's five values at
// random places, a 32-byte sector each. From kPackBodies bodies the key kernel,
// which has the positions in hand, writes them wrapped, with mass and species,
// as one 32-byte record, and the gather reads one sector (3 M bodies: keys 34 ->
// 47 us, gather 108 -> 46 us; a build 1161 -> 1118 us). At 131k bodies, all in L2,
// it is still 5 us of a 650 us force; smaller sizes were not tried.
__device__ __forceinline__ double4_32a pack_body(double x, double y, double z, float mass, uint8_t type) {
  const uint64_t mt = (uint64_t)type << 32 | __float_as_uint(mass);
  return make_double4_32a(x, y, z, __longlong_as_double((long long)mt));
}

__device__ __forceinline__ uint64_t body_key(const KeyArgs& a, int64_t i, uint8_t type) {
  return sort_key(a.pos[i], a.pos[a.n + i], a.pos[2 * a.n + i], type, a.L, a.invL, a.pow2, a.ebox);
}

// A species as the gather stores it (out of range: 0, flagged there).
__device__ __forceinline__ uint32_t stored_type(uint8_t t, int D) { return t < D ? t : 0u; }

// Words of the sort (c->sort_words): the digit histograms of the 8 passes,
// the species counts (kept until the next sort: the starts of the type-major
// order), and one tile ticket per pass and for the type order.
constexpr int kSwTypes = 8 * 256, kSwTickets = kSwTypes + 8, kSortWords = kSwTickets + 9;

// Keys of all bodies, the digit histograms of passes first..7 and the species
// counts; clears the look-back state of the first pass and of the type order.
__global__ void __launch_bounds__(512)
k_keys(KeyArgs a, int first, uint64_t* __restrict__ keys, uint32_t* words,
       uint64_t* __restrict__ lb, int64_t lb_words, uint64_t* __restrict__ lbt, int64_t lbt_words) {
  __shared__ uint32_t h[8][256];
  __shared__ uint32_t ht[8];
  for (int j = threadIdx.x; j < 8 * 256; j += blockDim.x) (&h[0][0])[j] = 0;
  if (threadIdx.x < 8) ht[threadIdx.x] = 0;
  __syncthreads();
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t j = t; j < lb_words; j += stride) lb[j] = 0;
  for (int64_t j = t; j < lbt_words; j += stride) lbt[j] = 0;
  for (int64_t i = t; i < a.n; i += stride) {
    const uint8_t ty = a.type[i];
    const double x = a.pos[i], y = a.pos[a.n + i], z = a.pos[2 * a.n + i];
    const uint64_t k = sort_key(x, y, z, ty, a.L, a.invL, a.pow2, a.ebox);
    keys[i] = k;
    if (a.rec)
      a.rec[i] = pack_body(wrap_box(x, a.L, a.invL, a.pow2), wrap_box(y, a.L, a.invL, a.pow2),
                           wrap_box(z, a.L, a.invL, a.pow2), a.mass[i], ty);
#pragma unroll
    for (int p = 0; p < 8; ++p)
      if (p >= first) atomicAdd(&h[p][(uint32_t)(k >> (8 * p)) & 0xffu], 1u);
    atomicAdd(&ht[stored_type(ty, a.D)], 1u);
  }
  __syncthreads();
  for (int j = threadIdx.x; j < 8 * 256; j += blockDim.x)
    if ((&h[0][0])[j]) atomicAdd(&words[j], (&h[0][0])[j]);
  if (threadIdx.x < 8 && ht[threadIdx.x]) atomicAdd(&words[kSwTypes + threadIdx.x], ht[threadIdx.x]);
}

// ---------------------------------------------------------- radix sort

// One stable pass on one 8-bit digit, in one launch: each block takes the
// next tile of kRsThreads * ITEMS keys, ranks it by digit (each warp its
// contiguous run in order, ballots group equal digits; then warps in order
// per digit), publishes the tile's digit counts, adds up those of the tiles
// before it until it meets one that published its prefix, and writes the keys
// out through shared memory, so that each digit's run of the tile leaves as
// one contiguous segment. It reads and writes 12 B a key once and waits mostly
// on its own phases (ranking, look-back, write-out). A histogram, a scan and a
// scatter launch per pass read the keys twice and cost two to three launches
// more (8 passes: 131k bodies 190 -> 75 us, 3 M 470 -> 320 us; 4096 bodies
// 145 -> 57 us). ITEMS is small for few keys, so that every SM has a tile.
constexpr int kRsThreads = 256;
constexpr int kRsWarps = kRsThreads / 32;
constexpr int kRsItemsSmall = 4, kRsItemsLarge = 16;
// two tiles of the larger kind per SM of a GB300. (Fixed, since the look-back state
// is sized by it: fewer bodies than this can need more of it than more bodies do.)
constexpr int64_t kRsLarge = (int64_t)2 * 152 * kRsThreads * kRsItemsLarge;

// Look-back state of one pass. Tiles form groups of kRsGroup: a tile adds up
// the tiles before it in its group (their states loaded together) and the
// groups before; the last tile of a group publishes the group's counts. The tiles of a wave publish at about the same time, so walking
// back tile by tile would cost a tile hundreds of loads in a row (3 M bodies:
// 53 us a pass, 40 us with groups and the tile size below).
constexpr int kRsGroup = 16;
struct RsLookback {
  uint64_t* tile;       // [tile][256]: aggregates
  uint64_t* group;      // [group][256]: aggregates, then prefixes
};

template <int ITEMS>
struct RsSmem {
  uint32_t wcnt[kRsWarps][256];   // per warp and digit: count, then place in the digit's run
  uint32_t dstart[256];           // tile position of each digit's run
  int64_t gdst[256];              // global position of each digit's run less its tile position
  uint32_t wsum[2][kRsWarps];
  uint32_t tile;
  uint64_t tk[kRsThreads * ITEMS];
  uint32_t tv[kRsThreads * ITEMS];
};

// Lanes of the warp whose 8-bit digit equals this lane's (of the lanes in
// `in`): one ballot per bit (match.any, which waits for the memory pipe: 66 us a
// 3 M pass, ballots 47 us).
__device__ __forceinline__ uint32_t digit_peers(uint32_t d, uint32_t in) {
  uint32_t p = in;
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    const uint32_t m = __ballot_sync(0xffffffffu, d >> b & 1u);
    p &= d >> b & 1u ? m : ~m;
  }
  return p;
}

template <int ITEMS>
__global__ void __launch_bounds__(kRsThreads, 3)
k_rs_pass(const uint64_t* __restrict__ kin, const uint32_t* __restrict__ vin,
          uint64_t* __restrict__ kout, uint32_t* __restrict__ vout, int64_t n, int shift,
          const uint32_t* __restrict__ hist, uint32_t* ticket, RsLookback lb, RsLookback lb_next) {
  extern __shared__ __align__(16) unsigned char rs_raw[];
  RsSmem<ITEMS>& sm = *reinterpret_cast<RsSmem<ITEMS>*>(rs_raw);
  constexpr int kTile = kRsThreads * ITEMS;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (tid == 0) sm.tile = atomicAdd(ticket, 1u);
  for (int j = tid; j < kRsWarps * 256; j += kRsThreads) (&sm.wcnt[0][0])[j] = 0;
  __syncthreads();
  const int64_t tile = sm.tile;
  const int64_t group = tile / kRsGroup, g0 = group * kRsGroup;
  const int64_t t0 = tile * kTile;
  const int64_t sub0 = t0 + (int64_t)w * (32 * ITEMS);
  const uint32_t lt = (1u << lane) - 1u;
  uint64_t k[ITEMS];
  uint32_t rank[ITEMS];
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    const int64_t i = sub0 + it * 32 + lane;
    k[it] = i < n ? kin[i] : 0ull;
  }
#pragma unroll
  for (int h = 0; h < ITEMS; h += 4) {
    // the ballots of four items overlap; their counts follow in order
    uint32_t peers[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const bool valid = sub0 + (h + j) * 32 + lane < n;
      peers[j] = digit_peers((uint32_t)(k[h + j] >> shift) & 0xffu, __ballot_sync(0xffffffffu, valid));
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const bool valid = sub0 + (h + j) * 32 + lane < n;
      const uint32_t d = (uint32_t)(k[h + j] >> shift) & 0xffu;
      const uint32_t prior = sm.wcnt[w][d];
      __syncwarp();
      rank[h + j] = prior + __popc(peers[j] & lt);
      if (valid && (peers[j] & lt) == 0) sm.wcnt[w][d] = prior + __popc(peers[j]);
      __syncwarp();
    }
  }
  __syncthreads();
  uint32_t total = 0, incl = 0, gincl = 0, gtot = 0;
  if (tid < 256) {
    // thread d: the digit's total in the tile, published at once
#pragma unroll
    for (int ww = 0; ww < kRsWarps; ++ww) {
      const uint32_t t = sm.wcnt[ww][tid];
      sm.wcnt[ww][tid] = total;
      total += t;
    }
    lb_store(&lb.tile[tile * 256 + tid], kLbAggregate | total);
    lb_next.tile[tile * 256 + tid] = 0;
    if (tile == g0) lb_next.group[group * 256 + tid] = 0;
    gtot = hist[tid];
    incl = total;
    gincl = gtot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o), y = __shfl_up_sync(0xffffffffu, gincl, o);
      if (lane >= o) {
        incl += x;
        gincl += y;
      }
    }
    if (lane == 31) {
      sm.wsum[0][w] = incl;
      sm.wsum[1][w] = gincl;
    }
  }
  __syncthreads();
  uint32_t base = incl - total, gbase = gincl - gtot;
  if (tid < 256) {
    for (int ww = 0; ww < w; ++ww) {
      base += sm.wsum[0][ww];
      gbase += sm.wsum[1][ww];
    }
    sm.dstart[tid] = base;
  }
  __syncthreads();
  // the tile by digit in shared memory, while the other tiles publish
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    if (sub0 + it * 32 + lane < n) {
      const uint32_t d = (uint32_t)(k[it] >> shift) & 0xffu;
      const uint32_t at = sm.dstart[d] + sm.wcnt[w][d] + rank[it];
      sm.tk[at] = k[it];
      sm.tv[at] = vin ? vin[sub0 + it * 32 + lane] : (uint32_t)(sub0 + it * 32 + lane);
    }
  }
  if (tid < 256) {
    // the digit's bodies in the tiles of the group before this one; several
    // states at a time, so that their loads overlap
    constexpr int kBatch = 8;
    uint64_t before = 0;
    for (int64_t t = g0; t < tile; t += kBatch) {
      uint64_t st[kBatch];
#pragma unroll
      for (int j = 0; j < kBatch; ++j)
        st[j] = t + j < tile ? lb_load(&lb.tile[(t + j) * 256 + tid]) : kLbAggregate;
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        for (int poll = 0; st[j] == 0 && poll < kLbPolls; ++poll)
          st[j] = lb_load(&lb.tile[(t + j) * 256 + tid]);
        if (st[j] == 0)
          for (int64_t i = (t + j) * kTile; i < (t + j + 1) * kTile; ++i)
            st[j] += ((uint32_t)(kin[i] >> shift) & 0xffu) == (uint32_t)tid;
        before += st[j] & kLbCount;
      }
    }
    // the last tile of a group publishes the group's count
    const bool last = tile == g0 + kRsGroup - 1;
    const uint64_t gsum = before + total;
    if (last) lb_store(&lb.group[group * 256 + tid], (group == 0 ? kLbPrefix : kLbAggregate) | gsum);
    // and in the groups before, back to the nearest prefix
    uint64_t gbefore = 0;
    bool done = false;
    for (int64_t t = group - 1; t >= 0 && !done; t -= kBatch) {
      uint64_t st[kBatch];
#pragma unroll
      for (int j = 0; j < kBatch; ++j)
        st[j] = t - j >= 0 ? lb_load(&lb.group[(t - j) * 256 + tid]) : kLbPrefix;
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        if (done) continue;
        for (int poll = 0; st[j] == 0 && poll < kLbPolls; ++poll)
          st[j] = lb_load(&lb.group[(t - j) * 256 + tid]);
        if (st[j] == 0) {
          for (int64_t i = 0; i < (t - j + 1) * kRsGroup * kTile; ++i)
            gbefore += ((uint32_t)(kin[i] >> shift) & 0xffu) == (uint32_t)tid;
          st[j] = kLbPrefix;
        }
        gbefore += st[j] & kLbCount;
        done = (st[j] & kLbPrefix) != 0;
      }
    }
    if (last && group > 0) lb_store(&lb.group[group * 256 + tid], kLbPrefix | (gbefore + gsum));
    sm.gdst[tid] = (int64_t)gbase + (int64_t)(before + gbefore) - (int64_t)base;
  }
  __syncthreads();
  const int valid = (int)((n - t0) < kTile ? (n - t0) : kTile);
  for (int p = tid; p < valid; p += kRsThreads) {
    const uint64_t key = sm.tk[p];
    const int64_t dst = sm.gdst[(uint32_t)(key >> shift) & 0xffu] + p;
    kout[dst] = key;
    vout[dst] = sm.tv[p];
  }
}

static bool rs_large(int64_t n) { return n >= kRsLarge; }
static int64_t rs_tiles(int64_t n) {
  const int64_t tile = kRsThreads * (rs_large(n) ? kRsItemsLarge : kRsItemsSmall);
  return (n + tile - 1) / tile;
}

static int64_t rs_groups(int64_t n) { return (rs_tiles(n) + kRsGroup - 1) / kRsGroup; }
// 64-bit words of one pass's look-back state, and its parts in them
static int64_t rs_lb_words(int64_t n) { return 256 * (rs_tiles(n) + rs_groups(n)); }
static RsLookback rs_lookback(uint64_t* w, int64_t n) { return RsLookback{w, w + 256 * rs_tiles(n)}; }

template <int ITEMS>
static int rs_pass(ng_ctx* c, const uint64_t* kin, const uint32_t* vin, uint64_t* kout, uint32_t* vout,
                   int64_t n, int pass, RsLookback lb, RsLookback lb_next) {
  uint32_t* words = as<uint32_t>(c->sort_words);
  const size_t smem = sizeof(RsSmem<ITEMS>);
  NG_CUDA(c, cudaFuncSetAttribute(k_rs_pass<ITEMS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  k_rs_pass<ITEMS><<<(int)rs_tiles(n), kRsThreads, smem, c->stream>>>(
      kin, vin, kout, vout, n, 8 * pass, words + 256 * pass, words + kSwTickets + pass, lb, lb_next);
  c->launches += 1;
  NG_CUDA(c, cudaGetLastError());
  return NG_OK;
}

// ------------------------------------------------------ type-major order

// tperm[j] = sorted index of the j-th body in type-major order (each species
// in key order): a stable partition by the stored species in one launch. A
// block ranks the bodies of its tile by ballots; one warp per species adds
// up the counts of the tiles before (32 states per load). 1 B read and 4 B
// written a body; as a radix pass on the keys' species bits with an index fill
// and its own histogram and scan it read 24 B and wrote 16 B in four launches.
constexpr int kToThreads = 512, kToItems = 8, kToTile = kToThreads * kToItems;
constexpr int kToChunks = kToTile / 32;

__global__ void __launch_bounds__(kToThreads)
k_type_order(int64_t n, int D, const uint8_t* __restrict__ stype, uint32_t* words, uint64_t* lb,
             uint32_t* __restrict__ tperm) {
  __shared__ uint32_t cnt[8][kToChunks];   // per species and chunk: bodies, then output position
  __shared__ uint32_t tile_s;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (tid == 0) tile_s = atomicAdd(&words[kSwTickets + 8], 1u);
  __syncthreads();
  const int64_t tile = tile_s, t0 = tile * kToTile;
  const uint32_t lt = (1u << lane) - 1u;
  int ty[kToItems];
  uint32_t rank[kToItems];
#pragma unroll
  for (int it = 0; it < kToItems; ++it) {
    const int64_t i = t0 + it * kToThreads + tid;
    ty[it] = i < n ? (int)stype[i] : -1;
  }
#pragma unroll
  for (int it = 0; it < kToItems; ++it) {
    const int chunk = it * (kToThreads / 32) + w;
    rank[it] = 0;
    for (int s = 0; s < D; ++s) {
      const uint32_t m = __ballot_sync(0xffffffffu, ty[it] == s);
      if (ty[it] == s) rank[it] = __popc(m & lt);
      if (lane == 0) cnt[s][chunk] = __popc(m);
    }
  }
  __syncthreads();
  if (w < D) {
    // warp w: species w. The chunks' exclusive scan, then the tiles before
    constexpr int kPer = kToChunks / 32;
    uint32_t v[kPer], sum = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      v[j] = cnt[w][lane * kPer + j];
      sum += v[j];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += x;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    if (lane == 0) lb_store(&lb[tile * 8 + w], (tile == 0 ? kLbPrefix : kLbAggregate) | total);
    const uint64_t before = lb_before(lb + w, 8, tile, [&] {
      uint64_t c = 0;
      for (int64_t i = lane; i < t0; i += 32) c += stype[i] == w;
      return c;
    });
    if (lane == 0 && tile > 0) lb_store(&lb[tile * 8 + w], kLbPrefix | (before + total));
    uint32_t run = (uint32_t)before + incl - sum;
    for (int s = 0; s < w; ++s) run += words[kSwTypes + s];
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      cnt[w][lane * kPer + j] = run;
      run += v[j];
    }
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < kToItems; ++it)
    if (ty[it] >= 0)
      tperm[cnt[ty[it]][it * (kToThreads / 32) + w] + rank[it]] =
          (uint32_t)(t0 + it * kToThreads + tid);
}

static int64_t to_tiles(int64_t n) { return (n + kToTile - 1) / kToTile; }

// -------------------------------------------------------------- gather

struct GatherArgs {
  int64_t n;
  // plain: caller arrays, wrapped and checked; resident: the previous state
  const double* pos;
  const float* mass;
  const uint8_t* type;
  const float* vel;
  const uint32_t* orig;
  const double4_32a* rec;   // packed bodies (nullptr: not packed)
  double* spos;
  float* smass;
  uint8_t* stype;
  float* svel;
  uint32_t* sorig;
  double L, invL;
  bool pow2;
  int D;
  uint32_t* status;
};

// Body i of the input becomes sorted body k. All of it is loaded before the
// first store: the compiler must assume that the arrays overlap, and in turn
// each load waited for the store before it (2^24 bodies, resident: 0.53 ms, now 0.26).
__device__ __forceinline__ void gather_plain(const GatherArgs& g, int64_t k, uint32_t i) {
  const int64_t n = g.n;
  const double x = g.pos[i], y = g.pos[n + i], z = g.pos[2 * n + i];
  const float m = g.mass[i];
  const uint8_t ti = g.type[i];
  g.spos[k] = wrap_box(x, g.L, g.invL, g.pow2);
  g.spos[n + k] = wrap_box(y, g.L, g.invL, g.pow2);
  g.spos[2 * n + k] = wrap_box(z, g.L, g.invL, g.pow2);
  g.smass[k] = m;
  if (ti >= g.D) atomicOr(&g.status[ST_FLAGS], (uint32_t)SF_BAD_TYPE);
  g.stype[k] = (uint8_t)stored_type(ti, g.D);    // out-of-range species: flagged, never used as an index
}

__device__ __forceinline__ void gather_packed(const GatherArgs& g, int64_t k, uint32_t i) {
  const int64_t n = g.n;
  const double4_32a r = g.rec[i];
  const uint64_t mt = (uint64_t)__double_as_longlong(r.w);
  g.spos[k] = r.x;
  g.spos[n + k] = r.y;
  g.spos[2 * n + k] = r.z;
  g.smass[k] = __uint_as_float((uint32_t)mt);
  const uint8_t ti = (uint8_t)(mt >> 32);
  if (ti >= g.D) atomicOr(&g.status[ST_FLAGS], (uint32_t)SF_BAD_TYPE);
  g.stype[k] = (uint8_t)stored_type(ti, g.D);
}

// The resident step's gather: the previous state (positions already wrapped
// by the drift, masses, species, velocities and caller indices, in the
// previous step's sorted order) into this step's sorted order. The bodies
// move little from step to step, so perm is close to the identity and every
// read is close to sequential.
__device__ __forceinline__ void gather_resident(const GatherArgs& g, int64_t k, uint32_t i) {
  const int64_t n = g.n;
  const double x = g.pos[i], y = g.pos[n + i], z = g.pos[2 * n + i];
  const float u = g.vel[i], v = g.vel[n + i], w = g.vel[2 * n + i], m = g.mass[i];
  const uint8_t t = g.type[i];
  const uint32_t o = g.orig[i];
  g.spos[k] = x;
  g.spos[n + k] = y;
  g.spos[2 * n + k] = z;
  g.svel[k] = u;
  g.svel[n + k] = v;
  g.svel[2 * n + k] = w;
  g.smass[k] = m;
  g.stype[k] = t;
  g.sorig[k] = o;
}

template <bool RESIDENT>
__global__ void k_gather(GatherArgs g, const uint32_t* __restrict__ perm) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < g.n;
       k += (int64_t)gridDim.x * blockDim.x) {
    if (RESIDENT) gather_resident(g, k, perm[k]);
    else if (g.rec) gather_packed(g, k, perm[k]);
    else gather_plain(g, k, perm[k]);
  }
}

// ------------------------------------------------------- small problems

// The whole sort stage of few bodies in one launch: a body's
// sorted place is the number of keys below its own (and of equal keys of lower
// index, so the order is that of the stable passes), counted by comparing it
// with every key; its place in the type-major order counts those of its own
// species. At these sizes a radix pass costs far more than its work: 4096
// bodies take 81 us of kernels in the 11 launches of the general path, and one
// block with the passes in shared memory took 44 us on one SM; this takes 20.
// The n^2 comparisons, five instructions each over the whole chip, set the limit.
// Each block forms all keys (the bodies are read from L2) and ranks 32 * ITEMS
// bodies, one per lane and item; its warps share out the keys they are compared with.
// In a box that is a power of two a key is integer work, and a build takes 129 us
// at 4096 bodies and 153 at 8192 (general path: 186 and 193). In other boxes it is
// six FP64 divisions, formed again by every block: 195 / 253 / 299 us at 4096 /
// 6144 / 8192 bodies against 223 / 226 / 229, so there the general path takes over
// where the two meet, at 5120.
constexpr int kRkThreads = 512, kRkWarps = kRkThreads / 32;
constexpr int kRkPad = 4 * kRkWarps;   // keys are padded to whole quads per warp
constexpr int64_t kSmallSort = 8192, kSmallSortAnyBox = 5120;

static size_t rank_smem(int64_t n) { return (size_t)((n + kRkPad - 1) / kRkPad * kRkPad) * 12; }

template <int ITEMS, bool RESIDENT>
__global__ void __launch_bounds__(kRkThreads)
k_sort_rank(KeyArgs a, GatherArgs g, int first, uint64_t* __restrict__ keys,
            uint32_t* __restrict__ perm, uint32_t* words, uint32_t* __restrict__ tperm) {
  extern __shared__ __align__(16) unsigned char rk_raw[];
  __shared__ uint32_t rank[32 * ITEMS], trank[32 * ITEMS], species[8];
  const int n = (int)a.n, npad = (n + kRkPad - 1) / kRkPad * kRkPad;
  uint64_t* sk = reinterpret_cast<uint64_t*>(rk_raw);          // keys, the sorted digits only
  uint32_t* st = reinterpret_cast<uint32_t*>(sk + npad);       // species
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int b0 = blockIdx.x * 32 * ITEMS, b1 = b0 + 32 * ITEMS;
  for (int j = tid; j < 32 * ITEMS; j += kRkThreads) rank[j] = trank[j] = 0;
  if (tid < 8) species[tid] = 0;
  __syncthreads();
#pragma unroll 2
  for (int j0 = 0; j0 < npad; j0 += kRkThreads) {   // whole warps: npad is a multiple of 64
    const int j = j0 + tid;
    if (j0 + (tid & ~31) >= npad) break;
    uint32_t t = 8;
    uint64_t k = ~0ull;                             // behind every key
    if (j < n) {
      const uint8_t ty = a.type[j];
      k = body_key(a, j, ty) >> (8 * first);
      t = stored_type(ty, a.D);
    }
    sk[j] = k;
    st[j] = t;
    for (int q = 0; q < a.D; ++q) {
      const uint32_t m = __ballot_sync(0xffffffffu, t == (uint32_t)q);
      if (lane == 0 && m) atomicAdd(&species[q], (uint32_t)__popc(m));
    }
  }
  __syncthreads();
  uint64_t key[ITEMS];
  uint32_t ty[ITEMS], r[ITEMS], tr[ITEMS];
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    const int i = min(b0 + it * 32 + lane, n - 1);
    key[it] = sk[i];
    ty[it] = st[i];
    r[it] = tr[it] = 0;
  }
  // keys j before the block's bodies count when not above, those behind when below
  auto count = [&](int j, auto below) {
    const ulonglong2 ka = *reinterpret_cast<const ulonglong2*>(sk + j);
    const ulonglong2 kb = *reinterpret_cast<const ulonglong2*>(sk + j + 2);
    const uint4 t = *reinterpret_cast<const uint4*>(st + j);
    const uint64_t kj[4] = {ka.x, ka.y, kb.x, kb.y};
    const uint32_t tj[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int it = 0; it < ITEMS; ++it) {
        const bool lt = kj[u] < below(it, j + u);
        r[it] += lt ? 1u : 0u;
        tr[it] += lt && tj[u] == ty[it] ? 1u : 0u;
      }
  };
  const int per = npad / kRkWarps, js = w * per, je = js + per;   // multiples of 4
  uint64_t next[ITEMS];   // keys are below 2^63: no overflow
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) next[it] = key[it] + 1;
#pragma unroll 2
  for (int j = js; j < min(je, b0); j += 4) count(j, [&](int it, int) { return next[it]; });
  for (int j = max(js, b0); j < min(je, b1); j += 4)
    count(j, [&](int it, int jj) { return jj < b0 + it * 32 + lane ? next[it] : key[it]; });
#pragma unroll 2
  for (int j = max(js, b1); j < je; j += 4) count(j, [&](int it, int) { return key[it]; });
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    atomicAdd(&rank[it * 32 + lane], r[it]);
    atomicAdd(&trank[it * 32 + lane], tr[it]);
  }
  __syncthreads();
  for (int b = tid; b < 32 * ITEMS; b += kRkThreads) {
    const int i = b0 + b;
    if (i >= n) break;
    const uint32_t k = rank[b], t = st[i];
    keys[k] = body_key(a, i, a.type[i]);
    perm[k] = (uint32_t)i;
    if (RESIDENT) gather_resident(g, k, (uint32_t)i);
    else gather_plain(g, k, (uint32_t)i);
    uint32_t at = trank[b];
    for (uint32_t q = 0; q < t; ++q) at += species[q];
    tperm[at] = k;
  }
  if (blockIdx.x == 0 && tid < 8) words[kSwTypes + tid] = species[tid];
}

int work_grid(ng_ctx* c, int64_t items, int per_sm) {
  const int64_t need = (items + 255) / 256;
  const int64_t most = (int64_t)c->nsm * per_sm;
  return (int)std::max<int64_t>(1, std::min(need, most));
}

bool box_is_pow2(double L) {
  int e = 0;
  return std::frexp(L, &e) == 0.5;
}

int reserve_sort(ng_ctx* c, int64_t n) {
  NG_TRY(ensure(c, c->keys_a, n * 8));
  NG_TRY(ensure(c, c->keys_b, n * 8));
  NG_TRY(ensure(c, c->vals_a, n * 4));
  NG_TRY(ensure(c, c->vals_b, n * 4));
  NG_TRY(ensure(c, c->sort_words, kSortWords * sizeof(uint32_t)));
  // two radix passes' states (one cleared while the other is in use), then the type order's
  NG_TRY(ensure(c, c->lookback, (size_t)(2 * rs_lb_words(n) + 8 * to_tiles(n)) * sizeof(uint64_t)));
  NG_TRY(ensure(c, c->spos, n * 24));
  NG_TRY(ensure(c, c->smass, n * 4));
  NG_TRY(ensure(c, c->stype, n));
  NG_TRY(ensure(c, c->tperm, n * 4));
  NG_TRY(ensure(c, c->scan_part, kScanBlocks * sizeof(uint32_t)));
  return NG_OK;
}

template <int ITEMS, bool RESIDENT>
static int sort_rank(ng_ctx* c, const KeyArgs& a, const GatherArgs& g, int first) {
  const size_t smem = rank_smem(a.n);
  NG_CUDA(c, cudaFuncSetAttribute(k_sort_rank<ITEMS, RESIDENT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)rank_smem(kSmallSort)));
  const int grid = (int)((a.n + 32 * ITEMS - 1) / (32 * ITEMS));
  k_sort_rank<ITEMS, RESIDENT><<<grid, kRkThreads, smem, c->stream>>>(
      a, g, first, as<uint64_t>(c->keys_a), as<uint32_t>(c->vals_a), as<uint32_t>(c->sort_words),
      as<uint32_t>(c->tperm));
  c->launches += 1;
  c->typed = true;
  NG_CUDA(c, cudaGetLastError());
  return NG_OK;
}

// Keys of the bodies at g.pos, their stable sort (sorted keys in keys_a, the
// permutation sorted index -> input index in vals_a) and the gather into
// sorted order.
template <bool RESIDENT>
static int sort_stage(ng_ctx* c, GatherArgs g) {
  const int64_t n = g.n;
  uint64_t *ka = as<uint64_t>(c->keys_a), *kb = as<uint64_t>(c->keys_b);
  uint32_t *va = as<uint32_t>(c->vals_a), *vb = as<uint32_t>(c->vals_b);
  // 8 passes of 8 bits: the result returns to (ka, va). A tree capped at
  // level_cap reads the Morton bits of its levels only (bits >= 3 + 3 (20 -
  // cap)), so the passes below them are skipped, keeping an even number of
  // passes: bodies that share those bits keep their previous relative order,
  // and every cell down to the cap is still one contiguous range.
  int first = 0;
  if (c->level_cap < kMaxLevel) {
    first = (3 + 3 * (kMaxLevel - std::max(c->level_cap, 0))) / 8;
    if ((8 - first) & 1) --first;
  }
  c->sort_passes = 8 - first;
  c->typed = false;
  KeyArgs a{n, g.pos, g.type, g.L, g.invL, g.pow2, g.pow2 ? std::ilogb(c->L) : 0, c->p.D, g.mass, nullptr};
  if (n <= (g.pow2 ? kSmallSort : kSmallSortAnyBox)) {
    stage_mark(c, NG_STAGE_KEYS);
    // at most 128 blocks: one round on the SMs
    return n <= kSmallSort / 2 ? sort_rank<1, RESIDENT>(c, a, g, first) : sort_rank<2, RESIDENT>(c, a, g, first);
  }
  if (!RESIDENT && n >= kPackBodies && c->rpack.bytes >= (size_t)n * sizeof(double4_32a))
    g.rec = a.rec = as<double4_32a>(c->rpack);
  const int64_t lbw = rs_lb_words(n), lbt = 8 * to_tiles(n);
  uint64_t* lb = as<uint64_t>(c->lookback);
  stage_mark(c, NG_STAGE_KEYS);
  NG_CUDA(c, cudaMemsetAsync(c->sort_words.p, 0, kSortWords * sizeof(uint32_t), c->stream));
  // blocks of at least 2048 bodies, at most two per SM: each adds its
  // histograms to the global ones
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)c->nsm * 2, (n + 2047) / 2048));
  k_keys<<<grid, 512, 0, c->stream>>>(a, first, ka, as<uint32_t>(c->sort_words),
                                      lb, lbw, lb + 2 * lbw, lbt);
  c->launches += 1;
  NG_CUDA(c, cudaGetLastError());
  stage_mark(c, NG_STAGE_RADIX);
  for (int pass = first; pass < 8; ++pass) {
    const bool even = ((pass - first) & 1) == 0;
    const uint64_t* kin = even ? ka : kb;
    const uint32_t* vin = pass == first ? nullptr : even ? va : vb;   // first pass: the index
    uint64_t* kout = even ? kb : ka;
    const RsLookback lin = rs_lookback(even ? lb : lb + lbw, n), lnext = rs_lookback(even ? lb + lbw : lb, n);
    uint32_t* vout = even ? vb : va;
    if (rs_large(n)) NG_TRY(rs_pass<kRsItemsLarge>(c, kin, vin, kout, vout, n, pass, lin, lnext));
    else NG_TRY(rs_pass<kRsItemsSmall>(c, kin, vin, kout, vout, n, pass, lin, lnext));
  }
  stage_mark(c, NG_STAGE_GATHER);
  k_gather<RESIDENT><<<work_grid(c, n, 8), 256, 0, c->stream>>>(g, va);
  c->launches += 1;
  NG_CUDA(c, cudaGetLastError());
  return NG_OK;
}

static GatherArgs gather_args(ng_ctx* c, int64_t n) {
  GatherArgs g{};
  g.n = n;
  g.spos = as<double>(c->spos);
  g.smass = as<float>(c->smass);
  g.stype = as<uint8_t>(c->stype);
  g.L = c->L;
  g.invL = 1.0 / c->L;
  g.pow2 = box_is_pow2(c->L);
  g.D = c->p.D;
  g.status = as<uint32_t>(c->status);
  return g;
}

int sort_resident(ng_ctx* c, int64_t n) {
  GatherArgs g = gather_args(c, n);
  g.pos = as<double>(c->spos_alt);
  g.mass = as<float>(c->smass_alt);
  g.type = as<uint8_t>(c->stype_alt);
  g.vel = as<float>(c->rvel_alt);
  g.orig = as<uint32_t>(c->rorig_alt);
  g.svel = as<float>(c->rvel);
  g.sorig = as<uint32_t>(c->rorig);
  return sort_stage<true>(c, g);
}

int sort_bodies(ng_ctx* c, int64_t n, const double* pos, const uint8_t* type, const float* mass) {
  NG_TRY(reserve_sort(c, n));
  GatherArgs g = gather_args(c, n);
  g.pos = pos;
  g.mass = mass;
  g.type = type;
  return sort_stage<false>(c, g);
}

int type_order(ng_ctx* c) {
  const int64_t n = c->n;
  stage_mark(c, NG_STAGE_TYPE_ORDER);
  // a tree rebuilt on the same sorted bodies keeps their order (the launch
  // takes its tickets and look-back state as the sort's key kernel left them)
  if (c->typed) return NG_OK;
  c->typed = true;
  k_type_order<<<(int)to_tiles(n), kToThreads, 0, c->stream>>>(
      n, c->p.D, as<uint8_t>(c->stype), as<uint32_t>(c->sort_words),
      as<uint64_t>(c->lookback) + 2 * rs_lb_words(n), as<uint32_t>(c->tperm));
  c->launches += 1;
  NG_CUDA(c, cudaGetLastError());
  return NG_OK;
}

const uint32_t* type_counts(const ng_ctx* c) { return as<uint32_t>(c->sort_words) + kSwTypes; }

}  // namespace ng
