// Pure tree mode (no TreePM split, no PM): the per-particle walk with the
// full laws, including the accumulator ("Mahalo") laws of Sec. 3.3 whose
// force depends on the number N_perp of bodies behind a monopole and on the
// passive mass, so it cannot be read from a table of separations.
//
// One warp per sorted body walks the tree with the criterion of the
// per-particle count (geometric or relative, decisions in FP64 as there),
// a node per lane, and evaluates every accepted species monopole and every
// body of an opened leaf, a term per lane, with the pair's law in FP32
// (offsets and |d|^2 + eps^2 from positions held as two floats each, correct
// to 2^-30 of |d| before their one rounding to FP32, and from the FP64
// positions where the pair is closer than that allows; the cut-off decided as
// in FP64):
//   Newton         f = 1
//   Yukawa (C=1)   f = 1 + a (1 + r/l) e^{-r/l}
//   pure Yukawa    f = a (1 + r/l) e^{-r/l}
//   Mahalo         f = (2/pi) [atan(x) - x / (1 + x^2)], x = 4 pi beta r / s,
//                  s = (active cored ? M / N_perp : 0) + (passive cored ? m : 0)
// and the acceleration G M f(rho) d / rho^3 at the softened separation rho,
// for rho < r_cut (minimum image, r_cut < L/2). A species is cored when its
// own pair law is the Mahalo law.
//
// Pure tree mode 2 (Sec. 2.3 lattice corrections): no cut-off, and every
// term adds the force of all other periodic images of its source, read by
// trilinear interpolation from a table of the correction over [0, L/2]^3
// (one per distinct law; each component odd in its own axis, even in the
// others). The tables are computed here in FP64: an Ewald sum for the
// Newtonian part, an image sum for Yukawa parts (yuk_l <= L/8).
#include "ng_internal.cuh"

namespace ng {

namespace {

struct ExactArgs {
  const float4* geo;       // [node] centre, half side (box units, exact in FP32)
  const int4* link;        // [node] child_first, nchild, body_first, body_count
  const double* m64;       // [node][D][4]: M, sum m x, sum m y, sum m z (box units)
  const uint32_t* cnt;     // [node][D]: N_perp
  // positions in box units as two floats, x = hi + lo to 2^-49: bodies
  // {hi, m}, {lo, species}; node species {com hi, M}, {com lo, N_perp}; and the
  // centre of mass of all species of a node, hi only
  float4* brec;            // [body][2]
  float4* nrec;            // [node][D][2]
  float4* arec;            // [node]
  const double* spos;      // [3][n] sorted, physical
  const float* smass;      // [n] sorted
  const uint8_t* stype;    // [n] sorted
  const uint32_t* perm;    // sorted -> caller (previous accelerations)
  const uint32_t* out;     // sorted -> output index (nullptr: sorted order)
  int64_t n;
  int D;
  double invL, L;
  double rcut2_box;        // cut-off^2 in box units (node skipping)
  double theta;
  const float* aold;
  double alphaL2, gmax;
  int relative;
  int ignore_nperp;
  double rcut2, eps2;           // physical units (cut-off decided in FP64, as the oracle)
  float beta4pi;
  int8_t kind[kMaxD][kMaxD];
  float G[kMaxD][kMaxD], ya[kMaxD][kMaxD], inv_l[kMaxD][kMaxD];
  uint8_t cored[kMaxD];
  const float4* lattice;   // [law][(N+1)^3] corrections per unit G M (box units), or nullptr
  int lat_n;               // N
  float lat_scale;         // 2 N / L
  float lat_inv_l2;        // 1 / L^2
  int8_t tabid[kMaxD][kMaxD];
  float* acc;              // [3][n] output order
  int accumulate;
  unsigned long long* counter;   // executed terms (optional)
  uint32_t* status;
  bool unit;               // L == 1
  float Lh, Ll;            // L = Lh + Ll
  float theta32;
  float eps2h, eps2l;      // eps2 = eps2h + eps2l
  float cut_lo2, cut_hi2;  // node cut-off^2 (box units) less and plus the FP32 margin
  float rc2f;              // rcut2, for the terms' FP32 decision
};

// One term within the cut-off: passive species s of mass mp, active species t
// of mass M behind which stand np bodies, offset (physical, source - target)
// and softened separation^2 q; the law is evaluated in FP32.
__device__ __forceinline__ void exact_term(const ExactArgs& a, int s, int t, float M, float np,
                                           float mp, float dx, float dy, float dz, float q, float& ax,
                                           float& ay, float& az) {
  const float rho = sqrtf(q);
  float f;
  const int kind = a.kind[s][t];
  if (kind == NG_MAHALO) {
    const float npu = a.ignore_nperp ? 1.f : np;
    const float scale = (a.cored[t] ? M / npu : 0.f) + (a.cored[s] ? mp : 0.f);
    const float x = a.beta4pi * rho / scale;
    f = 0.63661977236758134f * (atanf(x) - x / fmaf(x, x, 1.f));
  } else {
    f = kind == NG_YUKAWA_PURE ? 0.f : 1.f;
    if (kind == NG_YUKAWA || kind == NG_YUKAWA_PURE) {
      const float u = rho * a.inv_l[s][t];
      f = fmaf(a.ya[s][t] * (1.f + u), expf(-u), f);
    }
  }
  const float g = a.G[s][t] * M * f / (q * rho);
  ax = fmaf(g, dx, ax);
  ay = fmaf(g, dy, ay);
  az = fmaf(g, dz, az);
  if (a.lattice) {
    // all other images: trilinear interpolation at |d|, signs per axis
    const int N = a.lat_n, P = N + 1;
    const float4* T = a.lattice + (size_t)a.tabid[s][t] * P * P * P;
    const float dv[3] = {dx, dy, dz};
    int i0[3];
    float fr[3];
#pragma unroll
    for (int e = 0; e < 3; ++e) {
      const float u = fminf(fabsf(dv[e]) * a.lat_scale, (float)N);
      i0[e] = min((int)u, N - 1);
      fr[e] = u - (float)i0[e];
    }
    float cx = 0.f, cy = 0.f, cz = 0.f;
#pragma unroll
    for (int corner = 0; corner < 8; ++corner) {
      const int bx = corner >> 2, by = (corner >> 1) & 1, bz = corner & 1;
      const float w = (bx ? fr[0] : 1.f - fr[0]) * (by ? fr[1] : 1.f - fr[1]) *
                      (bz ? fr[2] : 1.f - fr[2]);
      const float4 v = __ldg(T + ((size_t)(i0[0] + bx) * P + (i0[1] + by)) * P + (i0[2] + bz));
      cx = fmaf(w, v.x, cx);
      cy = fmaf(w, v.y, cy);
      cz = fmaf(w, v.z, cz);
    }
    const float gc = a.G[s][t] * M * a.lat_inv_l2;
    // the table holds d_e >= 0; the component flips with the sign of d_e
    ax = fmaf(gc, dx < 0.f ? -cx : cx, ax);
    ay = fmaf(gc, dy < 0.f ? -cy : cy, ay);
    az = fmaf(gc, dz < 0.f ? -cz : cz, az);
  }
}

// hi + lo of a position (box units)
__device__ __forceinline__ void split(double p, float* hi, float* lo) {
  *hi = (float)p;
  *lo = (float)(p - (double)*hi);
}

// The two-float records of every body and node.
__global__ void k_exact_prep(ExactArgs a) {
  if (a.status[ST_FLAGS] & SF_NODE_OVERFLOW) return;
  const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t b = t0; b < a.n; b += stride) {
    float h[3], l[3];
    for (int e = 0; e < 3; ++e) split(a.spos[e * a.n + b] * a.invL, &h[e], &l[e]);
    a.brec[2 * b] = make_float4(h[0], h[1], h[2], a.smass[b]);
    a.brec[2 * b + 1] = make_float4(l[0], l[1], l[2], __int_as_float((int)a.stype[b]));
  }
  const uint32_t total = a.status[ST_LEVELS + kMaxLevel + 1];
  for (int64_t k = t0; k < (int64_t)total; k += stride) {
    double mt = 0.0, st[3] = {0.0, 0.0, 0.0};
    for (int t = 0; t < a.D; ++t) {
      const size_t r = (size_t)k * a.D + t;
      const double* m = a.m64 + r * 4;
      float h[3] = {0.f, 0.f, 0.f}, l[3] = {0.f, 0.f, 0.f};
      mt += m[0];
      for (int e = 0; e < 3; ++e) {
        st[e] += m[1 + e];
        if (m[0] > 0.0) split(m[1 + e] / m[0], &h[e], &l[e]);
      }
      // (a positive mass that is zero in FP32 still is a term)
      const float M = m[0] > 0.0 ? (float)m[0] : -1.f;
      a.nrec[2 * r] = make_float4(h[0], h[1], h[2], M);
      a.nrec[2 * r + 1] = make_float4(l[0], l[1], l[2], (float)a.cnt[r]);
    }
    a.arec[k] = make_float4((float)(st[0] / mt), (float)(st[1] / mt), (float)(st[2] / mt), 0.f);
  }
}

// FP32 offset wrapped to the nearest image (|d| < 1; exact)
__device__ __forceinline__ float image32(float d) { return fabsf(d) > 0.5f ? d - copysignf(1.f, d) : d; }

// Whether the per-particle walk accepts node nd for the body at x, decided in
// FP64 as the count decides: 0 beyond the cut-off, 1 accepted, 2 opened.
__device__ __noinline__ int exact_decide64(const ExactArgs& a, uint32_t nd, int64_t k) {
  const double x[3] = {a.spos[k] * a.invL, a.spos[a.n + k] * a.invL, a.spos[2 * a.n + k] * a.invL};
  const float4 ge = a.geo[nd];
  const double c[3] = {(double)ge.x, (double)ge.y, (double)ge.z};
  const double half = (double)ge.w, side = 2.0 * half;
  double g2 = 0.0, dcs[3];
  bool inside = true;
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    const double dc = nearest_image_unit(__dsub_rn(c[e], x[e]));
    dcs[e] = dc;
    double gap = __dsub_rn(fabs(dc), half);
    gap = gap > 0.0 ? gap : 0.0;
    g2 = __dadd_rn(g2, __dmul_rn(gap, gap));
    if (fabs(dc) > half) inside = false;
  }
  if (g2 >= a.rcut2_box) return 0;
  if (inside) return 2;
  double mt = 0.0, sx = 0.0, sy = 0.0, sz = 0.0;
  for (int t = 0; t < a.D; ++t) {
    const double* m = a.m64 + ((size_t)nd * a.D + t) * 4;
    mt += m[0];
    sx += m[1];
    sy += m[2];
    sz += m[3];
  }
  const double com[3] = {sx / mt, sy / mt, sz / mt};
  double dd2 = 0.0;
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    const double v = nearest_image_unit(__dsub_rn(com[e], x[e]));
    dd2 = __dadd_rn(dd2, __dmul_rn(v, v));
  }
  if (a.relative) {
    const double lim = __dmul_rn(0.6, side);
    bool near = true;
#pragma unroll
    for (int e = 0; e < 3; ++e)
      if (!(fabs(dcs[e]) < lim)) near = false;
    const double lhs = __dmul_rn(__dmul_rn(a.gmax, mt), __dmul_rn(side, side));
    const double rhs = __dmul_rn(__dmul_rn(a.alphaL2, (double)a.aold[a.perm[k]]), __dmul_rn(dd2, dd2));
    return !near && lhs <= rhs ? 1 : 2;
  }
  return side < __dmul_rn(a.theta, sqrt(dd2)) ? 1 : 2;
}

// The same in FP32 where it is certain, else -1 (geometric criterion). Error
// bounds, box units (coordinates below 1): a node centre is exact, x and the
// centre of mass are rounded by 2^-25, a difference by 2^-25 more, so that gaps
// and |offsets| per axis are known to 1e-7, distances to 2e-7 and to a few
// 2^-24 of themselves; the margins are at least twice that.
__device__ __forceinline__ int exact_decide32(const ExactArgs& a, const float4 ge, const float4 cm,
                                              const float xh[3]) {
  const float gx = fabsf(image32(ge.x - xh[0])) - ge.w, gy = fabsf(image32(ge.y - xh[1])) - ge.w,
              gz = fabsf(image32(ge.z - xh[2])) - ge.w;
  const float far = fmaxf(gx, fmaxf(gy, gz));
  const float px = fmaxf(gx, 0.f), py = fmaxf(gy, 0.f), pz = fmaxf(gz, 0.f);
  const float g2 = fmaf(px, px, fmaf(py, py, pz * pz));
  if (g2 > a.cut_hi2) return 0;
  if (!(g2 < a.cut_lo2)) return -1;
  if (far < -4e-7f) return 2;          // inside the cube
  if (!(far > 4e-7f)) return -1;
  const float ex = image32(cm.x - xh[0]), ey = image32(cm.y - xh[1]), ez = image32(cm.z - xh[2]);
  const float d = sqrtf(fmaf(ex, ex, fmaf(ey, ey, ez * ez)));
  const float m = fmaf(2e-6f, d, 6e-7f), side = 2.f * ge.w;
  if (side < a.theta32 * (d - m) * 0.999999f) return 1;
  if (side > a.theta32 * (d + m) * 1.000001f) return 2;
  return -1;
}

// Bodies closer than this (box units, largest component) take their offset from
// the FP64 positions: two floats hold a position to 2^-50 and leave an offset
// uncertain by 2^-47 with the roundings of their difference, 2^-31 of |d| here.
constexpr float kExactNear = 1.f / 65536.f;

// A term in FP64, in the operation order of the count: offset (physical) and
// |d|^2 + eps^2 of node species record or body src from body k, each rounded
// once; w < 0: beyond the cut-off.
__device__ __noinline__ float4 exact_pair64(const ExactArgs& a, bool mono, uint32_t src, int64_t k) {
  double d[3];
  const double* m = a.m64 + (size_t)src * 4;
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    const double p = mono ? m[1 + e] / m[0] : a.spos[e * a.n + src] * a.invL;
    d[e] = nearest_image_unit(__dsub_rn(p, a.spos[e * a.n + k] * a.invL)) * a.L;
  }
  const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1])),
                              __dmul_rn(d[2], d[2]));
  const double q = __dadd_rn(r2, a.eps2);
  return make_float4((float)d[0], (float)d[1], (float)d[2], q < a.rcut2 ? (float)q : -1.f);
}

// Offset of two-float position (ph, pl) from (xh, xl) as two floats: the
// difference of the high parts with its rounding error (Knuth's two-sum),
// wrapped exactly, plus the low parts; times L. x: the offset rounded to FP32,
// y: what the rounding left. far: the largest |component| so far, box units.
__device__ __forceinline__ float2 exact_offset(const ExactArgs& a, float ph, float pl, float xh, float xl,
                                               float& far) {
  const float s = __fsub_rn(ph, xh);
  const float bb = __fsub_rn(s, ph);
  const float err = __fsub_rn(__fsub_rn(ph, __fsub_rn(s, bb)), __fadd_rn(xh, bb));
  float w = image32(s), low = __fadd_rn(err, __fsub_rn(pl, xl));
  far = fmaxf(far, fabsf(w));
  if (!a.unit) {
    const float p = __fmul_rn(w, a.Lh);
    low = fmaf(w, a.Ll, fmaf(low, a.Lh, fmaf(w, a.Lh, -p)));
    w = p;
  }
  const float h = __fadd_rn(w, low);
  return make_float2(h, __fsub_rn(low, __fsub_rn(h, w)));
}

// |d|^2 + eps^2 of two-float offsets: squares with their rounding errors,
// summed with the errors of the sum (Knuth's two-sum), so that only the last
// rounding is left, as from an FP64 sum.
__device__ __forceinline__ float exact_q(const ExactArgs& a, float2 x, float2 y, float2 z) {
  const float px = __fmul_rn(x.x, x.x), py = __fmul_rn(y.x, y.x), pz = __fmul_rn(z.x, z.x);
  const float ex = fmaf(x.x + x.x, x.y, fmaf(x.x, x.x, -px));
  const float ey = fmaf(y.x + y.x, y.y, fmaf(y.x, y.x, -py));
  const float ez = fmaf(z.x + z.x, z.y, fmaf(z.x, z.x, -pz));
  float low = (ex + ey) + (ez + a.eps2l);
  float sum = px;
  const float add[3] = {py, pz, a.eps2h};
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const float s = __fadd_rn(sum, add[j]);
    const float bb = __fsub_rn(s, sum);
    low += __fadd_rn(__fsub_rn(sum, __fsub_rn(s, bb)), __fsub_rn(add[j], bb));
    sum = s;
  }
  return __fadd_rn(sum, low);
}

constexpr int kExactWarps = 4;

struct ExactWarp {
  uint32_t stack[kStackCap];
  uint32_t node[32];      // accepted nodes of the round
  uint32_t lfirst[32];    // opened leaves of the round: first body
  uint32_t loff[32];      // and exclusive prefix of body counts
};

// One warp per body. A thread per body left the threads of a warp on
// different nodes and leaves, and few warps in flight (30k bodies: 940); here
// the lanes of a warp take 32 nodes of the body's stack at a time, then the
// terms these rounds accept and open, 32 at a time. In FP64 (1/64 of the FP32
// rate) the decisions and offsets kept that pipe 85 % busy; they are now made
// in FP32 with error bounds, in FP64 only where FP32 cannot tell, with the same
// outcome. 30011 bodies, two species, leaf 8: 11.4 ms with a thread per body,
// 3.4 ms with a warp per body in FP64, 0.52 ms with FP32 throughout; offsets and
// |d|^2 with the digits of FP64 cost 6 % (30011 bodies in 8 spheres: a tree force
// 782 -> 832 us; at 72 and 80 registers, with less spilled, 862 and 901). The terms
// and their number are those of the per-particle count; each lane sums its terms
// in FP32, the lanes' sums are added at the end.
__global__ void __launch_bounds__(32 * kExactWarps, 8) k_walk_exact(ExactArgs a) {
  __shared__ ExactWarp sm[kExactWarps];
  if (a.status[ST_FLAGS] & SF_NODE_OVERFLOW) return;
  ExactWarp& ws = sm[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  const uint32_t nnodes = a.status[ST_LEVELS + kMaxLevel + 1];
  unsigned long long mine = 0;
  for (int64_t k = (int64_t)blockIdx.x * kExactWarps + (threadIdx.x >> 5); k < a.n;
       k += (int64_t)gridDim.x * kExactWarps) {
    const float4 bh = a.brec[2 * k], bl = a.brec[2 * k + 1];
    const float xh[3] = {bh.x, bh.y, bh.z};
    const int s = __float_as_int(bl.w);
    const float mp = bh.w;
    float ax = 0.f, ay = 0.f, az = 0.f;
    uint32_t terms = 0;
    if (lane == 0) ws.stack[0] = 0;
    int size = 1;
    uint32_t visits = 0;
    uint32_t bad = 0;
    __syncwarp();
    while (size > 0) {
      // the stack of the group walk: up to 32 nodes from the top; opened
      // nodes whose children do not fit are pushed back (see k_walk)
      if (size + 7 > kStackCap) { bad = SF_STACK_OVERFLOW; break; }
      if (visits > nnodes) { bad = SF_BAD_TREE; break; }
      int kk = min(32, size);
      int avail = (kStackCap - kStackReserve) - (size - kk);
      if (avail < 8) {
        kk = 1;
        avail = kStackCap - (size - 1);
      }
      visits += kk;
      const bool has = lane < kk;
      const uint32_t nd = has ? ws.stack[size - kk + lane] : 0u;
      size -= kk;
      __syncwarp();
      int cls = 0;   // 0 skip, 1 accept, 2 leaf, 3 open
      int4 lk = make_int4(0, 0, 0, 0);
      if (has) {
        const float4 ge = a.geo[nd];
        const float4 cm = a.arec[nd];
        lk = a.link[nd];
        int r = a.relative ? -1 : exact_decide32(a, ge, cm, xh);
        if (r < 0) r = exact_decide64(a, nd, k);
        cls = r == 2 ? (lk.y == 0 ? 2 : 3) : r;
      }
      const uint32_t nch = (uint32_t)lk.y;
      // opened nodes: children onto the stack
      {
        const uint32_t mych = cls == 3 ? nch : 0u;
        uint32_t incl = mych;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += t;
        }
        const bool fit = (int)incl <= avail;
        const uint32_t back = __ballot_sync(0xffffffffu, cls == 3 && !fit);
        const int used = (int)__reduce_max_sync(0xffffffffu, fit ? incl : 0u);
        if (cls == 3) {
          if (fit) {
            const uint32_t c0 = (uint32_t)lk.x;
            for (uint32_t j = 0; j < nch; ++j) ws.stack[size + (int)(incl - mych + j)] = c0 + j;
          } else {
            ws.stack[size + used + __popc(back & lt)] = nd;
          }
        }
        size += used + __popc(back);
        visits -= __popc(back);
      }
      // accepted nodes: a term per species with mass
      const uint32_t acc = __ballot_sync(0xffffffffu, cls == 1);
      if (cls == 1) ws.node[__popc(acc & lt)] = nd;
      // opened leaves: their bodies
      const uint32_t lm = __ballot_sync(0xffffffffu, cls == 2);
      uint32_t bodies = 0;
      if (lm) {
        const uint32_t nb = cls == 2 ? (uint32_t)lk.w : 0u;
        uint32_t incl = nb;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += t;
        }
        bodies = __shfl_sync(0xffffffffu, incl, 31);
        if (cls == 2) {
          const int at = __popc(lm & lt);
          ws.lfirst[at] = (uint32_t)lk.z;
          ws.loff[at] = incl - nb;
        }
      }
      __syncwarp();
      // monopole terms, then body terms, in one run of lanes
      const uint32_t monos = (uint32_t)__popc(acc) * (uint32_t)a.D;
      const int nl = __popc(lm);
      for (uint32_t f = lane; f < monos + bodies; f += 32) {
        float4 ph, pl;
        float np = 1.f;
        int t;
        uint32_t src;   // node species record, or body
        const bool mono = f < monos;
        if (mono) {
          const uint32_t i = f / (uint32_t)a.D;
          t = (int)(f - i * (uint32_t)a.D);
          src = ws.node[i] * (uint32_t)a.D + (uint32_t)t;
          ph = a.nrec[2 * (size_t)src];
          if (ph.w < 0.f) continue;   // no mass of this species
          pl = a.nrec[2 * (size_t)src + 1];
          np = pl.w;
        } else {
          const uint32_t h = f - monos;
          int lo = 0, hi = nl - 1;   // the last leaf that starts at or before h
          while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (ws.loff[mid] <= h) lo = mid; else hi = mid - 1;
          }
          src = ws.lfirst[lo] + (h - ws.loff[lo]);
          if ((int64_t)src == k) continue;
          ph = a.brec[2 * (size_t)src];
          pl = a.brec[2 * (size_t)src + 1];
          t = __float_as_int(pl.w);
        }
        float far = 0.f;
        const float2 x2 = exact_offset(a, ph.x, pl.x, xh[0], bl.x, far);
        const float2 y2 = exact_offset(a, ph.y, pl.y, xh[1], bl.y, far);
        const float2 z2 = exact_offset(a, ph.z, pl.z, xh[2], bl.z, far);
        float dx = x2.x, dy = y2.x, dz = z2.x, q = exact_q(a, x2, y2, z2);
        bool within = q < a.rc2f;
        // where two floats or FP32 cannot tell (both rare)
        if (far < kExactNear || (fabsf(q - a.rc2f) <= 2e-6f * a.rc2f && a.rc2f < 3.0e38f)) {
          const float4 d = exact_pair64(a, mono, src, k);
          dx = d.x;
          dy = d.y;
          dz = d.z;
          q = d.w;
          within = q >= 0.f;
        }
        if (within) exact_term(a, s, t, ph.w, np, mp, dx, dy, dz, q, ax, ay, az);
        ++terms;
      }
      __syncwarp();
    }
    if (bad && lane == 0) atomicOr(&a.status[ST_FLAGS], bad);
    __syncwarp();
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      ax += __shfl_xor_sync(0xffffffffu, ax, o);
      ay += __shfl_xor_sync(0xffffffffu, ay, o);
      az += __shfl_xor_sync(0xffffffffu, az, o);
    }
    mine += terms;
    if (lane < 3) {
      const uint32_t i = a.out ? a.out[k] : (uint32_t)k;
      const float v = lane == 0 ? ax : lane == 1 ? ay : az;
      float* o = a.acc + (size_t)lane * a.n + i;
      *o = a.accumulate ? *o + v : v;
    }
  }
  if (a.counter) {
    for (int o = 16; o; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
    if (lane == 0 && mine) atomicAdd(a.counter, mine);
  }
}

}  // namespace

int launch_walk_exact(ng_ctx* c, float* acc, bool accumulate, bool count) {
  ExactArgs a{};
  a.geo = as<float4>(c->n_geo);
  a.link = as<int4>(c->n_link);
  a.m64 = as<double>(c->n_m64);
  a.brec = as<float4>(c->exact_body);
  a.nrec = as<float4>(c->exact_node);
  a.arec = a.nrec + (size_t)c->cap_nodes * c->p.D * 2;
  a.cnt = as<uint32_t>(c->n_cnt);
  a.spos = as<double>(c->spos);
  a.smass = as<float>(c->smass);
  a.stype = as<uint8_t>(c->stype);
  a.perm = as<uint32_t>(c->vals_a);
  a.out = force_out(c);
  a.n = c->n;
  a.D = c->p.D;
  a.L = c->L;
  a.invL = 1.0 / c->L;
  const double rc = c->rcut / c->L;
  a.rcut2_box = rc * rc;
  a.theta = c->p.theta;
  a.relative = relative_active(c) ? 1 : 0;
  a.aold = as<float>(c->aold);
  a.alphaL2 = c->p.alpha * c->L * c->L;
  a.gmax = coupling_max(c);
  a.ignore_nperp = c->p.ignore_nperp;
  a.rcut2 = c->rcut * c->rcut;
  a.eps2 = c->p.eps * c->p.eps;
  a.beta4pi = (float)(4.0 * M_PI * c->p.beta);
  for (int i = 0; i < kMaxD; ++i) {
    a.cored[i] = i < c->p.D && c->p.law[i][i] == NG_MAHALO ? 1 : 0;
    for (int j = 0; j < kMaxD; ++j) {
      const bool in = i < c->p.D && j < c->p.D;
      a.kind[i][j] = (int8_t)(in ? c->p.law[i][j] : NG_NEWTON);
      a.G[i][j] = in ? (float)c->p.G[i][j] : 0.f;
      a.ya[i][j] = in ? (float)c->p.yuk_a[i][j] : 0.f;
      a.inv_l[i][j] = in && c->p.yuk_l[i][j] > 0 ? (float)(1.0 / c->p.yuk_l[i][j]) : 0.f;
    }
  }
  a.lattice = c->lattice_grid > 0 ? as<float4>(c->lattice) : nullptr;
  a.lat_n = c->lattice_grid;
  a.lat_scale = (float)(2.0 * c->lattice_grid / c->L);
  a.lat_inv_l2 = (float)(1.0 / (c->L * c->L));
  for (int i = 0; i < kMaxD; ++i)
    for (int j = 0; j < kMaxD; ++j) a.tabid[i][j] = c->tabid[i][j];
  a.acc = acc;
  a.accumulate = accumulate ? 1 : 0;
  a.counter = count ? as<unsigned long long>(c->counter) : nullptr;
  a.status = as<uint32_t>(c->status);
  a.unit = c->L == 1.0;
  a.Lh = (float)c->L;
  a.Ll = (float)(c->L - (double)a.Lh);
  a.theta32 = (float)a.theta;
  a.eps2h = (float)a.eps2;
  a.eps2l = (float)(a.eps2 - (double)a.eps2h);
  a.rc2f = (float)a.rcut2;
  a.cut_lo2 = (float)((rc - 2e-6) * (rc - 2e-6) * 0.999999);
  a.cut_hi2 = (float)((rc + 2e-6) * (rc + 2e-6) * 1.000001);
  if (!(rc > 4e-6)) a.cut_lo2 = -1.f;   // a cut-off near the margin: always in FP64
  k_exact_prep<<<work_grid(c, c->n, 8), 256, 0, c->stream>>>(a);
  // one warp a body, eight blocks per SM resident; bodies are taken in turns
  const int64_t blocks = (c->n + kExactWarps - 1) / kExactWarps;
  k_walk_exact<<<(int)std::min<int64_t>(blocks, (int64_t)c->nsm * 64), 32 * kExactWarps, 0, c->stream>>>(a);
  c->launches += 2;
  NG_CUDA(c, cudaGetLastError());
  return NG_OK;
}

// ------------------------------------------------ lattice-correction tables

// Correction of one law at grid point (i, j, k) of [0, 1/2]^3 (box units,
// L = 1), per unit G M, FP64: all images but the nearest. Newtonian part by
// Ewald summation (splitting 2; real-space images |n_i| <= 3, reciprocal
// vectors |m_i| <= 5); Yukawa part a (1 + mu r) e^{-mu r} / r^2 by images
// |n_i| <= 4.
__global__ void k_lattice_table(int kind, double ya, double mu, int N, float4* out) {
  const int P = N + 1;
  const int64_t total = (int64_t)P * P * P;
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < total;
       g += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(g / ((int64_t)P * P)), j = (int)((g / P) % P), k = (int)(g % P);
    const double d[3] = {0.5 * i / N, 0.5 * j / N, 0.5 * k / N};
    double acc[3] = {0.0, 0.0, 0.0};
    if (kind != NG_YUKAWA_PURE) {
      const double al = 2.0;
      for (int nx = -3; nx <= 3; ++nx)
        for (int ny = -3; ny <= 3; ++ny)
          for (int nz = -3; nz <= 3; ++nz) {
            const double v[3] = {d[0] + nx, d[1] + ny, d[2] + nz};
            const double r = sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
            if (r == 0.0) continue;
            const double f = (erfc(al * r) + 2.0 * al * r * 0.56418958354775628 *
                                                 exp(-al * al * r * r)) / (r * r * r);
            for (int e = 0; e < 3; ++e) acc[e] += f * v[e];
          }
      for (int mx = -5; mx <= 5; ++mx)
        for (int my = -5; my <= 5; ++my)
          for (int mz = -5; mz <= 5; ++mz) {
            if (mx == 0 && my == 0 && mz == 0) continue;
            const double kv[3] = {2.0 * M_PI * mx, 2.0 * M_PI * my, 2.0 * M_PI * mz};
            const double k2 = kv[0] * kv[0] + kv[1] * kv[1] + kv[2] * kv[2];
            const double w = 4.0 * M_PI / k2 * exp(-k2 / (4.0 * al * al)) *
                             sin(kv[0] * d[0] + kv[1] * d[1] + kv[2] * d[2]);
            for (int e = 0; e < 3; ++e) acc[e] += w * kv[e];
          }
      const double r = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
      if (r > 0.0)
        for (int e = 0; e < 3; ++e) acc[e] -= d[e] / (r * r * r);
    }
    if (kind == NG_YUKAWA || kind == NG_YUKAWA_PURE) {
      for (int nx = -4; nx <= 4; ++nx)
        for (int ny = -4; ny <= 4; ++ny)
          for (int nz = -4; nz <= 4; ++nz) {
            if (nx == 0 && ny == 0 && nz == 0) continue;
            const double v[3] = {d[0] + nx, d[1] + ny, d[2] + nz};
            const double r = sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
            const double f = ya * (1.0 + mu * r) * exp(-mu * r) / (r * r * r);
            for (int e = 0; e < 3; ++e) acc[e] += f * v[e];
          }
    }
    out[g] = make_float4((float)acc[0], (float)acc[1], (float)acc[2], 0.f);
  }
}

int build_lattice(ng_ctx* c, int nlaws, const int* kind, const double* a, const double* l) {
  constexpr int N = 64;
  const size_t P3 = (size_t)(N + 1) * (N + 1) * (N + 1);
  NG_TRY(ensure(c, c->lattice, (size_t)nlaws * P3 * sizeof(float4)));
  for (int u = 0; u < nlaws; ++u) {
    const bool yk = kind[u] == NG_YUKAWA || kind[u] == NG_YUKAWA_PURE;
    k_lattice_table<<<work_grid(c, (int64_t)P3, 4), 256, 0, c->stream>>>(
        kind[u], yk ? a[u] : 0.0, yk ? c->L / l[u] : 0.0, N, as<float4>(c->lattice) + u * P3);
    c->launches += 1;
    NG_CUDA(c, cudaGetLastError());
  }
  c->lattice_grid = N;
  return NG_OK;
}

// The short-range (or, in pure tree mode, the whole) tree force of a context:
// the exact-law walk in pure tree mode, the FP64 pair sum in direct mode
// (theta = 0), the FP32 group walk otherwise.
int launch_tree_force(ng_ctx* c, float* acc, bool accumulate, bool count) {
  stage_mark(c, NG_STAGE_WALK);
  if (c->p.pure_tree) return launch_walk_exact(c, acc, accumulate, count);
  if (direct_mode(c)) return launch_direct64(c, acc, accumulate, count);
  return launch_walk(c, acc, accumulate, count);
}

}  // namespace ng
