// composite_warp.cuh — the warp walk shared by the tile-order compositing forward
// (composite_fwd.cu) and backward (composite_bwd.cu).
//
// A block covers an image tile (or 256 pixels of a larger one), a warp 64 of its pixels (an 8 x 8
// square when the tile is made of such squares), a thread two of them; the pair's arithmetic runs in
// packed FP32 (fma.rn.f32x2: one issue slot for two FMAs, each rounded like fmaf).  Both kernels are
// bound by instruction issue, not by memory or FP32 rate, so the layout is the one that needs the
// fewest warp instructions per (pixel, particle): a particle's record and 48 SH coefficients are
// read from shared memory once for 64 pixels instead of 32, and the backward's shuffle reductions
// run once for 64 pixels.
//
// Warps do not share staged data: each takes the tile's list 32 entries at a time, one lane per
// entry, drops the entries that cannot reach its pixels (rect_near on the prefetched rectangles,
// block_misses after activation), and stages only the survivors in its own shared memory.  About
// half of the (warp, entry) pairs survive (0.43 for the multi-view 3M-particle scene, 0.54 for 1M
// particles on one rolling-shutter 1080p view), so re-activating a particle in
// each of a tile's warps costs less than the walk over the rest did, and no warp ever waits for
// another one: there is no block barrier (the leading stall of a shared staging buffer).
#pragma once

#include "composite_common.cuh"

namespace ut3d {
namespace {

constexpr unsigned kFull = 0xffffffffu;

// ---------------------------------------------------------------- packed pairs (one value per pixel)

__device__ __forceinline__ float2 dot3x2(const f3x2 &a, const f3x2 &b) {
  return fma2(a.x, b.x, fma2(a.y, b.y, mul2(a.z, b.z)));
}

// M v for the record's M (row-major in g0, g1, g2.x), as mat3_mul rounds it
__device__ __forceinline__ f3x2 rec_mul(float4 g0, float4 g1, float4 g2, const f3x2 &v) {
  f3x2 r;
  r.x = fma2(bc(g0.x), v.x, fma2(bc(g0.y), v.y, mul2(bc(g0.z), v.z)));
  r.y = fma2(bc(g0.w), v.x, fma2(bc(g1.x), v.y, mul2(bc(g1.y), v.z)));
  r.z = fma2(bc(g1.z), v.x, fma2(bc(g1.w), v.y, mul2(bc(g2.x), v.z)));
  return r;
}

__device__ __forceinline__ f3x2 cross3x2(const f3x2 &a, const f3x2 &b) {
  f3x2 c;
  c.x = fma2(a.y, b.z, neg2(mul2(a.z, b.y)));
  c.y = fma2(a.z, b.x, neg2(mul2(a.x, b.z)));
  c.z = fma2(a.x, b.y, neg2(mul2(a.y, b.x)));
  return c;
}

// The canonical-space rays of a pixel pair: o_g, d_g, |o_g x d_g|^2 and |d_g|^2 (eval_response's
// arithmetic).
struct PairEval {
  f3x2 og, dg;
  float2 cc, dd;
};

template <bool RS>
__device__ __forceinline__ PairEval eval_pair(float4 g0, float4 g1, float4 g2, const f3x2 &o, const f3x2 &d) {
  PairEval e;
  e.dg = rec_mul(g0, g1, g2, d);
  if (RS) {
    const f3x2 m = rec_mul(g0, g1, g2, o);
    e.og.x = add2(m.x, bc(-g2.y));
    e.og.y = add2(m.y, bc(-g2.z));
    e.og.z = add2(m.z, bc(-g2.w));
  } else {
    e.og.x = bc(g2.y);
    e.og.y = bc(g2.z);
    e.og.z = bc(g2.w);
  }
  const f3x2 c = cross3x2(e.og, e.dg);
  e.cc = dot3x2(c, c);
  e.dd = dot3x2(e.dg, e.dg);
  return e;
}

// The hardware's reciprocal and power of two, one instruction each: for arguments and results known
// to be normal numbers (subnormals count as zero).
__device__ __forceinline__ float rcp_normal(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float exp2_normal(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// x^(m/2) of both pixels for an integer m >= 0: repeated products (and a square root for odd m).
__device__ __forceinline__ float2 pow_half2(float2 x, int m) {
  float2 p = (m & 1) ? make_float2(sqrtf(x.x), sqrtf(x.y)) : bc(1.f);
  for (int i = 0; i < (m >> 1); ++i) p = mul2(p, x);
  return p;
}

// rho(omega^2) of both pixels as 2^(log2(e) x exponent); alpha = sigma rho.  A pixel that passes the
// threshold test has rho >= alpha_min / sigma >= alpha_min; where that is subnormal rho may read 0.
// Other pixels' values are not used.  The degree-n kernel's power is one loop for the pair: a loop
// each, run whether the pixel needs it or not, cost the forward of 200k faint particles of degree 4
// at 64x64 2879 us, 2326 so.
template <bool GEN>
__device__ __forceinline__ float2 response2(float2 w2, const DevOpts &op) {
  constexpr float log2e = 1.4426950408889634f;
  if (!GEN) return make_float2(exp2_normal((-0.5f * log2e) * w2.x), exp2_normal((-0.5f * log2e) * w2.y));
  const float2 x = mul2(bc(log2e), mul2(bc(-op.kernel_lambda), pow_half2(w2, op.kernel_degree)));
  return make_float2(exp2_normal(x.x), exp2_normal(x.y));
}

// d rho / d omega^2 times sigma of both pixels for the degree-n kernel, from a = sigma rho at w2.
__device__ __forceinline__ float2 dresponse2(const DevOpts &op, float2 a, float2 w2) {
  const float c = -op.kernel_lambda * 0.5f * (float)op.kernel_degree;
  return mul2(mul2(bc(c), pow_half2(w2, op.kernel_degree - 2)), a);
}

// Raw colour of a staged particle for the pixel pair (sh_colour's order of operations; the first
// term, fmaf(beta_0, Y_0, 1/2), is the same for every pixel and staged in beta_0's place).
template <int NSH>
__device__ __forceinline__ void sh_colour2(const float *shb, const float2 *Y, float2 &r0, float2 &r1, float2 &r2) {
  constexpr int NC = NSH * 3;
  if constexpr (NC % 4 == 0) {
    const float4 *s4 = reinterpret_cast<const float4 *>(shb);
#pragma unroll
    for (int j = 0; j < NC / 4; ++j) {
      const float4 c = s4[j];
      const float cv[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int idx = 4 * j + e, k = idx / 3, ch = idx % 3;
        float2 &r = ch == 0 ? r0 : (ch == 1 ? r1 : r2);
        r = k == 0 ? bc(cv[e]) : fma2(bc(cv[e]), Y[k], r);
      }
    }
  } else {
    r0 = bc(shb[0]);
    r1 = bc(shb[1]);
    r2 = bc(shb[2]);
#pragma unroll
    for (int k = 1; k < NSH; ++k) {
      r0 = fma2(bc(shb[3 * k]), Y[k], r0);
      r1 = fma2(bc(shb[3 * k + 1]), Y[k], r1);
      r2 = fma2(bc(shb[3 * k + 2]), Y[k], r2);
    }
  }
}

// ---------------------------------------------------------------- sums over a warp (the backwards)

// Reduce-scatter of 16 per-lane values over the 32 lanes: afterwards lanes 2i and 2i+1 hold
// the warp total of value i.
__device__ __forceinline__ void warp_reduce_scatter16(float (&v)[16], int lane) {
#pragma unroll
  for (int o = 16, L = 8; L >= 1; o >>= 1, L >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int j = 0; j < L; ++j) {
      float send = up ? v[j] : v[j + L];
      float keep = up ? v[j + L] : v[j];
      v[j] = keep + __shfl_xor_sync(kFull, send, o);
    }
  }
  v[0] += __shfl_xor_sync(kFull, v[0], 1);
}

// D += A B for one m16n8k16 BF16 tile (FP32 accumulate).
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// ---------------------------------------------------------------- pixels of a warp

// A block holds up to kBlockWarps of a tile's warps (tiles over 256 pixels take several blocks:
// warps share nothing but the L1), so one register budget fits every tile shape.
constexpr int kBlockWarps = 4;

__host__ __device__ inline int tile_warps(const DevOpts &op) { return (op.tile_w * op.tile_h + 63) / 64; }
__host__ __device__ inline int tile_blocks(const DevOpts &op) {
  return (tile_warps(op) + kBlockWarps - 1) / kBlockWarps;
}
inline int block_warps(const DevOpts &op) { return tile_warps(op) < kBlockWarps ? tile_warps(op) : kBlockWarps; }

__device__ __forceinline__ bool tile_is_8x8(const DevOpts &op) { return op.tile_w % 8 == 0 && op.tile_h % 8 == 0; }

// Pixel h (0, 1) of a lane within its tile; false past the tile's last pixel.  Squares of 8 x 8
// per warp when the tile is made of them, two 8 x 4 blocks when it is made of those, else
// row-major runs.  Results do not depend on the mapping: every pixel's walk is its own.
__device__ __forceinline__ bool tile_pixel2(const DevOpts &op, int warp, int lane, int h, int &lx, int &ly) {
  if (tile_is_8x8(op)) {
    const int bx = op.tile_w / 8;
    lx = (warp % bx) * 8 + (lane & 7);
    ly = (warp / bx) * 8 + 4 * h + (lane >> 3);
    return true;
  }
  if (op.tile_w % 8 == 0 && op.tile_h % 4 == 0) {
    const int bx = op.tile_w / 8, k = 2 * warp + h;
    lx = (k % bx) * 8 + (lane & 7);
    ly = (k / bx) * 4 + (lane >> 3);
    return k < bx * (op.tile_h / 4);
  }
  const int t = warp * 64 + h * 32 + lane;
  lx = t % op.tile_w;
  ly = t / op.tile_w;
  return t < op.tile_w * op.tile_h;
}

// A pixel as x | y << 16 (both below 2^15), or kDead: never inside a rectangle.
constexpr uint32_t kDead = 0x80008000u;

// The pair's pixels, rays and SH basis: px, py, whether each lies in its tile and image, whether it
// has a ray (pixel_setup's results, both pixels in step).
template <int DEG>
struct PixelPair {
  int px[2], py[2];
  bool in[2], valid[2];
  f3x2 o, d;
  float2 Y[(DEG + 1) * (DEG + 1)];
};

template <int DEG>
__device__ __forceinline__ void pixel_pair(const DevCam &cam, const DevOpts &op, int x0, int y0, int warp, int lane,
                                           PixelPair<DEG> &q) {
  constexpr int NSH = (DEG + 1) * (DEG + 1);
  PixelPlane p[2];
  float rd[2], x[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    int lx, ly;
    q.in[h] = tile_pixel2(op, warp, lane, h, lx, ly);
    q.px[h] = x0 + lx;
    q.py[h] = y0 + ly;
    q.in[h] = q.in[h] && q.px[h] < cam.W && q.py[h] < cam.H;
    p[h] = pixel_plane(cam, q.px[h], q.py[h]);
    rd[h] = p[h].rd;
    q.valid[h] = q.in[h] && imaged(cam, p[h]);
  }
  undistort<2>(cam, rd, q.valid, op.newton_iters, x);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float3 o = make_float3(0.f, 0.f, 1.f), d = o;
    float Y[NSH];
#pragma unroll
    for (int k = 0; k < NSH; ++k) Y[k] = 0.f;
    if (q.valid[h]) {
      ray_of(cam, q.py[h], p[h], x[h], o, d);
      const float in = rsqrtf(dot3(d, d));
      sh_basis<DEG>(d.x * in, d.y * in, d.z * in, Y);
    }
    (h ? q.o.x.y : q.o.x.x) = o.x; (h ? q.o.y.y : q.o.y.x) = o.y; (h ? q.o.z.y : q.o.z.x) = o.z;
    (h ? q.d.x.y : q.d.x.x) = d.x; (h ? q.d.y.y : q.d.y.x) = d.y; (h ? q.d.z.y : q.d.z.x) = d.z;
#pragma unroll
    for (int k = 0; k < NSH; ++k) (h ? q.Y[k].y : q.Y[k].x) = Y[k];
  }
}

__device__ __forceinline__ bool in_rect(uint32_t p, uint32_t r0, uint32_t r1) {
  return __vmins2(__vmaxs2(p, r0), r1) == p;  // per 16-bit half: clamping to [r0, r1] keeps p
}

// ---------------------------------------------------------------- culling
//
// Bounds of a warp's live pixels: bounding box, and rays (o, d) with
// d = dc + s e1 + t e2 + delta, |s|, |t| <= 1, |delta| <= r; |d| <= dn; |o - oc| <= ro; |o| <= on.
struct __align__(16) WarpRays {
  int x0, x1, y0, y1;
  float3 dc;
  float r;
  float3 e1;
  float dn;
  float3 e2;
  float ro;
  float3 oc;
  float on;
};

__device__ __forceinline__ float warp_max_nonneg(float x) {  // non-negative floats: bit order = value order
  return __uint_as_float(__reduce_max_sync(kFull, __float_as_uint(x)));
}

__device__ __forceinline__ float3 shfl3(float3 v, int l) {
  return make_float3(__shfl_sync(kFull, v.x, l), __shfl_sync(kFull, v.y, l), __shfl_sync(kFull, v.z, l));
}

__device__ __forceinline__ float3 pick(const f3x2 &v, int h) {
  return h ? make_float3(v.x.y, v.y.y, v.z.y) : make_float3(v.x.x, v.y.x, v.z.x);
}

// The WarpRays of the warp's live pixels (every lane calls it; lane 0 writes *out and the caller
// synchronises the warp).  rows: the warp's pixels are an 8 x rows block (8: two pixels a lane,
// tile_is_8x8; 4: pixel 0 of each lane, tile_pixel's blocks), or 0 for any other layout.
__device__ __forceinline__ void warp_rays(const uint32_t (&pk)[2], const f3x2 &o, const f3x2 &d, int rows, int lane,
                                          WarpRays *out) {
  WarpRays w;
  const bool l0 = pk[0] != kDead, l1 = pk[1] != kDead;
  const int a0 = (int)(pk[0] & 0xffffu), b0 = (int)(pk[0] >> 16), a1 = (int)(pk[1] & 0xffffu), b1 = (int)(pk[1] >> 16);
  constexpr int big = 0x7fffffff;
  w.x0 = __reduce_min_sync(kFull, min(l0 ? a0 : big, l1 ? a1 : big));
  w.x1 = __reduce_max_sync(kFull, max(l0 ? a0 : -1, l1 ? a1 : -1));
  w.y0 = __reduce_min_sync(kFull, min(l0 ? b0 : big, l1 ? b1 : big));
  w.y1 = __reduce_max_sync(kFull, max(l0 ? b0 : -1, l1 ? b1 : -1));
  const unsigned v0 = __ballot_sync(kFull, l0), v1 = __ballot_sync(kFull, l1);
  const bool plane = v0 == kFull && (rows == 4 || (rows == 8 && v1 == kFull));
  const int ref = v0 ? __ffs(v0) - 1 : (v1 ? __ffs(v1) - 1 : 0);
  w.oc = shfl3(pick(o, v0 ? 0 : 1), ref);
  if (plane) {  // the plane through the block's corner rays
    const float3 a = shfl3(pick(d, 0), 0), b = shfl3(pick(d, 0), 7), c = shfl3(pick(d, rows == 8), 24),
                 e = shfl3(pick(d, rows == 8), 31);
    w.dc = make_float3(0.25f * (a.x + b.x + c.x + e.x), 0.25f * (a.y + b.y + c.y + e.y),
                       0.25f * (a.z + b.z + c.z + e.z));
    w.e1 = make_float3(0.25f * (b.x + e.x - a.x - c.x), 0.25f * (b.y + e.y - a.y - c.y),
                       0.25f * (b.z + e.z - a.z - c.z));
    w.e2 = make_float3(0.25f * (c.x + e.x - a.x - b.x), 0.25f * (c.y + e.y - a.y - b.y),
                       0.25f * (c.z + e.z - a.z - b.z));
  } else {  // a ball around one live ray
    w.dc = shfl3(pick(d, v0 ? 0 : 1), ref);
    w.e1 = w.e2 = make_float3(0.f, 0.f, 0.f);
  }
  float r = 0.f, ro = 0.f, dn = 0.f, on = 0.f;
  const float s = ((float)(lane & 7) - 3.5f) * (1.f / 3.5f), hr = 0.5f * (float)(rows - 1);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    if (!(h ? l1 : l0)) continue;
    const float t = plane ? ((float)((lane >> 3) + 4 * h) - hr) / hr : 0.f;
    const float3 dh = pick(d, h), oh = pick(o, h);
    const float3 dd = make_float3(dh.x - fmaf(s, w.e1.x, fmaf(t, w.e2.x, w.dc.x)),
                                  dh.y - fmaf(s, w.e1.y, fmaf(t, w.e2.y, w.dc.y)),
                                  dh.z - fmaf(s, w.e1.z, fmaf(t, w.e2.z, w.dc.z)));
    const float3 od = make_float3(oh.x - w.oc.x, oh.y - w.oc.y, oh.z - w.oc.z);
    r = fmaxf(r, sqrtf(dot3(dd, dd)));
    ro = fmaxf(ro, sqrtf(dot3(od, od)));
    dn = fmaxf(dn, sqrtf(dot3(dh, dh)));
    on = fmaxf(on, sqrtf(dot3(oh, oh)));
  }
  w.dn = warp_max_nonneg(dn) * 1.0001f;
  w.on = warp_max_nonneg(on) * 1.0001f;
  w.r = warp_max_nonneg(r) * 1.0001f + 1e-6f * w.dn;
  w.ro = warp_max_nonneg(ro) * 1.0001f;
  if (lane == 0) *out = w;
}

__device__ __forceinline__ bool rect_near(const WarpRays &w, short4 r) {
  return w.x1 >= r.x && w.x0 <= r.z && w.y1 >= r.y && w.y0 <= r.w;
}

// The approximate square root: error below 1e-6, inside the factors 1.0001 of the bounds that use it.
__device__ __forceinline__ float sqrt_bound(float x) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// True if no live pixel of the warp can pass eval_response's test |c|^2 <= thr |d_g|^2,
// c = o_g x d_g, for the record g.  Over the warp's rays, with n = c0 / |c0| the direction of the
// centre ray's c0 = og0 x M dc and ci = og0 x M ei,
//   |c| >= n . c >= |c0| - |n . c1| - |n . c2| - |og0| |M| r - |M| ro |M| dn,
//   |d_g| <= |M dc| + |M e1| + |M e2| + |M| r       (|M|: Frobenius norm).
// The rounding of o_g, d_g and c in eval_pair is below 16 ulp of |M| dn (|o_g| + |M| on) (the
// staged M (o - mu) or M mu is shared by every pixel, so its own rounding cancels); twice that is
// the second term of the slack.  Infinite or NaN intermediates compare false and keep the
// particle, so only particles that eval_pair rejects for all 64 pixels are dropped: images do not
// depend on this test.  It drops nearly everything that can be dropped (88 to 98 % of the survivors
// of an 8 x 8 square reach a pixel that is still walking), at about 3 instructions per (warp, entry).
template <bool RS>
__device__ __forceinline__ bool block_misses(const float4 (&g)[4], const WarpRays &w) {
  const float4 g0 = g[0], g1 = g[1], g2 = g[2];
  auto mul = [&](float3 v) {
    return make_float3(fmaf(g0.x, v.x, fmaf(g0.y, v.y, g0.z * v.z)), fmaf(g0.w, v.x, fmaf(g1.x, v.y, g1.y * v.z)),
                       fmaf(g1.z, v.x, fmaf(g1.w, v.y, g2.x * v.z)));
  };
  const float m9[9] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w, g2.x};
  float nm = 0.f;
#pragma unroll
  for (int k = 0; k < 9; ++k) nm = fmaf(m9[k], m9[k], nm);
  nm = sqrt_bound(nm) * 1.0001f;
  float3 og = make_float3(g2.y, g2.z, g2.w);
  if (RS) {
    const float3 m = mul(w.oc);
    og = make_float3(m.x - og.x, m.y - og.y, m.z - og.z);
  }
  const float3 d0 = mul(w.dc), d1 = mul(w.e1), d2 = mul(w.e2);
  const float3 c0 = cross3(og, d0), c1 = cross3(og, d1), c2 = cross3(og, d2);
  const float cc = dot3(c0, c0);
  const float lhs = cc - fabsf(dot3(c0, c1)) - fabsf(dot3(c0, c2));
  const float on = sqrt_bound(dot3(og, og));
  const float dmax = sqrt_bound(dot3(d0, d0)) + sqrt_bound(dot3(d1, d1)) + sqrt_bound(dot3(d2, d2)) + nm * w.r;
  const float md = nm * w.dn;
  float slack = on * nm * w.r + 2e-6f * md * (on + nm * (RS ? w.on + w.ro : 0.f));
  if (RS) slack = fmaf(nm * w.ro, md, slack);
  return cc > 1e-30f && lhs > sqrt_bound(cc) * (slack + sqrt_bound(g[3].y) * dmax * 1.0001f);
}

// The entries of [c0, c0 + 32) of a batch of nb records staged by a block that can reach this warp's
// pixels, as a mask (every lane calls it).
template <bool RS>
__device__ __forceinline__ unsigned near_mask(const float4 (*geo)[4], int c0, int nb, const WarpRays &w, int lane) {
  bool near_ = false;
  if (c0 + lane < nb) {
    float4 g[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) g[q] = geo[c0 + lane][q];
    const int r0 = __float_as_int(g[3].z), r1 = __float_as_int(g[3].w);
    const short4 r = make_short4((short)(r0 & 0xffff), (short)(r0 >> 16), (short)(r1 & 0xffff), (short)(r1 >> 16));
    near_ = rect_near(w, r) && !block_misses<RS>(g, w);
  }
  return __ballot_sync(kFull, near_);
}

// The warp's WarpRays when every lane holds one pixel of a tile (tile_pixel).
__device__ __forceinline__ void warp_rays1(const DevOpts &op, int px, int py, float3 o, float3 d, bool live, int lane,
                                           WarpRays *out) {
  const uint32_t pk[2] = {live ? (uint32_t)px | ((uint32_t)py << 16) : kDead, kDead};
  const f3x2 o2 = {bc(o.x), bc(o.y), bc(o.z)}, d2 = {bc(d.x), bc(d.y), bc(d.z)};
  warp_rays(pk, o2, d2, op.tile_w % 8 == 0 && op.tile_h % 4 == 0 ? 4 : 0, lane, out);
}

// ---------------------------------------------------------------- list entries and SH staging

// Entry k of a tile's list for this lane, or 0 and an empty rectangle past the end.
__device__ __forceinline__ uint32_t list_index(const uint32_t *__restrict__ vals, uint32_t k, uint32_t end) {
  return k < end ? vals[k] : 0u;
}
__device__ __forceinline__ short4 list_rect(const short4 *__restrict__ rect, int part_off, uint32_t idx, uint32_t k,
                                            uint32_t end) {
  return k < end ? rect[part_off + idx] : make_short4(0, 0, -1, -1);
}

// SH coefficients of the n particles idx[] into the warp's dst, by asynchronous copies (16 bytes
// when the rows are 16-byte aligned, else 4), with beta_0 replaced by the colour's constant term
// (sh_colour2); complete, and visible to the warp, on return.  n is at most 32.
template <int NC>
__device__ __forceinline__ void stage_sh_warp(const DevScene &sc, const uint32_t *idx, int n, float *dst, int lane) {
  const uint32_t d0 = (uint32_t)__cvta_generic_to_shared(dst);
  if (NC % 4 == 0 && sc.sh_vec) {
    constexpr int N4 = NC % 4 == 0 ? NC / 4 : 1;
    for (int f = lane; f < n * N4; f += 32) {
      const int b = f / N4;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d0 + 16 * f),
                   "l"(sc.sh + (size_t)idx[b] * NC + 4 * (f - b * N4))
                   : "memory");
    }
  } else {
    for (int f = lane; f < n * NC; f += 32) {
      const int b = f / NC;
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d0 + 4 * f),
                   "l"(sc.sh + (size_t)idx[b] * NC + (f - b * NC))
                   : "memory");
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncwarp();
  float Y0[1];
  sh_basis<0>(0.f, 0.f, 1.f, Y0);
  if (lane < n) {
#pragma unroll
    for (int c = 0; c < 3; ++c) dst[lane * NC + c] = fmaf(dst[lane * NC + c], Y0[0], 0.5f);
  }
  __syncwarp();
}

}  // namespace
}  // namespace ut3d
