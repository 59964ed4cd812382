// composite_bwd.cu — hand-written backward of the compositing (supplementary Sec. B) for a
// batch of views.
//
// The backward replays the forward IN FORWARD ORDER: the stored rgb and T_final give the
// suffix sums S_i = C - sum_{j<=i} c_j alpha_j T_j without dividing transmittances,
// and n_used tells each pixel where the forward stopped.  Per (particle, warp) the 13
// geometry partials are reduced with a transposing reduce-scatter and the 3 x (deg+1)^2 SH
// partials with a tensor-core contraction over the warp's pixels; both go to the particle's
// accumulators in global memory as coalesced reductions.  A final per-particle kernel maps the
// accumulated dL/dM, dL/dmu, dL/dsigma onto log-scales, quaternions and logits.  Tiles run
// heaviest replay first.
#include <cuda_bf16.h>

#include "composite_warp.cuh"

namespace ut3d {
namespace {

// Two floats as bf16 pairs hi + lo (x = hi + lo to about 2^-17): the three-term products
// hi*hi + hi*lo + lo*hi keep FP32-level accuracy on the BF16 tensor-core path.
__device__ __forceinline__ void split_bf16x2(float x, float y, uint32_t &hi, uint32_t &lo) {
  __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  float2 hf = __bfloat1622float2(h);
  __nv_bfloat162 l = __floats2bfloat162_rn(x - hf.x, y - hf.y);
  hi = *reinterpret_cast<uint32_t *>(&h);
  lo = *reinterpret_cast<uint32_t *>(&l);
}

constexpr int kSlots = 8;     // particle columns of one tensor-core flush (the MMA's N)
constexpr int kRoundB = 24;   // survivors staged at a time: 17 KB a warp, 12 warps an SM

// Shared memory of one warp of the backward.
template <int DEG, bool PP>
struct __align__(16) BwdWarp {
  static constexpr int NSH = (DEG + 1) * (DEG + 1);
  static constexpr int NC = NSH * 3;
  static constexpr int ROWS = PP ? 1 : (NSH > 8 ? 16 : 8);  // basis rows of the MMA's A that can be non-zero
  static constexpr int COLS = PP ? 1 : 3 * kSlots;
  // gradient rows on their way out: stride 60 for the 48 floats of degree 3 keeps the fragment
  // writes free of bank conflicts, any multiple of 4 the 16-byte reads aligned
  static constexpr int OST = NC == 48 ? 60 : (NC % 4 == 0 ? NC + 4 : NC);
  WarpRays rays;
  float4 geo[kRoundB][5];                   // stage_particle's record; o - mu or mu, list position
  alignas(16) float col[kRoundB * (PP ? 4 : NC)];  // SH coefficients, or the colour (PP)
  uint32_t idx[kRoundB];
  uint32_t cidx[kSlots > kRoundB ? kSlots : kRoundB];  // particle of each column / outgoing row
  float dc[PP ? kRoundB : 1][3];            // PP: dL/dcolour of every survivor
  alignas(16) uint2 A[ROWS][32];                        // basis of the pixel pairs, (hi, lo) bf16 pairs
  union alignas(16) {
    uint2 W[COLS][32];                      // SH weights of the pixel pairs, row = channel x column
    float out[(PP ? kRoundB : kSlots) * OST];
  };
};

// Slot of pixel pair l in row `row` of A or W: the fragment loads read four consecutive pairs of
// eight rows, which the XOR spreads over all banks.
__device__ __forceinline__ int pair_slot(int row, int l) { return l ^ ((row & 7) << 2); }

// Adds n gradient rows of NC floats (row b at out + b * stride, particle idx[b]) to d_sh: 16-byte
// vector reductions when the rows are aligned, consecutive scalars otherwise (both coalesced; the
// L2 takes 1.3 T float reductions a second that way against 0.13 T scattered ones).
template <int NC>
__device__ __forceinline__ void add_rows(const DevScene &sc, const float *out, int stride, const uint32_t *idx, int n,
                                         int lane) {
  if (NC % 4 == 0 && sc.dsh_vec) {
    constexpr int N4 = NC % 4 == 0 ? NC / 4 : 1;
    for (int f = lane; f < n * N4; f += 32) {
      const int b = f / N4, j = 4 * (f - b * N4);
      const float4 v = *reinterpret_cast<const float4 *>(out + b * stride + j);
      asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(sc.d_sh + (size_t)idx[b] * NC + j), "f"(v.x),
                   "f"(v.y), "f"(v.z), "f"(v.w)
                   : "memory");
    }
  } else {
    for (int f = lane; f < n * NC; f += 32) {
      const int b = f / NC, j = f - b * NC;
      atomicAdd(sc.d_sh + (size_t)idx[b] * NC + j, out[b * stride + j]);
    }
  }
}

// Backward of k_composite_fwd for one tile, walked like the forward (composite_warp.cuh): two
// pixels a thread, survivors of the warp's own culling, no block barrier.  Per (pixel, particle)
// pair the partials are dL/dbeta_k,c = w_c Y_k (w_c = dL/dc_c alpha T where the colour is not
// clamped), the 9 products v x^T for dL/dM, v for dL/dmu and dL/dsigma.
//
// The SH part is a dense contraction over the warp's 64 pixels, D[k][j] = sum_p Y_k(p) W_c(p, j),
// run on the tensor cores (m16n8k16, BF16 hi/lo split with the three cross terms, FP32
// accumulate): A = Y^T (basis x pixels) is fixed for the tile; B = W (pixels x particles)
// collects, column by column, only particles that reach at least one pixel of the warp, and is
// contracted once kSlots columns are full.  A lane's two pixels are neighbours in the
// contraction's order, so each lane splits and stores its own pair.  The 13 geometry partials are
// summed over the pair, then with a 16-value reduce-scatter.  Both go straight to the particle's
// accumulators in global memory with coalesced reductions, which the L2 absorbs (about 20 G rows
// of 64 floats a second): no accumulators shared by the tile's warps, no flush, no barrier.
// Bound by instruction issue (59 % of the cycles at 12 warps an SM).  Compiled for 3 blocks of 128
// threads per SM (167 registers): at 4 blocks the pair's state spills (1M rolling-shutter 1080p
// training step 2558 us against 2520, backward of 200k particles at 640x480 890 against 780), at 5
// far more.  Against one pixel a thread with accumulators shared by the tile's warps: that step
// 3058 -> 2449 us, that backward 1143 -> 718 us, the 8-view step of 3M particles 58.9 -> 46.3 ms
// (with the forward's change); with one branch a survivor and each reciprocal taken once:
// 2415 -> 2269, 791 -> 669 us and 46.8 -> 42.4 ms.  The scaled reciprocal costs 0.8 % (that backward).
// PP (per-particle colour mode): the colour gradient dL/dc is one 3-vector per particle, summed
// in the three spare slots of the reduce-scatter; after each round it becomes
// dL/dbeta = dL/dc Y(dir) and the mean's gradient through the view direction.
template <int DEG, bool RS, bool PP, bool GEN>
__global__ void __launch_bounds__(32 * kBlockWarps, 3)
    k_composite_bwd(const __grid_constant__ BatchDesc bd, DevOpts op, const short4 *__restrict__ rect,
                    const uint32_t *__restrict__ vals, const uint2 *__restrict__ ranges, TileSched ts) {
  using L = BwdWarp<DEG, PP>;
  constexpr int NSH = L::NSH;
  constexpr int NC = L::NC;
  constexpr int PDEG = PP ? 0 : DEG;  // per-pixel SH basis only when colours are per pixel
  extern __shared__ __align__(16) unsigned char smem[];

  // tiles in the order k_tile_order gave them (most list entries to replay first)
  const uint32_t rank = blockIdx.x / (uint32_t)tile_blocks(op);
  if (rank >= *ts.n_work) return;
  const int tile = (int)ts.order[rank];
  UT_DBG_CHECK(tile < bd.total_tiles, UT_DBG_TILE_ID, tile, bd.total_tiles, 3);
  const DevView &view = bd.v[view_of_tile(bd, tile)];
  const DevScene &sc = bd.s[view.scene];
  const DevCam &cam = view.cam;
  const int lane = threadIdx.x & 31;
  const int warp = (int)(blockIdx.x % (uint32_t)tile_blocks(op)) * kBlockWarps + (int)(threadIdx.x >> 5);  // of the tile
  if (warp >= tile_warps(op)) return;  // warps never wait for each other
  const int g8 = lane >> 2, t4 = lane & 3;
  L &S = reinterpret_cast<L *>(smem)[threadIdx.x >> 5];
  const int lt = tile - view.tile_off;
  const int x0 = (lt % view.tiles_x) * op.tile_w, y0 = (lt / view.tiles_x) * op.tile_h;
  const uint2 rg = ranges[tile];

  PixelPair<PDEG> q;
  pixel_pair<PDEG>(cam, op, x0, y0, warp, lane, q);
  const f3x2 o = q.o, d = q.d;
  uint32_t pk[2], end[2];  // the pixels with something to replay (kDead: none), and where each stops
  float2 gr[3], Cf[3], gAT;  // upstream dL/drgb, composited colour, dL/dalpha T_final
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float u[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    end[h] = 0;
    if (q.valid[h]) {
      const size_t pix = (size_t)q.py[h] * cam.W + q.px[h], plane = (size_t)cam.W * cam.H;
      end[h] = view.n_used[pix];
      u[0] = view.d_rgb[pix]; u[1] = view.d_rgb[plane + pix]; u[2] = view.d_rgb[2 * plane + pix];
      u[3] = view.rgb[pix]; u[4] = view.rgb[plane + pix]; u[5] = view.rgb[2 * plane + pix];
      u[6] = view.d_alpha[pix] * view.tfinal[pix];
    }
    pk[h] = end[h] > rg.x ? (uint32_t)q.px[h] | ((uint32_t)q.py[h] << 16) : kDead;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      (h ? gr[c].y : gr[c].x) = u[c];
      (h ? Cf[c].y : Cf[c].x) = u[3 + c];
    }
    (h ? gAT.y : gAT.x) = u[6];
  }
  // no pixel of this warp blends a particle at or after `stop`
  const uint32_t stop = min(__reduce_max_sync(kFull, max(end[0], end[1])), rg.y);
  if (stop <= rg.x) return;  // warp-uniform
  warp_rays(pk, o, d, tile_is_8x8(op) ? 8 : 0, lane, &S.rays);
  if constexpr (!PP) {
#pragma unroll
    for (int k = 0; k < L::ROWS; ++k) {
      uint2 hl = make_uint2(0u, 0u);
      if (k < NSH) split_bf16x2(q.Y[k < NSH ? k : 0].x, q.Y[k < NSH ? k : 0].y, hl.x, hl.y);
      S.A[k][pair_slot(k, lane)] = hl;
    }
  }
  __syncwarp();

  // Contracts the first `cols` columns of W with Y and adds the rows to the particles' SH
  // gradients.  Columns past `cols` hold older values; they only feed their own, unread outputs.
  auto flush = [&](int cols) {
    __syncwarp();
    float acc[3][4];
#pragma unroll
    for (int c = 0; c < 3; ++c) acc[c][0] = acc[c][1] = acc[c][2] = acc[c][3] = 0.f;
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
      const int l0 = pair_slot(g8, 8 * ks + t4), l1 = pair_slot(g8, 8 * ks + 4 + t4);
      const uint2 z = make_uint2(0u, 0u);
      const uint2 a0 = S.A[g8][l0], a2 = S.A[g8][l1];
      const uint2 a1 = L::ROWS > 8 ? S.A[L::ROWS > 8 ? g8 + 8 : 0][l0] : z;
      const uint2 a3 = L::ROWS > 8 ? S.A[L::ROWS > 8 ? g8 + 8 : 0][l1] : z;
      const uint32_t ahi[4] = {a0.x, a1.x, a2.x, a3.x}, alo[4] = {a0.y, a1.y, a2.y, a3.y};
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const uint2 b0 = S.W[c * kSlots + g8][l0], b1 = S.W[c * kSlots + g8][l1];
        mma_bf16(acc[c], ahi, b0.x, b1.x);
        mma_bf16(acc[c], ahi, b0.y, b1.y);
        mma_bf16(acc[c], alo, b0.x, b1.x);
      }
    }
    __syncwarp();
    // acc[c][r]: basis g8 (+8 for r >= 2), column 2 t4 (+1 for odd r)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int k = g8 + (r >= 2 ? 8 : 0), col = 2 * t4 + (r & 1);
      if (k < NSH) {
#pragma unroll
        for (int c = 0; c < 3; ++c) S.out[col * L::OST + 3 * k + c] = acc[c][r];
      }
    }
    __syncwarp();
    add_rows<NC>(sc, S.out, L::OST, S.cidx, cols, lane);
    __syncwarp();
  };

  float2 T = bc(1.f), A[3] = {bc(0.f), bc(0.f), bc(0.f)};  // transmittance, running prefix of the colour
  int cols = 0;
  uint32_t idx = list_index(vals, rg.x + lane, stop), idx1 = list_index(vals, rg.x + 32 + lane, stop);
  short4 r = list_rect(rect, view.part_off, idx, rg.x + lane, stop);
  for (uint32_t p0 = rg.x; p0 < stop;) {
    const short4 r1 = list_rect(rect, view.part_off, idx1, p0 + 32 + lane, stop);
    const uint32_t idx2 = list_index(vals, p0 + 64 + lane, stop);
    bool near_ = rect_near(S.rays, r);
    float4 g[4], aux;
    if (near_) {
      stage_particle<RS>(sc, cam, op, r, idx, g, &aux);
      near_ = !block_misses<RS>(g, S.rays);
    }
    const unsigned m = __ballot_sync(kFull, near_);
    const int b0 = __popc(m & ((1u << lane) - 1u)), n = min(__popc(m), kRoundB);
    // survivors past the round's room are left to the next one
    const unsigned over = __ballot_sync(kFull, near_ && b0 >= kRoundB);
    if (near_ && b0 < kRoundB) {
#pragma unroll
      for (int q = 0; q < 4; ++q) S.geo[b0][q] = g[q];
      aux.w = __uint_as_float(p0 + lane);
      S.geo[b0][4] = aux;
      S.idx[b0] = idx;
      if (PP) {
        reinterpret_cast<float4 *>(S.col)[b0] = particle_colour<DEG, RS>(sc, cam, op, idx);
        S.dc[PP ? b0 : 0][0] = S.dc[PP ? b0 : 0][1] = S.dc[PP ? b0 : 0][2] = 0.f;
      }
    }
    __syncwarp();
    if (!PP) stage_sh_warp<NC>(sc, S.idx, n, S.col, lane);
    for (int b = 0; b < n; ++b) {  // warp-uniform
      const float4 g3 = S.geo[b][3], ax = S.geo[b][4];
      const uint32_t q0 = __float_as_uint(g3.z), q1 = __float_as_uint(g3.w), pos = __float_as_uint(ax.w);
      bool h0 = in_rect(pk[0], q0, q1) && pos < end[0], h1 = in_rect(pk[1], q0, q1) && pos < end[1];
      const PairEval e = eval_pair<RS>(S.geo[b][0], S.geo[b][1], S.geo[b][2], o, d);
      h0 = h0 && e.cc.x <= g3.y * e.dd.x;
      h1 = h1 && e.cc.y <= g3.y * e.dd.y;
      if (!__any_sync(kFull, h0 || h1)) continue;
      // straight-line from here: a pixel that the particle does not reach has alpha 0 and takes part
      // in no sum (its alpha, colour, dL/dalpha and tau are selected to 0, so that no infinity of its
      // own gets in)
      // 1 / |d_g|^2 is taken of 2^64 |d_g|^2, and multiplied by numerators scaled alike, where |d_g|^2
      // is small: a scale above 1e19 makes it subnormal, and its reciprocal an infinity
      const float2 up = make_float2(e.dd.x < 0x1p-63f ? 0x1p64f : 1.f, e.dd.y < 0x1p-63f ? 0x1p64f : 1.f);
      const float2 du = mul2(e.dd, up), rd = make_float2(rcp_normal(du.x), rcp_normal(du.y));
      const float2 w2 = mul2(mul2(e.cc, up), rd);
      const float2 rho = sel2(h0, h1, response2<GEN>(w2, op), bc(0.f));
      const float2 a = mul2(bc(g3.x), rho);
      const float2 al = make_float2(fminf(a.x, op.alpha_max), fminf(a.y, op.alpha_max));
      float2 c0, c1, c2;
      if (PP) {
        const float4 cr = reinterpret_cast<const float4 *>(S.col)[b];
        c0 = bc(cr.x); c1 = bc(cr.y); c2 = bc(cr.z);
      } else {
        sh_colour2<NSH>(S.col + b * NC, q.Y, c0, c1, c2);
      }
      c0 = make_float2(h0 ? fmaxf(c0.x, 0.f) : 0.f, h1 ? fmaxf(c0.y, 0.f) : 0.f);
      c1 = make_float2(h0 ? fmaxf(c1.x, 0.f) : 0.f, h1 ? fmaxf(c1.y, 0.f) : 0.f);
      c2 = make_float2(h0 ? fmaxf(c2.x, 0.f) : 0.f, h1 ? fmaxf(c2.y, 0.f) : 0.f);
      const float2 w = mul2(al, T);
      // the prefix repeats the forward's sums bit for bit, so that the colour still to come,
      // S = C - prefix, keeps its relative accuracy down to the last particles of a ray
      A[0] = fma2(c0, w, A[0]);
      A[1] = fma2(c1, w, A[1]);
      A[2] = fma2(c2, w, A[2]);
      const float2 om = make_float2(1.f - al.x, 1.f - al.y);  // >= 1 - alpha_max > 0
      const float2 inv = make_float2(rcp_normal(om.x), rcp_normal(om.y));
      // dL/dalpha = sum_c g_c c T + (g_A T_final - sum_c g_c S_c) / (1 - alpha)
      const float2 gc = fma2(gr[0], c0, fma2(gr[1], c1, mul2(gr[2], c2)));
      const float2 gs = fma2(gr[0], sub2(A[0], Cf[0]), fma2(gr[1], sub2(A[1], Cf[1]),
                                                              fma2(gr[2], sub2(A[2], Cf[2]), gAT)));
      const float2 dal = fma2(gc, T, mul2(gs, inv));
      const float2 wc[3] = {make_float2(c0.x > 0.f ? gr[0].x * w.x : 0.f, c0.y > 0.f ? gr[0].y * w.y : 0.f),
                            make_float2(c1.x > 0.f ? gr[1].x * w.x : 0.f, c1.y > 0.f ? gr[1].y * w.y : 0.f),
                            make_float2(c2.x > 0.f ? gr[2].x * w.x : 0.f, c2.y > 0.f ? gr[2].y * w.y : 0.f)};
      T = mul2(T, om);
      const float2 da = make_float2(!h0 || a.x > op.alpha_max ? 0.f : dal.x,
                                    !h1 || a.y > op.alpha_max ? 0.f : dal.y);
      float v[16];
      v[12] = fmaf(da.x, rho.x, da.y * rho.y);
      // 2 dL/domega^2
      float2 dw = make_float2(-a.x * da.x, -a.y * da.y);
      if (GEN) dw = mul2(mul2(bc(2.f), dresponse2(op, a, sel2(h0, h1, w2, bc(0.f)))), da);
      const float2 od = mul2(dot3x2(e.og, e.dg), up);
      const float2 tau = make_float2(h0 ? -(od.x * rd.x) : 0.f, h1 ? -(od.y * rd.y) : 0.f);
      const float2 vv[3] = {mul2(dw, fma2(tau, e.dg.x, e.og.x)), mul2(dw, fma2(tau, e.dg.y, e.og.y)),
                            mul2(dw, fma2(tau, e.dg.z, e.og.z))};
      f3x2 x;
      if (RS) {
        x.x = add2(o.x, bc(-ax.x));
        x.y = add2(o.y, bc(-ax.y));
        x.z = add2(o.z, bc(-ax.z));
      } else {
        x.x = bc(ax.x);
        x.y = bc(ax.y);
        x.z = bc(ax.z);
      }
      const float2 xx[3] = {fma2(tau, d.x, x.x), fma2(tau, d.y, x.y), fma2(tau, d.z, x.z)};
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        v[q] = vv[q].x + vv[q].y;
#pragma unroll
        for (int c = 0; c < 3; ++c) v[3 + 3 * q + c] = fmaf(vv[q].x, xx[c].x, vv[q].y * xx[c].y);
      }
      const uint32_t pi = S.idx[b];
      if (PP) {
#pragma unroll
        for (int c = 0; c < 3; ++c) v[13 + c] = wc[c].x + wc[c].y;
      } else {
        v[13] = v[14] = v[15] = 0.f;
        // SH weights into the next free column of W
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          uint2 hl;
          split_bf16x2(wc[c].x, wc[c].y, hl.x, hl.y);
          S.W[PP ? 0 : c * kSlots + cols][pair_slot(cols, lane)] = hl;
        }
        if (lane == 0) S.cidx[cols] = pi;
      }
      warp_reduce_scatter16(v, lane);
      const int vi = (lane >> 1) & 15;
      if (!(lane & 1)) {
        if (vi < 13) atomicAdd(&sc.gacc[(size_t)pi * 16 + vi], v[0]);
        else if (PP) S.dc[PP ? b : 0][vi - 13] = v[0];
      }
      if (!PP && ++cols == kSlots) {
        flush(kSlots);
        cols = 0;
      }
    }
    if constexpr (PP) {
      // dL/dc of this warp's pixels -> dL/dbeta_k,ch = dL/dc_ch Y_k(dir) and the mean's gradient
      // through dir = (mu - c) / |mu - c|: (I - dir dir^T) / |mu - c| sum_ch dL/dc_ch grad c_ch
      __syncwarp();
      const bool row = lane < n;
      const float g0c = row ? S.dc[row ? lane : 0][0] : 0.f, g1c = row ? S.dc[row ? lane : 0][1] : 0.f,
                  g2c = row ? S.dc[row ? lane : 0][2] : 0.f;
      const bool some = !(g0c == 0.f && g1c == 0.f && g2c == 0.f);
      const unsigned rows = __ballot_sync(kFull, some);
      if (some) {
        const uint32_t pi = S.idx[lane];
        const int b = __popc(rows & ((1u << lane) - 1u));
        const float3 mu = make_float3(sc.means[3 * pi], sc.means[3 * pi + 1], sc.means[3 * pi + 2]);
        float il;
        const float3 dir = particle_dir<RS>(cam, op, mu, il);
        float Yp[NSH], a[NSH];
        sh_basis<DEG>(dir.x, dir.y, dir.z, Yp);
        const float *beta = sc.sh + (size_t)pi * NC;
        float *dsh = S.out + b * L::OST;
        S.cidx[b] = pi;
#pragma unroll
        for (int k = 0; k < NSH; ++k) {
          a[k] = fmaf(g0c, beta[3 * k], fmaf(g1c, beta[3 * k + 1], g2c * beta[3 * k + 2]));
          dsh[3 * k] = g0c * Yp[k];
          dsh[3 * k + 1] = g1c * Yp[k];
          dsh[3 * k + 2] = g2c * Yp[k];
        }
        const float3 G = sh_poly_grad<DEG>(dir.x, dir.y, dir.z, a);
        const float gd = dot3(G, dir);
        atomicAdd(&sc.gacc[(size_t)pi * 16 + 13], (G.x - gd * dir.x) * il);
        atomicAdd(&sc.gacc[(size_t)pi * 16 + 14], (G.y - gd * dir.y) * il);
        atomicAdd(&sc.gacc[(size_t)pi * 16 + 15], (G.z - gd * dir.z) * il);
      }
      __syncwarp();
      add_rows<NC>(sc, S.out, L::OST, S.cidx, __popc(rows), lane);
    }
    __syncwarp();  // the survivors are read before the next round's are staged
    if (over) {
      p0 += __ffs(over) - 1;
      idx = list_index(vals, p0 + lane, stop);
      idx1 = list_index(vals, p0 + 32 + lane, stop);
      r = list_rect(rect, view.part_off, idx, p0 + lane, stop);
    } else {
      p0 += 32;
      idx = idx1;
      idx1 = idx2;
      r = r1;
    }
  }
  if (!PP && cols > 0) flush(cols);
}

// One warp per tile: work = list entries the backward replays (up to one past the last
// particle any of the tile's pixels blended, from n_used), and a histogram of the buckets.
__global__ void k_tile_work(const __grid_constant__ BatchDesc bd, DevOpts op, const uint2 *__restrict__ ranges,
                            TileSched ts) {
  const int tile = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (tile >= bd.total_tiles) return;
  const DevView &view = bd.v[view_of_tile(bd, tile)];
  const int lt = tile - view.tile_off;
  const int x0 = (lt % view.tiles_x) * op.tile_w, y0 = (lt / view.tiles_x) * op.tile_h;
  const int W = view.cam.W, H = view.cam.H;
  uint32_t m = 0;
  for (int i = lane; i < op.tile_w * op.tile_h; i += 32) {
    const int px = x0 + i % op.tile_w, py = y0 + i / op.tile_w;
    if (px < W && py < H) m = max(m, view.n_used[(size_t)py * W + px]);
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) {
    const uint2 rg = ranges[tile];
    const uint32_t w = m > rg.x ? min(m, rg.y) - rg.x : 0u;
    ts.work[tile] = w;
    if (w) atomicAdd(&ts.hist[work_bucket(w)], 1u);
  }
}

// d(rotation matrix)/d(unit quaternion) contracted with G = dL/dR (row-major).
__device__ __forceinline__ void rot_grad(const float *q, const float *G, float *gq) {
  float w = q[0], x = q[1], y = q[2], z = q[3];
  gq[0] = 2.f * (x * (G[7] - G[5]) + y * (G[2] - G[6]) + z * (G[3] - G[1]));
  gq[1] = 2.f * (-2.f * x * (G[4] + G[8]) + y * (G[1] + G[3]) + z * (G[2] + G[6]) + w * (G[7] - G[5]));
  gq[2] = 2.f * (x * (G[1] + G[3]) - 2.f * y * (G[0] + G[8]) + z * (G[5] + G[7]) + w * (G[2] - G[6]));
  gq[3] = 2.f * (x * (G[2] + G[6]) + y * (G[5] + G[7]) - 2.f * z * (G[0] + G[4]) + w * (G[3] - G[1]));
}

// Per particle of every scene in the batch: dL/dM, sum v, dL/dsigma -> parameter gradients.
__global__ void k_finalize(const __grid_constant__ BatchDesc bd, int total) {
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < total; g += gridDim.x * blockDim.x) {
    const DevScene &sc = bd.s[scene_of_grad(bd, g)];
    const int i = g - sc.grad_off;
    float3 mu = make_float3(sc.means[3 * i], sc.means[3 * i + 1], sc.means[3 * i + 2]);
    float3 ls = make_float3(sc.log_scales[3 * i], sc.log_scales[3 * i + 1], sc.log_scales[3 * i + 2]);
    Particle p;
    bool ok = activate(mu, ls, sc.quats[i], sc.logits[i], p);
    // the particle's 16 accumulators as four 16-byte loads (rows are 64-byte aligned)
    const float4 *A4 = reinterpret_cast<const float4 *>(sc.gacc + (size_t)i * 16);
    const float4 a0 = A4[0], a1 = A4[1], a2 = A4[2], a3 = A4[3];
    const float A[16] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w, a2.x, a2.y, a2.z, a2.w, a3.x, a3.y, a3.z, a3.w};
    float out_m[3] = {0.f, 0.f, 0.f}, out_s[3] = {0.f, 0.f, 0.f}, out_q[4] = {0.f, 0.f, 0.f, 0.f}, out_l = 0.f;
    if (ok) {
      float v0 = A[0], v1 = A[1], v2 = A[2];
      // slots 13..15: the mean's gradient through the per-particle view direction (zero in
      // the per-pixel colour mode)
      for (int j = 0; j < 3; ++j) out_m[j] = A[13 + j] - (p.M[j] * v0 + p.M[3 + j] * v1 + p.M[6 + j] * v2);
      float G[9];
      for (int k = 0; k < 3; ++k) {
        float acc = 0.f;
        const float is = 1.f / p.s[k];
        for (int j = 0; j < 3; ++j) {
          float dm = A[3 + 3 * k + j];
          acc = fmaf(dm, p.M[3 * k + j], acc);
          G[3 * j + k] = dm * is;
        }
        out_s[k] = -acc;
      }
      float gq[4];
      rot_grad(p.q, G, gq);
      float dot = gq[0] * p.q[0] + gq[1] * p.q[1] + gq[2] * p.q[2] + gq[3] * p.q[3];
      const float iqn = 1.f / p.qn;
      for (int j = 0; j < 4; ++j) out_q[j] = (gq[j] - p.q[j] * dot) * iqn;
      out_l = A[12] * p.sigma * (1.f - p.sigma);
    }
    for (int j = 0; j < 3; ++j) {
      sc.d_means[3 * i + j] = out_m[j];
      sc.d_log_scales[3 * i + j] = out_s[j];
    }
    for (int j = 0; j < 4; ++j) sc.d_quats[4 * i + j] = out_q[j];
    sc.d_logits[i] = out_l;
  }
}

template <int DEG, bool RS, bool PP, bool GEN>
void bwd_launch_k(const BatchDesc &bd, const DevOpts &op, const int16_t *rect, const uint32_t *vals,
                  const uint32_t *ranges, const TileSched &ts, cudaStream_t s) {
  const int warps = block_warps(op);
  const size_t smem = sizeof(BwdWarp<DEG, PP>) * (size_t)warps;
  cudaFuncSetAttribute(k_composite_bwd<DEG, RS, PP, GEN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  k_composite_bwd<DEG, RS, PP, GEN><<<bd.total_tiles * tile_blocks(op), 32 * warps, smem, s>>>(
      bd, op, reinterpret_cast<const short4 *>(rect), vals, reinterpret_cast<const uint2 *>(ranges), ts);
}

// Degree 0 colours do not depend on the direction: both colour modes run the per-pixel kernel.
// The degree-n kernels run with per-pixel colours (make_opts rejects the combination with
// per-particle colours).
template <int DEG, bool RS>
void bwd_launch(const BatchDesc &bd, const DevOpts &op, const int16_t *rect, const uint32_t *vals,
                const uint32_t *ranges, const TileSched &ts, cudaStream_t s) {
  if (op.kernel_degree != 2) {
    bwd_launch_k<DEG, RS, false, true>(bd, op, rect, vals, ranges, ts, s);
    return;
  }
  if constexpr (DEG > 0) {
    if (op.colour_mode == UT_COLOUR_PER_PARTICLE) {
      bwd_launch_k<DEG, RS, true, false>(bd, op, rect, vals, ranges, ts, s);
      return;
    }
  }
  bwd_launch_k<DEG, RS, false, false>(bd, op, rect, vals, ranges, ts, s);
}

}  // namespace

size_t backward_workspace_bytes(int n, bool kbuffer) {
  const size_t part = align256(sizeof(float) * 16 * (size_t)(n > 0 ? n : 1));
  return kbuffer ? 2 * part : part;
}

size_t tile_sched_bytes(int tiles) {
  const size_t t = (size_t)(tiles > 0 ? tiles : 1);
  return 2 * align256(sizeof(uint32_t) * t) + align256(sizeof(uint32_t) * (2 * kOrderBuckets + 1));
}


// Clears the scenes' accumulators and d_sh, orders the tiles by replay length, runs the
// backward over every tile with work, then finalize.
ut_status launch_composite_bwd(const BatchDesc &bd, const DevOpts &op, const int16_t *rect, const uint32_t *vals,
                               const uint32_t *ranges, void *sched, cudaStream_t s) {
  int total = 0;
  for (int k = 0; k < bd.ns; ++k) {
    const DevScene &sc = bd.s[k];
    if (sc.n <= 0) continue;
    const size_t nc = 3 * (size_t)(sc.deg + 1) * (sc.deg + 1);
    if (cudaMemsetAsync(sc.gacc, 0, sizeof(float) * 16 * (size_t)sc.n, s) != cudaSuccess) return UT_ERR_CUDA;
    if (cudaMemsetAsync(sc.d_sh, 0, sizeof(float) * nc * sc.n, s) != cudaSuccess) return UT_ERR_CUDA;
    total = sc.grad_off + sc.n > total ? sc.grad_off + sc.n : total;
  }
  if (op.kbuffer > 0) {  // "Ours (sorted)": its own replay of the per-ray k-buffer
    const ut_status st = launch_composite_bwd_kbuffer(bd, op, rect, vals, ranges, sched, s);
    if (st != UT_OK) return st;
  } else if (bd.total_tiles > 0) {
    const TileSched ts = carve_tile_sched(sched, bd.total_tiles);
    if (cudaMemsetAsync(ts.hist, 0, sizeof(uint32_t) * (2 * kOrderBuckets + 1), s) != cudaSuccess) return UT_ERR_CUDA;
    const auto *rg = reinterpret_cast<const uint2 *>(ranges);
    k_tile_work<<<(bd.total_tiles + 7) / 8, 256, 0, s>>>(bd, op, rg, ts);
    const int ob = (bd.total_tiles + kOrderBuckets - 1) / kOrderBuckets, cap = device_sm_count();
    k_tile_order<<<ob < cap ? ob : cap, kOrderBuckets, 0, s>>>(bd.total_tiles, ts);
    count_launches(2);
    const bool rs = any_rs(bd);
#define UT3D_BWD(D)                                                  \
  (rs ? bwd_launch<D, true>(bd, op, rect, vals, ranges, ts, s) \
      : bwd_launch<D, false>(bd, op, rect, vals, ranges, ts, s))
    switch (bd.s[0].deg) {
      case 0: UT3D_BWD(0); break;
      case 1: UT3D_BWD(1); break;
      case 2: UT3D_BWD(2); break;
      default: UT3D_BWD(3); break;
    }
#undef UT3D_BWD
    count_launches(1);
  }
  if (total > 0) {
    int g = (total + 255) / 256;
    int cap = device_sm_count() * 8;
    k_finalize<<<g < cap ? g : cap, 256, 0, s>>>(bd, total);
    count_launches(1);
  }
  return cudaGetLastError() == cudaSuccess ? UT_OK : UT_ERR_CUDA;
}

UT_DBG_READER(dbg_read_bwd)

}  // namespace ut3d
