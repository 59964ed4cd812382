// composite_fwd.cu — tile-based front-to-back compositing with 3D particle evaluation
// (Sec. 4.2, eq. GaussianMaxResponse; eq. QuadratureVolumeRendering) for a batch of views.
// Each block leaves its tile's list as soon as every pixel's transmittance has dropped below
// t_min; tiles run longest predicted walk first (k_fwd_predict + k_tile_order).
#include "composite_warp.cuh"

namespace ut3d {
namespace {

// Shared memory of one warp: its pixels' bounds and up to kRoundF staged survivors.
constexpr int kRoundF = 32;

template <int NST>
struct __align__(16) FwdWarp {
  WarpRays rays;
  float4 geo[kRoundF][4];       // stage_particle's record
  alignas(16) float col[kRoundF * NST];  // SH coefficients, or the colour (PP)
  uint32_t idx[kRoundF], pos[kRoundF];  // particle, list position
};

// A pixel's outputs (alpha is 0 where it has no ray: its T stays 1).
__device__ __forceinline__ void store_pixel(const DevView &view, const DevCam &cam, int px, int py, float c0, float c1,
                                            float c2, float T, uint32_t last) {
  const size_t pix = (size_t)py * cam.W + px, plane = (size_t)cam.W * cam.H;
  view.rgb[pix] = c0;
  view.rgb[plane + pix] = c1;
  view.rgb[2 * plane + pix] = c2;
  view.alpha[pix] = 1.f - T;
  if (view.tfinal) view.tfinal[pix] = T;
  if (view.n_used) view.n_used[pix] = last;
}

// Resident blocks of 128 threads per SM that the kernel is compiled for.  Bound by issue and by the
// latency of a chunk's loads, so more warps pay until the pixels' state spills.  Measured:
// degree 3 on the 1M rolling-shutter 1080p view 1021 us a frame at 4 blocks (124 registers), 1058
// at 5; per-particle colours (no SH basis in registers) composite_forward of 200k particles at
// 3840x2160 830 us at 6 blocks, 810 at 7, 802 at 8, but with a rolling shutter 948 us a frame at 5,
// 954 at 6, 1013 at 8; degree 1 536 us a frame (400k particles, 1080p) at 5, 521 at 6, 528 at 8.
constexpr int fwd_blocks(int deg, bool rs, bool pp) { return pp ? (rs ? 6 : 8) : (deg < 2 ? 6 : 4); }

// Forward compositing, two pixels a thread and 64 a warp (composite_warp.cuh).  Against one pixel a
// thread with the block's shared staging: 1M rolling-shutter 1080p, this kernel alone, 578 M -> 337 M
// warp instructions, 616 -> 459 us (issue 60 %, FMA pipe 59 % of the cycles at 16 warps an SM: bound
// by both); composite_forward of 200k particles at 3840x2160 964 -> 768 us; 8 views of 3M particles
// 13.4 -> 11 ms; the image is bit-identical.
// PP: per-particle colour mode (the colour of each staged particle is evaluated once, at its
// view direction, while staging; pixels read it from shared memory).
template <int DEG, bool RS, bool STATS, bool PP, bool GEN>
__global__ void __launch_bounds__(32 * kBlockWarps, fwd_blocks(DEG, RS, PP))
    k_composite_fwd(const __grid_constant__ BatchDesc bd, DevOpts op, const short4 *__restrict__ rect,
                    const uint32_t *__restrict__ vals, const uint2 *__restrict__ ranges,
                    unsigned long long *__restrict__ stats, TileSched ts) {
  constexpr int NSH = (DEG + 1) * (DEG + 1);
  constexpr int NC = NSH * 3;
  constexpr int PDEG = PP ? 0 : DEG;        // per-pixel SH basis only when colours are per pixel
  constexpr int NST = PP ? 4 : NC;          // staged colour floats per particle
  extern __shared__ __align__(16) unsigned char smem[];

  // tiles in the order k_tile_order gave them (longest predicted walk first); every tile is
  // in the order, so every pixel is written
  const uint32_t rank = blockIdx.x / (uint32_t)tile_blocks(op);
  const int tile = (int)(ts.order ? ts.order[rank] : rank);
  UT_DBG_CHECK(tile < bd.total_tiles, UT_DBG_TILE_ID, tile, bd.total_tiles, 2);
  const DevView &view = bd.v[view_of_tile(bd, tile)];
  const DevScene &sc = bd.s[view.scene];
  const DevCam &cam = view.cam;
  const int lane = threadIdx.x & 31;
  const int warp = (int)(blockIdx.x % (uint32_t)tile_blocks(op)) * kBlockWarps + (int)(threadIdx.x >> 5);  // of the tile
  if (warp >= tile_warps(op)) return;  // warps never wait for each other
  FwdWarp<NST> &S = reinterpret_cast<FwdWarp<NST> *>(smem)[threadIdx.x >> 5];
  const int lt = tile - view.tile_off;
  const int x0 = (lt % view.tiles_x) * op.tile_w, y0 = (lt / view.tiles_x) * op.tile_h;

  const uint2 rg = ranges[tile];
  if (rg.x >= rg.y) {  // nothing to composite: no rays needed
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      int lx, ly;
      if (tile_pixel2(op, warp, lane, h, lx, ly) && x0 + lx < cam.W && y0 + ly < cam.H)
        store_pixel(view, cam, x0 + lx, y0 + ly, 0.f, 0.f, 0.f, 1.f, 0u);
    }
    return;
  }
  // entries of this chunk of 32 and of the next one (their rectangles are loaded a chunk ahead)
  uint32_t idx = list_index(vals, rg.x + lane, rg.y), idx1 = list_index(vals, rg.x + 32 + lane, rg.y);
  short4 r = list_rect(rect, view.part_off, idx, rg.x + lane, rg.y);
  PixelPair<PDEG> q;
  pixel_pair<PDEG>(cam, op, x0, y0, warp, lane, q);
  const f3x2 o = q.o, d = q.d;
  uint32_t pk[2];  // the pixels still walking, kDead once stopped
#pragma unroll
  for (int h = 0; h < 2; ++h) pk[h] = q.valid[h] ? (uint32_t)q.px[h] | ((uint32_t)q.py[h] << 16) : kDead;
  warp_rays(pk, o, d, tile_is_8x8(op) ? 8 : 0, lane, &S.rays);
  __syncwarp();

  float T[2] = {1.f, 1.f}, C[2][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
  uint32_t last[2] = {0u, 0u};
  unsigned long long n_eval = 0, n_blend = 0;
  for (uint32_t p0 = rg.x; p0 < rg.y; p0 += 32) {
    if (__all_sync(kFull, pk[0] == kDead && pk[1] == kDead)) break;
    const short4 r1 = list_rect(rect, view.part_off, idx1, p0 + 32 + lane, rg.y);
    const uint32_t idx2 = list_index(vals, p0 + 64 + lane, rg.y);
    bool near_ = rect_near(S.rays, r);
    float4 g[4];
    if (near_) {
      stage_particle<RS>(sc, cam, op, r, idx, g, nullptr);
      near_ = !block_misses<RS>(g, S.rays) || STATS;  // the counting variant walks every rectangle
    }
    const unsigned m = __ballot_sync(kFull, near_);
    const int n = __popc(m);
    if (near_) {
      const int b = __popc(m & ((1u << lane) - 1u));
#pragma unroll
      for (int q = 0; q < 4; ++q) S.geo[b][q] = g[q];
      S.idx[b] = idx;
      S.pos[b] = p0 + lane;
      if (PP) reinterpret_cast<float4 *>(S.col)[b] = particle_colour<DEG, RS>(sc, cam, op, idx);
    }
    __syncwarp();
    if (!PP) stage_sh_warp<NC>(sc, S.idx, n, S.col, lane);
    int bl[2] = {-1, -1};  // last survivor blended by each pixel
    for (int b = 0; b < n; ++b) {
      // no branches: nearly every survivor reaches some pixel of the warp, and straight-line code lets
      // its loads start early; what a pixel does not blend is predicated off
      const float4 g3 = S.geo[b][3];
      const uint32_t r0 = __float_as_uint(g3.z), re = __float_as_uint(g3.w);
      bool h0 = in_rect(pk[0], r0, re), h1 = in_rect(pk[1], r0, re);
      if (STATS) n_eval += (int)h0 + (int)h1;
      const PairEval e = eval_pair<RS>(S.geo[b][0], S.geo[b][1], S.geo[b][2], o, d);
      h0 = h0 && e.cc.x <= g3.y * e.dd.x;
      h1 = h1 && e.cc.y <= g3.y * e.dd.y;
      const float2 rho = response2<GEN>(make_float2(__fdividef(e.cc.x, e.dd.x), __fdividef(e.cc.y, e.dd.y)), op);
      const float al0 = fminf(g3.x * rho.x, op.alpha_max), al1 = fminf(g3.x * rho.y, op.alpha_max);
      const float Tn0 = T[0] * (1.f - al0), Tn1 = T[1] * (1.f - al1);
      if (h0 && Tn0 < op.t_min) {
        pk[0] = kDead;
        h0 = false;
      }
      if (h1 && Tn1 < op.t_min) {
        pk[1] = kDead;
        h1 = false;
      }
      if (STATS) n_blend += (int)h0 + (int)h1;
      float2 c0, c1, c2;
      if (PP) {
        const float4 c = reinterpret_cast<const float4 *>(S.col)[b];
        c0 = bc(c.x); c1 = bc(c.y); c2 = bc(c.z);
      } else {
        sh_colour2<NSH>(S.col + b * NC, q.Y, c0, c1, c2);
      }
      if (h0) {
        const float w = al0 * T[0];
        C[0][0] = fmaf(fmaxf(c0.x, 0.f), w, C[0][0]);
        C[0][1] = fmaf(fmaxf(c1.x, 0.f), w, C[0][1]);
        C[0][2] = fmaf(fmaxf(c2.x, 0.f), w, C[0][2]);
        T[0] = Tn0;
        bl[0] = b;
      }
      if (h1) {
        const float w = al1 * T[1];
        C[1][0] = fmaf(fmaxf(c0.y, 0.f), w, C[1][0]);
        C[1][1] = fmaf(fmaxf(c1.y, 0.f), w, C[1][1]);
        C[1][2] = fmaf(fmaxf(c2.y, 0.f), w, C[1][2]);
        T[1] = Tn1;
        bl[1] = b;
      }
    }
    if (bl[0] >= 0) last[0] = S.pos[bl[0]] + 1;
    if (bl[1] >= 0) last[1] = S.pos[bl[1]] + 1;
    __syncwarp();  // the survivors are read before the next chunk's are staged
    idx = idx1;
    idx1 = idx2;
    r = r1;
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {  // (the coordinates are recomputed, not kept through the walk)
    int lx, ly;
    if (tile_pixel2(op, warp, lane, h, lx, ly) && x0 + lx < cam.W && y0 + ly < cam.H)
      store_pixel(view, cam, x0 + lx, y0 + ly, C[h][0], C[h][1], C[h][2], T[h], last[h]);
  }
  if (STATS) {
    for (int s = 16; s >= 1; s >>= 1) {
      n_eval += __shfl_xor_sync(kFull, n_eval, s);
      n_blend += __shfl_xor_sync(kFull, n_blend, s);
    }
    if (lane == 0) {
      atomicAdd(&stats[0], n_eval);
      atomicAdd(&stats[1], n_blend);
    }
  }
}

// "Ours (sorted)" (Sec. 4.4): compositing through a per-ray k-buffer (multi-layer alpha
// blending).  Hits (sigma rho >= alpha_min) met in the tile's depth order enter a buffer of at
// most k = op.kbuffer entries kept in shared memory (tau_max, alpha, rgb and the hit's position
// in the tile's list per entry); when a hit meets a full buffer, the closest of the buffered
// hits and the new one by tau_max -- the earlier arrival, i.e. the smaller list position, on
// equal tau_max -- is blended front to back (stop rule as in k_composite_fwd) and the new hit
// takes its slot unless it was itself the closest; at the end of the list the rest are blended
// in ascending (tau_max, arrival).
// n_used is written as 0 (the backward does not replay this variant).
template <int DEG, bool RS>
__global__ void __launch_bounds__(512, 1) k_composite_fwd_kbuffer(const __grid_constant__ BatchDesc bd, DevOpts op,
                                                               const short4 *__restrict__ rect,
                                                               const uint32_t *__restrict__ vals,
                                                               const uint2 *__restrict__ ranges, TileSched ts) {
  constexpr int NSH = (DEG + 1) * (DEG + 1);
  constexpr int NC = NSH * 3;
  __shared__ float4 s_geo[kBatchK][4];
  __shared__ __align__(16) float s_sh[kBatchK * NC];
  __shared__ uint32_t s_idx[kBatchK];
  extern __shared__ __align__(16) float s_kb[];  // [6][k][threads]: tau, alpha, r, g, b, list position; [warps] rays

  const int tile = (int)(ts.order ? ts.order[blockIdx.x] : blockIdx.x);
  UT_DBG_CHECK(tile < bd.total_tiles, UT_DBG_TILE_ID, tile, bd.total_tiles, 2);
  const DevView &view = bd.v[view_of_tile(bd, tile)];
  const DevScene &sc = bd.s[view.scene];
  const DevCam &cam = view.cam;
  const int lt = tile - view.tile_off;
  const int tx = lt % view.tiles_x, ty = lt / view.tiles_x;
  int lx, ly;
  tile_pixel(op, (int)threadIdx.x, lx, ly);
  const int px = tx * op.tile_w + lx;
  const int py = ty * op.tile_h + ly;
  const bool inside = px < cam.W && py < cam.H;
  const int K = op.kbuffer, nt = blockDim.x;
  float *kb_tau = s_kb + threadIdx.x, *kb_a = kb_tau + K * nt, *kb_r = kb_a + K * nt, *kb_g = kb_r + K * nt,
        *kb_b = kb_g + K * nt;  // entry j of this thread at [j * nt]
  uint32_t *kb_p = reinterpret_cast<uint32_t *>(kb_b + K * nt);
  float3 o, d;
  float Y[NSH];
  bool valid;
  pixel_setup<DEG>(cam, op, px, py, inside, o, d, Y, valid);

  const int lane = threadIdx.x & 31;
  WarpRays &rays = reinterpret_cast<WarpRays *>(s_kb + 6 * K * nt)[threadIdx.x >> 5];
  warp_rays1(op, px, py, o, d, valid, lane, &rays);

  float T = 1.f, C0 = 0.f, C1 = 0.f, C2 = 0.f;
  int nbuf = 0;
  bool done = !valid;
  auto blend = [&](float al, float r, float g, float b) {
    const float Tn = T * (1.f - al);
    if (Tn < op.t_min) {
      done = true;
      return;
    }
    const float w = al * T;
    C0 = fmaf(r, w, C0);
    C1 = fmaf(g, w, C1);
    C2 = fmaf(b, w, C2);
    T = Tn;
  };
  const uint2 rg = ranges[tile];
  for (uint32_t start = rg.x; start < rg.y; start += kBatchK) {
    if (__syncthreads_count(!done) == 0) break;
    const int nb = min((uint32_t)kBatchK, rg.y - start);
    for (int t = threadIdx.x; t < nb; t += blockDim.x) s_idx[t] = vals[start + t];
    __syncthreads();
    for (int t = threadIdx.x; t < nb; t += blockDim.x) {
      uint32_t idx = s_idx[t];
      stage_particle<RS>(sc, cam, op, rect[view.part_off + idx], idx, s_geo[t], nullptr);
    }
    stage_sh<NC>(sc, s_idx, nb, s_sh);
    __syncthreads();
    for (int c0 = 0; c0 < nb; c0 += 32) {
      if (__all_sync(kFull, done)) break;
      unsigned m = near_mask<RS>(s_geo, c0, nb, rays, lane);
      while (m && !done) {
        const int b = c0 + __ffs(m) - 1;
        m &= m - 1;
        float3 og, dg;
        float dd, a;
        if (!eval_response<RS>(s_geo[b], px, py, o, d, og, dg, dd, a)) continue;
        const float tau = -__fdividef(dot3(og, dg), dd);
        const float al = fminf(a, op.alpha_max);
        float r0, r1, r2;
        sh_colour<NSH>(s_sh + b * NC, Y, r0, r1, r2);
        r0 = fmaxf(r0, 0.f); r1 = fmaxf(r1, 0.f); r2 = fmaxf(r2, 0.f);
        const uint32_t pos = start + b;
        if (nbuf < K) {
          kb_tau[nbuf * nt] = tau; kb_a[nbuf * nt] = al;
          kb_r[nbuf * nt] = r0; kb_g[nbuf * nt] = r1; kb_b[nbuf * nt] = r2; kb_p[nbuf * nt] = pos;
          ++nbuf;
          continue;
        }
        // closest of the buffer and the new hit (the new hit arrived last: it wins only with a
        // strictly smaller tau_max)
        const int bi = kb_select(kb_tau, kb_p, nt, K, tau, true);
        if (bi < 0) {
          blend(al, r0, r1, r2);
        } else {
          blend(kb_a[bi * nt], kb_r[bi * nt], kb_g[bi * nt], kb_b[bi * nt]);
          kb_tau[bi * nt] = tau; kb_a[bi * nt] = al;
          kb_r[bi * nt] = r0; kb_g[bi * nt] = r1; kb_b[bi * nt] = r2; kb_p[bi * nt] = pos;
        }
      }
    }
  }
  // end of the list: the remaining hits in ascending (tau_max, arrival)
  while (!done && nbuf > 0) {
    const int bi = kb_select(kb_tau, kb_p, nt, nbuf, 0.f, false);
    blend(kb_a[bi * nt], kb_r[bi * nt], kb_g[bi * nt], kb_b[bi * nt]);
    --nbuf;
    kb_tau[bi * nt] = kb_tau[nbuf * nt]; kb_a[bi * nt] = kb_a[nbuf * nt];
    kb_r[bi * nt] = kb_r[nbuf * nt]; kb_g[bi * nt] = kb_g[nbuf * nt]; kb_b[bi * nt] = kb_b[nbuf * nt];
    kb_p[bi * nt] = kb_p[nbuf * nt];
  }
  if (inside) {
    size_t pix = (size_t)py * cam.W + px;
    size_t plane = (size_t)cam.W * cam.H;
    view.rgb[pix] = C0;
    view.rgb[plane + pix] = C1;
    view.rgb[2 * plane + pix] = C2;
    view.alpha[pix] = valid ? 1.f - T : 0.f;
    if (view.tfinal) view.tfinal[pix] = T;
    if (view.n_used) view.n_used[pix] = 0;
  }
}

// Forward schedule estimate, one warp per tile.  A heuristic that only orders the tiles (no
// result depends on it): a tile's pixels saturate after roughly a fixed optical depth of
// particles that cover the whole tile, so the estimate is the list position where
// sum -ln(1 - 0.3 sigma) over particles whose rect contains the tile's pixels reaches
// kFwdDepth, or the end of the first kFwdCap entries.  Every second entry stands for two: the
// kernel is bound by its gathers (two random L2 sectors an entry; 30 us of a 1044 us frame of 1M
// particles at 1080p, 1027 us with half of them), and half of them order the tiles as well.  Every
// tile gets work >= 1 so that every tile, even an empty one, is scheduled (its pixels must still
// be written).
constexpr int kFwdCap = 512;
constexpr float kFwdDepth = 40.f;

__global__ void k_fwd_predict(const __grid_constant__ BatchDesc bd, DevOpts op, const short4 *__restrict__ rect,
                              const uint32_t *__restrict__ vals, const uint2 *__restrict__ ranges, TileSched ts) {
  const int tile = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (tile >= bd.total_tiles) return;
  const DevView &view = bd.v[view_of_tile(bd, tile)];
  const float *logits = bd.s[view.scene].logits;
  const int lt = tile - view.tile_off;
  const int x0 = (lt % view.tiles_x) * op.tile_w, y0 = (lt / view.tiles_x) * op.tile_h;
  const int x1 = min(x0 + op.tile_w, view.cam.W) - 1, y1 = min(y0 + op.tile_h, view.cam.H) - 1;
  const uint2 rg = ranges[tile];
  const uint32_t end = min(rg.y, rg.x + (uint32_t)kFwdCap);
  uint32_t pred = end - rg.x;
  float tau = 0.f;
  bool found = false;
  for (uint32_t base = rg.x; base < end && !found; base += 256) {
    float c[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {  // four chunks of 32 entries in flight per step
      const uint32_t k = base + 64 * j + 2 * lane;
      c[j] = 0.f;
      if (k < end) {
        const uint32_t idx = vals[k];
        const short4 r = rect[view.part_off + idx];
        if (r.x <= x0 && r.y <= y0 && r.z >= x1 && r.w >= y1) {
          const float sg = 1.f / (1.f + __expf(-logits[idx]));
          c[j] = -2.f * __logf(1.f - fminf(0.3f * sg, 0.99f));
        }
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float incl = c[j];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const float y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      const unsigned hit = __ballot_sync(0xffffffffu, !found && tau + incl >= kFwdDepth);
      if (hit) {
        pred = min(base + 64 * j + 2 * __ffs(hit), end) - rg.x;
        found = true;
      }
      tau += __shfl_sync(0xffffffffu, incl, 31);
    }
  }
  if (lane == 0) {
    const uint32_t w = (rg.y > rg.x ? pred : 0u) + 1u;
    ts.work[tile] = w;
    atomicAdd(&ts.hist[work_bucket(w)], 1u);
  }
}

template <int DEG, bool RS, bool STATS, bool PP, bool GEN>
void fwd_launch_s(const BatchDesc &bd, const DevOpts &op, const int16_t *rect, const uint32_t *vals,
                  const uint32_t *ranges, unsigned long long *stats, const TileSched &ts, cudaStream_t s) {
  constexpr int NST = PP ? 4 : 3 * (DEG + 1) * (DEG + 1);
  const int warps = block_warps(op);
  const size_t smem = sizeof(FwdWarp<NST>) * (size_t)warps;
  static_assert(sizeof(FwdWarp<NST>) * kBlockWarps <= 48 * 1024, "a block's dynamic shared memory needs no opt-in");
  k_composite_fwd<DEG, RS, STATS, PP, GEN><<<bd.total_tiles * tile_blocks(op), 32 * warps, smem, s>>>(
      bd, op, reinterpret_cast<const short4 *>(rect), vals, reinterpret_cast<const uint2 *>(ranges), stats, ts);
}

template <int DEG, bool RS, bool PP, bool GEN>
void fwd_launch_k(const BatchDesc &bd, const DevOpts &op, const int16_t *rect, const uint32_t *vals,
                  const uint32_t *ranges, unsigned long long *stats, const TileSched &ts, cudaStream_t s) {
  if (stats) fwd_launch_s<DEG, RS, true, PP, GEN>(bd, op, rect, vals, ranges, stats, ts, s);
  else fwd_launch_s<DEG, RS, false, PP, GEN>(bd, op, rect, vals, ranges, stats, ts, s);
}

// Degree 0 colours do not depend on the direction: both colour modes run the per-pixel kernel.
// The degree-n kernels and the k-buffer run with per-pixel colours (make_opts rejects the
// other combinations).
template <int DEG, bool RS>
void fwd_launch(const BatchDesc &bd, const DevOpts &op, const int16_t *rect, const uint32_t *vals,
                const uint32_t *ranges, unsigned long long *stats, const TileSched &ts, cudaStream_t s) {
  if (op.kbuffer > 0) {
    const int threads = op.tile_w * op.tile_h;
    const size_t smem = sizeof(float) * 6 * (size_t)op.kbuffer * threads + sizeof(WarpRays) * (threads / 32);
    cudaFuncSetAttribute(k_composite_fwd_kbuffer<DEG, RS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaFuncSetAttribute(k_composite_fwd_kbuffer<DEG, RS>, cudaFuncAttributePreferredSharedMemoryCarveout,
                         cudaSharedmemCarveoutMaxShared);
    k_composite_fwd_kbuffer<DEG, RS><<<bd.total_tiles, threads, smem, s>>>(
        bd, op, reinterpret_cast<const short4 *>(rect), vals, reinterpret_cast<const uint2 *>(ranges), ts);
    return;
  }
  if (op.kernel_degree != 2) {
    fwd_launch_k<DEG, RS, false, true>(bd, op, rect, vals, ranges, stats, ts, s);
    return;
  }
  if constexpr (DEG > 0) {
    if (op.colour_mode == UT_COLOUR_PER_PARTICLE) {
      fwd_launch_k<DEG, RS, true, false>(bd, op, rect, vals, ranges, stats, ts, s);
      return;
    }
  }
  fwd_launch_k<DEG, RS, false, false>(bd, op, rect, vals, ranges, stats, ts, s);
}

}  // namespace

// Predicts each tile's walk and orders the tiles longest first (into sched, carve_tile_sched).
ut_status launch_walk_order(const BatchDesc &bd, const DevOpts &op, const int16_t *rect, const uint32_t *vals,
                            const uint32_t *ranges, void *sched, cudaStream_t s) {
  const TileSched ts = carve_tile_sched(sched, bd.total_tiles);
  if (cudaMemsetAsync(ts.hist, 0, sizeof(uint32_t) * (2 * kOrderBuckets + 1), s) != cudaSuccess) return UT_ERR_CUDA;
  k_fwd_predict<<<(bd.total_tiles + 7) / 8, 256, 0, s>>>(bd, op, reinterpret_cast<const short4 *>(rect), vals,
                                                         reinterpret_cast<const uint2 *>(ranges), ts);
  const int ob = (bd.total_tiles + kOrderBuckets - 1) / kOrderBuckets, sms = device_sm_count();
  k_tile_order<<<ob < sms ? ob : sms, kOrderBuckets, 0, s>>>(bd.total_tiles, ts);
  count_launches(2);
  return UT_OK;
}

// Composites the tiles, longest predicted walk first.
ut_status launch_composite_fwd(const BatchDesc &bd, const DevOpts &op, const int16_t *rect, const uint32_t *vals,
                               const uint32_t *ranges, unsigned long long *stats, void *sched, bool fixed_sequence,
                               cudaStream_t s) {
  if (op.kbuffer > 0 && stats) return UT_ERR_UNSUPPORTED;
  if (bd.total_tiles == 0) return UT_OK;
  // when every block is resident at once (4 a SM at least, 1 for the k-buffer) the order does not
  // matter: the prediction's launches would only delay the frame (1000 particles at 64x64: 8 us)
  const long long blocks = (long long)bd.total_tiles * (op.kbuffer > 0 ? 1 : tile_blocks(op));
  TileSched ts = carve_tile_sched(sched, bd.total_tiles);
  if (!fixed_sequence && blocks <= (op.kbuffer > 0 ? 1 : 4) * device_sm_count()) ts.order = nullptr;
  else if (ut_status st = launch_walk_order(bd, op, rect, vals, ranges, sched, s); st != UT_OK) return st;
  const bool rs = any_rs(bd);
#define UT3D_FWD(D)                                                     \
  (rs ? fwd_launch<D, true>(bd, op, rect, vals, ranges, stats, ts, s) \
      : fwd_launch<D, false>(bd, op, rect, vals, ranges, stats, ts, s))
  switch (bd.s[0].deg) {
    case 0: UT3D_FWD(0); break;
    case 1: UT3D_FWD(1); break;
    case 2: UT3D_FWD(2); break;
    default: UT3D_FWD(3); break;
  }
#undef UT3D_FWD
  count_launches(1);
  return cudaGetLastError() == cudaSuccess ? UT_OK : UT_ERR_CUDA;
}

UT_DBG_READER(dbg_read_fwd)

}  // namespace ut3d
