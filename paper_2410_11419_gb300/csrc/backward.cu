// Backward of the frame (differentiation form): gradients of a loss with
// respect to every scene parameter and MLP weight, given dL/d(image).
//
// Reverse order of the forward, reading the forward's workspace:
//   K9b  camera composite, back to front per pixel from the stored final
//        transmittance, recovering T by division (per-tile recomputation; no
//        per-pixel lists are stored)                          (Eq. 2, Sec. 4)
//   K8b  Psi and Phi (mlp_x3_bwd.cu; widths of 16: mlp_bwd.cu): forward
//        recomputed, backward through the layers, weight gradients as per-block
//        partials summed in a fixed order                        (Sec. 4.2, 4.3)
//   K6b  shadow splat (shadow_bwd.cu)                                 (Sec. 4.2)
//   K1b  per Gaussian: both EWA projections and the shading back to the
//        parameters                                       (Eq. 1-5, Sec. 3, 4.1)
// Per-Gaussian accumulators are summed with float atomics (after warp
// reductions); the result is deterministic up to the order of those atomics.
#include "gs3_internal.cuh"
#include "splat_eval.cuh"
#include "shadow_bwd.cuh"
#include "f32x2.cuh"

namespace gs3 {
namespace {

constexpr int kGeom = 8;    // dgamma, sums of w dx, w dy, w dx dy, w dx^2, w dy^2
constexpr int kColor = 8;   // dshade rgb, dT', dres rgb
constexpr int kMlpIn = 24;  // Phi: dmu 3, dwi 3, dl 6; Psi: dmu 3, dwo 3, dl 6

struct BwdBufs {
  float* cam_geom;    // [N][8]
  float* light_geom;  // [N][8]
  float* color;       // [N][8]
  float* dT;          // [N]
  float* mlp_in;      // [N][24]
};

__host__ __device__ size_t mlp_params(const MlpDev& m) {
  size_t s = 0;
  int din = m.in_dim;
  for (int l = 0; l <= m.n_hidden; ++l) {
    const int dout = l == m.n_hidden ? m.out_dim : m.width;
    s += (size_t)dout * din + dout;
    din = dout;
  }
  return s;
}

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

struct BwdPlan {
  size_t cam_geom, light_geom, color, dT, mlp_in, wred[2], ticket, mlp_scratch, ct, total;
};

BwdPlan plan_bwd(int n, const MlpDev& phi, const MlpDev& psi) {
  BwdPlan p;
  size_t c = 0;
  auto take = [&](size_t b) { size_t o = c; c = align256(c + b); return o; };
  p.cam_geom = take(4ull * kGeom * n);
  p.light_geom = take(4ull * kGeom * n);
  p.color = take(4ull * kColor * n);
  p.dT = take(4ull * n);
  p.mlp_in = take(4ull * kMlpIn * n);
  p.wred[0] = take(4ull * mlp_params(phi));
  p.wred[1] = take(4ull * mlp_params(psi));
  p.ticket = take(16);
  const size_t sa = mlp_bwd_scratch_bytes(n, phi), sb = mlp_bwd_scratch_bytes(n, psi);
  p.mlp_scratch = take(sa > sb ? sa : sb);  // Phi and Psi use it in turn
  p.ct = take(8ull * n);
  p.total = c;
  return p;
}

// ---------------------------------------------------------------------------
// K9b: camera composite backward.
// Per pixel, back to front over the entries the forward's ray took, T
// recovered by division from its final value.  With (gr, gg, gb) = dL/d(image),
// an entry of colours c (shading, T', residual) has
//   G      = Sh (g . c_shade) + (g . S) c_T' + g . c_res
//   dalpha = T G - D / (1 - alpha),  D = the sum of w G over the entries behind it
// and its colours get w Sh g, w (g . S) and w g (w = alpha T).  Geometry as in
// the shadow splat's backward (shadow_bwd.cu): only the sums of
// t = dalpha beta (dL/dgamma) and of gamma t times dx, dy, dx dy, dx^2, dy^2 are
// accumulated; k_prep_bwd applies the conic.
//
// A warp takes one half (16 x 8) of a tile on its own: lane l column l & 15 and
// rows (l >> 4) + 2 i, i = 0..3, so that a lane adds four pixels before the
// warp adds its lanes; an image too small to fill the chip that way goes by
// quarters (16 x 4, two pixels per lane), which halves a warp's serial walk
// (256 x 256, 20k Gaussians: 117 -> 94 us, 105 if the entries are still picked by
// halves).  The pixel pairs go through packed FP32 instructions;
// the next 32 entries are staged (those whose box and ellipse reach the half)
// while the current ones are walked, as in the forward.  The 14 terms of four
// entries are added over the 32 lanes through shared-memory rows.
// Bound: issue slots.  Object workload (300k Gaussians, 800 x 800): 1.24 ms with
// a pixel per thread and a 16-shuffle butterfly per entry and warp, 0.60 ms so
// (0.57 with T times the reciprocal in place of a rounded quotient).
// ---------------------------------------------------------------------------
constexpr int kCbWarps = 4;  // independent warps per block
constexpr int kCbRows = 4;   // entries whose lane sums are added together
constexpr int kCbTerms = 7;  // pairs of terms per entry

struct CamBwdParams {
  const uint32_t* list;
  const uint32_t* tile_start;
  const uint32_t* tile_order;  // the forward's launch order of the camera tiles
  const SplatRec* rrec;
  const float4* ccol;
  const uint32_t* order;
  const float* final_t;
  const uint32_t* n_contrib;
  const float4* pix_aux;
  const float* dimg;
  float* cam_geom;  // [N][8] by index: dL/dgamma, sums of w dx, w dy, w dx dy, w dx^2, w dy^2
  float* color;
  const uint32_t* nonfinite;  // some colour is infinite or not a number
  int W, H, gx, ntiles;
  float amax;
};

struct CamBwdStage {
  float4 yc[32];    // -y, -y, c, c
  float4 xart[32];  // x, a, r, threshold
  float2 gi[32];    // gamma, place in the list (as bits)
  float4 c0[32], c1[32];
  uint32_t g[32];   // Gaussian
};
struct CamBwdSmem {  // one warp's
  CamBwdStage e[2];
  f32x2 rows[kCbTerms][kCbRows][33];  // per term pair, entry and lane
  float row_gamma[kCbRows];
  uint32_t row_g[kCbRows];
};

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// MASK: a colour or a pixel's gradient is infinite or not a number, so that a
// zero weight does not cancel it: a pixel adds only the entries it takes.  Without
// MASK, false if a pixel asks for it (nothing is added then).
template <int NQ, bool MASK>
__device__ __forceinline__ bool camera_bwd_strip(const CamBwdParams& p, CamBwdSmem& B, int tile, int part) {
  const int lane = threadIdx.x & 31;
  const int half = part * NQ / 2;
  const int tx = tile % p.gx, ty = tile / p.gx;
  const uint32_t hbits = 3u << (2 * half);
  const float ox = (float)(tx * kTile), oy = (float)(ty * kTile);
  const int cx = lane & 15, cy = 4 * NQ * part + (lane >> 4);
  const int px = tx * kTile + cx;
  const float lx = cx + 0.5f;
  const uint32_t b = p.tile_start[tile];
  // per pixel pair q (rows 4 q and 4 q + 2 of the lane): row (far away until the
  // sweep reaches the pixel's last entry), T, D, dL/d(image), Sh, g . S
  f32x2 ly[NQ], T[NQ], D[NQ], gr[NQ], gg[NQ], gb[NQ], sh[NQ], gs[NQ];
  uint32_t nc[2 * NQ], next = 0u;
  float sum_in = 0.f;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    float t2[2], r2[2], g2[2], b2[2], h2[2], s2[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int py = ty * kTile + cy + 4 * q + 2 * h;
      nc[2 * q + h] = 0u;
      t2[h] = 1.f;
      r2[h] = g2[h] = b2[h] = h2[h] = s2[h] = 0.f;
      if (px < p.W && py < p.H) {
        const size_t pix = (size_t)py * p.W + px;
        nc[2 * q + h] = p.n_contrib[pix];
        t2[h] = p.final_t[pix];
        const float4 s = p.pix_aux[2 * pix];
        r2[h] = p.dimg[3 * pix]; g2[h] = p.dimg[3 * pix + 1]; b2[h] = p.dimg[3 * pix + 2];
        h2[h] = s.w;
        s2[h] = r2[h] * s.x + g2[h] * s.y + b2[h] * s.z;
        sum_in += ((r2[h] + g2[h]) + (b2[h] + h2[h])) + s2[h];
      }
      next = max(next, nc[2 * q + h]);
    }
    ly[q] = dup2(kFarRow);
    D[q] = 0ull;
    T[q] = pk2(t2[0], t2[1]);
    gr[q] = pk2(r2[0], r2[1]); gg[q] = pk2(g2[0], g2[1]); gb[q] = pk2(b2[0], b2[1]);
    sh[q] = pk2(h2[0], h2[1]); gs[q] = pk2(s2[0], s2[1]);
  }
  if (!MASK && __any_sync(0xffffffffu, non_finite(sum_in))) return false;
  const uint32_t end = __reduce_max_sync(0xffffffffu, next);  // entries some pixel of the strip took

  int nrow = 0;
  auto flush = [&]() {
    __syncwarp();
    const int r = lane & 3, c = lane >> 2;
    if (r < nrow && c < kCbTerms) {
      const f32x2* row = B.rows[c][r];
      f32x2 s0 = row[0], s1 = row[1];
#pragma unroll
      for (int l = 2; l < 32; l += 2) {
        s0 = add2(s0, row[l]);
        s1 = add2(s1, row[l + 1]);
      }
      const f32x2 s = add2(s0, s1);
      float x = lo2(s), y = hi2(s);
      const size_t g = B.row_g[r];
      if (c < 3) {
        const float gamma = B.row_gamma[r];
        if (c > 0) x *= gamma;  // the first term is dL/dgamma itself
        y *= gamma;
      }
      if (x != 0.f || y != 0.f) {
        float* dst = c < 3 ? p.cam_geom + kGeom * g + 2 * c : p.color + kColor * g + 2 * (c - 3);
        asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(dst), "f"(x), "f"(y) : "memory");
      }
    }
    __syncwarp();  // the rows are free again
    nrow = 0;
  };

  // entries below hi, last first: lane l takes entry hi - 1 - l
  auto rank_at = [&](uint32_t hi) { return hi > (uint32_t)lane ? p.list[b + hi - 1 - lane] : 0u; };
  struct Rec {
    float4 a, b, c;
  };
  auto rec_at = [&](uint32_t r) { return Rec{p.rrec[r].a, p.rrec[r].b, p.rrec[r].c}; };
  auto stage = [&](CamBwdStage& E, uint32_t hi, uint32_t rank, const Rec& rec) {
    SplatRec q;
    q.a = rec.a; q.b = rec.b; q.c = rec.c;
    float4 e0, e1;
    make_entry(q, ox, oy, e0, e1);
    // the halves (and no fewer) that the forward's quadrants lie in, or the strip's rows
    const uint32_t bits = __float_as_uint(e1.w) & hbits;
    bool hit = hi > (uint32_t)lane;
    if constexpr (NQ == 2) hit = hit && (bits & ellipse_halves(e0, e1)) != 0u;
    else hit = hit && bits != 0u && ellipse_rows(e0, e1, (float)(4 * part), (float)(4 * part + 3));
    const uint32_t m = __ballot_sync(0xffffffffu, hit);
    const int slot = __popc(m & ((1u << lane) - 1u));
    if (hit) {
      E.yc[slot] = make_float4(-e0.y, -e0.y, e0.w, e0.w);
      E.xart[slot] = make_float4(e0.x, e0.z, e1.x, e1.y);
      E.gi[slot] = make_float2(e1.z, __uint_as_float(hi - 1 - lane));
      cp_async16(&E.c0[slot], p.ccol + 2 * (size_t)rank);
      cp_async16(&E.c1[slot], p.ccol + 2 * (size_t)rank + 1);
      cp_async4(&E.g[slot], p.order + rank);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    return __popc(m);
  };
  auto below = [](uint32_t hi, uint32_t d) { return hi > d ? hi - d : 0u; };

  uint32_t rank = rank_at(end);
  Rec rec = rec_at(rank);
  uint32_t rank2 = rank_at(below(end, 32));
  int n = stage(B.e[0], end, rank, rec), buf = 0;
  rank = rank2;
  rec = rec_at(rank);
  rank2 = rank_at(below(end, 64));
  for (uint32_t hi = end; hi > 0; hi = below(hi, 32)) {
    int n2 = 0;
    if (hi > 32) {
      n2 = stage(B.e[buf ^ 1], hi - 32, rank, rec);
      rank = rank2;
      rec = rec_at(rank);
      rank2 = rank_at(below(hi, 96));
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncwarp();
    const CamBwdStage& E = B.e[buf];
    for (int t = 0; t < n; ++t) {
      const float2 gi = E.gi[t];
      const uint32_t idx = __float_as_uint(gi.y);
      if (idx < next) {  // pixels whose last entry this is, or lies ahead: once per pixel
        next = 0u;
#pragma unroll
        for (int i = 0; i < 2 * NQ; ++i) {
          const float y = (float)(cy + 2 * i) + 0.5f;
          if (idx < nc[i]) {
            ly[i / 2] = i & 1 ? pk2(lo2(ly[i / 2]), y) : pk2(y, hi2(ly[i / 2]));
            nc[i] = 0u;
          }
          next = max(next, nc[i]);
        }
      }
      const ulonglong2 yc = *reinterpret_cast<const ulonglong2*>(&E.yc[t]);
      const float4 qx = E.xart[t], c0 = E.c0[t], c1 = E.c1[t];
      const float dx = lx - qx.x;
      const f32x2 v = dup2(qx.z * dx), sx = dup2((qx.y * dx) * dx);
      const bool clampable = !(gi.x * 1.00001f < p.amax);
      f32x2 m0 = 0ull, m1 = 0ull, m2 = 0ull, k0 = 0ull, k1 = 0ull, k2 = 0ull, k3 = 0ull, k4 = 0ull, k5 = 0ull, k6 = 0ull;
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const f32x2 dy = add2(ly[q], yc.x);
        const f32x2 pw = power2_pair(dy, yc.y, v, sx);
        f32x2 beta = pk2(lo2(pw) >= qx.w ? ex2(lo2(pw)) : 0.f, hi2(pw) >= qx.w ? ex2(hi2(pw)) : 0.f);
        f32x2 alpha = mul2(dup2(gi.x), beta);
        if (clampable) {  // the same for the warp: alpha = alpha_max passes no gradient to the geometry
          const float a0 = lo2(alpha), a1 = hi2(alpha);
          beta = pk2(a0 < p.amax ? lo2(beta) : 0.f, a1 < p.amax ? hi2(beta) : 0.f);
          alpha = pk2(fminf(p.amax, a0), fminf(p.amax, a1));
        }
        auto taken = [&](f32x2 v) { return MASK ? pk2(lo2(alpha) != 0.f ? lo2(v) : 0.f, hi2(alpha) != 0.f ? hi2(v) : 0.f) : v; };
        const f32x2 om = fma2(alpha, dup2(-1.f), dup2(1.f));
        float ia, ib;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(ia) : "f"(lo2(om)));
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(ib) : "f"(hi2(om)));
        // the reciprocal by a Newton step (exactly 1 for alpha = 0), and with it the
        // quotient T / (1 - alpha), corrected by its remainder, which rounds it as a
        // division does (Markstein 1990): T times the reciprocal repeats the
        // reciprocal's rounding at every entry of that alpha
        const f32x2 nom = pk2(-lo2(om), -hi2(om));
        f32x2 inv = pk2(ia, ib);
        inv = fma2(inv, fma2(nom, inv, dup2(1.f)), inv);
        const f32x2 quot = mul2(T[q], inv);
        T[q] = fma2(fma2(nom, quot, T[q]), inv, quot);
        const f32x2 w = mul2(alpha, T[q]);
        f32x2 G = mul2(gr[q], dup2(c0.x));
        G = fma2(gg[q], dup2(c0.y), G);
        G = mul2(sh[q], fma2(gb[q], dup2(c0.z), G));
        G = fma2(gs[q], dup2(c0.w), G);
        G = fma2(gr[q], dup2(c1.x), G);
        G = fma2(gg[q], dup2(c1.y), G);
        G = taken(fma2(gb[q], dup2(c1.z), G));
        const f32x2 dalpha = fma2(T[q], G, mul2(mul2(inv, dup2(-1.f)), D[q]));
        D[q] = fma2(w, G, D[q]);
        const f32x2 ws = taken(mul2(w, sh[q])), pr = taken(gr[q]), pg = taken(gg[q]), pb = taken(gb[q]);
        k0 = fma2(ws, pr, k0);
        k1 = fma2(ws, pg, k1);
        k2 = fma2(ws, pb, k2);
        k3 = fma2(w, taken(gs[q]), k3);
        k4 = fma2(w, pr, k4);
        k5 = fma2(w, pg, k5);
        k6 = fma2(w, pb, k6);
        f32x2 tt = mul2(dalpha, beta);
        if (MASK) tt = pk2(lo2(beta) != 0.f ? lo2(tt) : 0.f, hi2(beta) != 0.f ? hi2(tt) : 0.f);
        const f32x2 td = mul2(tt, dy);
        m0 = add2(m0, tt);
        m1 = add2(m1, td);
        m2 = fma2(td, dy, m2);
      }
      auto sum = [](f32x2 x) { return lo2(x) + hi2(x); };
      const float s0 = sum(m0), s1 = sum(m1), x1 = s0 * dx;
      B.rows[0][nrow][lane] = pk2(s0, x1);
      B.rows[1][nrow][lane] = pk2(s1, s1 * dx);
      B.rows[2][nrow][lane] = pk2(x1 * dx, sum(m2));
      B.rows[3][nrow][lane] = pk2(sum(k0), sum(k1));
      B.rows[4][nrow][lane] = pk2(sum(k2), sum(k3));
      B.rows[5][nrow][lane] = pk2(sum(k4), sum(k5));
      B.rows[6][nrow][lane] = pk2(sum(k6), 0.f);
      if (lane == 0) {
        B.row_gamma[nrow] = gi.x;
        B.row_g[nrow] = E.g[t];
      }
      if (++nrow == kCbRows) flush();
    }
    __syncwarp();  // the buffer is free again
    n = n2;
    buf ^= 1;
  }
  if (nrow) flush();
  asm volatile("cp.async.wait_all;" ::: "memory");
  return true;
}

// (a call, which leaves the other form as it is without this one)
template <int NQ>
__device__ __noinline__ void camera_bwd_strip_masked(const CamBwdParams& p, CamBwdSmem& B, int tile, int part) {
  camera_bwd_strip<NQ, true>(p, B, tile, part);
}

template <int NQ>
__global__ void __launch_bounds__(kCbWarps * 32, 4) k_camera_bwd(const __grid_constant__ CamBwdParams p) {
  __shared__ CamBwdSmem smem[kCbWarps];
  CamBwdSmem& B = smem[threadIdx.x >> 5];
  const uint32_t unit = blockIdx.x * kCbWarps + (threadIdx.x >> 5);  // (tile in launch order, strip)
  constexpr uint32_t kParts = 4 / NQ;  // strips of 4 NQ rows
  if (unit >= kParts * (uint32_t)p.ntiles) return;
  const int tile = (int)p.tile_order[unit / kParts], part = (int)(unit % kParts);
  if (*p.nonfinite || !camera_bwd_strip<NQ, false>(p, B, tile, part)) camera_bwd_strip_masked<NQ>(p, B, tile, part);
}

__global__ void k_copy_strided(const float* src, int stride, int off, float* dst, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = src[(size_t)stride * i + off];
}

// ---------------------------------------------------------------------------
// K1b: per-Gaussian backward of both projections and the shading
// ---------------------------------------------------------------------------
struct M3 {
  float m[9];
};

__device__ __forceinline__ void quat_rot(const float4 qr, float Rm[9], float qn[4], float& len) {
  len = sqrtf(qr.x * qr.x + qr.y * qr.y + qr.z * qr.z + qr.w * qr.w);
  const float w = qr.x / len, x = qr.y / len, y = qr.z / len, z = qr.w / len;
  qn[0] = w; qn[1] = x; qn[2] = y; qn[3] = z;
  Rm[0] = 1.f - 2.f * (y * y + z * z); Rm[1] = 2.f * (x * y - w * z);       Rm[2] = 2.f * (x * z + w * y);
  Rm[3] = 2.f * (x * y + w * z);       Rm[4] = 1.f - 2.f * (x * x + z * z); Rm[5] = 2.f * (y * z - w * x);
  Rm[6] = 2.f * (x * z - w * y);       Rm[7] = 2.f * (y * z + w * x);       Rm[8] = 1.f - 2.f * (x * x + y * y);
}

// dL/dR (row-major) of R(q / |q|) -> dL/dq
__device__ __forceinline__ float4 quat_bwd(const float G[9], const float qn[4], float len) {
  const float w = qn[0], x = qn[1], y = qn[2], z = qn[3];
  float dw = 2.f * (-z * G[1] + y * G[2] + z * G[3] - x * G[5] - y * G[6] + x * G[7]);
  float dx = 2.f * (y * G[1] + z * G[2] + y * G[3] - 2.f * x * G[4] - w * G[5] + z * G[6] + w * G[7] - 2.f * x * G[8]);
  float dy = 2.f * (-2.f * y * G[0] + x * G[1] + w * G[2] + x * G[3] + z * G[5] - w * G[6] + z * G[7] - 2.f * y * G[8]);
  float dz = 2.f * (-2.f * z * G[0] - w * G[1] + x * G[2] + w * G[3] - 2.f * z * G[4] + y * G[5] + x * G[6] + y * G[7]);
  const float dot = w * dw + x * dx + y * dy + z * dz;
  return make_float4((dw - w * dot) / len, (dx - x * dot) / len, (dy - y * dot) / len, (dz - z * dot) / len);
}

struct ViewB {
  float R[9], t[3];
  float fx, fy, lowpass;
  float ortho;  // > 0: orthographic view with this many pixels per world unit
};

// one EWA projection's backward; adds to dmu, ds and dR (of R(q))
__device__ void proj_bwd(const float4 m, const float4 s, const float Rq[9], const ViewB& v, const float* gg,
                         float dmu[3], float ds[3], float dRq[9]) {
  const float* R = v.R;
  const float x = R[0] * m.x + R[1] * m.y + R[2] * m.z + v.t[0];
  const float y = R[3] * m.x + R[4] * m.y + R[5] * m.z + v.t[1];
  const float z = R[6] * m.x + R[7] * m.y + R[8] * m.z + v.t[2];
  const bool ortho = v.ortho > 0.f;
  const float iz = 1.f / z, iz2 = iz * iz;
  const float sv[3] = {s.x, s.y, s.z};
  float M[9], Sg[9];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) M[3 * i + j] = Rq[3 * i + j] * sv[j];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) Sg[3 * i + j] = M[3 * i] * M[3 * j] + M[3 * i + 1] * M[3 * j + 1] + M[3 * i + 2] * M[3 * j + 2];
  // J = [[fx / z, 0, -fx x / z^2], [0, fy / z, -fy y / z^2]], or [[s, 0, 0], [0, s, 0]]
  const float J00 = ortho ? v.ortho : v.fx * iz, J02 = ortho ? 0.f : -v.fx * x * iz2;
  const float J11 = ortho ? v.ortho : v.fy * iz, J12 = ortho ? 0.f : -v.fy * y * iz2;
  float T[6];
  for (int k = 0; k < 3; ++k) {
    T[k] = J00 * R[k] + J02 * R[6 + k];
    T[3 + k] = J11 * R[3 + k] + J12 * R[6 + k];
  }
  float TS[6];  // T Sigma
  for (int i = 0; i < 2; ++i)
    for (int k = 0; k < 3; ++k)
      TS[3 * i + k] = T[3 * i] * Sg[k] + T[3 * i + 1] * Sg[3 + k] + T[3 * i + 2] * Sg[6 + k];
  const float a = TS[0] * T[0] + TS[1] * T[1] + TS[2] * T[2] + v.lowpass;
  const float b = TS[0] * T[3] + TS[1] * T[4] + TS[2] * T[5];
  const float c = TS[3] * T[3] + TS[4] * T[4] + TS[5] * T[5] + v.lowpass;
  const float det = a * c - b * b, id = 1.f / det;
  const float CA = c * id, CB = -b * id, CC = a * id;
  // d/d(a, b, c) = -C Gs C with Gs = [[dA, dB/2], [dB/2, dC]]
  const float gA = gg[2], gB = 0.5f * gg[3], gC = gg[4];
  const float X00 = CA * gA + CB * gB, X01 = CA * gB + CB * gC;
  const float X10 = CB * gA + CC * gB, X11 = CB * gB + CC * gC;
  const float D00 = -(X00 * CA + X01 * CB), D01 = -(X00 * CB + X01 * CC), D11 = -(X10 * CB + X11 * CC);
  // G2 (symmetric) = [[D00, D01], [D01, D11]];  dT = 2 G2 T Sigma;  dSigma = T^T G2 T
  float dT[6];
  for (int k = 0; k < 3; ++k) {
    dT[k] = 2.f * (D00 * TS[k] + D01 * TS[3 + k]);
    dT[3 + k] = 2.f * (D01 * TS[k] + D11 * TS[3 + k]);
  }
  float dS[9];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j)
      dS[3 * i + j] = T[i] * (D00 * T[j] + D01 * T[3 + j]) + T[3 + i] * (D01 * T[j] + D11 * T[3 + j]);
  // dM = 2 dSigma M;  M = Rq diag(s)
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      const float dM = 2.f * (dS[3 * i] * M[j] + dS[3 * i + 1] * M[3 + j] + dS[3 * i + 2] * M[6 + j]);
      dRq[3 * i + j] += dM * sv[j];
      ds[j] += dM * Rq[3 * i + j];
    }
  // T = J R:  dJ = dT R^T
  const float dJ00 = dT[0] * R[0] + dT[1] * R[1] + dT[2] * R[2];
  const float dJ02 = dT[0] * R[6] + dT[1] * R[7] + dT[2] * R[8];
  const float dJ11 = dT[3] * R[3] + dT[4] * R[4] + dT[5] * R[5];
  const float dJ12 = dT[3] * R[6] + dT[4] * R[7] + dT[5] * R[8];
  const float du = gg[0], dv = gg[1];
  if (ortho) {  // u = s x + cx, v = s y + cy; J constant
    const float dx = du * v.ortho, dy = dv * v.ortho;
    dmu[0] += R[0] * dx + R[3] * dy;
    dmu[1] += R[1] * dx + R[4] * dy;
    dmu[2] += R[2] * dx + R[5] * dy;
    return;
  }
  const float dx = du * v.fx * iz + dJ02 * (-v.fx * iz2);
  const float dy = dv * v.fy * iz + dJ12 * (-v.fy * iz2);
  const float dz = du * (-v.fx * x * iz2) + dv * (-v.fy * y * iz2) + dJ00 * (-v.fx * iz2) +
                   dJ02 * (2.f * v.fx * x * iz2 * iz) + dJ11 * (-v.fy * iz2) + dJ12 * (2.f * v.fy * y * iz2 * iz);
  dmu[0] += R[0] * dx + R[3] * dy + R[6] * dz;
  dmu[1] += R[1] * dx + R[4] * dy + R[7] * dz;
  dmu[2] += R[2] * dx + R[5] * dy + R[8] * dz;
}

struct PrepBwdParams {
  SceneDev sc;
  ViewB cam, light;  // the light view's R, t and scale come from the forward's header
  const float* header_view;  // R (9), t (3) at H_LIGHT_VIEW, scale at H_LIGHT_ORTHO
  float4 lh;                 // homogeneous light (light_h)
  float cam_pos[3], intensity;
  int ablate;
  int falloff;
  const float* cam_geom;
  const float* light_geom;
  const SplatRec *cam_rec, *light_rec;  // by index
  const float* color;
  const float* mlp_in;
  gs3_grads out;
};

// One Gaussian of K1b.  With a shared lobe basis the frame and deviation
// gradients of lobe j go to the block's accumulators sacc[8 j + 0..6]
// (rotation 4, sigma 3) instead of per-Gaussian outputs.
__device__ __forceinline__ void prep_bwd_one(const PrepBwdParams& p, int g, float* sacc) {
  const int n = p.sc.n;
  const float4 m = p.sc.mean_op[g], s = p.sc.scale[g];
  const float gamma = 1.f / (1.f + expf(-m.w));
  // a splat's sums of w dx, ... (K9b, shadow_bwd.cuh) times its conic (A, B, C),
  // with d/du = A dx + B dy, d/dv = C dy + B dx, d/dA = -dx^2 / 2,
  // d/dB = -dx dy, d/dC = -dy^2 / 2: (du, dv, dA, dB, dC, dgamma)
  float gc[6], gl[6];
  auto geometry = [&](const float* sum, const float4 c, float* out) {
    out[0] = c.x * sum[1] + c.y * sum[2];
    out[1] = c.z * sum[2] + c.y * sum[1];
    out[2] = -0.5f * sum[4];
    out[3] = -sum[3];
    out[4] = -0.5f * sum[5];
    out[5] = sum[0];
  };
  geometry(p.cam_geom + (size_t)kGeom * g, p.cam_rec[g].b, gc);
  geometry(p.light_geom + (size_t)kGeom * g, p.light_rec[g].b, gl);
  float dmu[3] = {0, 0, 0}, ds[3] = {0, 0, 0}, dRq[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
  float Rq[9], qn[4], qlen;
  quat_rot(p.sc.rot[g], Rq, qn, qlen);
  ViewB lv = p.light;
#pragma unroll
  for (int i = 0; i < 12; ++i) (i < 9 ? lv.R[i] : lv.t[i - 9]) = p.header_view[H_LIGHT_VIEW + i];
  lv.ortho = p.header_view[H_LIGHT_ORTHO];
  proj_bwd(m, s, Rq, p.cam, gc, dmu, ds, dRq);
  proj_bwd(m, s, Rq, lv, gl, dmu, ds, dRq);
  const float4 dq = quat_bwd(dRq, qn, qlen);
  const float dgamma = gc[5] + gl[5];
  const float dlogit = dgamma * gamma * (1.f - gamma);

  // ---- shading backward (Eq. 2-5) ----
  const float* dcol = p.color + (size_t)kColor * g;
  const float lx = p.lh.x - p.lh.w * m.x, ly = p.lh.y - p.lh.w * m.y, lz = p.lh.z - p.lh.w * m.z;
  const float d2 = lx * lx + ly * ly + lz * lz, dl = sqrtf(d2);
  const float wi[3] = {lx / dl, ly / dl, lz / dl};
  const float vx = p.cam_pos[0] - m.x, vy = p.cam_pos[1] - m.y, vz = p.cam_pos[2] - m.z;
  const float dvn = sqrtf(vx * vx + vy * vy + vz * vz);
  const float wo[3] = {vx / dvn, vy / dvn, vz / dvn};
  float Rs[9], qs[4], qslen;
  quat_rot(p.sc.shade_rot[g], Rs, qs, qslen);
  float wil[3], wol[3];
  for (int i = 0; i < 3; ++i) {
    wil[i] = Rs[3 * i] * wi[0] + Rs[3 * i + 1] * wi[1] + Rs[3 * i + 2] * wi[2];
    wol[i] = Rs[3 * i] * wo[0] + Rs[3 * i + 1] * wo[1] + Rs[3 * i + 2] * wo[2];
  }
  const float off = 0.01f * (1.f - 0.36787944117144233f);
  const float xz = wil[2];
  const float fd = ((xz > 0.f ? xz : 0.01f * expm1f(xz)) + off) / ((1.f + off) * 3.14159265358979323846f);
  const float dfd_dx = (xz > 0.f ? 1.f : 0.01f * expf(xz)) / ((1.f + off) * 3.14159265358979323846f);
  float hs[3] = {wil[0] + wol[0], wil[1] + wol[1], wil[2] + wol[2]};
  const float hn = sqrtf(hs[0] * hs[0] + hs[1] * hs[1] + hs[2] * hs[2]);
  // the Lambertian-only stage has no lobes: no specular term and no lobe gradients
  const bool have_h = hn * hn >= 1e-24f && !(p.ablate & GS3_ABLATE_SPECULAR);
  float h[3] = {0, 0, 0};
  if (have_h) { h[0] = hs[0] / hn; h[1] = hs[1] / hn; h[2] = hs[2] / hn; }
  const bool falloff = p.falloff && p.lh.w != 0.f;  // a directional light's E is constant
  const float E = falloff ? p.intensity / d2 : p.intensity;
  const float4 rd = p.sc.albedo_d[g], rsp = p.sc.albedo_s[g];
  const float rdv[3] = {rd.x, rd.y, rd.z}, rsv[3] = {rsp.x, rsp.y, rsp.z};
  // f_s (recomputed) and the lobe gradients
  float fs[3] = {0, 0, 0};
  const int K = p.sc.k;
  float dfs[3];
  for (int c = 0; c < 3; ++c) dfs[c] = dcol[c] * E * rsv[c];
  float dh[3] = {0, 0, 0};
  if (have_h) {
    for (int j = 0; j < K; ++j) {
      const size_t li = (size_t)j * n + g;
      float Rl[9], ql[4], qllen;
      const size_t ls = p.sc.lobe_shared ? (size_t)j : li;
      quat_rot(p.sc.lobe_rot[ls], Rl, ql, qllen);
      const float4 sig = p.sc.lobe_sigma[ls];
      const float4 amp = p.sc.lobe_amp[li];
      const float hx = Rl[0] * h[0] + Rl[3] * h[1] + Rl[6] * h[2];
      const float hy = Rl[1] * h[0] + Rl[4] * h[1] + Rl[7] * h[2];
      const float hz = Rl[2] * h[0] + Rl[5] * h[1] + Rl[8] * h[2];
      const float sxy = sqrtf(hx * hx + hy * hy);
      const float theta = atan2f(sxy, hz);
      float Pq = 0.f, e2 = 0.f, G;
      const float iz = 1.f / sig.z;
      if (sxy > 1e-20f) {
        Pq = (hx / sig.x) * (hx / sig.x) + (hy / sig.y) * (hy / sig.y);
        e2 = theta * theta / (sxy * sxy) * Pq * iz * iz;
      } else if (hz < 0.f) {
        e2 = (3.14159265358979323846f / sig.x) * (3.14159265358979323846f / sig.x) * iz * iz;
      }
      G = expf(-0.5f * e2) * iz;
      fs[0] += amp.x * G; fs[1] += amp.y * G; fs[2] += amp.z * G;
      const float dG = dfs[0] * amp.x + dfs[1] * amp.y + dfs[2] * amp.z;
      p.out.lobe_amp[4 * li + 0] = dfs[0] * G;
      p.out.lobe_amp[4 * li + 1] = dfs[1] * G;
      p.out.lobe_amp[4 * li + 2] = dfs[2] * G;
      p.out.lobe_amp[4 * li + 3] = 0.f;
      float dsx = 0.f, dsy = 0.f, dsz = dG * G * (e2 - 1.f) * iz;
      float dhl[3] = {0.f, 0.f, 0.f};
      if (sxy > 1e-20f) {
        const float de2 = dG * (-0.5f * G);
        const float dF = de2 * iz * iz;
        const float is2 = 1.f / (sxy * sxy);
        dsx = dF * theta * theta * is2 * (-2.f * hx * hx / (sig.x * sig.x * sig.x));
        dsy = dF * theta * theta * is2 * (-2.f * hy * hy / (sig.y * sig.y * sig.y));
        const float r2 = sxy * sxy + hz * hz;
        const float th_s = hz / r2, th_z = -sxy / r2;
        const float dF_dsxy = 2.f * theta * th_s * Pq * is2 - 2.f * theta * theta * Pq * is2 / sxy;
        dhl[0] = dF * (dF_dsxy * hx / sxy + theta * theta * is2 * 2.f * hx / (sig.x * sig.x));
        dhl[1] = dF * (dF_dsxy * hy / sxy + theta * theta * is2 * 2.f * hy / (sig.y * sig.y));
        dhl[2] = dF * 2.f * theta * th_z * Pq * is2;
      }
      if (!p.sc.lobe_shared) {
        p.out.lobe_sigma[4 * li + 0] = dsx;
        p.out.lobe_sigma[4 * li + 1] = dsy;
        p.out.lobe_sigma[4 * li + 2] = dsz;
        p.out.lobe_sigma[4 * li + 3] = 0.f;
      }
      // hl = Rl^T h: dh += Rl dhl; dRl[k][i] += h_k dhl_i
      float dRl[9];
      for (int k = 0; k < 3; ++k) {
        dh[k] += Rl[3 * k] * dhl[0] + Rl[3 * k + 1] * dhl[1] + Rl[3 * k + 2] * dhl[2];
        for (int i = 0; i < 3; ++i) dRl[3 * k + i] = h[k] * dhl[i];
      }
      const float4 dql = quat_bwd(dRl, ql, qllen);
      if (p.sc.lobe_shared) {
        float* a = sacc + 8 * j;
        atomicAdd(a + 0, dql.x); atomicAdd(a + 1, dql.y); atomicAdd(a + 2, dql.z); atomicAdd(a + 3, dql.w);
        atomicAdd(a + 4, dsx); atomicAdd(a + 5, dsy); atomicAdd(a + 6, dsz);
      } else {
        reinterpret_cast<float4*>(p.out.lobe_rot)[li] = dql;
      }
    }
  } else {
    for (int j = 0; j < K; ++j) {
      const size_t li = (size_t)j * n + g;
      reinterpret_cast<float4*>(p.out.lobe_amp)[li] = make_float4(0, 0, 0, 0);
      if (!p.sc.lobe_shared) {
        reinterpret_cast<float4*>(p.out.lobe_sigma)[li] = make_float4(0, 0, 0, 0);
        reinterpret_cast<float4*>(p.out.lobe_rot)[li] = make_float4(0, 0, 0, 0);
      }
    }
  }
  float dE = 0.f, dfd = 0.f;
  float drd[3], drs[3];
  for (int c = 0; c < 3; ++c) {
    drd[c] = dcol[c] * E * fd;
    drs[c] = dcol[c] * E * fs[c];
    dE += dcol[c] * (rdv[c] * fd + rsv[c] * fs[c]);
    dfd += dcol[c] * E * rdv[c];
  }
  reinterpret_cast<float4*>(p.out.albedo_d)[g] = make_float4(drd[0], drd[1], drd[2], 0.f);
  reinterpret_cast<float4*>(p.out.albedo_s)[g] = make_float4(drs[0], drs[1], drs[2], 0.f);
  // h = hs / |hs|
  float dwil[3] = {0, 0, 0}, dwol[3] = {0, 0, 0};
  if (have_h) {
    const float hd = h[0] * dh[0] + h[1] * dh[1] + h[2] * dh[2];
    for (int i = 0; i < 3; ++i) {
      const float dhs = (dh[i] - h[i] * hd) / hn;
      dwil[i] = dhs;
      dwol[i] = dhs;
    }
  }
  dwil[2] += dfd * dfd_dx;
  // local = Rs w
  float dRs[9];
  float dwi[3], dwo[3];
  for (int i = 0; i < 3; ++i)
    for (int k = 0; k < 3; ++k) dRs[3 * i + k] = dwil[i] * wi[k] + dwol[i] * wo[k];
  for (int k = 0; k < 3; ++k) {
    dwi[k] = Rs[k] * dwil[0] + Rs[3 + k] * dwil[1] + Rs[6 + k] * dwil[2];
    dwo[k] = Rs[k] * dwol[0] + Rs[3 + k] * dwol[1] + Rs[6 + k] * dwol[2];
  }
  const float4 dqs = quat_bwd(dRs, qs, qslen);
  // MLP inputs
  const float* mi = p.mlp_in + (size_t)kMlpIn * g;
  for (int k = 0; k < 3; ++k) {
    dmu[k] += mi[k] + mi[12 + k];
    dwi[k] += mi[3 + k];
    dwo[k] += mi[15 + k];
  }
  // w_i = (L.xyz - L.w mu)/|.|, w_o = (pC - mu)/|.|, E = I / |pL - mu|^2 (point light)
  const float wid = wi[0] * dwi[0] + wi[1] * dwi[1] + wi[2] * dwi[2];
  const float wod = wo[0] * dwo[0] + wo[1] * dwo[1] + wo[2] * dwo[2];
  const float dd2 = falloff ? -dE * E / d2 : 0.f;
  const float lvv[3] = {lx, ly, lz};
  for (int k = 0; k < 3; ++k) {
    dmu[k] -= p.lh.w * (dwi[k] - wi[k] * wid) / dl;
    dmu[k] -= (dwo[k] - wo[k] * wod) / dvn;
    dmu[k] -= 2.f * lvv[k] * dd2;
  }
  reinterpret_cast<float4*>(p.out.mean_op)[g] = make_float4(dmu[0], dmu[1], dmu[2], dlogit);
  reinterpret_cast<float4*>(p.out.scale)[g] = make_float4(ds[0], ds[1], ds[2], 0.f);
  reinterpret_cast<float4*>(p.out.rot)[g] = dq;
  reinterpret_cast<float4*>(p.out.shade_rot)[g] = dqs;
  reinterpret_cast<float4*>(p.out.latent)[g] =
      make_float4(mi[6] + mi[18], mi[7] + mi[19], mi[8] + mi[20], mi[9] + mi[21]);
  reinterpret_cast<float4*>(p.out.latent)[n + g] = make_float4(mi[10] + mi[22], mi[11] + mi[23], 0.f, 0.f);
}

__global__ void __launch_bounds__(128) k_prep_bwd(PrepBwdParams p) {
  __shared__ float sacc[8 * kMaxLobes];
  const bool shared = p.sc.lobe_shared != 0;
  if (shared) {
    for (int i = threadIdx.x; i < 8 * p.sc.k; i += blockDim.x) sacc[i] = 0.f;
    __syncthreads();
  }
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g < p.sc.n) prep_bwd_one(p, g, sacc);
  if (shared) {  // the block's sums of the shared basis gradients
    __syncthreads();
    for (int i = threadIdx.x; i < 8 * p.sc.k; i += blockDim.x) {
      const int j = i >> 3, c = i & 7;
      if (c < 4) atomicAdd(p.out.lobe_rot + 4 * j + c, sacc[i]);
      else if (c < 7) atomicAdd(p.out.lobe_sigma + 4 * j + (c - 4), sacc[i]);
    }
  }
}

// scatter the reduced MLP parameter gradients into the (weights, biases) layout
__global__ void k_split_params(const float* red, int in_dim, int width, int nh, int out_dim, float* dw, float* db) {
  // red holds, per layer: W (out x in) then b (out)
  size_t ro = 0, wo = 0, bo = 0;
  int din = in_dim;
  for (int l = 0; l <= nh; ++l) {
    const int dout = l == nh ? out_dim : width;
    const size_t nw = (size_t)dout * din;
    for (size_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nw; i += gridDim.x * blockDim.x)
      dw[wo + i] = red[ro + i];
    for (size_t i = blockIdx.x * blockDim.x + threadIdx.x; i < (size_t)dout; i += gridDim.x * blockDim.x)
      db[bo + i] = red[ro + nw + i];
    ro += nw + dout;
    wo += nw;
    bo += dout;
    din = dout;
  }
}

}  // namespace

size_t backward_workspace_bytes(int n, const MlpDev& phi, const MlpDev& psi) {
  return plan_bwd(n, phi, psi).total;
}

gs3_status run_backward(const FrameArgs& f, const float* dimg, void* bws, size_t bws_bytes,
                        const gs3_grads& out, cudaStream_t s, SideStream* side) {
  const int n = f.sc.n;
  const BwdPlan bp = plan_bwd(n, f.sc.phi, f.sc.psi);
  if (bws_bytes < bp.total) return GS3_ERR_INVALID_ARG;
  unsigned char* B = static_cast<unsigned char*>(bws);
  float* cam_geom = reinterpret_cast<float*>(B + bp.cam_geom);
  float* light_geom = reinterpret_cast<float*>(B + bp.light_geom);
  float* color = reinterpret_cast<float*>(B + bp.color);
  float* dT = reinterpret_cast<float*>(B + bp.dT);
  float* mlp_in = reinterpret_cast<float*>(B + bp.mlp_in);
  cudaMemsetAsync(B, 0, bp.mlp_scratch, s);  // per-Gaussian accumulators start at zero
  unsigned char* ws = f.ws;
  const Workspace& L = *f.L;
  const int fin = (L.ntiles <= 256 ? 1 : 2) & 1;
  // K9b
  {
    CamBwdParams p;
    p.list = at<uint32_t>(ws, L.sp[0].tv[fin]);
    p.tile_start = at<uint32_t>(ws, L.sp[0].tile_start);
    p.tile_order = at<uint32_t>(ws, L.tile_order[0]);
    p.rrec = at<SplatRec>(ws, L.sp[0].rrec);
    p.ccol = at<float4>(ws, L.ccol);
    p.order = at<uint32_t>(ws, L.sp[0].sv[1]);
    p.final_t = at<float>(ws, L.final_t);
    p.n_contrib = at<uint32_t>(ws, L.n_contrib);
    p.pix_aux = at<float4>(ws, L.pix_aux);
    p.dimg = dimg;
    p.cam_geom = cam_geom;
    p.color = color;
    p.nonfinite = at<uint32_t>(ws, L.header) + H_NONFINITE;
    p.W = L.width; p.H = L.height; p.gx = L.gx; p.ntiles = L.ntiles;
    p.amax = f.opts.alpha_max;
    // quarter tiles while halves leave warp slots free (three blocks per SM); on every
    // image they cost the step of 300k at 800 x 800 2 % (5.05 -> 5.14 ms)
    if (2 * L.ntiles < 3 * kCbWarps * device_sm_count())
      k_camera_bwd<1><<<L.ntiles, kCbWarps * 32, 0, s>>>(p);
    else
      k_camera_bwd<2><<<(2 * L.ntiles + kCbWarps - 1) / kCbWarps, kCbWarps * 32, 0, s>>>(p);
    count_launch();
  }
  // K8b: one network's backward, then its weight gradients in fixed block order
  auto mlp_bwd = [&](int which, cudaStream_t st) {
    const MlpDev& m = which == 0 ? f.sc.phi : f.sc.psi;
    float* wred = reinterpret_cast<float*>(B + bp.wred[which]);
    const bool identity = (f.opts.ablate & (which == 0 ? GS3_ABLATE_PHI : GS3_ABLATE_PSI)) != 0;
    float* dw = which == 0 ? out.phi_w : out.psi_w;
    float* db = which == 0 ? out.phi_b : out.psi_b;
    const size_t np = mlp_params(m);
    if (identity) {
      cudaMemsetAsync(wred, 0, 4 * np, st);
      if (which == 0) {  // T' = T: the gradient passes straight through
        k_copy_strided<<<(n + 255) / 256, 256, 0, st>>>(color, kColor, 3, dT, n);
        count_launch();
      }
    } else {
      MlpArgs a;
      a.net = m;
      a.n = n;
      a.which = which;
      a.mean_op = f.sc.mean_op;
      a.latent = f.sc.latent;
      a.T = at<float>(ws, L.T);
      const float4 lh = light_h(f.light);
      a.light_pos[0] = lh.x; a.light_pos[1] = lh.y; a.light_pos[2] = lh.z; a.light_w = lh.w;
      for (int i = 0; i < 3; ++i) a.cam_pos[i] = f.cam.pos[i];
      a.color = color;
      a.dT = dT;
      a.mlp_in = mlp_in;
      a.status = at<uint32_t>(ws, L.header) + H_STATUS;
      run_mlp_backward(a, B + bp.mlp_scratch, wred, st);
    }
    k_split_params<<<64, 256, 0, st>>>(wred, m.in_dim, m.width, m.n_hidden, m.out_dim, dw, db);
    count_launch();
  };
  // Phi first: the shadow backward takes its dL/dT.  Then Psi, which the
  // shadow backward does not need, runs on the side stream beside it (the
  // networks share the MLP scratch, so they run in turn), after the receivers
  // of the stopped segments.  (Phi's weight gradients there too: 5.25 -> 5.34 ms
  // for the step of 300k.)
  mlp_bwd(0, s);
  cudaStream_t ss = side ? side->s : s;
  // K6b
  if (!(f.opts.ablate & GS3_ABLATE_SHADOW_SPLAT)) {
    ShadowBwdArgs a;
    a.dT = dT;
    a.ct = reinterpret_cast<float2*>(B + bp.ct);
    a.ticket = reinterpret_cast<uint32_t*>(B + bp.ticket);
    a.light_geom = light_geom;
    a.fork = side ? side->fork : nullptr;
    launch_shadow_backward(f, a, s, ss);
  } else if (side) {
    cudaEventRecord(side->fork, s);
    cudaStreamWaitEvent(ss, side->fork, 0);
  }
  mlp_bwd(1, ss);
  if (side) {
    cudaEventRecord(side->join, ss);
    cudaStreamWaitEvent(s, side->join, 0);
  }
  // K1b
  {
    PrepBwdParams p;
    p.sc = f.sc;
    p.header_view = reinterpret_cast<const float*>(at<uint32_t>(ws, L.header));
    for (int i = 0; i < 9; ++i) p.cam.R[i] = f.cam.R[i];
    for (int i = 0; i < 3; ++i) p.cam.t[i] = f.cam.t[i];
    p.cam.fx = f.cam.fx; p.cam.fy = f.cam.fy; p.cam.lowpass = f.opts.lowpass;
    p.cam.ortho = 0.f;
    p.light = p.cam;  // rotation, translation and scale are read from the header
    p.lh = light_h(f.light);
    p.ablate = f.opts.ablate;
    for (int i = 0; i < 3; ++i) p.cam_pos[i] = f.cam.pos[i];
    p.intensity = f.light.intensity;
    p.falloff = f.opts.falloff;
    p.cam_geom = cam_geom;
    p.light_geom = light_geom;
    p.cam_rec = at<SplatRec>(ws, L.sp[0].rec);
    p.light_rec = at<SplatRec>(ws, L.sp[1].rec);
    p.color = color;
    p.mlp_in = mlp_in;
    p.out = out;
    if (f.sc.lobe_shared && f.sc.k > 0) {  // accumulated with atomics
      cudaMemsetAsync(out.lobe_rot, 0, 16ull * f.sc.k, s);
      cudaMemsetAsync(out.lobe_sigma, 0, 16ull * f.sc.k, s);
    }
    k_prep_bwd<<<(n + 127) / 128, 128, 0, s>>>(p);
    count_launch();
  }
  return GS3_OK;
}

}  // namespace gs3
