// Segments of the light tiles' lists: what the shadow composite (composite.cu)
// and its backward (shadow_bwd.cu) share, so that both take every alpha
// decision with the same arithmetic and the same rays per lane.
#pragma once
#include "gs3_internal.cuh"
#include "splat_eval.cuh"
#include "f32x2.cuh"

namespace gs3 {
namespace {

constexpr int kPx = 8;  // rays per lane: lane l owns column l & 15, rows (l >> 4) + 2 i
constexpr uint32_t kSegLast = 0x80000000u;  // desc.x: the tile's last segment
constexpr uint32_t kNoItem = 0xFFFFFFFFu;   // desc.w: the tile's first segment

// Entries staged for a warp's rays, the terms that pair up duplicated so that
// they load as packed operands.
struct StagedEntries {
  float4 yc[32];   // -y, -y, c, c
  float4 xart[32]; // x, a, r, threshold
  float2 gb[32];   // -gamma, halves (as bits)
};

// Stages one entry in slot t: make_entry's record, and the halves its box
// and ellipse both reach, which are returned.
__device__ __forceinline__ uint32_t stage_entry(const SplatRec& q, float ox, float oy, StagedEntries& E, int t) {
  float4 e0, e1;
  make_entry(q, ox, oy, e0, e1);
  const uint32_t bits = __float_as_uint(e1.w) & ellipse_halves(e0, e1);
  E.yc[t] = make_float4(-e0.y, -e0.y, e0.w, e0.w);
  E.xart[t] = make_float4(e0.x, e0.z, e1.x, e1.y);
  E.gb[t] = make_float2(-e1.z, __uint_as_float(bits));
  return bits;
}

// beta of one pixel: 2^pw where it passes (pw >= thr), else 0
__device__ __forceinline__ float beta_of(float pw, float thr) { return pw >= thr ? ex2(pw) : 0.f; }

// (beta, beta) of two pixels from their packed powers
__device__ __forceinline__ f32x2 beta2_of(f32x2 pw, float thr) {
  return pk2(beta_of(lo2(pw), thr), beta_of(hi2(pw), thr));
}

// An entry's terms that a lane's rays share (one column): with dy = ly - y,
// power2 = fma(dy, fma(c, dy, v), sx), the arithmetic of splat_eval.cuh.
struct ColTerms {
  f32x2 ny, c, v, s;
  float thr;
};
__device__ __forceinline__ ColTerms col_terms(float lx, const StagedEntries& E, int t) {
  const ulonglong2 yc = *reinterpret_cast<const ulonglong2*>(&E.yc[t]);
  const float4 q = E.xart[t];
  const float dx = lx - q.x;
  return {yc.x, yc.y, dup2(q.z * dx), dup2((q.y * dx) * dx), q.w};
}
__device__ __forceinline__ f32x2 beta2_at(const ColTerms& e, f32x2 ly) {
  const f32x2 dy = add2(ly, e.ny);
  return beta2_of(power2_pair(dy, e.c, e.v, e.s), e.thr);
}

// An occluder on four rays of one half: P *= max(omin, 1 - gamma beta), which
// is P itself where it does not pass.
template <int H>
__device__ __forceinline__ void occ_half(const f32x2 (&ly)[kPx / 2], f32x2 (&P)[kPx / 2], const ColTerms& e,
                                         float ngamma, float omin) {
#pragma unroll
  for (int q = 2 * H; q < 2 * H + 2; ++q) {
    const f32x2 f = fma2(dup2(ngamma), beta2_at(e, ly[q]), dup2(1.f));
    P[q] = mul2(P[q], pk2(fmaxf(lo2(f), omin), fmaxf(hi2(f), omin)));
  }
}

// The lane's rays in pairs: the row offset of ray i (row (lane >> 4) + 2 i),
// far away where the ray is not in the image
__device__ __forceinline__ void lane_rows(int lane, int rows_in, f32x2 (&ly)[kPx / 2]) {
#pragma unroll
  for (int q = 0; q < kPx / 2; ++q) {
    const float y = (float)(lane >> 4) + 4 * q + 0.5f;
    ly[q] = pk2(2 * q < rows_in ? y : kFarRow, 2 * q + 1 < rows_in ? y + 2.f : kFarRow);
  }
}

// halves (0x3, 0xC) with a ray whose product is still >= the stop
__device__ __forceinline__ uint32_t live_halves(const f32x2 (&P)[kPx / 2]) {
  const bool h0 = fmaxf(fmaxf(lo2(P[0]), hi2(P[0])), fmaxf(lo2(P[1]), hi2(P[1]))) >= kShadowStop;
  const bool h1 = fmaxf(fmaxf(lo2(P[2]), hi2(P[2])), fmaxf(lo2(P[3]), hi2(P[3]))) >= kShadowStop;
  return (__any_sync(0xffffffffu, h0) ? 0x3u : 0u) | (__any_sync(0xffffffffu, h1) ? 0xCu : 0u);
}

// Where segment w's products for the next segment lie (256 floats each), and the
// backward's sums of the segments after it.  Items are numbered level by level, a
// level's tiles by decreasing segment count: the first segments of tiles with
// no other, which have neither, are the last of level 0 and take no room.
struct Links {
  uint32_t more, gap;  // tiles with a second segment, and without
  __device__ __forceinline__ size_t operator()(uint32_t w) const { return (size_t)(w < more ? w : w - gap) * 256; }
};
__device__ __forceinline__ Links frame_links(const uint32_t* lvl_off) {  // once per warp, not per item
  const uint32_t tiles = lvl_off[1], more = lvl_off[2] - tiles;
  return {more, tiles - more};
}

// A(C_s) of the lane's rays: 1 / 0 (in / outside the image) for a tile's
// first segment, else the predecessor's publication (read from L2: it was
// written on another SM); flag 2 publishes that every ray stopped.
template <typename P, typename L>
__device__ __forceinline__ void load_entering(const P& p, const L& link_slot, bool first, uint32_t wpred, uint32_t flag, int lane,
                                              int rows_in, f32x2 (&A)[kPx / 2]) {
  const float* in = p.pub_a + (first ? 0 : link_slot(wpred)) + lane;
  auto one = [&](int i) { return first ? (i < rows_in ? 1.f : 0.f) : (flag == 2u ? 0.f : __ldcg(in + 32 * i)); };
#pragma unroll
  for (int q = 0; q < kPx / 2; ++q) A[q] = pk2(one(2 * q), one(2 * q + 1));
}

// The segment a work item names.
struct SegItem {
  int tx, ty, rows_in;
  uint32_t R0, R1, C0, C1, wpred;
  bool first, last;
};

template <typename P>
__device__ __forceinline__ SegItem seg_item(const P& p, uint32_t w, int lane) {
  const uint4 d = p.desc[w];
  SegItem it;
  const int tile = (int)(d.x & ~kSegLast);
  it.last = (d.x & kSegLast) != 0u;
  it.first = d.w == kNoItem;
  it.tx = tile % p.gx;
  it.ty = tile / p.gx;
  it.R0 = d.y;
  it.R1 = d.z;
  it.wpred = d.w;
  it.C0 = it.C1 = it.R0;
  if (it.R1 > it.R0) {  // an empty tile has one segment without entries
    it.C0 = p.kbound[it.R0];
    it.C1 = p.kbound[it.last ? it.R1 - 1 : it.R1];
  }
  // ray i of the lane is row (lane >> 4) + 2 i: rows below the image hold no ray
  const int lxi = lane & 15, lyi = lane >> 4;
  it.rows_in = it.tx * kTile + lxi < p.W ? min(kPx, (p.H - it.ty * kTile - lyi + 1) / 2) : 0;
  return it;
}

// The next work item of the warp (a ticket), or false past the last.
__device__ __forceinline__ bool next_item(uint32_t* ticket, uint32_t total, int lane, uint32_t& w) {
  uint32_t t = 0;
  if (lane == 0) t = atomicAdd(ticket, 1u);
  w = __shfl_sync(0xffffffffu, t, 0);
  return w < total;
}

}  // namespace
}  // namespace gs3
