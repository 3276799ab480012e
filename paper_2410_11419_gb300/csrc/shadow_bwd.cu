// K6 backward: the shadow splat's gradients (Sec. 4.2), given dL/dT.
//
// Per shadow ray m and tile, in list order: receiver j saw T_m(j), the product
// of (1 - alpha_k) over its occluders k < K(j), and T_j = sum beta T_m / sum
// beta.  With coef_j = dL/dT_j / den_j:
//   receiver j (passing):  dL/dbeta_jm = coef_j (T_m(j) - T_j)
//   occluder k (passing):  dL/dalpha_km = -S_m(k) / (1 - alpha_k),
//                          S_m(k) = sum over receivers j with K(j) > k of coef_j beta_jm T_m(j)
// The work is the forward's segments (composite.cu), which are independent but
// for S: a segment needs, per ray, the sum over the receivers of the tile's
// later segments.  So:
//   k_shadow_bwd_sums    each open segment's own sum per ray (but a tile's
//                        first, which nothing before it needs), walked
//                        forward from the products K6a published;
//   k_shadow_bwd_suffix  those sums added up from the tile's last open segment
//                        backwards;
//   k_shadow_bwd         each open segment back to front, from the product the
//                        ray leaves it with (K6a's) or, where it stopped in
//                        it, from where it stopped (K6b's record), and the sum
//                        over the later segments: undoing occluder k divides it
//                        out, receivers add to S;
//   k_shadow_bwd_stopped the receivers of the segments that every ray enters
//                        stopped: T_m = 0, so they carry coef_j (0 - T_j) and
//                        take no occluder.
// Entries, rays per lane, batches of 32 and packed pixel pairs are the
// forward's.  With dL/dpower = w at a pixel (dx, dy) from the splat centre,
// the centre and conic gradients are linear in the sums of w dx, w dy,
// w dx^2, w dx dy and w dy^2 with coefficients that belong to the Gaussian, so
// only those sums (and dL/dgamma) are accumulated here, and k_prep_bwd forms
// the gradients.  A lane's eight pixels share dx, so it keeps (w, w dy, w dy^2)
// and multiplies by dx once per entry; the warp's 32 lanes are added through
// shared-memory rows, eight entries at a time, and added to the Gaussian with
// two-float reductions.
//
// Bound: issue slots.  Object workload (300k Gaussians, 800 x 800): 0.24 +
// 0.02 + 0.76 ms (0.10 for the stopped segments beside them), against 2.57 ms
// (0.31) with one warp per tile over the tile's whole list, scalar; 20k
// Gaussians at 256 x 256, where that left 256 warps on the chip, 0.13 ms
// against 0.84.
#include "shadow_bwd.cuh"
#include "shadow_seg.cuh"

namespace gs3 {
namespace {

constexpr int kBwdWarps = 4;  // independent warps per block
constexpr int kRows = 8;      // entries whose lane sums are added together

struct BwdParams {
  const uint32_t* list;
  const uint32_t* tile_start;
  const SplatRec* rrec;
  const uint32_t* order;
  const uint32_t* kbound;
  const uint32_t* tile_order;
  const uint32_t* lvl_off;
  const uint32_t* counts;  // [2] items in open_list and dead_list
  const uint4* desc;
  const uint32_t* open_list;
  const uint32_t* dead_list;
  const float* pub_a;
  const uint32_t* pub_flag;
  const uint8_t* pass_mask;
  const float* light_final;
  const uint32_t* light_stop;
  const float2* ct;    // by light rank: (coef_j, T_j)
  float* seg_sum;      // [link_slot][256]: a segment's own sum per ray, then the later segments'
  uint32_t* ticket;    // [4]: three tickets, and whether some coef_j is infinite or not a number
  float* light_geom;   // [N][8] by index: dL/dgamma, sums of w dx, w dy, w dx dy, w dx^2, w dy^2
  int W, H, gx, ntiles;
  float amax;
};

__global__ void k_bwd_coef(const uint32_t* __restrict__ order, const float* __restrict__ dT,
                           const float* __restrict__ den, const float* __restrict__ T, float2* __restrict__ ct, uint32_t* nonfinite, int n) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n) return;
  const uint32_t g = order[r];
  const float d = den[g];
  const float c = d > 0.f ? dT[g] / d : 0.f;
  ct[r] = make_float2(c, T[g]);
  if (non_finite(c)) *nonfinite = 1u;
}

__device__ __forceinline__ void red_add2(float* p, float x, float y) {
  asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(x), "f"(y) : "memory");
}

// ---- a segment's own sum per ray -------------------------------------------
struct SumSmem {  // one warp's
  StagedEntries e;
  float coef[32];
};

// x where b is not 0, else 0.  With MASK (here and below) a coefficient is
// infinite or not a number, and a pixel that does not pass must not see it.
template <bool MASK>
__device__ __forceinline__ f32x2 where_passing(f32x2 b, f32x2 x) {
  return MASK ? pk2(lo2(b) != 0.f ? lo2(x) : 0.f, hi2(b) != 0.f ? hi2(x) : 0.f) : x;
}

template <bool MASK>
__device__ __forceinline__ void sum_item(const BwdParams& p, const Links& link_slot, uint32_t w, SumSmem& S, int lane) {
  const SegItem it = seg_item(p, w, lane);
  if (it.first) return;
  const float lx = (lane & 15) + 0.5f, omin = 1.f - p.amax;
  const float ox = (float)(it.tx * kTile), oy = (float)(it.ty * kTile);
  f32x2 ly[kPx / 2], P[kPx / 2], sum[kPx / 2];
  lane_rows(lane, it.rows_in, ly);
  load_entering(p, link_slot, false, it.wpred, __ldcg(p.pub_flag + it.wpred), lane, it.rows_in, P);
#pragma unroll
  for (int q = 0; q < kPx / 2; ++q) sum[q] = 0ull;
  uint32_t j = it.R0, k = it.C0;
  const uint32_t kend = p.kbound[it.R1 - 1];
  for (;;) {
    // a stopped ray's receivers see 0
#pragma unroll
    for (int q = 0; q < kPx / 2; ++q)
      P[q] = pk2(lo2(P[q]) >= kShadowStop ? lo2(P[q]) : 0.f, hi2(P[q]) >= kShadowStop ? hi2(P[q]) : 0.f);
    const uint32_t live = live_halves(P);
    if (!live || j >= it.R1) break;
    const int nops = (int)min(32u, (it.R1 - j) + (kend - k));
    uint32_t pos = 32u;
    if (j + lane < it.R1) pos = lane + (p.kbound[j + lane] - k);
    const uint32_t M = __reduce_or_sync(0xffffffffu, pos < 32u ? 1u << pos : 0u);
    const int nrecv = __popc(M), mine = __popc(M & ((1u << lane) - 1u));
    __syncwarp();  // the previous batch is consumed
    if (lane < nops) {
      const bool is_recv = (M >> lane) & 1u;
      const uint32_t rank = p.list[is_recv ? j + mine : k + (lane - mine)];
      stage_entry(p.rrec[rank], ox, oy, S.e, lane);
      const float coef = is_recv ? p.ct[rank].x : 0.f;
      S.coef[lane] = coef;
      if (is_recv && coef == 0.f) S.e.gb[lane].y = 0.f;  // no half
    }
    __syncwarp();
    for (int t = 0; t < nops; ++t) {
      const float2 gb = S.e.gb[t];
      const uint32_t bits = __float_as_uint(gb.y) & live;
      if (!bits) continue;
      const ColTerms e = col_terms(lx, S.e, t);
      if ((M >> t) & 1u) {
        const f32x2 c = dup2(S.coef[t]);
#pragma unroll
        for (int q = 0; q < kPx / 2; ++q)
          if (bits & (q < 2 ? 0x3u : 0xCu)) {
            const f32x2 b = beta2_at(e, ly[q]);
            sum[q] = fma2(where_passing<MASK>(b, mul2(c, b)), P[q], sum[q]);
          }
      } else {
        if (bits & 0x3u) occ_half<0>(ly, P, e, gb.x, omin);
        if (bits & 0xCu) occ_half<1>(ly, P, e, gb.x, omin);
      }
    }
    j += nrecv;
    k += nops - nrecv;
  }
  float* out = p.seg_sum + link_slot(w) + lane;
#pragma unroll
  for (int q = 0; q < kPx / 2; ++q) {
    out[64 * q] = lo2(sum[q]);
    out[64 * q + 32] = hi2(sum[q]);
  }
}

// (the masked forms are calls, which leaves the others as they are without them)
__device__ __noinline__ void sum_item_masked(const BwdParams& p, const Links& link_slot, uint32_t w, SumSmem& S, int lane) {
  sum_item<true>(p, link_slot, w, S, lane);
}

__global__ void __launch_bounds__(kBwdWarps * 32, 6) k_shadow_bwd_sums(const __grid_constant__ BwdParams p) {
  __shared__ SumSmem smem[kBwdWarps];
  const int lane = threadIdx.x & 31;
  const uint32_t total = p.counts[0];
  const bool mask = p.ticket[3] != 0u;
  const Links links = frame_links(p.lvl_off);
  uint32_t w;
  while (next_item(p.ticket, total, lane, w)) {
    if (mask) sum_item_masked(p, links, p.open_list[w], smem[threadIdx.x >> 5], lane);
    else sum_item<false>(p, links, p.open_list[w], smem[threadIdx.x >> 5], lane);
  }
}

// One warp per tile: seg_sum of each open segment becomes the sum over the
// tile's later open segments (the open ones are a prefix of the segments).
__global__ void __launch_bounds__(128) k_shadow_bwd_suffix(const BwdParams p) {
  after_previous();
  const uint32_t pos = blockIdx.x * 4 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (pos >= (uint32_t)p.ntiles) return;
  const int tile = (int)p.tile_order[pos];
  const uint32_t nseg = seg_count(p.tile_start[tile + 1] - p.tile_start[tile], p.lvl_off[kSegWord]);
  if (nseg < 2u) return;
  uint32_t nopen = nseg;
  for (uint32_t s0 = 1; s0 < nseg && nopen == nseg; s0 += 32) {
    const uint32_t s = s0 + (uint32_t)lane;
    const bool dead = s < nseg && __ldcg(p.pub_flag + p.lvl_off[s - 1] + pos) == 2u;
    const uint32_t m = __ballot_sync(0xffffffffu, dead);
    if (m) nopen = s0 + (uint32_t)(__ffs(m) - 1);
  }
  const Links link_slot = frame_links(p.lvl_off);
  float4 acc[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
  for (uint32_t s = nopen; s-- > 0;) {
    float4* v = reinterpret_cast<float4*>(p.seg_sum + link_slot(p.lvl_off[s] + pos)) + 2 * lane;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float4 own = s > 0 ? v[i] : make_float4(0.f, 0.f, 0.f, 0.f);
      v[i] = acc[i];
      acc[i] = make_float4(acc[i].x + own.x, acc[i].y + own.y, acc[i].z + own.z, acc[i].w + own.w);
    }
  }
}

// ---- open segments, back to front -------------------------------------------
struct BwdSmem {  // one warp's
  StagedEntries e;
  float2 ct[32];
  uint32_t g[32];
  f32x2 rows[3][kRows][33];  // per term pair, entry and lane: (w, w dx), (w dy, w dx dy), (w dx^2, w dy^2)
  uint8_t op[kRows];         // the rows' places in the batch
};

// 1 / f, rounded to nearest for every f in [0.01, 1] (compared with __frcp_rn over all
// of them), so exactly 1 for f = 1
__device__ __forceinline__ f32x2 rcp2(f32x2 f) {
  float a, b;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(a) : "f"(lo2(f)));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(b) : "f"(hi2(f)));
  const f32x2 r = pk2(a, b);
  return fma2(r, fma2(pk2(-lo2(f), -hi2(f)), r, dup2(1.f)), r);
}

struct Moments {
  f32x2 m0, m1, m2;  // sums of w, w dy, w dy^2
};

// A receiver's four rays of one half
template <int H, bool MASK>
__device__ __forceinline__ void recv_bwd(const f32x2 (&ly)[kPx / 2], const f32x2 (&A)[kPx / 2], f32x2 (&S)[kPx / 2],
                                         const ColTerms& e, f32x2 coef, f32x2 nT, Moments& m) {
#pragma unroll
  for (int q = 2 * H; q < 2 * H + 2; ++q) {
    const f32x2 dy = add2(ly[q], e.ny);
    const f32x2 b = beta2_of(power2_pair(dy, e.c, e.v, e.s), e.thr);
    const f32x2 cb = where_passing<MASK>(b, mul2(coef, b));
    S[q] = fma2(cb, A[q], S[q]);
    const f32x2 w = mul2(cb, add2(A[q], nT)), wd = mul2(w, dy);
    m.m0 = add2(m.m0, w);
    m.m1 = add2(m.m1, wd);
    m.m2 = fma2(wd, dy, m.m2);
  }
}

// Undoing an occluder on four rays of one half; the moments are those of
// S beta / (1 - alpha) (its factor -gamma is applied to their sums).  CLAMP:
// gamma may reach alpha_max, where alpha is clamped and passes no gradient.
template <int H, bool CLAMP, bool MASK>
__device__ __forceinline__ void occ_bwd(const f32x2 (&ly)[kPx / 2], f32x2 (&A)[kPx / 2], const f32x2 (&S)[kPx / 2],
                                        const ColTerms& e, float ngamma, float amax, Moments& m) {
#pragma unroll
  for (int q = 2 * H; q < 2 * H + 2; ++q) {
    const f32x2 dy = add2(ly[q], e.ny);
    f32x2 b = beta2_of(power2_pair(dy, e.c, e.v, e.s), e.thr);
    f32x2 f = fma2(dup2(ngamma), b, dup2(1.f));
    if (CLAMP) {
      f = pk2(fmaxf(lo2(f), 1.f - amax), fmaxf(hi2(f), 1.f - amax));
      b = pk2(-ngamma * lo2(b) < amax ? lo2(b) : 0.f, -ngamma * hi2(b) < amax ? hi2(b) : 0.f);
    }
    const f32x2 inv = rcp2(f);
    A[q] = mul2(A[q], inv);
    const f32x2 w = where_passing<MASK>(b, mul2(mul2(S[q], inv), b)), wd = mul2(w, dy);
    m.m0 = add2(m.m0, w);
    m.m1 = add2(m.m1, wd);
    m.m2 = fma2(wd, dy, m.m2);
  }
}

template <bool MASK>
__device__ __forceinline__ void bwd_item(const BwdParams& p, const Links& link_slot, uint32_t w, BwdSmem& B, int lane) {
  const SegItem it = seg_item(p, w, lane);
  if (it.R1 <= it.R0) return;
  const int lxi = lane & 15, lyi = lane >> 4;
  const float lx = lxi + 0.5f;
  const float ox = (float)(it.tx * kTile), oy = (float)(it.ty * kTile);
  const size_t pix0 = (size_t)(it.ty * kTile + lyi) * p.W + it.tx * kTile + lxi;
  f32x2 ly[kPx / 2], A[kPx / 2], S[kPx / 2];
  lane_rows(lane, it.rows_in, ly);
  load_entering(p, link_slot, it.first, it.wpred, it.first ? 1u : __ldcg(p.pub_flag + it.wpred), lane, it.rows_in, A);
  // the product each ray leaves the segment with; one that ends in it gets its
  // product when the walk reaches the occluder it ended at (pending: those
  // rays, next: the largest such limit; kNoStop: it ran through the list)
  const uint32_t fl_out = it.last ? 2u : __ldcg(p.pub_flag + w);
  uint32_t pending = 0u, next = 0u;
  const bool only = it.first && it.last;  // the tile's only segment
  const size_t link = only ? 0 : link_slot(w);
#pragma unroll
  for (int i = 0; i < kPx; ++i) {
    float a = i & 1 ? hi2(A[i / 2]) : lo2(A[i / 2]);
    if (a >= kShadowStop) {
      a = fl_out == 2u ? 0.f : __ldcg(p.pub_a + link + 32 * i + lane);
      if (a == 0.f) {
        const uint32_t lim = p.light_stop[pix0 + (size_t)2 * i * p.W];
        if (lim == kNoStop) {
          a = p.light_final[pix0 + (size_t)2 * i * p.W];
        } else {
          pending |= 1u << i;
          next = max(next, lim);
        }
      }
    } else {
      a = 0.f;
    }
    A[i / 2] = i & 1 ? pk2(lo2(A[i / 2]), a) : pk2(a, hi2(A[i / 2]));
  }
#pragma unroll
  for (int q = 0; q < kPx / 2; ++q)
    S[q] = only ? 0ull : pk2(__ldcg(p.seg_sum + link + 64 * q + lane), __ldcg(p.seg_sum + link + 64 * q + 32 + lane));

  // the rows' sums over the 32 lanes: lane l < 24 takes term pair l >> 3 of
  // entry l & 7, in lane order
  int nrow = 0;
  uint32_t M = 0u;
  auto flush = [&]() {
    __syncwarp();
    const int r = lane & 7, c = lane >> 3;
    if (r < nrow && c < 3) {
      const f32x2* row = B.rows[c][r];
      f32x2 s0 = row[0], s1 = row[1];
#pragma unroll
      for (int l = 2; l < 32; l += 2) {
        s0 = add2(s0, row[l]);
        s1 = add2(s1, row[l + 1]);
      }
      const f32x2 s = add2(s0, s1);
      const int t = B.op[r];
      float x = lo2(s), y = hi2(s);
      if ((M >> t) & 1u) {
        if (c == 0) x = 0.f;  // a receiver has no part in dL/dgamma
      } else {
        const float ng = B.e.gb[t].x;
        x = c == 0 ? -x : x * ng;
        y *= ng;
      }
      if (x != 0.f || y != 0.f) red_add2(p.light_geom + 8 * (size_t)B.g[t] + 2 * c, x, y);
    }
    __syncwarp();  // the rows are free again
    nrow = 0;
  };
  auto push = [&](int t, const Moments& m, float dx) {
    const float m0 = lo2(m.m0) + hi2(m.m0), m1 = lo2(m.m1) + hi2(m.m1), m2 = lo2(m.m2) + hi2(m.m2);
    const float x1 = m0 * dx;
    B.rows[0][nrow][lane] = pk2(m0, x1);
    B.rows[1][nrow][lane] = pk2(m1, m1 * dx);
    B.rows[2][nrow][lane] = pk2(x1 * dx, m2);
    if (lane == 0) B.op[nrow] = (uint8_t)t;
    if (++nrow == kRows) flush();
  };

  uint32_t j = it.R1, k = it.C1;  // receivers and occluders below these are left
  for (;;) {
    const uint32_t left = (j - it.R0) + (k - it.C0);
    if (left == 0u) break;
    const int nops = (int)min(32u, left);
    // the receivers' places, counted from the end
    uint32_t pos = 32u;
    if (j - it.R0 > (uint32_t)lane) pos = lane + (k - p.kbound[j - 1 - lane]);
    M = __reduce_or_sync(0xffffffffu, pos < 32u ? 1u << pos : 0u);
    const int nrecv = __popc(M), mine = __popc(M & ((1u << lane) - 1u));
    // halves with a ray that took occluders here
    const bool h0 = fmaxf(fmaxf(lo2(A[0]), hi2(A[0])), fmaxf(lo2(A[1]), hi2(A[1]))) > 0.f || (pending & 0x0Fu);
    const bool h1 = fmaxf(fmaxf(lo2(A[2]), hi2(A[2])), fmaxf(lo2(A[3]), hi2(A[3]))) > 0.f || (pending & 0xF0u);
    const uint32_t live = (__any_sync(0xffffffffu, h0) ? 0x3u : 0u) | (__any_sync(0xffffffffu, h1) ? 0xCu : 0u);
    __syncwarp();  // the previous batch is consumed
    if (lane < nops) {
      const bool is_recv = (M >> lane) & 1u;
      const uint32_t rank = p.list[is_recv ? j - 1 - mine : k - 1 - (lane - mine)];
      stage_entry(p.rrec[rank], ox, oy, B.e, lane);
      if (is_recv) {
        const float2 ct = p.ct[rank];
        B.ct[lane] = ct;
        if (ct.x == 0.f) B.e.gb[lane].y = 0.f;  // no half
      }
      B.g[lane] = p.order[rank];
    }
    __syncwarp();
    for (int t = 0; t < nops; ++t) {
      const float2 gb = B.e.gb[t];
      uint32_t bits = __float_as_uint(gb.y);
      Moments m{0ull, 0ull, 0ull};
      if ((M >> t) & 1u) {
        if (!bits) continue;
        const ColTerms e = col_terms(lx, B.e, t);
        const float2 ct = B.ct[t];
        if (bits & 0x3u) recv_bwd<0, MASK>(ly, A, S, e, dup2(ct.x), dup2(-ct.y), m);
        if (bits & 0xCu) recv_bwd<1, MASK>(ly, A, S, e, dup2(ct.x), dup2(-ct.y), m);
      } else {
        const uint32_t kk = k - 1u - (uint32_t)(t - __popc(M & ((1u << t) - 1u)));
        if (next == kk + 1u) {  // rays that ended at this occluder: once per ray
          next = 0u;
#pragma unroll
          for (int i = 0; i < kPx; ++i) {
            if (!(pending & (1u << i))) continue;
            const uint32_t lim = p.light_stop[pix0 + (size_t)2 * i * p.W];
            if (lim == kk + 1u) {
              const float a = p.light_final[pix0 + (size_t)2 * i * p.W];
              A[i / 2] = i & 1 ? pk2(lo2(A[i / 2]), a) : pk2(a, hi2(A[i / 2]));
              pending &= ~(1u << i);
            } else {
              next = max(next, lim);
            }
          }
        }
        bits &= live;
        if (!bits) continue;
        const ColTerms e = col_terms(lx, B.e, t);
        if (-gb.x * 1.00001f < p.amax) {  // gamma beta stays below alpha_max (beta <= 1 up to rounding)
          if (bits & 0x3u) occ_bwd<0, false, MASK>(ly, A, S, e, gb.x, p.amax, m);
          if (bits & 0xCu) occ_bwd<1, false, MASK>(ly, A, S, e, gb.x, p.amax, m);
        } else {
          if (bits & 0x3u) occ_bwd<0, true, MASK>(ly, A, S, e, gb.x, p.amax, m);
          if (bits & 0xCu) occ_bwd<1, true, MASK>(ly, A, S, e, gb.x, p.amax, m);
        }
      }
      push(t, m, lx - B.e.xart[t].x);
    }
    if (nrow) flush();  // the rows name this batch's entries
    j -= nrecv;
    k -= nops - nrecv;
  }
}

__device__ __noinline__ void bwd_item_masked(const BwdParams& p, const Links& link_slot, uint32_t w, BwdSmem& B, int lane) {
  bwd_item<true>(p, link_slot, w, B, lane);
}

__global__ void __launch_bounds__(kBwdWarps * 32, 4) k_shadow_bwd(const __grid_constant__ BwdParams p) {
  after_previous();
  __shared__ BwdSmem smem[kBwdWarps];
  const int lane = threadIdx.x & 31;
  const uint32_t total = p.counts[0];
  uint32_t w;
  const bool mask = p.ticket[3] != 0u;
  const Links links = frame_links(p.lvl_off);
  while (next_item(p.ticket + 1, total, lane, w)) {
    if (mask) bwd_item_masked(p, links, p.open_list[w], smem[threadIdx.x >> 5], lane);
    else bwd_item<false>(p, links, p.open_list[w], smem[threadIdx.x >> 5], lane);
  }
}

// ---- stopped segments ---------------------------------------------------------
// A warp takes a segment and lists its (receiver, half) units: the halves the
// forward found passing, of the receivers whose coef_j T_j is not 0; a lane
// walks the 16 x 8 pixels of one unit at a time (w = -coef_j T_j beta, the
// factor applied to the sums) and adds its sums to the Gaussian.
constexpr int kStopScan = 128;  // receivers listed at a time

struct StopSmem {  // one warp's
  uint16_t unit[2 * kStopScan];  // receiver (bits 0-7) and half (bit 8)
};

__device__ __forceinline__ void stopped_unit(const BwdParams& p, uint32_t idx, int h, float ox, float oy, int ncol,
                                             int nrow) {
  const uint32_t rank = p.list[idx];
  const float2 ct = p.ct[rank];
  float4 e0, e1;
  make_entry(p.rrec[rank], ox, oy, e0, e1);
  f32x2 dy[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int y = 8 * h + 2 * q;  // rows below the image lie far away
    dy[q] = pk2((y < nrow ? (float)y + 0.5f : kFarRow) - e0.y, (y + 1 < nrow ? (float)y + 1.5f : kFarRow) - e0.y);
  }
  const f32x2 c = dup2(e0.w);
  float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f, s4 = 0.f;  // beta dx, beta dy, beta dx dy, beta dx^2, beta dy^2
  float fx = 0.5f;
#pragma unroll 1
  for (int x = 0; x < ncol; ++x, fx += 1.f) {
    const float dx = fx - e0.x;
    const f32x2 sx = dup2((e0.z * dx) * dx), v = dup2(e1.x * dx);
    Moments m{0ull, 0ull, 0ull};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const f32x2 b = beta2_of(power2_pair(dy[q], c, v, sx), e1.y), bd = mul2(b, dy[q]);
      m.m0 = add2(m.m0, b);
      m.m1 = add2(m.m1, bd);
      m.m2 = fma2(bd, dy[q], m.m2);
    }
    const float m0 = lo2(m.m0) + hi2(m.m0), m1 = lo2(m.m1) + hi2(m.m1);
    s0 = fmaf(m0, dx, s0);
    s1 += m1;
    s2 = fmaf(m1, dx, s2);
    s3 = fmaf(m0 * dx, dx, s3);
    s4 += lo2(m.m2) + hi2(m.m2);
  }
  const float w = -ct.x * ct.y;
  float* out = p.light_geom + 8 * (size_t)p.order[rank];
  red_add2(out, 0.f, w * s0);
  red_add2(out + 2, w * s1, w * s2);
  red_add2(out + 4, w * s3, w * s4);
}

__global__ void __launch_bounds__(kBwdWarps * 32) k_shadow_bwd_stopped(const BwdParams p) {
  __shared__ StopSmem smem[kBwdWarps];
  StopSmem& S = smem[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const uint32_t total = p.counts[1], below = (1u << lane) - 1u;
  uint32_t ticket;
  while (next_item(p.ticket + 2, total, lane, ticket)) {
    const uint4 d = p.desc[p.dead_list[ticket]];
    const int tile = (int)(d.x & ~kSegLast), tx = tile % p.gx, ty = tile / p.gx;
    const int ncol = min(kTile, p.W - tx * kTile), nrow = min(kTile, p.H - ty * kTile);
    for (uint32_t rs = d.y; rs < d.z; rs += kStopScan) {
      int n = 0;
      __syncwarp();
#pragma unroll
      for (int c = 0; c < kStopScan / 32; ++c) {
        const uint32_t i = rs + 32 * c + lane;
        uint32_t bits = i < d.z ? p.pass_mask[i] : 0u;
        if (bits) {
          const float2 ct = p.ct[p.list[i]];
          if (ct.x * ct.y == 0.f) bits = 0u;
        }
        const uint32_t m0 = __ballot_sync(0xffffffffu, bits & 0x3u), m1 = __ballot_sync(0xffffffffu, bits & 0xCu);
        if (bits & 0x3u) S.unit[n + __popc(m0 & below)] = (uint16_t)(32 * c + lane);
        n += __popc(m0);
        if (bits & 0xCu) S.unit[n + __popc(m1 & below)] = (uint16_t)((32 * c + lane) | 0x100);
        n += __popc(m1);
      }
      __syncwarp();
      for (int u = lane; u < n; u += 32) {
        const int code = S.unit[u];
        stopped_unit(p, rs + (code & 0xFF), code >> 8, (float)(tx * kTile), (float)(ty * kTile), ncol, nrow);
      }
    }
  }
}

// Blocks per SM of the persistent kernels (per device, looked up once).
struct BwdOccupancy {
  int sums, open, stopped;
};
BwdOccupancy bwd_occupancy() {
  static DeviceOnce once;
  static BwdOccupancy occ[kMaxDevices];
  int d = 0;
  cudaGetDevice(&d);
  once.run([d] {
    bool ok = true;
    for (const void* k : {(const void*)k_shadow_bwd_sums, (const void*)k_shadow_bwd})
      ok = ok && cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout,
                                      (int)cudaSharedmemCarveoutMaxShared) == cudaSuccess;
    if (d >= 0 && d < kMaxDevices) {
      BwdOccupancy& o = occ[d];
      ok = ok &&
           cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o.sums, k_shadow_bwd_sums, kBwdWarps * 32, 0) == cudaSuccess &&
           cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o.open, k_shadow_bwd, kBwdWarps * 32, 0) == cudaSuccess &&
           cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o.stopped, k_shadow_bwd_stopped, kBwdWarps * 32, 0) ==
               cudaSuccess;
    }
    return ok;
  });
  BwdOccupancy o{1, 1, 1};
  if (d >= 0 && d < kMaxDevices) o = occ[d];
  o.sums = o.sums < 1 ? 1 : o.sums;
  o.open = o.open < 1 ? 1 : o.open;
  o.stopped = o.stopped < 1 ? 1 : o.stopped;
  return o;
}

}  // namespace

void launch_shadow_backward(const FrameArgs& f, const ShadowBwdArgs& a, cudaStream_t s, cudaStream_t side) {
  const Workspace& L = *f.L;
  unsigned char* ws = f.ws;
  const int n = f.sc.n, fin = (L.ntiles <= 256 ? 1 : 2) & 1;
  BwdParams p;
  p.list = at<uint32_t>(ws, L.sp[1].tv[fin]);
  p.tile_start = at<uint32_t>(ws, L.sp[1].tile_start);
  p.rrec = at<SplatRec>(ws, L.sp[1].rrec);
  p.order = at<uint32_t>(ws, L.sp[1].sv[1]);
  p.kbound = at<uint32_t>(ws, L.sp[1].tv[1 - fin]);
  p.tile_order = at<uint32_t>(ws, L.tile_order[1]);
  p.lvl_off = at<uint32_t>(ws, L.seg_lvl);
  p.counts = p.lvl_off + kSegLevels + 4;
  p.desc = at<uint4>(ws, L.seg_desc);
  p.open_list = at<uint32_t>(ws, L.seg_lists);
  p.dead_list = p.open_list + shadow_seg_items(L.ntiles, L.cap);
  p.pub_a = at<float>(ws, L.seg_pub);
  p.pub_flag = at<uint32_t>(ws, L.seg_flag);
  p.pass_mask = at<uint8_t>(ws, L.sp[1].tk[1 - fin]);
  p.light_final = at<float>(ws, L.light_final);
  p.light_stop = at<uint32_t>(ws, L.light_stop);
  p.ct = a.ct;
  p.seg_sum = at<float>(ws, L.seg_sum);
  p.ticket = a.ticket;
  p.light_geom = a.light_geom;
  p.W = L.width; p.H = L.height; p.gx = L.gx; p.ntiles = L.ntiles;
  p.amax = f.opts.alpha_max;
  const BwdOccupancy o = bwd_occupancy();
  const int nsm = device_sm_count();
  k_bwd_coef<<<(n + 255) / 256, 256, 0, s>>>(p.order, a.dT, at<float>(ws, L.shadow_den), at<float>(ws, L.T), a.ct, a.ticket + 3, n);
  if (side != s) {
    cudaEventRecord(a.fork, s);
    cudaStreamWaitEvent(side, a.fork, 0);
  }
  k_shadow_bwd_stopped<<<nsm * o.stopped, kBwdWarps * 32, 0, side>>>(p);
  k_shadow_bwd_sums<<<nsm * o.sums, kBwdWarps * 32, 0, s>>>(p);
  launch_after(k_shadow_bwd_suffix, (L.ntiles + 3) / 4, 128, 0, s, p);
  launch_after(k_shadow_bwd, nsm * o.open, kBwdWarps * 32, 0, s, p);
  count_launch(5);
}

}  // namespace gs3
