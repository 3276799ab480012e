// K6, K7: shadow splatting (Sec. 4.2, Fig. 3) and K9: camera compositing
// (Sec. 3, Eq. 2) with the deferred per-pixel combination (Sec. 4).
//
// Both composites stream a 16x16 tile's depth-ordered list through shared
// memory as tile-relative entries (splat_eval.cuh): the shadow composite
// over segments of the list with eight rays per lane, the camera composite
// with a warp per 8x8 quadrant (two pixels per lane, 32 records at a time).
#include "gs3_internal.cuh"
#include "shadow_seg.cuh"

namespace gs3 {
namespace {

// ---------------------------------------------------------------------------
// K6: shadow composite.
// For every shadow ray m (light pixel) and every list entry j that passes the
// alpha test, T_m(j) = prod (1 - alpha_k,m) over passing k with
// d_k < d_j - bias.  The list is ordered by distance, so the occluders of j
// form a prefix of the tile's list; its end K(j) is precomputed per entry
// (k_bound_starts, k_bound_rest, from each Gaussian's bound among the depth
// ranks) and is non-decreasing in j.
//
// Work is split into segments of a tile's list: segment s holds receivers
// [R_s, R_s+1) (32 to 256 entries; the last takes the rest) and needs the
// occluders [C_s, C_s+1) on top of the product A(C_s) that every ray carries
// into it, with C_s = K(R_s).  Persistent warps take one segment at a time
// from a ticket counter, in three kernels:
//   K6a  computes each of the 256 rays' product Q over the occluder range,
//        takes A(C_s) from the segment before it (published by that warp; a
//        bounded wait) and publishes A(C_s+1) = A(C_s) Q for the next one.  Q
//        comes before the wait, so the segments of a long list run side by
//        side and only the last step is chained.
//   K6b  walks the receivers of the segments that some ray enters open, with
//        the products P = A(C_s) q, q the running product of the range's
//        occluders, summing (beta P, beta) per receiver into the (tile,
//        Gaussian) partials.
//   K6c  adds up beta alone in the segments that every ray enters stopped.
//
// Ray stop: a ray takes occluders only while its product P stays >=
// kShadowStop; the occluder that takes it below is the ray's last, and the
// receivers behind it see 0 (an exact product there is below kShadowStop as
// well).  K6a decides which segment a ray stops in (it publishes 0 from there
// on) and that segment's K6b records where: at the occluder whose factor takes
// P below the stop or, should the two products round to different sides of
// it, at the end of the range.  Thread layout as in the splat evaluation:
// lane l owns column l & 15, rows (l >> 4) + 2 i, i = 0..7, which is ray
// 32 i + l of the tile.
//
// Bound: issue slots and the FMA pipe (every pixel test is a power, an ex2 and
// a select).  So rays go in pairs through the packed FP32 instructions, an
// occluder updates P alone (a retired ray holds -0.0, which no factor changes
// and an unsigned minimum passes over, so no pixel needs a test of its own),
// and receivers and occluders come from one merged list, staged 32 at a time.
// Object workload (300k Gaussians, 800 x 800, 12.8 M light entries): K6a 0.377
// -> 0.272 ms, K6b 0.784 -> 0.466 ms, K6c 0.326 -> 0.165 ms (entries picked
// by their Gaussian's flags before their records are read, and only of
// Gaussians with a positive numerator), reduction 0.034 -> 0.020 ms; at 1 M and
// 1024 x 1024 K6a 1.095 -> 0.758, K6b 2.119 -> 1.154, K6c 2.081 -> 0.896 ms.
// ---------------------------------------------------------------------------
constexpr int kSegWarps = 4;        // independent warps per block
constexpr int kOccWin = 32;         // occluder window
constexpr int kSegSpin = 1 << 20;   // polls of a predecessor's publication before giving up


struct ShadowParams {
  const uint32_t* list;
  const uint32_t* tile_start;
  const SplatRec* rrec;
  const uint32_t* off;
  const uint32_t* kbound;
  const uint32_t* tile_order;  // tiles by decreasing segment count
  const uint32_t* lvl_off;     // [kSegLevels + 1]: first work item of each segment level
  uint32_t* ticket;            // [3] work counters of K6a, K6b and K6c (zeroed per frame)
  uint32_t* counts;            // [2] items in open_list and dead_list (zeroed per frame)
  uint4* desc;                 // [item]: tile and kSegLast, first and past-the-last receiver, preceding item
  uint32_t* open_list;         // items some ray enters open (K6b's), in no particular order
  uint32_t* dead_list;         // items every ray enters stopped (K6c's)
  float* pub_a;                // [link_slot][256]: A(C_s+1) published by an item
  uint32_t* pub_flag;          // [item]: 0 not yet, 1 published, 2 published and every ray stopped
  uint8_t* pass_mask;  // per list entry of a stopped segment: halves with a passing pixel, 0x3 rows 0-7, 0xC rows 8-15
  float2* partial;
  float* light_final;     // per light pixel: the product where the ray ended
  uint32_t* light_stop;   // per light pixel: 1 + index of the occluder that stopped it, or kNoStop
  uint32_t* status;
  uchar2* rank_flags;  // per light rank: (some receiver's sum beta P > 0, some pixel known to pass)
  int W, H, gx;
  float amax;
};

constexpr int kRowPad = 17;                 // a receiver's row of 16 lane sums, padded

struct ShadowSmem {  // one warp's
  StagedEntries e;
  f32x2 red[32][kRowPad];  // per receiver of the batch, per lane pair: (num, den)
};

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* a) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(uint32_t* a, uint32_t v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(a), "r"(v) : "memory");
}

// A receiver's four rays of one half: den += beta and num += beta P.
template <int H>
__device__ __forceinline__ void recv_half(const f32x2 (&ly)[kPx / 2], const f32x2 (&P)[kPx / 2], const ColTerms& e,
                                          f32x2& num, f32x2& den) {
#pragma unroll
  for (int q = 2 * H; q < 2 * H + 2; ++q) {
    const f32x2 b = beta2_at(e, ly[q]);
    den = add2(den, b);
    num = fma2(b, P[q], num);
  }
}

// The smallest product among the lane's rays, as bits: a retired ray holds
// -0.0, whose bits are above every positive product's.
__device__ __forceinline__ uint32_t min_bits(const f32x2 (&P)[kPx / 2]) {
  uint32_t m = __vimin3_u32((uint32_t)P[0], (uint32_t)(P[0] >> 32), (uint32_t)P[1]);
  m = __vimin3_u32(m, (uint32_t)(P[1] >> 32), (uint32_t)P[2]);
  m = __vimin3_u32(m, (uint32_t)(P[2] >> 32), (uint32_t)P[3]);
  return min(m, (uint32_t)(P[3] >> 32));
}

// K6a: A(C_s+1) of every segment but a tile's last, chained from A(C_s).
template <typename L>
__device__ __forceinline__ void chain_item(const ShadowParams& p, const L& link_slot, uint32_t w, StagedEntries& S, int lane) {
  const float lx = (lane & 15) + 0.5f, omin = 1.f - p.amax;
  const SegItem it = seg_item(p, w, lane);
  if (it.last) return;  // nothing follows it
  const float ox = (float)(it.tx * kTile), oy = (float)(it.ty * kTile);
  f32x2 ly[kPx / 2];
  lane_rows(lane, it.rows_in, ly);
  // A(C_s): known now for the first segment, or when the predecessor
  // published already; until then A = 1 stands in (A <= 1)
  uint32_t flag = 1u;
  if (!it.first && lane == 0) flag = ld_acquire(p.pub_flag + it.wpred);
  flag = __shfl_sync(0xffffffffu, flag, 0);
  __syncwarp();  // orders every lane's reads after lane 0's acquire
  bool known = flag != 0u;
  f32x2 A[kPx / 2];
  load_entering(p, link_slot, it.first || !known, it.wpred, flag, lane, it.rows_in, A);
  // the range's products Q; once no ray's A Q stays at the stop the rest of
  // the range changes nothing (each ray stops in it either way)
  f32x2 Q[kPx / 2];
#pragma unroll
  for (int q = 0; q < kPx / 2; ++q) Q[q] = dup2(1.f);
  uint32_t live = live_halves(A);
  for (uint32_t wb = it.C0; wb < it.C1 && live; wb += kOccWin) {
    if (!known) {  // the predecessor may have published meanwhile
      uint32_t fl = 0u;
      if (lane == 0) fl = ld_acquire(p.pub_flag + it.wpred);
      fl = __shfl_sync(0xffffffffu, fl, 0);
      __syncwarp();
      if (fl != 0u) {
        known = true;
        load_entering(p, link_slot, false, it.wpred, fl, lane, it.rows_in, A);
      }
    }
    f32x2 AQ[kPx / 2];
#pragma unroll
    for (int q = 0; q < kPx / 2; ++q) AQ[q] = mul2(A[q], Q[q]);
    live = live_halves(AQ);
    if (!live) break;
    const int wc = (int)min((uint32_t)kOccWin, it.C1 - wb);
    __syncwarp();
    if (lane < wc) stage_entry(p.rrec[p.list[wb + lane]], ox, oy, S, lane);
    __syncwarp();
    for (int t = 0; t < wc; ++t) {
      const float2 gb = S.gb[t];
      const uint32_t bits = __float_as_uint(gb.y) & live;
      if (!bits) continue;
      const ColTerms e = col_terms(lx, S, t);
      if (bits & 0x3u) occ_half<0>(ly, Q, e, gb.x, omin);
      if (bits & 0xCu) occ_half<1>(ly, Q, e, gb.x, omin);
    }
  }
  // A(C_s) from the predecessor (bounded wait), then A(C_s+1) for the successor
  if (!known) {
    uint32_t fl = 0u;
    if (lane == 0) {
      int spins = 0;
      while ((fl = ld_acquire(p.pub_flag + it.wpred)) == 0u) {
        if (++spins > kSegSpin) {
          atomicCAS(p.status, 0u, (uint32_t)GS3_ERR_TIMEOUT);
          fl = 2u;  // give up: the frame is reported invalid, the warp finishes
          break;
        }
        __nanosleep(64);
      }
    }
    fl = __shfl_sync(0xffffffffu, fl, 0);
    __syncwarp();
    load_entering(p, link_slot, false, it.wpred, fl, lane, it.rows_in, A);
  }
  const bool dead_in = live_halves(A) == 0u;
  bool any = false;
  float* out = p.pub_a + link_slot(w) + lane;
#pragma unroll
  for (int q = 0; q < kPx / 2; ++q) {
    const f32x2 AQ = mul2(A[q], Q[q]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float a = h ? hi2(AQ) : lo2(AQ);
      if (!(a >= kShadowStop)) a = 0.f;  // the ray stopped in this range or before it
      any |= a != 0.f;
      if (!dead_in) out[64 * q + 32 * h] = a;
    }
  }
  const bool any_out = __any_sync(0xffffffffu, any);
  __threadfence();  // every lane's products before the flag
  __syncwarp();
  if (lane == 0) st_release(p.pub_flag + w, any_out ? 1u : 2u);
}

// The work items of a batch of frames: the tickets run over every frame's
// items in turn; locate() maps a ticket to its frame and the frame's item
// (or, for K6b and K6c, its place in the frame's list of such items).
enum { kAllItems = 0, kOpenItems = 1, kDeadItems = 2 };
__device__ __forceinline__ uint32_t item_count(const ShadowParams& p, int kind) {
  return kind == kAllItems ? p.lvl_off[kSegLevels] : p.counts[kind - 1];
}
__device__ __forceinline__ uint32_t batch_items(const ShadowParams* reqs, int nreq, int kind) {
  uint32_t t = 0;
  for (int r = 0; r < nreq; ++r) t += item_count(reqs[r], kind);
  return t;
}
__device__ __forceinline__ int locate(const ShadowParams* reqs, int nreq, int kind, uint32_t& w) {
  int r = 0;
  for (; r < nreq - 1; ++r) {
    const uint32_t t = item_count(reqs[r], kind);
    if (w < t) break;
    w -= t;
  }
  return r;
}

// Links from shared memory where they are used, which leaves k_shadow_chain its registers
struct SharedLinks {
  const volatile Links* at;
  __device__ __forceinline__ size_t operator()(uint32_t w) const {
    return (size_t)(w < at->more ? w : w - at->gap) * 256;
  }
};

// One frame (p) or a batch of nreq frames (reqs, in device memory; p is the
// first, whose tickets the batch shares).  5 blocks per SM: 0.272 ms against
// 0.279 at 4, 0.287 at 6 and 0.314 at 8.  Past 88 registers they leave too few for
// another stream's blocks (eight lights side by side: 2,630 us with 96, 2,615 with 88).
template <bool BATCH>
__global__ void __launch_bounds__(kSegWarps * 32, 5) k_shadow_chain(const ShadowParams p, const ShadowParams* reqs,
                                                                    int nreq) {
  after_previous();
  __shared__ StagedEntries smem[kSegWarps];
  __shared__ Links links[kSegWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  StagedEntries& S = smem[warp];
  const uint32_t total = BATCH ? batch_items(reqs, nreq, kAllItems) : item_count(p, kAllItems);
  if (!BATCH && lane == 0) links[warp] = frame_links(p.lvl_off);
  __syncwarp();
  uint32_t w;
  while (next_item(p.ticket, total, lane, w)) {
    if (BATCH) {
      const int r = locate(reqs, nreq, kAllItems, w);
      chain_item(reqs[r], frame_links(reqs[r].lvl_off), w, S, lane);
    } else {
      chain_item(p, SharedLinks{links + warp}, w, S, lane);
    }
  }
}

// K6c: the receivers of the segments every ray of which stopped before the
// segment (A(C_s) = 0 throughout, as K6a published).  The products are 0,
// so a receiver needs only its beta sum over the tile, which depends on no
// other entry, and only if its Gaussian's numerator is not 0: K6b marked the
// Gaussians with a positive one (rank_flags.x).  Of any other Gaussian the
// shadow value is 0 if some pixel passes and 1 if none does, so its entries
// are needed only until one is known to pass (rank_flags.y: K6b or
// k_dead_probe found one, or a unit here did), and its partials are neither
// written nor read.  A warp takes a segment, picks the entries it needs from
// their flags (before it reads any record), stages up to kDeadBatch of them,
// lists their (receiver, half) units (the halves their box and ellipse
// reach), and each lane walks the 16 x 8 pixels of one unit at a time, with
// the power arithmetic of the ray layout (pixel centres x + 0.5, y + 0.5);
// the two halves of a receiver are then added in a fixed order.  Which
// entries of an unmarked Gaussian are evaluated depends on timing; T does not.
constexpr int kDeadBatch = 128;
constexpr int kDeadWarps = 4;
constexpr int kDeadScan = 256;  // entries whose flags are read at a time

struct DeadSmem {  // one warp's
  float4 e0[kDeadBatch], e1[kDeadBatch];
  float den[2][kDeadBatch];
  uint32_t slot[kDeadBatch];      // the receiver's partial slot
  uint32_t rank[kDeadScan];       // needed entries: depth rank, bit 31 set if K6b marked it
  uint8_t at[kDeadScan];          // and their places among the entries read
  uint16_t unit[2 * kDeadBatch];  // receiver (bits 0-7) and half (bit 8) of each unit
};

// The beta sum of one receiver entry over the 16 x 8 pixels of half h of an
// interior tile, column by column, pixel pairs in packed registers.
__device__ __forceinline__ float dead_half(const float4 e0, const float4 e1, int h) {
  f32x2 dy[4];
  const float y0 = 8.f * h + 0.5f;
#pragma unroll
  for (int q = 0; q < 4; ++q) dy[q] = pk2((y0 + 2.f * q) - e0.y, (y0 + 2.f * q + 1.f) - e0.y);
  const f32x2 c = dup2(e0.w);
  f32x2 den = 0ull;
  float fx = 0.5f;
#pragma unroll 1
  for (int x = 0; x < kTile; ++x) {
    const float dx = fx - e0.x;
    fx += 1.f;
    const f32x2 sx = dup2((e0.z * dx) * dx), v = dup2(e1.x * dx);
#pragma unroll
    for (int q = 0; q < 4; ++q) den = add2(den, beta2_of(power2_pair(dy[q], c, v, sx), e1.y));
  }
  return lo2(den) + hi2(den);
}

// the same over the pixels of half h that lie inside the image (edge tiles)
__device__ __forceinline__ float dead_half_edge(const float4 e0, const float4 e1, int h, int ncol, int nrow) {
  float den = 0.f, fx = 0.5f;
  const int y1 = min(8 * h + 8, nrow);
  for (int x = 0; x < ncol; ++x, fx += 1.f) {
    const float dx = fx - e0.x;
    const float sx = (e0.z * dx) * dx, v = e1.x * dx;
    float fy = 8.f * h + 0.5f;
    for (int y = 8 * h; y < y1; ++y, fy += 1.f) {
      const float dy = fy - e0.y;
      den += beta_of(fmaf(dy, fmaf(e0.w, dy, v), sx), e1.y);
    }
  }
  return den;
}

__device__ __forceinline__ void dead_item(const ShadowParams& p, uint32_t w, DeadSmem& D, int lane) {

    const uint4 d = p.desc[w];
    const int tile = (int)(d.x & ~kSegLast);
    const int tx = tile % p.gx, ty = tile / p.gx;
    const float ox = (float)(tx * kTile), oy = (float)(ty * kTile);
    const uint32_t R0 = d.y, R1 = d.z;
    const int ncol = min(kTile, p.W - tx * kTile), nrow = min(kTile, p.H - ty * kTile);
    const bool interior = ncol == kTile && nrow == kTile;
    const uint32_t below = (1u << lane) - 1u;
    for (uint32_t rs = R0; rs < R1; rs += kDeadScan) {
      // the entries needed, from their Gaussians' flags
      uint32_t rank[kDeadScan / 32];
      uchar2 fl[kDeadScan / 32];
#pragma unroll
      for (int c = 0; c < kDeadScan / 32; ++c) {
        const uint32_t i = rs + 32 * c + lane;
        rank[c] = i < R1 ? p.list[i] : 0u;
      }
#pragma unroll
      for (int c = 0; c < kDeadScan / 32; ++c) {
        // the second flag may be set meanwhile: read past the L1
        const uint16_t f = __ldcg(reinterpret_cast<const uint16_t*>(p.rank_flags) + rank[c]);
        fl[c] = make_uchar2((uint8_t)f, (uint8_t)(f >> 8));
      }
      int nq = 0;
      __syncwarp();
#pragma unroll
      for (int c = 0; c < kDeadScan / 32; ++c) {
        const uint32_t i = rs + 32 * c + lane;
        const bool need = i < R1 && (fl[c].x || !fl[c].y);
        const uint32_t m = __ballot_sync(0xffffffffu, need);
        if (need) {
          D.rank[nq + __popc(m & below)] = rank[c] | (fl[c].x ? 0x80000000u : 0u);
          D.at[nq + __popc(m & below)] = (uint8_t)(32 * c + lane);
        } else if (i < R1) {
          p.pass_mask[i] = 0;
        }
        nq += __popc(m);
      }
      __syncwarp();
      for (int q0 = 0; q0 < nq; q0 += kDeadBatch) {
        const int rc = min(kDeadBatch, nq - q0);
        // stage the receivers; list the units of half 0, then of half 1
        int n0 = 0, n1 = 0;
        uint32_t box[kDeadBatch / 32];
#pragma unroll
        for (int c = 0; c < kDeadBatch / 32; ++c) {
          const int t = 32 * c + lane;
          box[c] = 0u;
          if (t < rc) {
            const uint32_t r = D.rank[q0 + t] & 0x7FFFFFFFu;
            const SplatRec q = p.rrec[r];
            float4 e0, e1;
            make_entry(q, ox, oy, e0, e1);
            box[c] = __float_as_uint(e1.w) & ellipse_halves(e0, e1);
            D.e0[t] = e0;
            D.e1[t] = e1;
            D.slot[t] = p.off[r] + (uint32_t)((ty - q.r.y) * (q.r.z - q.r.x + 1) + (tx - q.r.x));
          }
          n0 += __popc(__ballot_sync(0xffffffffu, (box[c] & 0x3u) != 0u));
          n1 += __popc(__ballot_sync(0xffffffffu, (box[c] & 0xCu) != 0u));
        }
        int b0 = 0, b1 = n0;  // next unit slot of each half
#pragma unroll
        for (int c = 0; c < kDeadBatch / 32; ++c) {
          const int t = 32 * c + lane;
          const uint32_t m0 = __ballot_sync(0xffffffffu, (box[c] & 0x3u) != 0u);
          const uint32_t m1 = __ballot_sync(0xffffffffu, (box[c] & 0xCu) != 0u);
          if (box[c] & 0x3u) D.unit[b0 + __popc(m0 & below)] = (uint16_t)t;
          if (box[c] & 0xCu) D.unit[b1 + __popc(m1 & below)] = (uint16_t)(t | 0x100);
          b0 += __popc(m0);
          b1 += __popc(m1);
          if (t < rc) D.den[0][t] = D.den[1][t] = 0.f;
        }
        __syncwarp();
        const int nu = n0 + n1;
        for (int u = lane; u < nu; u += 32) {
          const int code = D.unit[u];
          const int t = code & 0xFF, h = code >> 8;
          const float4 e0 = D.e0[t], e1 = D.e1[t];
          D.den[h][t] = interior ? dead_half(e0, e1, h) : dead_half_edge(e0, e1, h, ncol, nrow);
        }
        __syncwarp();
        for (int t = lane; t < rc; t += 32) {
          const float d0 = D.den[0][t], d1 = D.den[1][t];
          const uint32_t r = D.rank[q0 + t];
          const bool live = (r >> 31) != 0u;
          if (live) p.partial[D.slot[t]] = make_float2(0.f, d0 + d1);
          else if (d0 + d1 > 0.f) reinterpret_cast<volatile uchar2*>(p.rank_flags)[r].y = 1;
          p.pass_mask[rs + D.at[q0 + t]] = live ? (uint8_t)((d0 > 0.f ? 0x3u : 0u) | (d1 > 0.f ? 0xCu : 0u)) : 0;
        }
        __syncwarp();
      }
    }
  }

// Before K6c: a Gaussian of which K6b found neither a positive numerator nor
// a passing pixel has its pixel nearest the splat centre tested with K6c's
// exact arithmetic (the entry of that tile, the pixel's power against the
// threshold); if it passes, K6c can skip every entry of the Gaussian.  Only a
// pixel that K6c itself would evaluate counts: inside the image, in a tile of
// the Gaussian's rectangle, in a half its box and ellipse reach.
__global__ void k_dead_probe(const ShadowParams p, int n) {
  after_previous();
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n || p.rank_flags[r].x || p.rank_flags[r].y) return;
  const SplatRec q = p.rrec[r];
  if (q.r.x < 0) return;  // not in the light view
  const float cx = q.a.x + q.b.w, cy = q.a.y + q.c.x;
  if (!(cx >= 0.f && cy >= 0.f && cx < (float)p.W && cy < (float)p.H)) return;
  const int px = (int)cx, py = (int)cy;
  const int tx = px / kTile, ty = py / kTile;
  if (tx < q.r.x || tx > q.r.z || ty < q.r.y || ty > q.r.w) return;
  float4 e0, e1;
  make_entry(q, (float)(tx * kTile), (float)(ty * kTile), e0, e1);
  const int x = px - tx * kTile, y = py - ty * kTile, h = y >> 3;
  // K6c evaluates the half only if the entry's box and ellipse reach it
  if (!(__float_as_uint(e1.w) & ellipse_halves(e0, e1) & (3u << (2 * h)))) return;
  const float dx = (0.5f + (float)x) - e0.x;
  const float sx = (e0.z * dx) * dx, v = e1.x * dx;
  const float dy = ((8.f * h + 0.5f) + (float)(y & 7)) - e0.y;
  const float pw = fmaf(dy, fmaf(e0.w, dy, v), sx);
  if (pw >= e1.y) p.rank_flags[r].y = 1;
}

template <bool BATCH>
__global__ void __launch_bounds__(kDeadWarps * 32, 7) k_shadow_dead(const ShadowParams p, const ShadowParams* reqs,
                                                                    int nreq) {
  after_previous();
  __shared__ DeadSmem smem[kDeadWarps];
  DeadSmem& D = smem[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const uint32_t total = BATCH ? batch_items(reqs, nreq, kDeadItems) : item_count(p, kDeadItems);
  uint32_t w;
  while (next_item(p.ticket + 2, total, lane, w)) {
    if (BATCH) {
      const int r = locate(reqs, nreq, kDeadItems, w);
      dead_item(reqs[r], reqs[r].dead_list[w], D, lane);
    } else {
      dead_item(p, p.dead_list[w], D, lane);
    }
  }
}

// K6b: the receivers of a segment that some ray enters open, with the
// products P = A(C_s) times the running product of the range's occluders.
// The occluders of the range and the receivers are merged into one sequence
// (occluder k before receiver j where k < K(j)) and taken 32 at a time: the
// place of receiver j is (j - R0) + (K(j) - C0), the other places are the
// occluders', so each lane finds and stages one entry of the batch; the warp
// then walks the 32 entries.  A receiver's per-lane sums go to a row of shared
// memory; after the walk the lane that staged it adds up the row (in a fixed
// order) and writes its partial.
__device__ __forceinline__ void live_item(const ShadowParams& p, const Links& link_slot, uint32_t w, ShadowSmem& S, int lane) {
  const int lxi = lane & 15, lyi = lane >> 4;
  const float lx = lxi + 0.5f, omin = 1.f - p.amax;
  const SegItem it = seg_item(p, w, lane);
  const float ox = (float)(it.tx * kTile), oy = (float)(it.ty * kTile);
  f32x2 ly[kPx / 2];
  lane_rows(lane, it.rows_in, ly);
  // A(C_s) and A(C_s+1), as K6a published them
  const uint32_t fl_in = it.first ? 1u : __ldcg(p.pub_flag + it.wpred);
  const uint32_t fl_out = it.last ? 1u : __ldcg(p.pub_flag + w);
  f32x2 P[kPx / 2];
  load_entering(p, link_slot, it.first, it.wpred, fl_in, lane, it.rows_in, P);
  uint32_t live = live_halves(P);
  // where a ray ended is recorded by the segment K6a has it stop in, or by
  // the tile's last one (ends: the lane's rays that this segment records)
  uint32_t ends = 0u;
  const float* handed_on = p.pub_a + (it.last ? 0 : link_slot(w)) + lane;
#pragma unroll
  for (int i = 0; i < kPx; ++i) {
    const float a = i & 1 ? hi2(P[i / 2]) : lo2(P[i / 2]);
    bool end = a >= kShadowStop;
    if (end && !it.last && fl_out != 2u) end = __ldcg(handed_on + 32 * i) == 0.f;
    ends |= end ? 1u << i : 0u;
  }
#pragma unroll
  for (int q = 0; q < kPx / 2; ++q)  // rays that are stopped or outside the image hold -0.0
    P[q] = pk2(lo2(P[q]) >= kShadowStop ? lo2(P[q]) : -0.f, hi2(P[q]) >= kShadowStop ? hi2(P[q]) : -0.f);
  const size_t pix0 = (size_t)(it.ty * kTile + lyi) * p.W + it.tx * kTile + lxi;
  auto record = [&](int i, float a, uint32_t lim) {  // ray i ended with product a; it took the occluders below lim
    p.light_final[pix0 + (size_t)2 * i * p.W] = a;
    p.light_stop[pix0 + (size_t)2 * i * p.W] = lim;
  };
  // occluders past the last receiver's are walked only for rays that stop in
  // the rest of the range
  const bool tail = !it.last && __any_sync(0xffffffffu, ends != 0u);
  uint32_t j = it.R0, k = it.C0;
  uint32_t kend = it.R1 > it.R0 ? (tail ? it.C1 : p.kbound[it.R1 - 1]) : it.C0;
  for (;;) {
    if (!live) kend = k;  // no ray takes occluders any more
    const uint32_t left = (it.R1 - j) + (kend - k);
    if (left == 0u) break;
    const int nops = (int)min(32u, left);
    // the receivers' places among the batch's 32
    uint32_t pos = 32u;
    if (j + lane < it.R1) pos = live ? lane + (p.kbound[j + lane] - k) : (uint32_t)lane;
    const uint32_t M = __reduce_or_sync(0xffffffffu, pos < 32u ? 1u << pos : 0u);
    const int nrecv = __popc(M), mine = __popc(M & ((1u << lane) - 1u));
    const bool is_recv = (M >> lane) & 1u;
    uint32_t rank = 0u, slot = 0u;
    __syncwarp();  // the previous batch is consumed
    if (lane < nops) {
      const uint32_t idx = is_recv ? j + mine : k + (lane - mine);
      rank = p.list[idx];
      const SplatRec q = p.rrec[rank];
      stage_entry(q, ox, oy, S.e, lane);
      if (is_recv) {
        slot = p.off[rank] + (uint32_t)((it.ty - q.r.y) * (q.r.z - q.r.x + 1) + (it.tx - q.r.x));
      }
    }
    __syncwarp();
    int row = 0;
    for (int t = 0; t < nops; ++t) {
      const float2 gb = S.e.gb[t];
      const uint32_t bits = __float_as_uint(gb.y);
      if ((M >> t) & 1u) {
        f32x2 num = 0ull, den = 0ull;
        if (bits) {
          const ColTerms e = col_terms(lx, S.e, t);
          if (bits & 0x3u) recv_half<0>(ly, P, e, num, den);
          if (bits & 0xCu) recv_half<1>(ly, P, e, num, den);
        }
        const float n1 = lo2(num) + hi2(num), d1 = lo2(den) + hi2(den);
        const float n2 = __shfl_xor_sync(0xffffffffu, n1, 16), d2 = __shfl_xor_sync(0xffffffffu, d1, 16);
        S.red[row][lxi] = pk2(n1 + n2, d1 + d2);  // lanes l and l + 16 hold the same sums
        ++row;
      } else {
        const uint32_t b = bits & live;
        if (!b) continue;
        const ColTerms e = col_terms(lx, S.e, t);
        if (b & 0x3u) occ_half<0>(ly, P, e, gb.x, omin);
        if (b & 0xCu) occ_half<1>(ly, P, e, gb.x, omin);
        // the occluder that takes a ray's product below the stop is its last:
        // P becomes -0.0, where it stays, and the receivers behind see 0
        if (min_bits(P) < __float_as_uint(kShadowStop)) {
          const uint32_t lim = k + (uint32_t)(t - row) + 1u;
#pragma unroll
          for (int i = 0; i < kPx; ++i) {
            const float a = i & 1 ? hi2(P[i / 2]) : lo2(P[i / 2]);
            if (__float_as_uint(a) < __float_as_uint(kShadowStop)) {
              if (ends & (1u << i)) record(i, a, lim);
              ends &= ~(1u << i);
              P[i / 2] = i & 1 ? pk2(lo2(P[i / 2]), -0.f) : pk2(-0.f, hi2(P[i / 2]));
            }
          }
        }
      }
    }
    __syncwarp();
    if (is_recv && lane < nops) {
      f32x2 s0 = S.red[mine][0], s1 = S.red[mine][1];
#pragma unroll
      for (int c = 2; c < 16; c += 2) {
        s0 = add2(s0, S.red[mine][c]);
        s1 = add2(s1, S.red[mine][c + 1]);
      }
      const f32x2 nd = add2(s0, s1);
      p.partial[slot] = make_float2(lo2(nd), hi2(nd));
      if (lo2(nd) > 0.f) p.rank_flags[rank].x = 1;
      if (hi2(nd) > 0.f) p.rank_flags[rank].y = 1;
    }
    j += nrecv;
    k += nops - nrecv;
    live = live_halves(P);
  }
  // rays that end past this segment's last occluder
#pragma unroll
  for (int i = 0; i < kPx; ++i)
    if (ends & (1u << i)) record(i, i & 1 ? hi2(P[i / 2]) : lo2(P[i / 2]), it.last ? kNoStop : it.C1);
}

// 6 blocks per SM (80 registers): 5 took 5 % longer and 4 took 16 % longer
// (object workload).
template <bool BATCH>
__global__ void __launch_bounds__(kSegWarps * 32, 6) k_shadow(const ShadowParams p, const ShadowParams* reqs, int nreq) {
  after_previous();
  __shared__ ShadowSmem smem[kSegWarps];
  ShadowSmem& S = smem[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const uint32_t total = BATCH ? batch_items(reqs, nreq, kOpenItems) : item_count(p, kOpenItems);
  const Links links = frame_links(p.lvl_off);
  uint32_t w;
  while (next_item(p.ticket + 1, total, lane, w)) {
    if (BATCH) {
      const int r = locate(reqs, nreq, kOpenItems, w);
      live_item(reqs[r], frame_links(reqs[r].lvl_off), reqs[r].open_list[w], S, lane);
    } else {
      live_item(p, links, p.open_list[w], S, lane);
    }
  }
}

// The ranks that shadow rank r's Gaussian are those of smaller distance:
// bound[r] = the first rank whose distance is >= d_r - bias (at most r).  The
// depth sort leaves the distances' bit patterns in rank order.  The ranks' flags
// are cleared on the way.
__global__ void __launch_bounds__(256) k_rank_bound(const float* __restrict__ dist, uint32_t* __restrict__ bound,
                                                    uchar2* __restrict__ flags, int n, float bias) {
  after_previous();
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n) return;
  flags[r] = make_uchar2(0, 0);
  const float thr = __fsub_rn(dist[r], bias);
  uint32_t lo = 0u, hi = (uint32_t)r;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (dist[mid] < thr) lo = mid + 1; else hi = mid;
  }
  bound[r] = lo;
}

// K(i) of an entry of a light list whose Gaussian's rank bound is `first`: the
// first index of the tile's list with a rank >= first, the end of the
// entry's occluder prefix, which lies in [lo, hi].
__device__ __forceinline__ uint32_t occ_bound(const uint32_t* __restrict__ list, uint32_t lo, uint32_t hi,
                                              uint32_t first) {
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (list[mid] < first) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// The level s of work item w and the item's tile position (lvl_off holds
// each level's first item).
__device__ __forceinline__ int item_level(const uint32_t* lvl_off, uint32_t w) {
  int lo = 0, hi = kSegLevels;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (lvl_off[mid] <= w) lo = mid; else hi = mid;
  }
  return lo;
}

// The items' descriptors and cleared flags, and K at the entries the segment plan reads (every
// segment's first entry and every tile's last), one thread per segment,
// before K6a.
__global__ void __launch_bounds__(256) k_bound_starts(const ShadowParams p,
                                                      const uint32_t* __restrict__ bound, uint32_t* __restrict__ kb) {
  after_previous();
  const uint32_t w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= p.lvl_off[kSegLevels]) return;
  p.pub_flag[w] = 0u;
  const int s = item_level(p.lvl_off, w);
  const uint32_t pos = w - p.lvl_off[s];
  const int tile = (int)p.tile_order[pos];
  const uint32_t b = p.tile_start[tile], e = p.tile_start[tile + 1];
  const uint32_t seg = p.lvl_off[kSegWord];
  const bool last = (uint32_t)s == seg_count(e - b, seg) - 1;
  const uint32_t r0 = b + (uint32_t)s * seg, r1 = last ? e : r0 + seg;
  p.desc[w] = make_uint4((uint32_t)tile | (last ? kSegLast : 0u), r0, r1, s > 0 ? p.lvl_off[s - 1] + pos : kNoItem);
  if (e <= b) return;
  kb[r0] = occ_bound(p.list, b, r0, bound[p.list[r0]]);
  if (last && e - 1 > r0) kb[e - 1] = occ_bound(p.list, b, e - 1, bound[p.list[e - 1]]);
}

// After K6a, one warp per segment: the lists of the segments with an open
// ray (K6b's) and of those every ray enters stopped (K6c's), and K of the
// open segments' other entries (K6b reads it per receiver), which lies
// between the segment's first bound and the next segment's.  No kernel takes
// an occluder for the entries of a stopped segment, so theirs stay unwritten
// past the first.
__global__ void __launch_bounds__(256) k_bound_rest(const ShadowParams p, const uint32_t* __restrict__ bound,
                                                    uint32_t* __restrict__ kb) {
  after_previous();
  __shared__ uint32_t cnt[2], base[2];
  const uint32_t total = p.lvl_off[kSegLevels];
  if (blockIdx.x * 8u >= total) return;
  const uint32_t w = blockIdx.x * 8u + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (threadIdx.x < 2) cnt[threadIdx.x] = 0u;
  __syncthreads();
  uint4 d = make_uint4(0u, 0u, 0u, kNoItem);
  int dead = -1;
  uint32_t at = 0u;
  if (w < total) {
    d = p.desc[w];
    dead = d.w != kNoItem && __ldcg(p.pub_flag + d.w) == 2u ? 1 : 0;
    if (lane == 0) at = atomicAdd(&cnt[dead], 1u);
  }
  __syncthreads();
  if (threadIdx.x < 2) base[threadIdx.x] = cnt[threadIdx.x] ? atomicAdd(p.counts + threadIdx.x, cnt[threadIdx.x]) : 0u;
  __syncthreads();
  if (dead >= 0 && lane == 0) (dead ? p.dead_list : p.open_list)[base[dead] + at] = w;
  if (dead != 0 || d.z <= d.y) return;
  const bool last = (d.x & kSegLast) != 0u;
  const uint32_t c0 = kb[d.y], c1 = kb[last ? d.z - 1 : d.z];
  for (uint32_t j = d.y + 1 + lane; j < d.z - (last ? 1u : 0u); j += 32)
    kb[j] = occ_bound(p.list, c0, min(c1, j), bound[p.list[j]]);
}

// K7: per Gaussian, sum its (tile) partials; T = num / den, or 1 when the
// Gaussian meets no shadow ray.  A Gaussian that K6b did not mark has a zero
// numerator and no sum to add: T is 0 if a pixel of it passes, else 1, and
// its den is stored as 0 (its gradients through the shadow splat are 0).
// Eight lanes per Gaussian rank (four per warp): lane s adds partials s,
// s + 8, ... in order, then three shuffle levels combine the eight sums in a
// fixed order.
__global__ void __launch_bounds__(256) k_shadow_reduce(int n, const uint32_t* __restrict__ off,
                                                       const uint32_t* __restrict__ cnt,
                                                       const float2* __restrict__ partial,
                                                       const uchar2* __restrict__ flags,
                                                       const uint32_t* __restrict__ order,
                                                       const uint32_t* header, float* __restrict__ T,
                                                       float* __restrict__ den_out) {
  after_previous();
  const int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 3;
  const int sub = threadIdx.x & 7;
  const bool valid = r < n;
  const uint32_t P = header[H_PAIRS_LIGHT];
  const uchar2 fl = valid ? flags[r] : make_uchar2(0, 0);
  float num = 0.f, den = 0.f;
  if (fl.x) {
    const uint32_t o = off[r], c = cnt[r];
    if (o + c <= P) {
      for (uint32_t i = sub; i < c; i += 8) {
        const float2 v = partial[o + i];
        num += v.x;
        den += v.y;
      }
    }
  }
#pragma unroll
  for (int sh = 4; sh > 0; sh >>= 1) {
    num += __shfl_xor_sync(0xffffffffu, num, sh);
    den += __shfl_xor_sync(0xffffffffu, den, sh);
  }
  if (valid && sub == 0) {
    const uint32_t g = order[r];
    T[g] = den > 0.f ? num / den : (fl.y ? 0.f : 1.f);
    den_out[g] = den;
  }
}

__global__ void k_fill(float* x, int n, float v) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) x[i] = v;
}

// ---------------------------------------------------------------------------
// K9: camera composite of seven channels (shading rgb, refined shadow,
// residual rgb) front to back; a ray stops before the transmittance would
// fall below t_stop; the block leaves a batch loop once all rays stopped.
// Output: shading * shadow + residual per pixel.
// ---------------------------------------------------------------------------
constexpr int kCamThreads = 128;  // two pixels per thread

struct CamParams {
  const uint32_t* list;
  const uint32_t* tile_start;
  const uint32_t* tile_order;  // block b renders tile tile_order[b] (longest list first)
  const SplatRec* rrec;
  const float4* ccol;
  float* out;
  float* final_t;
  uint32_t* n_contrib;
  float4* pix_aux;
  const uint32_t* nonfinite;  // some colour is infinite or not a number
  int W, H, gx;
  float amax, tstop;
};

// Entries staged for a warp's quadrant, as the shadow splat's (centre relative
// to the tile, conic times log2 e), the terms that pair up duplicated, with
// COLS colour quadruples each; the slots past the last are filled up to a
// whole group of G with entries that never pass.
template <int COLS, int G>
struct CamEntries {
  float4 yc[32];          // -y, -y, c, c
  float4 xart[32];        // x, a, r, threshold
  float2 gi[32];          // gamma, place in the list (as bits)
  float4 col[32][COLS];
};

// A thread's two pixels (one column, rows cy and cy + 4) in packed registers.
struct CamPixels {
  float lx;
  f32x2 ly;  // far away where the pixel is outside the image or its ray stopped
  f32x2 T;
  uint32_t done;  // bit k: pixel k takes no more entries
  uint32_t consumed[2];
};

// The weights alpha T with which entries t .. t + G - 1 enter the two pixels, 0
// where they do not pass; T goes on behind them.  The alpha is gamma 2^power2.  A
// ray stops before T would fall below tstop: it keeps its T, and its row moves
// far away, so that nothing passes from there on.  The alphas of a group do
// not depend on one another; only the product T is a chain.
template <int COLS, int G>
__device__ __forceinline__ void camera_weights(const CamEntries<COLS, G>& E, int t, float amax, float tstop,
                                               CamPixels& px, f32x2 (&w)[G]) {
  f32x2 alpha[G], T[G + 1];
  T[0] = px.T;
#pragma unroll
  for (int i = 0; i < G; ++i) {
    const ulonglong2 yc = *reinterpret_cast<const ulonglong2*>(&E.yc[t + i]);
    const float4 q = E.xart[t + i];
    const float dx = px.lx - q.x;
    const f32x2 dy = add2(px.ly, yc.x);
    const f32x2 pw = power2_pair(dy, yc.y, dup2(q.z * dx), dup2((q.y * dx) * dx));
    const f32x2 ga = mul2(dup2(E.gi[t + i].x), beta2_of(pw, q.w));
    alpha[i] = pk2(fminf(amax, lo2(ga)), fminf(amax, hi2(ga)));
    T[i + 1] = mul2(T[i], fma2(alpha[i], dup2(-1.f), dup2(1.f)));
  }
  px.T = T[G];
  if (fminf(lo2(T[G]), hi2(T[G])) < tstop) {  // once per ray: it stopped at an entry of this group
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      bool stopped = false;
      float Tk = k ? hi2(T[G]) : lo2(T[G]);
#pragma unroll
      for (int i = 0; i < G; ++i) {
        const float Tn = k ? hi2(T[i + 1]) : lo2(T[i + 1]);
        if (!stopped && Tn < tstop) {
          stopped = true;
          Tk = k ? hi2(T[i]) : lo2(T[i]);
          px.consumed[k] = __float_as_uint(E.gi[t + i].y);
        }
        if (stopped) alpha[i] = k ? pk2(lo2(alpha[i]), 0.f) : pk2(0.f, hi2(alpha[i]));
      }
      if (stopped) {
        px.done |= 1u << k;
        px.ly = k ? pk2(lo2(px.ly), kFarRow) : pk2(kFarRow, hi2(px.ly));
        px.T = k ? pk2(lo2(px.T), Tk) : pk2(Tk, hi2(px.T));
      }
    }
  }
#pragma unroll
  for (int i = 0; i < G; ++i) w[i] = mul2(alpha[i], T[i]);
}

struct CamTile {
  float ox, oy;
  uint32_t b, e, wq;
  int px, py0;
};

// A block takes a tile (the longest lists first).  128 threads, two pixels
// each: warp w covers quadrant w (the 8x8 block at (8 (w & 1), 8 (w >> 1))), lane
// l column l & 7 and rows l >> 3 and (l >> 3) + 4 of it, so the two pixels share
// the entry's dx terms.
__device__ __forceinline__ CamTile camera_tile_of(const CamParams& p, int tile, CamPixels& x) {
  const int tx = tile % p.gx, ty = tile / p.gx;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int cx = 8 * (w & 1) + (lane & 7), cy = 8 * (w >> 1) + (lane >> 3);
  CamTile t{(float)(tx * kTile), (float)(ty * kTile), p.tile_start[tile], p.tile_start[tile + 1], 1u << w,
            tx * kTile + cx, ty * kTile + cy};
  const bool in0 = t.px < p.W && t.py0 < p.H, in1 = t.px < p.W && t.py0 + 4 < p.H;
  x.lx = cx + 0.5f;
  x.ly = pk2(in0 ? cy + 0.5f : kFarRow, in1 ? cy + 4.5f : kFarRow);
  x.T = dup2(1.f);
  x.done = (in0 ? 0u : 1u) | (in1 ? 0u : 2u);
  x.consumed[0] = x.consumed[1] = t.e - t.b;
  return t;
}

// 16 bytes from global to shared memory, asynchronously (cp.async)
__device__ __forceinline__ void copy16_async(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// Composites a quadrant's list: each warp on its own takes 32 entries at a
// time, one per lane, keeps those whose box and ellipse reach its quadrant,
// stages them side by side and walks them G at a time; cols(E, slot, rank)
// starts the copies of an entry's colours, use(E, t, w) adds G weighted
// entries.  It leaves when every pixel is done.  The next 32 entries are
// staged, and the records and ranks of those behind them asked for, before
// the current ones are walked.  No block barrier: a quadrant does not wait
// for another.
template <int COLS, int G, typename Cols, typename Use>
__device__ __forceinline__ void camera_walk(const CamParams& p, const CamTile& t, CamPixels& x,
                                            CamEntries<COLS, G> (&E)[2], Cols&& cols, Use&& use) {
  const int lane = threadIdx.x & 31;
  auto rank_at = [&](uint32_t i) { return i < t.e ? p.list[i] : 0u; };
  struct Rec {
    float4 a, b, c;
  };
  auto rec_at = [&](uint32_t r) { return Rec{p.rrec[r].a, p.rrec[r].b, p.rrec[r].c}; };
  // entries [rb, rb + 32) into a buffer; returns how many reach the quadrant
  auto stage = [&](CamEntries<COLS, G>& B, uint32_t rb, uint32_t rank, const Rec& rec) {
    SplatRec q;
    q.a = rec.a; q.b = rec.b; q.c = rec.c;
    float4 e0, e1;
    make_entry(q, t.ox, t.oy, e0, e1);
    const bool hit = rb + lane < t.e && (__float_as_uint(e1.w) & ellipse_halves(e0, e1) & t.wq) != 0u;
    const uint32_t m = __ballot_sync(0xffffffffu, hit);
    const int n = __popc(m), slot = __popc(m & ((1u << lane) - 1u));
    if (hit) {
      B.yc[slot] = make_float4(-e0.y, -e0.y, e0.w, e0.w);
      B.xart[slot] = make_float4(e0.x, e0.z, e1.x, e1.y);
      B.gi[slot] = make_float2(e1.z, __uint_as_float(rb - t.b + lane));
      cols(B, slot, rank);
    } else {  // lanes without a hit fill the last group
      const int fill = n + lane - slot;
      if (fill < (n + G - 1) / G * G) {
        B.yc[fill] = make_float4(0.f, 0.f, 0.f, 0.f);
        B.xart[fill] = make_float4(0.f, 0.f, 0.f, 1.f);  // power 0, below its threshold
        B.gi[fill] = make_float2(0.f, 0.f);
#pragma unroll
        for (int c = 0; c < COLS; ++c) B.col[fill][c] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    return n;
  };
  if (t.b >= t.e) return;
  uint32_t rank = rank_at(t.b + lane);
  Rec rec = rec_at(rank);
  uint32_t rank2 = rank_at(t.b + 32 + lane);
  int n = stage(E[0], t.b, rank, rec), buf = 0;
  rank = rank2;
  rec = rec_at(rank);
  rank2 = rank_at(t.b + 64 + lane);
  for (uint32_t rb = t.b; rb < t.e; rb += 32) {
    if (__all_sync(0xffffffffu, x.done == 3u)) break;
    int next = 0;
    if (rb + 32 < t.e) {
      next = stage(E[buf ^ 1], rb + 32, rank, rec);
      rank = rank2;
      rec = rec_at(rank);
      rank2 = rank_at(rb + 128 + lane - 32);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncwarp();
    for (int k = 0; k < n; k += G) {
      f32x2 w[G];
      camera_weights(E[buf], k, p.amax, p.tstop, x, w);
      use(E[buf], k, w);
    }
    __syncwarp();  // the buffer is free again
    n = next;
    buf ^= 1;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// Bound: issue slots and the FMA pipe, once a warp has independent work.
// Object workload (443 entries per quadrant and 5,100 in its list) / 1 M at
// 1024 x 1024: 0.400 / 0.797 ms with block-wide batches of 256 records and
// scalar updates under branches (0.406 / 0.797 with the updates packed and
// without branches: a warp waited on its loads and the chain of T); 0.297 /
// 0.620 with a list per quadrant and four entries at a time; 0.255 / 0.535
// with the next entries staged ahead.  Two entries at a time take the same
// time, eight 5 % longer.
constexpr int kCamGroup = 4;
using CamSmem = CamEntries<2, kCamGroup>;

// MASK: the frame has colours that a zero weight does not cancel, so a pixel
// adds only the entries it takes (their weights are positive).
template <bool MASK>
__device__ __forceinline__ void camera_tile(const CamParams& p, int tile, CamSmem (*smem)[2]) {
  CamPixels x;
  const CamTile t = camera_tile_of(p, tile, x);
  f32x2 acc[2][4];  // per pixel: (S r, g), (S b, Sh), (R r, g), (R b, -)
#pragma unroll
  for (int k = 0; k < 2; ++k)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[k][c] = 0ull;
  camera_walk<2, kCamGroup>(
      p, t, x, smem[threadIdx.x >> 5],
      [&](CamSmem& E, int slot, uint32_t rank) {
        copy16_async(&E.col[slot][0], &p.ccol[2 * (size_t)rank]);
        copy16_async(&E.col[slot][1], &p.ccol[2 * (size_t)rank + 1]);
      },
      [&](const CamSmem& E, int k0, const f32x2 (&w)[kCamGroup]) {
#pragma unroll
        for (int i = 0; i < kCamGroup; ++i) {
          const ulonglong2 c0 = *reinterpret_cast<const ulonglong2*>(&E.col[k0 + i][0]);
          const ulonglong2 c1 = *reinterpret_cast<const ulonglong2*>(&E.col[k0 + i][1]);
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const f32x2 wk = dup2(k ? hi2(w[i]) : lo2(w[i]));
            if (MASK && lo2(wk) == 0.f) continue;
            acc[k][0] = fma2(wk, c0.x, acc[k][0]);
            acc[k][1] = fma2(wk, c0.y, acc[k][1]);
            acc[k][2] = fma2(wk, c1.x, acc[k][2]);
            acc[k][3] = fma2(wk, c1.y, acc[k][3]);
          }
        }
      });
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int py = t.py0 + 4 * k;
    if (t.px < p.W && py < p.H) {
      const size_t pix = (size_t)py * p.W + t.px;
      const float a[8] = {lo2(acc[k][0]), hi2(acc[k][0]), lo2(acc[k][1]), hi2(acc[k][1]),
                          lo2(acc[k][2]), hi2(acc[k][2]), lo2(acc[k][3]), 0.f};
      p.out[3 * pix + 0] = a[0] * a[3] + a[4];
      p.out[3 * pix + 1] = a[1] * a[3] + a[5];
      p.out[3 * pix + 2] = a[2] * a[3] + a[6];
      p.final_t[pix] = k ? hi2(x.T) : lo2(x.T);
      p.n_contrib[pix] = x.consumed[k];
      p.pix_aux[2 * pix] = make_float4(a[0], a[1], a[2], a[3]);
      p.pix_aux[2 * pix + 1] = make_float4(a[4], a[5], a[6], 0.f);
    }
  }
}

// One frame (p), or a batch of nreq frames (reqs in device memory) whose
// tiles follow one another: frame r owns blocks [tile_prefix[r], tile_prefix[r + 1]).
// 6 blocks per SM whatever the second form takes.
template <bool BATCH>
__global__ void __launch_bounds__(kCamThreads, 6) k_camera(const __grid_constant__ CamParams p, const CamParams* reqs, const uint32_t* tile_prefix,
                                                int nreq) {
  after_previous();
  __shared__ CamSmem M[kCamThreads / 32][2];
  if (BATCH) {
    int r = 0;
    while (r < nreq - 1 && blockIdx.x >= tile_prefix[r + 1]) ++r;
    const CamParams& q = reqs[r];
    const int tile = (int)q.tile_order[blockIdx.x - tile_prefix[r]];  // (asked for together with the flag)
    if (*q.nonfinite) camera_tile<true>(q, tile, M);
    else camera_tile<false>(q, tile, M);
  } else {
    const int tile = (int)p.tile_order[blockIdx.x];
    if (*p.nonfinite) camera_tile<true>(p, tile, M);
    else camera_tile<false>(p, tile, M);
  }
}

// ---------------------------------------------------------------------------
// K9 for an environment light (Sec. 4.5): the camera composite of nl <= 8
// lights in one pass.  The camera splat (alphas, order, stops) does not
// depend on the light, so every light's shading S_l and refined shadow Sh_l
// are composited on the same weights, each into its own accumulators, in the
// order camera_tile uses (each light's sums equal that light's own frame's);
// the residual R, which does not see the light, is composited once.
// out (+)= sum_l w_l (S_l Sh_l + R).
// ---------------------------------------------------------------------------
constexpr int kEnvGroup = 2;  // entries taken together

struct EnvCamParams {
  CamParams c;           // the first light's workspace: camera splat, residual colours, final T
  const float4* envcol;  // [rank][nl]: (shade_l rgb, T'_l)
  float w[kMaxBatch];
  int nl;
  int accumulate;  // add to out (a later group of lights)
};

using EnvSmem = CamEntries<kMaxBatch + 1, kEnvGroup>;  // colours: the lights', then R

// The thread layout and entry arithmetic of camera_tile, with 4 accumulators
// per light and pixel plus 3 for R.
template <bool MASK>
__device__ __forceinline__ void camera_env_tile(const EnvCamParams& e, int tile, EnvSmem (*M)[2]) {
  const CamParams& p = e.c;
  const int nl = e.nl;
  CamPixels x;
  const CamTile t = camera_tile_of(p, tile, x);
  f32x2 R[2][2], S[2][kMaxBatch][2];  // per pixel: (R r, g), (R b, -); per light (S r, g), (S b, Sh)
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    R[k][0] = R[k][1] = 0ull;
#pragma unroll
    for (int l = 0; l < kMaxBatch; ++l) S[k][l][0] = S[k][l][1] = 0ull;
  }
  camera_walk<kMaxBatch + 1, kEnvGroup>(
      p, t, x, M[threadIdx.x >> 5],
      [&](EnvSmem& E, int slot, uint32_t rank) {
        const float4* src = e.envcol + (size_t)rank * nl;
#pragma unroll
        for (int l = 0; l < kMaxBatch; ++l)
          if (l < nl) copy16_async(&E.col[slot][l], src + l);
        copy16_async(&E.col[slot][kMaxBatch], &p.ccol[2 * (size_t)rank + 1]);
      },
      [&](const EnvSmem& E, int k0, const f32x2 (&w)[kEnvGroup]) {
#pragma unroll
        for (int i = 0; i < kEnvGroup; ++i) {
          if (!__any_sync(0xffffffffu, w[i] != 0ull)) continue;
          const f32x2 wk[2] = {dup2(lo2(w[i])), dup2(hi2(w[i]))};
          const ulonglong2 r = *reinterpret_cast<const ulonglong2*>(&E.col[k0 + i][kMaxBatch]);
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            if (MASK && lo2(wk[k]) == 0.f) continue;
            R[k][0] = fma2(wk[k], r.x, R[k][0]);
            R[k][1] = fma2(wk[k], r.y, R[k][1]);
          }
#pragma unroll
          for (int l = 0; l < kMaxBatch; ++l) {
            if (l < nl) {
              const ulonglong2 c = *reinterpret_cast<const ulonglong2*>(&E.col[k0 + i][l]);
#pragma unroll
              for (int k = 0; k < 2; ++k) {
                if (MASK && lo2(wk[k]) == 0.f) continue;
                S[k][l][0] = fma2(wk[k], c.x, S[k][l][0]);
                S[k][l][1] = fma2(wk[k], c.y, S[k][l][1]);
              }
            }
          }
        }
      });
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int py = t.py0 + 4 * k;
    if (!(t.px < p.W && py < p.H)) continue;
    const size_t pix = (size_t)py * p.W + t.px;
    float o0 = 0.f, o1 = 0.f, o2 = 0.f;
#pragma unroll
    for (int l = 0; l < kMaxBatch; ++l) {
      if (l < nl) {
        // the image light l's own frame gives, then its weight
        const float sh = hi2(S[k][l][1]);
        const float i0 = lo2(S[k][l][0]) * sh + lo2(R[k][0]), i1 = hi2(S[k][l][0]) * sh + hi2(R[k][0]),
                    i2 = lo2(S[k][l][1]) * sh + lo2(R[k][1]);
        o0 = fmaf(e.w[l], i0, o0);
        o1 = fmaf(e.w[l], i1, o1);
        o2 = fmaf(e.w[l], i2, o2);
      }
    }
    if (e.accumulate) {
      o0 += p.out[3 * pix + 0];
      o1 += p.out[3 * pix + 1];
      o2 += p.out[3 * pix + 2];
    }
    p.out[3 * pix + 0] = o0;
    p.out[3 * pix + 1] = o1;
    p.out[3 * pix + 2] = o2;
    p.final_t[pix] = k ? hi2(x.T) : lo2(x.T);
    p.n_contrib[pix] = x.consumed[k];
  }
}

// (a call, which leaves the other form as it is without this one)
__device__ __noinline__ void camera_env_tile_masked(const EnvCamParams& e, int tile, EnvSmem (*M)[2]) {
  camera_env_tile<true>(e, tile, M);
}

__global__ void __launch_bounds__(kCamThreads) k_camera_env(const __grid_constant__ EnvCamParams e) {
  __shared__ EnvSmem M[kCamThreads / 32][2];
  const int tile = (int)e.c.tile_order[blockIdx.x];
  if (*e.c.nonfinite) camera_env_tile_masked(e, tile, M);
  else camera_env_tile<false>(e, tile, M);
}

// Launch order of a splat's tiles: longest list first, so that the last
// blocks to start are the short ones and the final partial wave stays short
// (a longest-processing-time-first schedule).  One block: a counting sort on
// a key of the list length (1024 buckets, the largest first), placed by
// shared-memory atomics.  The key is the length in steps of 8 (longer lists
// share the top bucket), or with lvl_off the tile's number of shadow segments,
// seg_count(length, seg), whose seg is chosen here; then lvl_off[s] (s =
// 0..1024) also receives the first work item of segment level s: the number
// of segments of levels below s, level s holding every tile with more than s
// segments (a prefix of the order).  The order within a bucket may vary from run to run; no result
// depends on it.
__global__ void __launch_bounds__(1024) k_tile_order(const uint32_t* __restrict__ tile_start, int ntiles,
                                                     uint32_t* __restrict__ order, uint32_t* __restrict__ lvl_off) {
  after_previous();
  constexpr int kBuckets = 1024;
  __shared__ uint32_t cnt[kBuckets];
  __shared__ uint32_t wsum[32];
  __shared__ uint32_t longest;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  uint32_t seg_len = 0u;
  if (lvl_off) {
    if (t == 0) longest = 0u;
    __syncthreads();
    uint32_t len = 0u;
    for (int i = t; i < ntiles; i += blockDim.x) len = max(len, tile_start[i + 1] - tile_start[i]);
    len = __reduce_max_sync(0xffffffffu, len);
    if (lane == 0) atomicMax(&longest, len);
    __syncthreads();
    const uint32_t pairs = tile_start[ntiles];
    seg_len = kSegMin;
    while (seg_len < kSegLen && (pairs / seg_len > kSegTarget || longest > seg_len * (uint32_t)(kSegLevels - 1)))
      seg_len *= 2u;
    if (t == 0) lvl_off[kSegWord] = seg_len;
    if (t > 0 && t < (int)(kSegWord - kSegLevels)) lvl_off[kSegLevels + t] = 0u;  // the tickets and list counts
  }
  auto bucket = [&](int i) {
    const uint32_t len = tile_start[i + 1] - tile_start[i];
    const uint32_t key = seg_len ? seg_count(len, seg_len) : min(len >> 3, (uint32_t)(kBuckets - 1));
    return (uint32_t)(kBuckets - 1) - key;  // largest key first
  };
  // exclusive scan of one value per thread over the block
  auto block_scan = [&](uint32_t c) -> uint32_t {
    uint32_t x = c;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    if (warp == 0) {
      uint32_t v = wsum[lane];
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
      }
      wsum[lane] = v;
    }
    __syncthreads();
    const uint32_t r = (warp ? wsum[warp - 1] : 0u) + x - c;
    __syncthreads();  // wsum is free for the next scan
    return r;
  };
  cnt[t] = 0u;
  __syncthreads();
  for (int i = t; i < ntiles; i += blockDim.x) atomicAdd(&cnt[bucket(i)], 1u);
  __syncthreads();
  const uint32_t before = block_scan(cnt[t]);  // tiles in buckets < t: key > 1023 - t
  __syncthreads();
  cnt[t] = before;
  __syncthreads();
  if (lvl_off) {
    // level s holds the tiles with more than s segments: cnt[1023 - s] of them
    const uint32_t c = t < kBuckets - 1 ? cnt[kBuckets - 1 - t] : 0u;
    const uint32_t off = block_scan(c);
    lvl_off[t] = off;
    if (t == kBuckets - 1) lvl_off[kBuckets] = off + c;
  }
  __syncthreads();
  for (int i = t; i < ntiles; i += blockDim.x) order[atomicAdd(&cnt[bucket(i)], 1u)] = (uint32_t)i;
}

}  // namespace

void launch_tile_order(const FrameArgs& f, int splat, cudaStream_t s) {
  const Workspace& L = *f.L;
  uint32_t* order = at<uint32_t>(f.ws, L.tile_order[splat]);
  launch_after(k_tile_order, 1, 1024, 0, s, at<uint32_t>(f.ws, L.sp[splat].tile_start), L.ntiles, order, nullptr);
  count_launch();
}

// Segments past each tile's first: no more than pairs / seg, for the seg that
// k_tile_order chooses (kSegTarget of them, or seg is kSegLen).
static size_t later_segments(size_t cap) {
  const size_t few = cap / kSegMin, many = cap / kSegLen > kSegTarget ? cap / kSegLen : kSegTarget;
  return (few < many ? few : many) + 1;
}
size_t shadow_seg_items(int ntiles, size_t cap) { return (size_t)ntiles + later_segments(cap); }
size_t shadow_seg_links(int ntiles, size_t cap) {
  const size_t later = later_segments(cap), firsts = (size_t)ntiles < later ? (size_t)ntiles : later;
  return firsts + later;
}

namespace {

// The shadow composite's parameters of a prepared frame.
ShadowParams shadow_params(const FrameArgs& f) {
  const SplatBufs& b = f.L->sp[1];
  unsigned char* ws = f.ws;
  const int fin = (f.L->ntiles <= 256 ? 1 : 2) & 1;
  uint32_t* lvl = at<uint32_t>(ws, f.L->seg_lvl);
  uint32_t* header = at<uint32_t>(ws, f.L->header);
  ShadowParams p;
  p.tile_order = at<uint32_t>(ws, f.L->tile_order[1]);
  p.lvl_off = lvl;
  p.ticket = lvl + kSegLevels + 1;
  p.counts = lvl + kSegLevels + 4;
  p.desc = at<uint4>(ws, f.L->seg_desc);
  p.open_list = at<uint32_t>(ws, f.L->seg_lists);
  p.dead_list = p.open_list + shadow_seg_items(f.L->ntiles, f.L->cap);
  p.pub_a = at<float>(ws, f.L->seg_pub);
  p.pub_flag = at<uint32_t>(ws, f.L->seg_flag);
  p.list = at<uint32_t>(ws, b.tv[fin]);
  p.tile_start = at<uint32_t>(ws, b.tile_start);
  p.rrec = at<SplatRec>(ws, b.rrec);
  p.off = at<uint32_t>(ws, b.off);
  p.kbound = at<uint32_t>(ws, b.tv[1 - fin]);
  p.pass_mask = at<uint8_t>(ws, b.tk[1 - fin]);
  p.partial = at<float2>(ws, f.L->partial);
  p.light_final = at<float>(ws, f.L->light_final);
  p.light_stop = at<uint32_t>(ws, f.L->light_stop);
  p.status = header + H_STATUS;
  p.rank_flags = at<uchar2>(ws, f.L->rank_flags);
  p.W = f.L->width; p.H = f.L->height; p.gx = f.L->gx;
  p.amax = f.opts.alpha_max;
  return p;
}

CamParams camera_params(const FrameArgs& f, float* out_rgb) {
  const SplatBufs& b = f.L->sp[0];
  unsigned char* ws = f.ws;
  const int fin = (f.L->ntiles <= 256 ? 1 : 2) & 1;
  CamParams p;
  p.list = at<uint32_t>(ws, b.tv[fin]);
  p.tile_start = at<uint32_t>(ws, b.tile_start);
  p.rrec = at<SplatRec>(ws, b.rrec);
  p.ccol = at<float4>(ws, f.L->ccol);
  p.out = out_rgb;
  p.final_t = at<float>(ws, f.L->final_t);
  p.n_contrib = at<uint32_t>(ws, f.L->n_contrib);
  p.pix_aux = at<float4>(ws, f.L->pix_aux);
  p.nonfinite = at<uint32_t>(ws, f.L->header) + H_NONFINITE;
  p.W = f.L->width; p.H = f.L->height; p.gx = f.L->gx;
  p.amax = f.opts.alpha_max; p.tstop = f.opts.t_stop;
  p.tile_order = at<uint32_t>(ws, f.L->tile_order[0]);  // from the camera binning stage
  return p;
}

// Blocks per SM of the persistent segment kernels (per device, looked up once).
struct SegOccupancy {
  int chain, live, dead;
};
SegOccupancy seg_occupancy() {
  static DeviceOnce once;
  static SegOccupancy occ[kMaxDevices];
  once.run([] {
    int d = 0;
    cudaGetDevice(&d);
    bool ok = true;
    for (const void* k : {(const void*)k_shadow<false>, (const void*)k_shadow<true>, (const void*)k_shadow_chain<false>,
                          (const void*)k_shadow_chain<true>})
      ok = ok && cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout,
                                      (int)cudaSharedmemCarveoutMaxShared) == cudaSuccess;
    if (d >= 0 && d < kMaxDevices) {
      SegOccupancy& o = occ[d];
      ok = ok &&
           cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o.chain, k_shadow_chain<true>, kSegWarps * 32, 0) ==
               cudaSuccess &&
           cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o.live, k_shadow<true>, kSegWarps * 32, 0) == cudaSuccess &&
           cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o.dead, k_shadow_dead<true>, kDeadWarps * 32, 0) ==
               cudaSuccess;
    }
    return ok;
  });
  int d = 0;
  cudaGetDevice(&d);
  SegOccupancy o{1, 1, 1};
  if (d >= 0 && d < kMaxDevices) o = occ[d];
  if (o.chain < 1) o.chain = 1;
  if (o.live < 1) o.live = 1;
  if (o.dead < 1) o.dead = 1;
  return o;
}

// Layout of a batch's parameter block (device, and its pinned host staging).
struct BatchLayout {
  static constexpr size_t shadow = 0;
  static constexpr size_t camera = ((sizeof(ShadowParams) * kMaxBatch + 255) / 256) * 256;
  static constexpr size_t prefix = camera + ((sizeof(CamParams) * kMaxBatch + 255) / 256) * 256;
  static constexpr size_t total = prefix + 4 * (kMaxBatch + 1);
};

}  // namespace

size_t batch_param_bytes() { return BatchLayout::total; }

void prepare_shadow_composite(const FrameArgs& f, cudaStream_t s) {
  const SplatBufs& b = f.L->sp[1];
  unsigned char* ws = f.ws;
  const int fin = (f.L->ntiles <= 256 ? 1 : 2) & 1;
  uint32_t* kb = at<uint32_t>(ws, b.tv[1 - fin]);
  // the light tiles by segment count, and the work items of each segment level
  uint32_t* lvl = at<uint32_t>(ws, f.L->seg_lvl);
  launch_after(k_tile_order, 1, 1024, 0, s, at<uint32_t>(ws, b.tile_start), f.L->ntiles, at<uint32_t>(ws, f.L->tile_order[1]), lvl);
  // the occluder bounds the segment plan reads; the rest follow K6a
  const size_t items = shadow_seg_items(f.L->ntiles, f.L->cap);
  const int n = f.sc.n;
  uint32_t* bound = at<uint32_t>(ws, b.sk[0]);  // free once the depths are sorted
  launch_after(k_rank_bound, (n + 255) / 256, 256, 0, s, at<float>(ws, b.sk[1]), bound,
               at<uchar2>(ws, f.L->rank_flags), n, f.opts.shadow_bias);
  launch_after(k_bound_starts, (int)((items + 255) / 256), 256, 0, s, shadow_params(f), bound, kb);
  count_launch(3);
}

// the occluder bounds of the open segments' other entries (after K6a)
void launch_bound_rest(const FrameArgs& f, const ShadowParams& p, cudaStream_t s) {
  const SplatBufs& b = f.L->sp[1];
  const int fin = (f.L->ntiles <= 256 ? 1 : 2) & 1;
  const size_t items = shadow_seg_items(f.L->ntiles, f.L->cap);
  launch_after(k_bound_rest, (int)((items * 32 + 255) / 256), 256, 0, s, p, at<uint32_t>(f.ws, b.sk[0]),
                                                               at<uint32_t>(f.ws, b.tv[1 - fin]));
  count_launch();
}

void launch_shadow_composite(const FrameArgs& f, cudaStream_t s) {
  prepare_shadow_composite(f, s);
  const ShadowParams p = shadow_params(f);
  const SegOccupancy o = seg_occupancy();
  const int nsm = device_sm_count();
  // persistent warps: every resident warp slot takes segments from a ticket
  launch_after(k_shadow_chain<false>, nsm * o.chain, kSegWarps * 32, 0, s, p, nullptr, 1);
  launch_bound_rest(f, p, s);
  launch_after(k_shadow<false>, nsm * o.live, kSegWarps * 32, 0, s, p, nullptr, 1);
  launch_after(k_dead_probe, (f.L->n + 255) / 256, 256, 0, s, p, f.L->n);
  launch_after(k_shadow_dead<false>, nsm * o.dead, kDeadWarps * 32, 0, s, p, nullptr, 1);
  count_launch(4);
}

// Self-test of the chain's bounded waits: the segment plan of a frame whose
// light binning ran, then K6a with its ticket starting at the second segment
// level, so that no first segment ever publishes and every second segment's
// wait runs out (each then publishes its rays as stopped).
__global__ void k_skip_first_level(const uint32_t* lvl_off, uint32_t* ticket) {
  if (threadIdx.x == 0) ticket[0] = lvl_off[1];
}

void launch_shadow_chain_selftest(const FrameArgs& f, cudaStream_t s) {
  prepare_shadow_composite(f, s);
  const ShadowParams p = shadow_params(f);
  k_skip_first_level<<<1, 32, 0, s>>>(p.lvl_off, p.ticket);
  const SegOccupancy o = seg_occupancy();
  launch_after(k_shadow_chain<false>, device_sm_count() * o.chain, kSegWarps * 32, 0, s, p, nullptr, 1);
  count_launch(2);
}

void launch_shadow_composite_batch(const FrameArgs* const* f, int n, unsigned char* dev, unsigned char* host,
                                   cudaStream_t s) {
  ShadowParams* hp = reinterpret_cast<ShadowParams*>(host + BatchLayout::shadow);
  for (int r = 0; r < n; ++r) hp[r] = shadow_params(*f[r]);
  cudaMemcpyAsync(dev + BatchLayout::shadow, hp, sizeof(ShadowParams) * n, cudaMemcpyHostToDevice, s);
  const ShadowParams* dp = reinterpret_cast<const ShadowParams*>(dev + BatchLayout::shadow);
  // the batch shares the first frame's tickets; every frame's flags were zeroed when it was prepared
  const SegOccupancy o = seg_occupancy();
  const int nsm = device_sm_count();
  k_shadow_chain<true><<<nsm * o.chain, kSegWarps * 32, 0, s>>>(hp[0], dp, n);
  for (int r = 0; r < n; ++r) launch_bound_rest(*f[r], hp[r], s);
  launch_after(k_shadow<true>, nsm * o.live, kSegWarps * 32, 0, s, hp[0], dp, n);
  for (int r = 0; r < n; ++r) launch_after(k_dead_probe, (f[r]->L->n + 255) / 256, 256, 0, s, hp[r], f[r]->L->n);
  launch_after(k_shadow_dead<true>, nsm * o.dead, kDeadWarps * 32, 0, s, hp[0], dp, n);
  count_launch(2 + n + 1);
}

void launch_shadow_reduce(const FrameArgs& f, cudaStream_t s, bool wait) {
  const SplatBufs& b = f.L->sp[1];
  unsigned char* ws = f.ws;
  const int n = f.sc.n;
  launch_behind(wait, k_shadow_reduce, (n * 8 + 255) / 256, 256, 0, s, n, at<uint32_t>(ws, b.off), at<uint32_t>(ws, b.cnt), at<float2>(ws, f.L->partial),
      at<uchar2>(ws, f.L->rank_flags), at<uint32_t>(ws, b.sv[1]), at<uint32_t>(ws, f.L->header), at<float>(ws, f.L->T),
      at<float>(ws, f.L->shadow_den));
  count_launch();
}

void launch_fill_shadow_one(const FrameArgs& f, cudaStream_t s) {
  const int n = f.sc.n;
  k_fill<<<(n + 255) / 256, 256, 0, s>>>(at<float>(f.ws, f.L->T), n, 1.f);
  k_fill<<<(n + 255) / 256, 256, 0, s>>>(at<float>(f.ws, f.L->shadow_den), n, 0.f);
  count_launch();
  count_launch();
}

void launch_camera_composite(const FrameArgs& f, float* out_rgb, bool wait, cudaStream_t s) {
  launch_behind(wait, k_camera<false>, f.L->ntiles, kCamThreads, 0, s, camera_params(f, out_rgb), nullptr, nullptr, 1);
  count_launch();
}

void launch_camera_env(const FrameArgs& f0, const float4* envcol, int nl, const float* w, bool accumulate,
                       float* out_rgb, cudaStream_t s) {
  EnvCamParams e;
  e.c = camera_params(f0, out_rgb);
  e.envcol = envcol;
  e.nl = nl;
  for (int l = 0; l < kMaxBatch; ++l) e.w[l] = l < nl ? w[l] : 0.f;
  e.accumulate = accumulate ? 1 : 0;
  k_camera_env<<<f0.L->ntiles, kCamThreads, 0, s>>>(e);
  count_launch();
}

void launch_camera_composite_batch(const FrameArgs* const* f, float* const* out, int n, unsigned char* dev,
                                   unsigned char* host, cudaStream_t s) {
  CamParams* hp = reinterpret_cast<CamParams*>(host + BatchLayout::camera);
  uint32_t* pre = reinterpret_cast<uint32_t*>(host + BatchLayout::prefix);
  pre[0] = 0;
  for (int r = 0; r < n; ++r) {
    hp[r] = camera_params(*f[r], out[r]);
    pre[r + 1] = pre[r] + (uint32_t)f[r]->L->ntiles;
  }
  cudaMemcpyAsync(dev + BatchLayout::camera, hp, sizeof(CamParams) * n, cudaMemcpyHostToDevice, s);
  cudaMemcpyAsync(dev + BatchLayout::prefix, pre, 4 * (n + 1), cudaMemcpyHostToDevice, s);
  k_camera<true><<<pre[n], kCamThreads, 0, s>>>(hp[0], reinterpret_cast<const CamParams*>(dev + BatchLayout::camera),
                                         reinterpret_cast<const uint32_t*>(dev + BatchLayout::prefix), n);
  count_launch();
}

}  // namespace gs3
