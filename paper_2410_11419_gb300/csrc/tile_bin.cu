// K4-K5: tile binning of one splat (camera or light): for every tile, the
// depth ranks of the Gaussians whose tile rectangle covers it, in rank order,
// and the tiles' [start, end) ranges (Sec. 3; the light view is binned the
// same way, Sec. 4.2).
//
// A rank's (tile, rank) pairs are the tiles of its rectangle, so the lists
// are built from the rectangles by two stable counting passes instead of
// emitting the pairs and sorting them on the tile bits:
//   rows     the ranks covering tile row y, for every y, in rank order, with
//            each rank's column span beside it: the counts per (row, block
//            of kBinBlock ranks) come from k_reorder; k_bin_plan scans each
//            row's counts and the row totals; k_bin_rows places;
//   columns  each row's sequence is cut into chunks of bin_chunk(gx) items;
//            k_bin_count counts the items per (row, column, chunk);
//            k_bin_rowscan scans each row's counts in (column, chunk) order,
//            after the pairs of the rows above, which gives every tile's
//            start and every chunk's offset in each of its tiles; k_bin_place
//            writes the list entries.
// Up to kScanBuckets rows or columns, each placement goes over the buckets
// (scan_place): a warp holds 256 items, eight per lane, and for every bucket
// it owns asks which of them cover it (a ballot per 32 items), which gives the
// bucket's entries in item order, side by side in memory, without shared
// memory or barriers (the counts come from difference arrays).  That is 64 instructions per bucket and 256 items
// whatever the spans, so past that many buckets it loses to going over the
// (item, bucket) pairs (place_spans), about 4.6 instructions each: 256 items,
// one per thread; a warp's offset in bucket x is the bucket's running offset
// plus the items of earlier warps covering x (per-warp difference arrays);
// inside a warp the pairs are dealt 32 per round in item order, and a pair's
// rank among the round's pairs of the same bucket (match_any) is added to a
// per-bucket counter.  Either way every list is in rank order, the result a
// stable sort of the pairs by tile would give, and no step depends on timing
// or waits on another block.
// Bound: the scattered 4-byte stores of the list (a bucket's run of 256 items
// holds about 36 entries) and the ballots.  Rows + counts + placement of the
// camera splat alone, 300k Gaussians at 800 x 800: 19 + 9 + 68 us; of both splats
// beside the shadow composite, 1 M at 1024 x 1024: 0.13 + 0.13 + 0.83 ms, where
// all three over the pairs take 0.19 + 0.54 + 1.57.
#include <climits>

#include "gs3_internal.cuh"

namespace gs3 {
namespace {

constexpr int kBinThreads = 256;  // 8 warps
constexpr int kBinWarps = kBinThreads / 32;

__device__ __forceinline__ uint32_t warp_inclusive_sum(uint32_t v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t u = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += u;
  }
  return v;
}

// Exclusive scan of v[0, len) in place, starting at carry, by one block of
// NT threads (four consecutive words per thread per step); returns carry plus
// the sum.  sm: 32 words of shared memory.  Every thread must call it.
template <int NT>
__device__ uint32_t block_scan_inplace(uint32_t* v, size_t len, uint32_t carry, uint32_t* sm) {
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  constexpr int kWarps = NT / 32;
  for (size_t base = 0; base < len; base += 4 * NT) {
    uint32_t x[4], s = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const size_t i = base + 4 * (size_t)t + j;
      x[j] = i < len ? v[i] : 0u;
      s += x[j];
    }
    const uint32_t inc = warp_inclusive_sum(s, lane);
    if (lane == 31) sm[w] = inc;
    __syncthreads();
    if (w == 0) {
      const uint32_t u = warp_inclusive_sum(lane < kWarps ? sm[lane] : 0u, lane);
      if (lane < kWarps) sm[lane] = u;
    }
    __syncthreads();
    uint32_t pre = carry + (w ? sm[w - 1] : 0u) + inc - s;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const size_t i = base + 4 * (size_t)t + j;
      if (i < len) v[i] = pre;
      pre += x[j];
    }
    carry += sm[kWarps - 1];
    __syncthreads();  // sm is rewritten by the next step
  }
  return carry;
}

// the sum of every thread's x over a block of NT threads (all threads get it)
template <int NT>
__device__ uint32_t block_sum(uint32_t x, uint32_t* sm) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = x;
  __syncthreads();
  uint32_t s = 0;
#pragma unroll
  for (int k = 0; k < NT / 32; ++k) s += sm[k];
  __syncthreads();
  return s;
}

// The plan words: rs[gy + 1] row starts in the row sequence, cb[gy + 1]
// chunk starts (every row has at least one chunk), pairs[gy] list entries
// per row, ok (the pairs fit the capacity), ticket (cleared by k_reorder).
struct BinPlan {
  uint32_t *rs, *cb, *pairs, *ok, *ticket;
  __device__ BinPlan(uint32_t* p, int gy)
      : rs(p), cb(p + gy + 1), pairs(p + 2 * gy + 2), ok(p + 3 * gy + 2), ticket(p + 3 * gy + 3) {}
};

// the row of chunk kg: the largest y with cb[y] <= kg (cb[0] = 0 <= kg < cb[gy])
__device__ __forceinline__ int chunk_row(const uint32_t* cb, int gy, uint32_t kg) {
  int lo = 0, hi = gy;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (cb[mid] <= kg) lo = mid; else hi = mid;
  }
  return lo;
}

// Shared memory of a span placement (about 41 KB).
struct SpanSmem {
  int cnt[kBinWarps][kMaxTileAxis + 1];  // per warp: difference array, counts, then offsets per bucket
  uint32_t run[kMaxTileAxis];            // per bucket: the running offset
  uint32_t ex[kBinWarps][32];            // per warp: exclusive prefix of the lanes' span widths
  int lo[kBinWarps][32];                 // per warp: the lanes' first buckets
  uint32_t v0[kBinWarps][32], v1[kBinWarps][32];  // per warp: the lanes' payloads
};

// Stable placement of 256 items, one per thread in thread order: an item with
// a <= b covers buckets a..b, and its copy for bucket x goes to
// out0 / out1[S.run[x] + the items of lower threads covering x].  S.run must
// hold the buckets' offsets and is advanced past the items.  Every thread of
// the block calls it.
__device__ void place_spans(SpanSmem& S, int nbk, int a, int b, uint32_t v0, uint32_t v1,
                            uint32_t* __restrict__ out0, uint32_t* __restrict__ out1, size_t cap) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int* c = S.cnt[w];
  for (int x = lane; x <= nbk; x += 32) c[x] = 0;
  __syncwarp();
  const bool has = a <= b;
  if (has) {
    atomicAdd(&c[a], 1);
    atomicAdd(&c[b + 1], -1);
  }
  __syncwarp();
  uint32_t carry = 0;  // the warp's items per bucket: running sum of the difference array
  for (int x0 = 0; x0 < nbk; x0 += 32) {
    const int x = x0 + lane;
    const uint32_t v = warp_inclusive_sum(x < nbk ? (uint32_t)c[x] : 0u, lane);
    if (x < nbk) c[x] = (int)(carry + v);
    carry += __shfl_sync(0xffffffffu, v, 31);
  }
  __syncthreads();
  for (int x = threadIdx.x; x < nbk; x += kBinThreads) {  // warp k starts after warps 0..k-1
    uint32_t base = S.run[x];
#pragma unroll
    for (int k = 0; k < kBinWarps; ++k) {
      const uint32_t n = (uint32_t)S.cnt[k][x];
      S.cnt[k][x] = (int)base;
      base += n;
    }
    S.run[x] = base;
  }
  __syncthreads();
  // the warp's (item, bucket) pairs in item order, 32 per round
  const uint32_t wid = has ? (uint32_t)(b - a + 1) : 0u;
  const uint32_t inc = warp_inclusive_sum(wid, lane);
  const uint32_t total = __shfl_sync(0xffffffffu, inc, 31);
  S.ex[w][lane] = inc - wid;
  S.lo[w][lane] = a;
  S.v0[w][lane] = v0;
  S.v1[w][lane] = v1;
  __syncwarp();
  const uint32_t lt = (1u << lane) - 1u;
  // four rounds at a time: their item searches are independent, so they run
  // side by side; the counters are then read and advanced round by round
  for (uint32_t p0 = 0; p0 < total; p0 += 128) {
    int jq[4], xq[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t p = p0 + 32 * q + lane;
      int j = 0;  // the item of pair p: the last lane j with ex[j] <= p
#pragma unroll
      for (int s = 16; s > 0; s >>= 1)
        if (S.ex[w][j + s] <= p) j += s;
      jq[q] = j;
      xq[q] = S.lo[w][j] + (int)(p - S.ex[w][j]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (p0 + 32 * q >= total) break;  // the same for every lane
      const bool act = p0 + 32 * q + lane < total;
      const int j = jq[q], x = xq[q];
      const uint32_t m = __match_any_sync(0xffffffffu, act ? x : -1 - lane);
      if (act) {
        const uint32_t pos = (uint32_t)c[x] + (uint32_t)__popc(m & lt);
        if (pos < cap) {
          out0[pos] = S.v0[w][j];
          if (out1) out1[pos] = S.v1[w][j];
        }
      }
      __syncwarp();  // every lane has read its bucket's counter
      if (act && (m >> lane) == 1u) c[x] += __popc(m);
      __syncwarp();
    }
  }
  __syncthreads();  // S is rewritten by the next call
}

// A warp's 256 items in order, eight per lane (item 32 c + lane at c): item c
// covers buckets lo .. lo + wid (lo = kNoSpan: none).
constexpr int kScanBuckets = 128;
constexpr uint32_t kNoSpan = 0x80000000u;
struct WarpSpans {
  uint32_t lo[8], wid[8], v0[8];
};

// Stable placement of a warp's 256 items into the buckets x = first, first +
// step, ... < nbk, `first + step l` starting at lane l's base: an item's copy
// for bucket x goes to out0[base + the earlier items covering x], and
// v1 likewise to out1 if out1 is given.
template <bool TWO>
__device__ __forceinline__ void scan_place(const WarpSpans& S, const uint32_t (&v1)[8], int nbk, int first, int step,
                                           uint32_t base, uint32_t* __restrict__ out0, uint32_t* __restrict__ out1,
                                           size_t cap) {
  const uint32_t below = (1u << (threadIdx.x & 31)) - 1u;
  for (int x = first, l = 0; x < nbk; x += step, ++l) {
    uint32_t at = __shfl_sync(0xffffffffu, base, l);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const bool in = (uint32_t)x - S.lo[c] <= S.wid[c];
      const uint32_t m = __ballot_sync(0xffffffffu, in);
      const uint32_t pos = at + (uint32_t)__popc(m & below);
      if (in && pos < cap) {
        out0[pos] = S.v0[c];
        if (TWO) out1[pos] = v1[c];
      }
      at += (uint32_t)__popc(m);
    }
  }
}

// Blocks y < gy: the row's block counts scanned in place (exclusive, within the
// row), its total to rs[y]; block gy: the blocks' pairs likewise (every rank's
// first list slot starts there).  The last block to finish makes the plan, four
// rows per thread (gy <= 1024): row starts from the row totals, chunks per row and
// their starts, and the capacity check.  No block waits for another.
// Bound: launches; with the ranks' slots scanned by k_bin_rows this is one kernel
// where a scan of all ranks, this scan and the plan were five.
__global__ void __launch_bounds__(kBinThreads) k_bin_plan(uint32_t* __restrict__ row_cnt, int nb, int gy, uint32_t ch,
                                                          size_t tab_words, int gx, uint32_t* __restrict__ plan,
                                                          uint32_t* header, int h_need, int h_pairs, size_t cap) {
  after_previous();
  __shared__ uint32_t sm[32];
  __shared__ uint32_t rows[kMaxTileAxis], chunks[kMaxTileAxis];
  __shared__ bool last;
  BinPlan P(plan, gy);
  const int y = blockIdx.x, t = threadIdx.x;
  const uint32_t total = block_scan_inplace<kBinThreads>(row_cnt + (size_t)y * nb, (size_t)nb, 0u, sm);
  if (t == 0) {
    if (y < gy) P.rs[y] = total;
    else header[h_need] = total;
    __threadfence();
    last = atomicAdd(P.ticket, 1u) == (uint32_t)gy;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int i = t; i < gy; i += kBinThreads) {
    const uint32_t m = __ldcg(P.rs + i), c = (uint32_t)(((uint64_t)m + ch - 1) / ch);
    rows[i] = m;
    chunks[i] = c > 1u ? c : 1u;
    P.pairs[i] = 0u;
  }
  __syncthreads();
  const uint32_t M = block_scan_inplace<kBinThreads>(rows, (size_t)gy, 0u, sm);
  const uint32_t C = block_scan_inplace<kBinThreads>(chunks, (size_t)gy, 0u, sm);
  for (int i = t; i < gy; i += kBinThreads) {
    P.rs[i] = rows[i];
    P.cb[i] = chunks[i];
  }
  if (t == 0) {
    P.rs[gy] = M;
    P.cb[gy] = C;
    const uint32_t need = __ldcg(header + h_need);
    const bool ok = need <= cap && (size_t)C * (size_t)gx <= tab_words;
    header[h_pairs] = ok ? need : 0u;
    if (!ok) atomicCAS(&header[H_STATUS], 0u, (uint32_t)GS3_ERR_CAPACITY);
    *P.ok = ok ? 1u : 0u;
  }
}

__device__ __forceinline__ uint32_t tiles_of(int4 q) {
  return q.x >= 0 ? (uint32_t)(q.z - q.x + 1) * (uint32_t)(q.w - q.y + 1) : 0u;
}

// The row sequence: the block's 256 ranks over their rows, each copy with the
// rank's column span (x0 | x1 << 16) beside it; row y's offset for this block
// is the row's start plus the row's counts of the blocks before.  Also off[r], rank r's
// first slot among all pairs in rank order (the shadow partials' slots).
__global__ void __launch_bounds__(kBinThreads) k_bin_rows(int n, const SplatRec* __restrict__ rrec,
                                                          const uint32_t* __restrict__ row_cnt, int nb, int gy,
                                                          const uint32_t* __restrict__ plan,
                                                          uint32_t* __restrict__ rowseq, uint32_t* __restrict__ rowspan,
                                                          uint32_t* __restrict__ off, size_t cap) {
  after_previous();
  __shared__ SpanSmem S;
  __shared__ uint32_t sm[kBinWarps];
  for (int y = threadIdx.x; y < gy; y += kBinThreads) S.run[y] = plan[y] + row_cnt[(size_t)y * nb + blockIdx.x];
  const int r = blockIdx.x * kBinThreads + threadIdx.x;
  int a = 0, b = -1;
  uint32_t span = 0, c = 0;
  if (r < n) {
    const int4 q = rrec[r].r;
    c = tiles_of(q);
    if (q.x >= 0) {
      a = q.y;
      b = q.w;
      span = (uint32_t)q.x | ((uint32_t)q.z << 16);
    }
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t inc = warp_inclusive_sum(c, lane);
  if (lane == 31) sm[w] = inc;
  __syncthreads();
  uint32_t slot = row_cnt[(size_t)gy * nb + blockIdx.x] + inc - c;
  for (int k = 0; k < w; ++k) slot += sm[k];
  if (r < n) off[r] = slot;
  if (plan[3 * gy + 2] == 0u) return;
  place_spans(S, gy, a, b, (uint32_t)r, span, rowseq, rowspan, cap);
}

// k_bin_rows going over the rows (gy <= kScanBuckets).
__global__ void __launch_bounds__(kBinThreads) k_bin_rows_scan(int n, const SplatRec* __restrict__ rrec,
                                                               const uint32_t* __restrict__ row_cnt, int nb, int gy,
                                                               const uint32_t* __restrict__ plan,
                                                               uint32_t* __restrict__ rowseq,
                                                               uint32_t* __restrict__ rowspan,
                                                               uint32_t* __restrict__ off, size_t cap) {
  after_previous();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  WarpSpans S;
  uint32_t span[8];
  uint32_t slot = row_cnt[(size_t)gy * nb + blockIdx.x], own = 0u;  // warp w takes the slots of ranks 32 w ..
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int r = blockIdx.x * kBinThreads + 32 * c + lane;
    int4 q = make_int4(-1, 0, 0, 0);
    if (r < n) q = rrec[r].r;
    const uint32_t tiles = tiles_of(q);
    if (c < w) slot += __reduce_add_sync(0xffffffffu, tiles);
    if (c == w) own = tiles;
    S.lo[c] = q.x >= 0 ? (uint32_t)q.y : kNoSpan;
    S.wid[c] = q.x >= 0 ? (uint32_t)(q.w - q.y) : 0u;
    S.v0[c] = (uint32_t)r;
    span[c] = (uint32_t)q.x | ((uint32_t)q.z << 16);
  }
  slot += warp_inclusive_sum(own, lane) - own;
  if (blockIdx.x * kBinThreads + 32 * w + lane < n) off[blockIdx.x * kBinThreads + 32 * w + lane] = slot;
  if (plan[3 * gy + 2] == 0u) return;
  const int y = w + kBinWarps * lane;
  const uint32_t base = y < gy ? plan[y] + row_cnt[(size_t)y * nb + blockIdx.x] : 0u;
  scan_place<true>(S, span, gy, w, kBinWarps, base, rowseq, rowspan, cap);
}

// A chunk of at most 256 items of a row's sequence, for a warp
__device__ __forceinline__ void load_chunk(const uint32_t* __restrict__ rowspan, uint32_t i0, uint32_t i1, int lane,
                                           WarpSpans& S) {
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const uint32_t i = i0 + 32 * c + lane;
    const uint32_t sp = i < i1 ? rowspan[i] : kNoSpan;
    S.lo[c] = i < i1 ? sp & 0xFFFFu : kNoSpan;
    S.wid[c] = i < i1 ? (sp >> 16) - (sp & 0xFFFFu) : 0u;
  }
}

// k_bin_count for chunks of 256 (gx <= kScanBuckets), a warp per chunk: the
// difference array takes two shared-memory adds per item where a ballot per 32
// items and column took three instructions.  Camera of 300k Gaussians at
// 800 x 800: 35 -> 9 us.
__global__ void __launch_bounds__(kBinThreads) k_bin_count_warp(const uint32_t* __restrict__ rowspan,
                                                                uint32_t* __restrict__ plan, int gx, int gy,
                                                                uint32_t* __restrict__ tab) {
  after_previous();
  __shared__ int diff[kBinWarps][kScanBuckets + 1];
  BinPlan P(plan, gy);
  if (*P.ok == 0u) return;
  const uint32_t C = P.cb[gy];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int* d = diff[w];
  for (uint32_t kg = blockIdx.x * kBinWarps + w; kg < C; kg += gridDim.x * kBinWarps) {
    const int y = chunk_row(P.cb, gy, kg);
    const uint32_t c0 = P.cb[y], nch = P.cb[y + 1] - c0, k = kg - c0;
    const uint32_t i0 = P.rs[y] + 256u * k, i1 = min(P.rs[y + 1], i0 + 256u);
    for (int x = lane; x <= gx; x += 32) d[x] = 0;
    __syncwarp();
    uint32_t total = 0u;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const uint32_t i = i0 + 32 * c + lane;
      if (i < i1) {
        const uint32_t sp = rowspan[i];
        const int x0 = (int)(sp & 0xFFFFu), x1 = (int)(sp >> 16);
        atomicAdd(&d[x0], 1);
        atomicAdd(&d[x1 + 1], -1);
        total += (uint32_t)(x1 - x0 + 1);
      }
    }
    __syncwarp();
    uint32_t* out = tab + (size_t)c0 * gx + k;
    uint32_t run = 0u;
    for (int x0 = 0; x0 < gx; x0 += 32) {
      const int x = x0 + lane;
      const uint32_t v = warp_inclusive_sum(x < gx ? (uint32_t)d[x] : 0u, lane);
      if (x < gx) out[(size_t)x * nch] = run + v;
      run += __shfl_sync(0xffffffffu, v, 31);
    }
    total = __reduce_add_sync(0xffffffffu, total);
    if (lane == 0 && total) atomicAdd(P.pairs + y, total);
    __syncwarp();  // d is cleared for the next chunk
  }
}

// k_bin_place going over the columns (gx <= kScanBuckets, chunks of 256).
__global__ void __launch_bounds__(kBinThreads) k_bin_place_scan(const uint32_t* __restrict__ rowseq,
                                                                const uint32_t* __restrict__ rowspan,
                                                                const uint32_t* __restrict__ plan,
                                                                const uint32_t* __restrict__ tab, int gx, int gy,
                                                                uint32_t* __restrict__ list, size_t cap) {
  after_previous();
  const uint32_t* rs = plan;
  const uint32_t* cb = plan + gy + 1;
  if (plan[3 * gy + 2] == 0u) return;
  const uint32_t C = cb[gy];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (uint32_t kg = blockIdx.x; kg < C; kg += gridDim.x) {
    const int y = chunk_row(cb, gy, kg);
    const uint32_t c0 = cb[y], nch = cb[y + 1] - c0, k = kg - c0;
    const uint32_t i0 = rs[y] + 256u * k, i1 = min(rs[y + 1], i0 + 256u);
    WarpSpans S;
    load_chunk(rowspan, i0, i1, lane, S);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const uint32_t i = i0 + 32 * c + lane;
      S.v0[c] = i < i1 ? rowseq[i] : 0u;
    }
    const int x = w + kBinWarps * lane;
    const uint32_t base = x < gx ? tab[(size_t)c0 * gx + (size_t)x * nch + k] : 0u;
    scan_place<false>(S, S.v0, gx, w, kBinWarps, base, list, nullptr, cap);
  }
}

// Counts per (row, column, chunk): a difference array over the columns of
// the chunk's spans, then its running sum, at tab[cb[y] gx + x nch + k]
// (row y's counts in (column, chunk) order); adds the chunk's list entries
// to the row's pairs.
__global__ void __launch_bounds__(kBinThreads) k_bin_count(const uint32_t* __restrict__ rowspan,
                                                           uint32_t* __restrict__ plan, int gx, int gy, uint32_t ch,
                                                           uint32_t* __restrict__ tab) {
  after_previous();
  __shared__ int d[kMaxTileAxis + 1];
  __shared__ uint32_t sm[32];
  BinPlan P(plan, gy);
  if (*P.ok == 0u) return;
  const uint32_t C = P.cb[gy];
  for (uint32_t kg = blockIdx.x; kg < C; kg += gridDim.x) {
    const int y = chunk_row(P.cb, gy, kg);
    const uint32_t c0 = P.cb[y], nch = P.cb[y + 1] - c0, k = kg - c0;
    const uint32_t i0 = P.rs[y] + k * ch, i1 = min(P.rs[y + 1], i0 + ch);
    for (int x = threadIdx.x; x <= gx; x += kBinThreads) d[x] = 0;
    __syncthreads();
    uint32_t width = 0;
    for (uint32_t i = i0 + threadIdx.x; i < i1; i += kBinThreads) {
      const uint32_t sp = rowspan[i];
      const int x0 = (int)(sp & 0xFFFFu), x1 = (int)(sp >> 16);
      atomicAdd(&d[x0], 1);
      atomicAdd(&d[x1 + 1], -1);
      width += (uint32_t)(x1 - x0 + 1);
    }
    const uint32_t total = block_sum<kBinThreads>(width, sm);  // also orders the difference array's updates
    if (threadIdx.x == 0 && total) atomicAdd(P.pairs + y, total);
    if (threadIdx.x < 32) {
      const int lane = threadIdx.x;
      uint32_t* out = tab + (size_t)c0 * gx + k;
      uint32_t run = 0;
      for (int x0 = 0; x0 < gx; x0 += 32) {
        const int x = x0 + lane;
        const uint32_t v = warp_inclusive_sum(x < gx ? (uint32_t)d[x] : 0u, lane);
        if (x < gx) out[(size_t)x * nch] = run + v;
        run += __shfl_sync(0xffffffffu, v, 31);
      }
    }
    __syncthreads();  // d is cleared for the next chunk
  }
}

constexpr int kRowscanThreads = 512;  // a block of 1024 finds no room beside a networks' block

// One block per row: the row's counts scanned in (column, chunk) order after
// the list entries of the rows above; tile (y, x) starts at the scanned count
// of its first chunk.  The last row also writes the end of the last tile.
__global__ void __launch_bounds__(kRowscanThreads) k_bin_rowscan(uint32_t* __restrict__ tab, const uint32_t* __restrict__ plan,
                                                      int gx, int gy, uint32_t* __restrict__ tile_start) {
  after_previous();
  __shared__ uint32_t sm[32];
  const int y = blockIdx.x;
  const uint32_t* cb = plan + gy + 1;
  const uint32_t* pairs = plan + 2 * gy + 2;
  uint32_t* ts = tile_start + (size_t)y * gx;
  if (plan[3 * gy + 2] == 0u) {  // over capacity: every list empty
    for (int x = threadIdx.x; x < gx; x += blockDim.x) ts[x] = 0u;
    if (y == gy - 1 && threadIdx.x == 0) tile_start[(size_t)gx * gy] = 0u;
    return;
  }
  uint32_t above = 0;
  for (int t = threadIdx.x; t < y; t += blockDim.x) above += pairs[t];
  above = block_sum<kRowscanThreads>(above, sm);
  const uint32_t c0 = cb[y], nch = cb[y + 1] - c0;
  uint32_t* seg = tab + (size_t)c0 * gx;
  const uint32_t end = block_scan_inplace<kRowscanThreads>(seg, (size_t)nch * gx, above, sm);
  for (int x = threadIdx.x; x < gx; x += blockDim.x) ts[x] = seg[(size_t)x * nch];
  if (y == gy - 1 && threadIdx.x == 0) tile_start[(size_t)gx * gy] = end;
}

// The list entries: each chunk in steps of 256 items over their columns,
// starting at the chunk's offsets in its tiles.
__global__ void __launch_bounds__(kBinThreads) k_bin_place(const uint32_t* __restrict__ rowseq,
                                                           const uint32_t* __restrict__ rowspan,
                                                           const uint32_t* __restrict__ plan,
                                                           const uint32_t* __restrict__ tab, int gx, int gy,
                                                           uint32_t ch, uint32_t* __restrict__ list, size_t cap) {
  after_previous();
  __shared__ SpanSmem S;
  const uint32_t* rs = plan;
  const uint32_t* cb = plan + gy + 1;
  if (plan[3 * gy + 2] == 0u) return;
  const uint32_t C = cb[gy];
  for (uint32_t kg = blockIdx.x; kg < C; kg += gridDim.x) {
    const int y = chunk_row(cb, gy, kg);
    const uint32_t c0 = cb[y], nch = cb[y + 1] - c0, k = kg - c0;
    const uint32_t i0 = rs[y] + k * ch, i1 = min(rs[y + 1], i0 + ch);
    for (int x = threadIdx.x; x < gx; x += kBinThreads) S.run[x] = tab[(size_t)c0 * gx + (size_t)x * nch + k];
    __syncthreads();
    for (uint32_t sub = i0; sub < i1; sub += kBinThreads) {
      const uint32_t i = sub + threadIdx.x;
      int a = 0, b = -1;
      uint32_t r = 0;
      if (i < i1) {
        r = rowseq[i];
        const uint32_t sp = rowspan[i];
        a = (int)(sp & 0xFFFFu);
        b = (int)(sp >> 16);
      }
      place_spans(S, gx, a, b, r, 0u, list, nullptr, cap);
    }
    __syncthreads();  // S.run is rewritten for the next chunk
  }
}

}  // namespace

void launch_binning(const FrameArgs& f, int sp, cudaStream_t s) {
  const SplatBufs& b = f.L->sp[sp];
  unsigned char* ws = f.ws;
  const int n = f.sc.n;
  const int gx = f.L->gx, gy = f.L->gy, nb = f.L->nb_rows;
  const size_t cap = f.L->cap;
  uint32_t* header = at<uint32_t>(ws, f.L->header);
  const int h_need = sp ? H_NEED_LIGHT : H_NEED_CAM;
  const int h_pairs = sp ? H_PAIRS_LIGHT : H_PAIRS_CAM;
  // the lists go where the composites and the backward read them; the row
  // sequence and spans use buffers that are free until then
  const int fin = (f.L->ntiles <= 256 ? 1 : 2) & 1;
  uint32_t* list = at<uint32_t>(ws, b.tv[fin]);
  uint32_t* rowseq = at<uint32_t>(ws, b.tk[fin]);
  uint32_t* rowspan = at<uint32_t>(ws, b.tv[1 - fin]);
  uint32_t* row_cnt = at<uint32_t>(ws, b.row_cnt);
  uint32_t* plan = at<uint32_t>(ws, b.bin_plan);
  uint32_t* tab = at<uint32_t>(ws, b.bin_tab);
  const uint32_t ch = bin_chunk(gx);
  launch_after(k_bin_plan, gy + 1, kBinThreads, 0, s, row_cnt, nb, gy, ch, bin_tab_words(cap, gx, gy), gx, plan, header,
               h_need, h_pairs, cap);
  uint32_t* off = at<uint32_t>(ws, b.off);
  const SplatRec* rrec = at<SplatRec>(ws, b.rrec);
  if (gy <= kScanBuckets)
    launch_after(k_bin_rows_scan, nb, kBinThreads, 0, s, n, rrec, row_cnt, nb, gy, plan, rowseq, rowspan, off, cap);
  else
    launch_after(k_bin_rows, nb, kBinThreads, 0, s, n, rrec, row_cnt, nb, gy, plan, rowseq, rowspan, off, cap);
  const size_t chunks = cap / ch + (size_t)gy + 1;
  const bool scan = gx <= kScanBuckets;  // chunks of 256 items
  int grid = device_sm_count() * (scan ? 8 : 5);
  if ((size_t)grid > chunks) grid = (int)chunks;
  const int wgrid = (int)((chunks + kBinWarps - 1) / kBinWarps);
  if (scan) launch_after(k_bin_count_warp, wgrid < grid ? wgrid : grid, kBinThreads, 0, s, rowspan, plan, gx, gy, tab);
  else launch_after(k_bin_count, grid, kBinThreads, 0, s, rowspan, plan, gx, gy, ch, tab);
  launch_after(k_bin_rowscan, gy, kRowscanThreads, 0, s, tab, plan, gx, gy, at<uint32_t>(ws, b.tile_start));
  if (scan) launch_after(k_bin_place_scan, grid, kBinThreads, 0, s, rowseq, rowspan, plan, tab, gx, gy, list, cap);
  else launch_after(k_bin_place, grid, kBinThreads, 0, s, rowseq, rowspan, plan, tab, gx, gy, ch, list, cap);
  count_launch(5);
}

}  // namespace gs3
