// K2-K3: the depth sort of one splat (camera or light) and the records in
// depth-rank order; the paper bins the light view with the same splatting
// pipeline as the camera view (Sec. 3, Sec. 4.2).
//
//   1. stable radix sort of the N FP32 depth keys (index payload, emitted in
//      index order), one pass per 8-bit digit with decoupled look-back
//      -> rank r, order[r]
//   2. records gathered into rank order, tile counts per rank, and the counts
//      per (tile row, block of ranks) that the binning by counting
//      (tile_bin.cu) starts from
// Ties in depth keep index order, so a tile's list is ascending (depth bits,
// index), as a stable sort of 64-bit (tile << 32 | depth) keys emitted in
// index order would give.
#include "gs3_internal.cuh"

namespace gs3 {
namespace {

// ---------------------------------------------------------------------------
// Stable LSD radix sort pass, 8-bit digit, u32 key + u32 value.
// ---------------------------------------------------------------------------
// ---------------------------------------------------------------------------
// The depth sorts, one kernel per digit pass (decoupled look-back).  Each
// block takes the next kSortThreads * ROUNDS items in order by a ticket, ranks
// them within their digit and stages them in shared memory sorted by digit,
// so that each digit's run of the block leaves as contiguous stores.  Warp w
// ranks its own 32 * ROUNDS consecutive items against its own digit counters
// (no block barrier per round); a block scan over (digit, warp) then places
// the warps' runs, so the order within a digit is the items' order (stable).
// The block publishes its count of every digit, and adds up the counts of the
// blocks before it from their published words: a block's own count (flag 2
// pass + 1) or, once that block finished its look-back, the count of it and of
// every block before it (flag 2 pass + 2); the words of an earlier pass have
// lower flags, so one region, zeroed once, serves all passes.  Four words are
// read at a time, so a look-back over blocks that have not finished theirs
// waits for a quarter of the loads (a pass over 300k keys: 13.0 -> 11.5 us).  A block waits only on blocks with
// smaller tickets, which have started and never wait on it; every wait is
// bounded: past kLookSpin polls the block records GS3_ERR_TIMEOUT in the
// header and goes on.  The digits' global starts come from totals counted once
// before the first pass, so no histogram pass or device-wide scan runs between
// the passes.
// ---------------------------------------------------------------------------
constexpr int kLookSpin = 1 << 20;
constexpr int kLookWords = 4;

// Every digit of every pass (PASSES eight-bit digits), counted over the n keys.  Warp-private counters; a warp whose 32 keys share a digit (usual
// for the top digits of the depth keys) adds it once.
template <int PASSES>
__global__ void __launch_bounds__(256) k_digit_totals(const uint32_t* __restrict__ keys, uint32_t n,
                                                      uint32_t* __restrict__ totals) {
  __shared__ uint32_t h[PASSES][kSortThreads / 32][256];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
#pragma unroll
  for (int p = 0; p < PASSES; ++p)
#pragma unroll
    for (int w = 0; w < kSortThreads / 32; ++w) h[p][w][t] = 0;
  __syncthreads();
  // each warp takes 128 consecutive keys per step, four coalesced loads in flight per lane
  for (uint32_t wb = (blockIdx.x * (kSortThreads / 32) + warp) * 128u; wb < n; wb += gridDim.x * kSortThreads * 4u) {
    uint32_t k[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t i = wb + 32u * u + lane;
      k[u] = i < n ? keys[i] : 0u;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const bool valid = wb + 32u * u + lane < n;
      const uint32_t vm = __ballot_sync(0xffffffffu, valid);
      if (!vm) break;
#pragma unroll
      for (int p = 0; p < PASSES; ++p) {
        const uint32_t d = (k[u] >> (8 * p)) & 255u;
        const uint32_t first = __shfl_sync(0xffffffffu, d, 0);
        if (__all_sync(0xffffffffu, !valid || d == first)) {
          if (lane == 0) h[p][warp][first] += __popc(vm);
        } else if (valid) {
          atomicAdd(&h[p][warp][d], 1u);
        }
        __syncwarp();
      }
    }
  }
  __syncthreads();
  for (int p = 0; p < PASSES; ++p) {
    uint32_t c = 0;
#pragma unroll
    for (int w = 0; w < kSortThreads / 32; ++w) c += h[p][w][t];
    if (c) atomicAdd(&totals[p * 256 + t], c);
  }
}

template <int ROUNDS>
struct OnesweepSmem {
  uint32_t base[256];    // the block's first output slot per digit
  uint32_t start[256];   // first staging slot per digit
  uint32_t cnt[kSortThreads / 32][256];  // per warp and digit: items so far, then the warp's first slot
  uint32_t wsum[kSortThreads / 32], gsum[kSortThreads / 32];
  uint32_t ticket;
  uint32_t key[kSortThreads * ROUNDS], val[kSortThreads * ROUNDS];
};

template <int ROUNDS>
__global__ void __launch_bounds__(kSortThreads, 3) k_onesweep(
    const uint32_t* __restrict__ kin, const uint32_t* __restrict__ vin, uint32_t* __restrict__ kout,
    uint32_t* __restrict__ vout, uint32_t n, int shift,
    const uint32_t* __restrict__ totals, unsigned long long* look, uint32_t* ticket, uint32_t* header) {
  after_previous();
  constexpr int kItems = kSortThreads * ROUNDS;
  constexpr int kWarps = kSortThreads / 32;
  extern __shared__ uint4 onesweep_raw[];
  OnesweepSmem<ROUNDS>& S = *reinterpret_cast<OnesweepSmem<ROUNDS>*>(onesweep_raw);
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  if (t == 0) S.ticket = atomicAdd(ticket, 1u);
#pragma unroll
  for (int w = 0; w < kWarps; ++w) S.cnt[w][t] = 0;
  __syncthreads();
  const uint32_t blk = S.ticket;
  const uint32_t base = blk * (uint32_t)kItems;
  if (base >= n) return;  // every later ticket is past the end as well
  const uint32_t lt = (1u << lane) - 1u;
  const uint32_t wbase = base + (uint32_t)warp * (32u * ROUNDS);
  uint32_t kk[ROUNDS], vv[ROUNDS];
  uint32_t rk[(ROUNDS + 1) / 2];  // two 16-bit ranks per word
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) {
    const uint32_t i = wbase + r * 32 + lane;
    const bool valid = i < n;
    kk[r] = valid ? kin[i] : 0u;
    vv[r] = valid ? (vin ? vin[i] : i) : 0u;
  }
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) {
    const bool valid = wbase + r * 32 + lane < n;
    const uint32_t d = valid ? (kk[r] >> shift) & 255u : 256u;
    const uint32_t peers = __match_any_sync(0xffffffffu, d);
    const int leader = __ffs(peers) - 1;
    uint32_t c = 0;
    if (valid && lane == leader) c = S.cnt[warp][d];
    c = __shfl_sync(0xffffffffu, c, leader);
    const uint32_t rank = c + __popc(peers & lt);
    rk[r >> 1] = (r & 1) ? (rk[r >> 1] | (rank << 16)) : rank;
    if (valid && lane == leader) S.cnt[warp][d] = c + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  {
    // thread t = digit t: the block's count, published at once
    uint32_t tot = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const uint32_t c = S.cnt[w][t];
      S.cnt[w][t] = tot;
      tot += c;
    }
    volatile unsigned long long* mine = look + (size_t)blk * 256 + t;
    const uint32_t agg = 2u * ((uint32_t)shift / 8u) + 1u, pre = agg + 1u;  // this pass's flags
    *mine = (unsigned long long)(blk == 0 ? pre : agg) << 32 | tot;
    // staging starts (scan of the block's counts) and the digit's start over
    // all items (scan of the totals)
    const uint32_t g = totals[t];
    uint32_t x = tot, y = g;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t a = __shfl_up_sync(0xffffffffu, x, o);
      const uint32_t b = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= o) { x += a; y += b; }
    }
    if (lane == 31) { S.wsum[warp] = x; S.gsum[warp] = y; }
    // the blocks before this one
    uint32_t excl = 0;
    if (blk > 0) {
      uint32_t j = blk;  // blocks [0, j) are still to be added
      int spins = 0;
      while (j > 0) {
        unsigned long long v[kLookWords];
#pragma unroll
        for (int i = 0; i < kLookWords; ++i)
          v[i] = *(volatile const unsigned long long*)(look + (size_t)(j > (uint32_t)i ? j - 1 - i : 0) * 256 + t);
        bool wait = false;
#pragma unroll
        for (int i = 0; i < kLookWords; ++i) {
          if (wait || j == 0) continue;
          const uint32_t flag = (uint32_t)(v[i] >> 32);
          if (flag < agg) {
            wait = true;
          } else {
            excl += (uint32_t)v[i];
            j = flag == pre ? 0 : j - 1;
          }
        }
        if (wait) {
          if (++spins > kLookSpin) {
            atomicCAS(header + H_STATUS, 0u, (uint32_t)GS3_ERR_TIMEOUT);
            break;
          }
          __nanosleep(32);
        }
      }
      *mine = (unsigned long long)pre << 32 | (excl + tot);
    }
    __syncthreads();
    uint32_t before = 0, gbefore = 0;
    for (int w = 0; w < warp; ++w) { before += S.wsum[w]; gbefore += S.gsum[w]; }
    const uint32_t st = before + x - tot;
    S.start[t] = st;
    S.base[t] = gbefore + y - g + excl;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) S.cnt[w][t] += st;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) {
    if (wbase + r * 32 + lane < n) {
      const uint32_t lp = S.cnt[warp][(kk[r] >> shift) & 255u] + ((rk[r >> 1] >> (16 * (r & 1))) & 0xFFFFu);
      S.key[lp] = kk[r];
      S.val[lp] = vv[r];
    }
  }
  __syncthreads();
  const uint32_t cnt = min((uint32_t)kItems, n - base);
  for (uint32_t i = t; i < cnt; i += kSortThreads) {
    const uint32_t k = S.key[i];
    const uint32_t d = (k >> shift) & 255u;
    const uint32_t pos = S.base[d] + (i - S.start[d]);
    if (pos < n) {
      kout[pos] = k;
      vout[pos] = S.val[i];
    }
  }
}

// ---------------------------------------------------------------------------
// The whole depth sort of at most kSmallSort keys by one block: the four passes
// of k_onesweep with the keys in registers and shared memory between them, and
// no look-back.  Warp w holds the 32 R consecutive keys from 32 R w on.  It waits for
// nothing, and sets *status (if given) to 0.
// Bound: the passes' chains of barriers.  1000 / 4000 keys: 9 / 19 us, against 21 / 23
// in six launches (4096: 19.3 against 22.8); past that several blocks gain.
constexpr int kSmallSort = 4096;
constexpr int kSmallThreads = 512;
__global__ void __launch_bounds__(kSmallThreads) k_sort_small(const uint32_t* __restrict__ kin,
                                                              uint32_t* __restrict__ kout,
                                                              uint32_t* __restrict__ vout, uint32_t n,
                                                              uint32_t* status) {
  after_previous();
  if (status && threadIdx.x == 0) *status = 0u;
  constexpr int kWarps = kSmallThreads / 32, kRounds = kSmallSort / kSmallThreads;
  __shared__ uint32_t key[kSmallSort];
  __shared__ uint16_t val[kSmallSort];
  __shared__ uint32_t cnt[kWarps][256];  // per warp and digit: items so far, then the warp's first slot
  __shared__ uint32_t low[256], start[256], wsum[8];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31, digit = t & 255, half = t >> 8;
  const uint32_t R = (n + kSmallThreads - 1) / kSmallThreads, lt = (1u << lane) - 1u;
  const uint32_t first = (uint32_t)warp * 32u * R + lane;
  uint32_t kk[kRounds], vv[kRounds], rk[kRounds];
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    const uint32_t i = first + 32u * r;
    kk[r] = (uint32_t)r < R && i < n ? kin[i] : 0u;
    vv[r] = i;
  }
  for (int shift = 0; shift < 32; shift += 8) {
#pragma unroll
    for (int w = 0; w < kWarps; w += 2) cnt[w + half][digit] = 0u;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
      if ((uint32_t)r >= R) break;  // the same for every lane
      const bool valid = first + 32u * r < n;
      const uint32_t d = valid ? (kk[r] >> shift) & 255u : 256u;
      const uint32_t peers = __match_any_sync(0xffffffffu, d);
      const int leader = __ffs(peers) - 1;
      uint32_t c = 0;
      if (valid && lane == leader) c = cnt[warp][d];
      c = __shfl_sync(0xffffffffu, c, leader);
      rk[r] = c + __popc(peers & lt);
      if (valid && lane == leader) cnt[warp][d] = c + __popc(peers);
      __syncwarp();
    }
    __syncthreads();
    // two threads per digit, eight warps each; the upper ones scan the digits
    uint32_t tot = 0;
#pragma unroll
    for (int w = 0; w < kWarps / 2; ++w) {
      const uint32_t c = cnt[8 * half + w][digit];
      cnt[8 * half + w][digit] = tot;
      tot += c;
    }
    if (half == 0) low[digit] = tot;
    __syncthreads();
    uint32_t x = 0, all = 0;
    if (half == 1) {
      all = x = low[digit] + tot;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      if (lane == 31) wsum[warp & 7] = x;
    }
    __syncthreads();
    if (half == 1) {
      uint32_t before = 0;
      for (int w = 0; w < (warp & 7); ++w) before += wsum[w];
      start[digit] = before + x - all;
    }
    __syncthreads();
    const uint32_t base = start[digit] + (half ? low[digit] : 0u);
#pragma unroll
    for (int w = 0; w < kWarps / 2; ++w) cnt[8 * half + w][digit] += base;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
      if ((uint32_t)r < R && first + 32u * r < n) {
        const uint32_t pos = cnt[warp][(kk[r] >> shift) & 255u] + rk[r];
        if (shift == 24) {
          kout[pos] = kk[r];
          vout[pos] = vv[r];
        } else {
          key[pos] = kk[r];
          val[pos] = (uint16_t)vv[r];
        }
      }
    }
    __syncthreads();
    if (shift == 24) break;
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
      const uint32_t i = first + 32u * r;
      if ((uint32_t)r < R && i < n) {
        kk[r] = key[i];
        vv[r] = val[i];
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Rank order and counts
// ---------------------------------------------------------------------------
// Records into depth-rank order and the tile count of each rank.  Also
// counts, for the block's kBinBlock ranks, the ranks whose rectangle covers
// each tile row y (a difference array over the rows, then its running sum),
// into row_cnt[y][block], and adds up the block's tile counts into
// row_cnt[gy][block].  Clears the binning's ticket (the plan's last word).
__global__ void __launch_bounds__(kBinBlock) k_reorder(int n, const uint32_t* __restrict__ order,
                                                       const SplatRec* __restrict__ rec, SplatRec* __restrict__ rrec,
                                                       uint32_t* __restrict__ rank_of, uint32_t* __restrict__ cnt,
                                                       const float4* __restrict__ shade, float4* __restrict__ ccol,
                                                       uint32_t* __restrict__ row_cnt, int gy, uint32_t* __restrict__ ticket,
                                                       uint32_t* nonfinite) {
  after_previous();
  __shared__ int d[kMaxTileAxis + 1];
  __shared__ uint32_t tiles;
  if (threadIdx.x == 0) {
    tiles = 0u;
    if (blockIdx.x == 0) *ticket = 0u;
  }
  for (int y = threadIdx.x; y <= gy; y += blockDim.x) d[y] = 0;
  __syncthreads();
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t g = r < n ? order[r] : 0xFFFFFFFFu;
  uint32_t c = 0u;  // the rank's tiles
  if (g < (uint32_t)n) {
    const SplatRec q = rec[g];
    rrec[r] = q;
    rank_of[g] = r;
    const bool in = q.r.x >= 0;
    c = in ? (uint32_t)(q.r.z - q.r.x + 1) * (uint32_t)(q.r.w - q.r.y + 1) : 0u;
    cnt[r] = c;
    if (in) {
      atomicAdd(&d[q.r.y], 1);
      atomicAdd(&d[q.r.w + 1], -1);
    }
    if (ccol) {
      const float4 col = shade[g];
      ccol[2 * r] = make_float4(col.x, col.y, col.z, 0.f);
      if (non_finite(col.x + col.y + col.z)) *nonfinite = 1u;
    }
  }
  c = __reduce_add_sync(0xffffffffu, c);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(&tiles, c);
  __syncthreads();
  if (threadIdx.x == 32) row_cnt[(size_t)gy * gridDim.x + blockIdx.x] = tiles;
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    int run = 0;
    for (int y0 = 0; y0 < gy; y0 += 32) {
      const int y = y0 + lane;
      int v = y < gy ? d[y] : 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
      }
      if (y < gy) row_cnt[(size_t)y * gridDim.x + blockIdx.x] = (uint32_t)(run + v);
      run += __shfl_sync(0xffffffffu, v, 31);
    }
  }
}

// Stable LSD sort of n keys with their positions on the low 8 * PASSES bits: one
// k_digit_totals, then one k_onesweep per pass.  Even passes write (k0, v0),
// odd passes (k1, v1), each reading the previous pass's output (pass 0 reads
// kin and the positions).  look_region: onesweep_bytes(nblocks, PASSES) bytes, zeroed
// here.  Up to kSmallSort keys: one launch of k_sort_small, whose output is (k1, v1).
// own_status: the kOrderFront bytes before look_region belong to the sort and start
// with `header`, the word for its status, which is cleared as well.  first_ticket: of
// the first pass (past 0: a self-test, its waits run out).
template <int ROUNDS>
void onesweep_sort(const uint32_t* kin, uint32_t* k0, uint32_t* v0, uint32_t* k1, uint32_t* v1, uint32_t n, int nblocks,
                   unsigned char* look_region, uint32_t* header, cudaStream_t s, bool wait = false,
                   bool own_status = false, int first_ticket = 0) {
  constexpr int PASSES = 4;
  if (n <= kSmallSort) {
    launch_behind(wait, k_sort_small, 1, kSmallThreads, 0, s, kin, k1, v1, n, own_status ? header : nullptr);
    count_launch();
    return;
  }
  static DeviceOnce once;
  once.run([] {
    return cudaFuncSetAttribute(k_onesweep<ROUNDS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)sizeof(OnesweepSmem<ROUNDS>)) == cudaSuccess;
  });
  unsigned long long* look = reinterpret_cast<unsigned long long*>(look_region);
  uint32_t* tickets = reinterpret_cast<uint32_t*>(look + 256 * (size_t)nblocks);
  uint32_t* totals = tickets + PASSES;
  const size_t front = own_status ? kOrderFront : 0;
  cudaMemsetAsync(look_region - front, 0, front + onesweep_bytes(nblocks, PASSES), s);
  if (first_ticket) cudaMemsetAsync(tickets, first_ticket, 1, s);
  const int tb_cap = device_sm_count() * 4, tb = (int)((n + 1023) / 1024);
  k_digit_totals<PASSES><<<tb < tb_cap ? tb : tb_cap, kSortThreads, 0, s>>>(kin, n, totals);
  const uint32_t* ki = kin;
  const uint32_t* vi = nullptr;
  for (int p = 0; p < PASSES; ++p) {
    uint32_t* ko = (p & 1) ? k1 : k0;
    uint32_t* vo = (p & 1) ? v1 : v0;
    launch_after(k_onesweep<ROUNDS>, nblocks, kSortThreads, sizeof(OnesweepSmem<ROUNDS>), s, ki, vi, ko, vo, n, 8 * p,
                 totals + 256 * p, look, tickets + p, header);
    ki = ko;
    vi = vo;
  }
  count_launch(1 + PASSES);
}

}  // namespace

// gs3_depth_order_static: 1024 keys per block up to 512 blocks, 2048 past that
// (GS3_STATIC_SORT_MAX_KEYS is 512 such blocks), so that a few hundred thousand
// keys fill the chip and the look-back region stays at 1 MB.
void depth_order(const uint32_t* keys, uint32_t n, uint32_t* k0, uint32_t* v0, uint32_t* k1, uint32_t* order,
                 unsigned char* front, cudaStream_t s, int first_ticket) {
  unsigned char* look = front + kOrderFront;
  uint32_t* status = reinterpret_cast<uint32_t*>(front);
  auto blocks = [&](int rounds) { return (int)((n + kSortThreads * rounds - 1) / (kSortThreads * rounds)); };
  if (blocks(4) <= kDepthOrderBlocks)
    onesweep_sort<4>(keys, k0, v0, k1, order, n, blocks(4), look, status, s, false, true, first_ticket);
  else
    onesweep_sort<8>(keys, k0, v0, k1, order, n, blocks(8), look, status, s, false, true, first_ticket);
}

void launch_depth_sort(const FrameArgs& f, int sp, cudaStream_t s, bool wait) {
  const SplatBufs& b = f.L->sp[sp];
  unsigned char* ws = f.ws;
  const int n = f.sc.n;
  // 1024 keys per block, so that a few hundred thousand keys fill the SMs
  onesweep_sort<kDepthSortRounds>(at<uint32_t>(ws, b.key), at<uint32_t>(ws, b.sk[0]), at<uint32_t>(ws, b.sv[0]),
                                  at<uint32_t>(ws, b.sk[1]), at<uint32_t>(ws, b.sv[1]), (uint32_t)n, f.L->nb_n,
                                  at<unsigned char>(ws, b.dlook), at<uint32_t>(ws, f.L->header), s, wait);
  // 4 passes end in buffer 1: sv[1] holds the index of each depth rank
  launch_after(k_reorder, f.L->nb_rows, kBinBlock, 0, s, n, at<uint32_t>(ws, b.sv[1]), at<SplatRec>(ws, b.rec), at<SplatRec>(ws, b.rrec),
      at<uint32_t>(ws, b.rank_of), at<uint32_t>(ws, b.cnt), at<float4>(ws, f.L->shade),
      sp == 0 ? at<float4>(ws, f.L->ccol) : nullptr, at<uint32_t>(ws, b.row_cnt), f.L->gy,
               at<uint32_t>(ws, b.bin_plan) + 3 * f.L->gy + 3, at<uint32_t>(ws, f.L->header) + H_NONFINITE);
  count_launch();
}

}  // namespace gs3

// Self-test of the bounded waits: one look-back pass over n zero keys whose
// tickets start at 1, so every block's look-back reaches ticket 0's words,
// which no block writes.  Each such wait must give up after kLookSpin polls
// and record GS3_ERR_TIMEOUT; the pass then finishes.
extern "C" gs3_status gs3_selftest_wait_timeout(uint32_t n, uint32_t* status_out) {
  using namespace gs3;
  if (!status_out || n <= (uint32_t)kTileSortItems || n > (1u << 20)) {
    set_last_error("gs3_selftest_wait_timeout: need status_out and 4096 < n <= 1 << 20");
    return GS3_ERR_INVALID_ARG;
  }
  const int nblocks = (int)((n + kTileSortItems - 1) / kTileSortItems);
  const size_t look = onesweep_bytes(nblocks, 1);
  const size_t bytes = 16ull * n + look + 16;
  unsigned char* d = nullptr;
  if (cudaMalloc(&d, bytes) != cudaSuccess) {
    set_last_error("gs3_selftest_wait_timeout: cudaMalloc failed");
    return GS3_ERR_OOM;
  }
  uint32_t* kin = reinterpret_cast<uint32_t*>(d);
  uint32_t* vin = kin + n;
  uint32_t* kout = vin + n;
  uint32_t* vout = kout + n;
  unsigned long long* lk = reinterpret_cast<unsigned long long*>(d + 16ull * n);
  uint32_t* tickets = reinterpret_cast<uint32_t*>(lk + 256ull * nblocks);
  uint32_t* totals = tickets + 1;
  uint32_t* status = reinterpret_cast<uint32_t*>(d + 16ull * n + look);
  const uint32_t first_ticket = 1;
  cudaError_t e = cudaMemset(d, 0, bytes);
  if (e == cudaSuccess) e = cudaMemcpy(tickets, &first_ticket, 4, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    cudaFuncSetAttribute(k_onesweep<kTileSortRounds>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sizeof(OnesweepSmem<kTileSortRounds>));
    k_onesweep<kTileSortRounds><<<nblocks, kSortThreads, sizeof(OnesweepSmem<kTileSortRounds>)>>>(
        kin, vin, kout, vout, n, 0, totals, lk, tickets, status);
    count_launch();
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e == cudaSuccess) e = cudaMemcpy(status_out, status, 4, cudaMemcpyDeviceToHost);
  cudaFree(d);
  if (e != cudaSuccess) {
    set_last_error("gs3_selftest_wait_timeout: CUDA call failed");
    return GS3_ERR_CUDA;
  }
  return GS3_OK;
}
