// K8b: backward of the Phi (Sec. 4.2) and Psi (Sec. 4.3) MLPs with hidden widths
// of 32, 64 or 128, on the tensor cores, every FP32 operand as three BF16 values
// (mlp_x3.cu has the split and its products; widths of 16: mlp_bwd.cu).
//
// With h_0 = encode(Gaussian), h_l = act(W_l h_{l-1} + b_l), y = sigmoid(W_o h_L + b_o):
//   dz_o = dL/dy y (1 - y),  dz_L = (dz_o W_o) act'(h_L),  dz_l = (dz_{l+1} W_{l+1}) act'(h_l),
//   dh_0 = dz_1 W_1,  dW_l = sum over the Gaussians of dz_l h_{l-1}^T,  db_l = sum of dz_l.
//
// k_mlp_x3_rows carries a tile of 128 Gaussians through the whole chain, with
// the forward kernel's arrangement: encoded inputs, the hidden layers forward,
// the output layer and its gradient, the data gradients down to the inputs and
// through the encoding.  The forward products are three-pass TF32 (x as its 10
// leading mantissa bits and the rest, small' terms first, one accumulator), as in a
// GEMM per layer: the signs of h decide act', and a pre-activation within rounding
// of zero keeps the side that form gives it.  BF16 triples would be nearer to
// float64, and the frame's own networks use them (mlp_x3.cu), so for a few such
// pre-activations this side is not the frame's.  On the way back only the signs are
// needed; they stay in shared memory.  The activations (h_0 .. h_{L-1},
// dz_L .. dz_1) go to global memory as the weight gradients contract them: h from
// registers (eight lanes fill a 128-byte core matrix), dz, which lies in shared
// memory in that form, by one warp's bulk copies under the next layer's MMAs.
// dW_o: a warp adds dz_o h_L over its 32 rows by a transposing butterfly (16
// shuffles per 16 columns and output).
//
// k_mlp_x3_wgrad contracts those tiles over the Gaussians: the same bytes read
// as MN-major operands (a core matrix of 8 Gaussians x 8 units serves both
// ways), so that a step is bulk copies and MMAs alone; db_l from 16 columns of
// ones.  CTAs own contiguous row ranges, k_mlp_x3_sum adds their partials in
// order: no result depends on scheduling.
//
// The tiles pass in batches of kBatchTiles, which bounds the stored activations (at
// most 1.3 GB for 3 x 128, 1.8 GB for 4 x 128); the weight partials are kept per
// batch (3 x 128: 25 MB per 311,296 Gaussians).  Smaller batches, down to those that
// stay in L2, take 4 to 20 % longer: a launch's last tiles leave SMs idle.
//
// Bound: k_mlp_x3_rows by the chain of its 2 L products, one tile per SM at a time
// (the hand-overs; a third of its MMAs less changes nothing), k_mlp_x3_wgrad by
// reading the tiles (6.2 TB/s).  300k Gaussians, 3 x 128, both networks: rows 1.11,
// weight gradients 0.40, sums and weights 0.04 ms, against 2.70 ms as one three-pass
// TF32 GEMM per layer and direction with FP32 activations in between.  Gradients
// against float64: the same error (a product keeps 2^-26 here, 2^-21 there).
// Forward products split into BF16 as well take 0.15 ms less, but then the signs
// of a few pre-activations differ, and single Gaussians' gradients with them.
#include "mlp_x3.cuh"

namespace gs3 {
namespace {

using namespace x3;

constexpr int kThreads = kEpiThreads + 96;  // and the MMA, weight and store warps
constexpr int kColorStride = 8;
constexpr int kMlpInStride = 24;
constexpr int kMaxCtas = 152;      // one per SM
constexpr int kBatchTiles = 16 * kMaxCtas;

__host__ __device__ inline int wide(int W) { return W > kK0 ? W : kK0; }
// activations in shared memory: forward two TF32 parts, backward three BF16 splits
__host__ __device__ inline uint32_t act_bytes(int W) { return 2u * kRows * 4u * (uint32_t)wide(W); }
// a tile's stored activations: h_0, h_1 .. h_{nh-1}, dz_1 .. dz_nh
__host__ __device__ inline size_t tile_bytes(int W, int nh) { return 3ull * kRows * 2 * (kK0 + (2 * nh - 1) * (size_t)W); }
__host__ __device__ inline size_t h_off(int W, int l) { return l == 0 ? 0 : 3ull * kRows * 2 * (kK0 + (l - 1) * (size_t)W); }
__host__ __device__ inline size_t dz_off(int W, int nh, int l) { return 3ull * kRows * 2 * (kK0 + (nh - 1 + l) * (size_t)W); }
// weight chunks (16 inputs) of a tile's products: W_l forward as two TF32 parts,
// then W_l^T from the last to the first, which alone has 64 output units, as
// three BF16 splits
constexpr int kStep = 16;
__host__ __device__ inline uint32_t fwd_bytes(int rows) { return (uint32_t)rows * kStep * 8u; }
__host__ __device__ inline uint32_t bwd_bytes(int rows) { return (uint32_t)rows * kStep * 6u; }
__host__ __device__ inline uint32_t slot_bytes(int W) { return fwd_bytes(W) > bwd_bytes(kK0) ? fwd_bytes(W) : bwd_bytes(kK0); }
struct Chunks {
  int fwd, bwd, last;  // forward ones, transposed ones with W output units, those with 64
  __host__ __device__ Chunks(int W, int nh)
      : fwd((kK0 + (nh - 1) * W) / kStep), bwd((nh - 1) * W / kStep), last(W / kStep) {}
  __host__ __device__ int total() const { return fwd + bwd + last; }
  __host__ __device__ uint32_t bytes(int W, int c) const {
    return c < fwd ? fwd_bytes(W) : bwd_bytes(c < fwd + bwd ? W : kK0);
  }
  __host__ __device__ size_t offset(int W, int c) const {
    const size_t f = (size_t)(c < fwd ? c : fwd) * fwd_bytes(W);
    if (c <= fwd) return f;
    const int k = c - fwd;
    return f + (size_t)(k < bwd ? k : bwd) * bwd_bytes(W) + (size_t)(k < bwd ? 0 : k - bwd) * bwd_bytes(kK0);
  }
};
__host__ __device__ inline int layer_params(int W, int in_dim, int l) { return W * ((l == 0 ? in_dim : W) + 1); }

// ---- weights -------------------------------------------------------------------
__device__ __forceinline__ float tf32_part(float x) { return __uint_as_float(__float_as_uint(x) & 0xFFFFE000u); }

// One block per chunk, its parts one after the other, each [output units][16
// inputs] in the K-major canonical layout.
__global__ void __launch_bounds__(256) k_x3_pack_bwd(const float* w, int in_dim, int W, int nh, unsigned char* dst) {
  const Chunks ch(W, nh);
  const int c = blockIdx.x, cn = W / kStep;
  const bool tr = c >= ch.fwd;
  int l, k0, rows = W;
  if (!tr) {
    l = c < kK0 / kStep ? 0 : 1 + (c - kK0 / kStep) / cn;
    k0 = kStep * (l == 0 ? c : (c - kK0 / kStep) % cn);
  } else {
    l = nh - 1 - (c - ch.fwd) / cn;
    k0 = kStep * ((c - ch.fwd) % cn);
    if (l == 0) rows = kK0;
  }
  const int din = l == 0 ? in_dim : W;
  const float* wl = w + (l == 0 ? 0 : (size_t)W * in_dim + (size_t)(l - 1) * W * W);
  unsigned char* o = dst + ch.offset(W, c);
  for (int i = threadIdx.x; i < rows * kStep; i += blockDim.x) {
    // consecutive threads read consecutive inputs of W_l in both directions
    const int r = tr ? i % rows : i / kStep, k = tr ? i / rows : i % kStep;
    const float x = tr ? (r < din ? wl[(size_t)(k0 + k) * din + r] : 0.f)
                       : (k0 + k < din ? wl[(size_t)r * din + k0 + k] : 0.f);
    if (!tr) {
      const float b = tf32_part(x);
      unsigned char* d = o + canon_off(r, 4 * k, 4 * kStep);
      *reinterpret_cast<float*>(d) = b;
      *reinterpret_cast<float*>(d + rows * kStep * 4) = x - b;
    } else {
      __nv_bfloat16 s[3];
      split3(x, s[0], s[1], s[2]);
#pragma unroll
      for (int j = 0; j < 3; ++j)
        *reinterpret_cast<__nv_bfloat16*>(o + j * rows * kStep * 2 + canon_off(r, 2 * k, 2 * kStep)) = s[j];
    }
  }
}

// Eight values of row `row`, columns k0 .. k0 + 7, as two TF32 parts (the big one
// its 10 leading mantissa bits, the rest exact in FP32)
__device__ __forceinline__ void store_tf32x8(unsigned char* A, uint32_t part_bytes, int row, int k0, int kdim,
                                             const float* v) {
#pragma unroll
  for (int q = 0; q < 8; q += 4) {
    const float4 b = make_float4(tf32_part(v[q]), tf32_part(v[q + 1]), tf32_part(v[q + 2]), tf32_part(v[q + 3]));
    unsigned char* d = A + canon_off(row, 4 * (k0 + q), 4 * kdim);
    *reinterpret_cast<float4*>(d) = b;
    *reinterpret_cast<float4*>(d + part_bytes) =
        make_float4(v[q] - b.x, v[q + 1] - b.y, v[q + 2] - b.z, v[q + 3] - b.w);
  }
}

// ---- the chain over the rows ------------------------------------------------------
struct RowsParams {
  int n, nh, width, act, tile0, tile1;  // this batch's tiles
  const unsigned char* blob;
  const float* bias;
  const float* wout;
  const float* bout;
  X3Input in;
  const float* color;    // [N][8]: dT' at 3, dres at 4..6
  unsigned char* tiles;  // the batch's stored activations
  float* opart;          // per CTA: dW_o (row-major), db_o
  float* dT;
  float* mlp_in;  // [N][24]
  uint32_t* status;
};

__device__ __forceinline__ void bulk_s2g(void* dst, uint32_t src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, %0;" ::"r"(kEpiThreads) : "memory"); }

// The sums over the warp's lanes of 16 values: lane l gets value l >> 1's
__device__ __forceinline__ float butterfly16(float (&q)[16], int lane) {
#pragma unroll
  for (int h = 8, off = 16; h >= 1; h >>= 1, off >>= 1) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const float send = up ? q[i] : q[i + h], keep = up ? q[i + h] : q[i];
      q[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
  return q[0] + __shfl_xor_sync(0xffffffffu, q[0], 1);
}

// d/dv of PE(v), from the gradients of its features at rows `base` .. of a
// [feature][128] array
__device__ __forceinline__ void pe_grad(const float* d, const float (&v)[3], float (&out)[3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float g = d[c * kRows];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float f = (float)(1 << q);
      float s, co;
      sincospif(f * v[c], &s, &co);
      g += f * 3.14159265358979323846f * (co * d[(3 + 6 * q + c) * kRows] - s * d[(6 + 6 * q + c) * kRows]);
    }
    out[c] = g;
  }
}

template <int WHICH>
__global__ void __launch_bounds__(kThreads, 1) k_mlp_x3_rows(RowsParams p) {
  after_previous();
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ __align__(8) uint64_t bar_full[kStages], bar_empty[kStages], bar_a[4], bar_d[2], bar_z, bar_s;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int failed;
  constexpr int kOut = WHICH == 0 ? 1 : 3;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int W = p.width, nh = p.nh, cn = W / kChunk, Wm = wide(W);
  const Chunks ch(W, nh);
  const uint32_t slot = slot_bytes(W), ncols = 4u * (uint32_t)Wm;
  const uint32_t asz = kRows * 2u * (uint32_t)Wm, fsz = kRows * 4u * (uint32_t)Wm;  // a BF16 split, a TF32 part
  // [activations][weight ring][bias][wout][bout][output sums][dW_o sums][signs]
  unsigned char* A = sm;
  unsigned char* ring = sm + act_bytes(W);
  float* bsm = reinterpret_cast<float*>(ring + kStages * slot);
  float* wosm = bsm + nh * W;
  float* bosm = wosm + kOut * W;
  float* part = bosm + 4;                  // [2][128][kOut]
  float* wsum = part + 2 * kRows * kOut;   // [8 warps][kOut][W / 2]
  uint16_t* sign = reinterpret_cast<uint16_t*>(wsum + 4 * kOut * W);  // [nh][cn][256]
  if (warp == 0) {
    tmem_alloc(smem_u32(&tmem_slot), ncols);
    tmem_relinquish();
  }
  if (t == 0) {
    for (int i = 0; i < kStages; ++i) {
      mbar_init(smem_u32(&bar_full[i]), 1);
      mbar_init(smem_u32(&bar_empty[i]), 1);
    }
    for (int i = 0; i < 4; ++i) mbar_init(smem_u32(&bar_a[i]), kEpiThreads / 32);
    for (int i = 0; i < 2; ++i) mbar_init(smem_u32(&bar_d[i]), 1);
    mbar_init(smem_u32(&bar_z), kEpiThreads / 32);
    mbar_init(smem_u32(&bar_s), 1);
    fence_mbar_init();
    failed = 0;
  }
  for (int i = t; i < nh * W; i += kThreads) bsm[i] = p.bias[i];
  for (int i = t; i < kOut * W; i += kThreads) wosm[i] = p.wout[i];
  for (int i = t; i < 4 * kOut * W; i += kThreads) wsum[i] = 0.f;
  if (t < kOut) bosm[t] = p.bout[t];
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const int mine = (p.tile1 - p.tile0 - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;  // this CTA's tiles

  if (warp == kEpiThreads / 32 + 1) {
    // ---- weights: chunk after chunk, every tile anew --------------------------
    if (lane == 0) {
      const int per_tile = ch.total(), total = mine * per_tile;
      int g = 0;
      for (; g < total && !failed; ++g) {
        const int st = g % kStages, c = g % per_tile;
        if (g >= kStages && !mbar_wait_bounded(smem_u32(&bar_empty[st]), ((g / kStages) & 1) ^ 1)) {
          failed = 1;
          break;
        }
        const uint32_t bytes = ch.bytes(W, c);
        mbar_expect_tx(smem_u32(&bar_full[st]), bytes);
        bulk_g2s(smem_u32(ring + st * slot), p.blob + ch.offset(W, c), bytes, smem_u32(&bar_full[st]));
      }
      if (failed)  // our own copies land before the CTA leaves
        for (int k = g > kStages ? g - kStages : 0; k < g; ++k)
          mbar_wait_bounded(smem_u32(&bar_full[k % kStages]), (k / kStages) & 1);
    }
  } else if (warp == kEpiThreads / 32) {
    // ---- MMAs: 2 nh products per tile ---------------------------------------------
    if (lane == 0) {
      const uint32_t ring0 = smem_u32(ring), a0 = smem_u32(A);
      uint32_t a_phase = 0u;  // bit c: parity of chunk c's barrier
      int g = 0, seq = 0;
      for (int it = 0; it < mine && !failed; ++it) {
        for (int q = 0; q < 2 * nh && !failed; ++q, ++seq) {
          const int kdim = q == 0 ? kK0 : W, nk = kdim / kChunk, N = q == 2 * nh - 1 ? kK0 : W;
          const uint32_t idesc = q < nh ? idesc_tf32(kRows, N) : idesc_mma(2, kRows, N);
          const uint32_t sbo = (uint32_t)kdim * (q < nh ? 32u : 16u);
          const uint32_t big = tmem + (uint32_t)(seq & 1) * 2u * (uint32_t)Wm, small = big + (uint32_t)Wm;
          for (int c = 0; c < nk && !failed; ++c) {
            if (!mbar_wait_bounded(smem_u32(&bar_a[c]), (a_phase >> c) & 1u)) {
              failed = 1;
              break;
            }
            a_phase ^= 1u << c;
            for (int h = 0; h < kChunk / kStep; ++h, ++g) {
              const int st = g % kStages;
              if (!mbar_wait_bounded(smem_u32(&bar_full[st]), (g / kStages) & 1)) {
                failed = 1;
                break;
              }
              tc_fence_after();
              const uint32_t b0 = ring0 + (uint32_t)st * slot;
              const uint32_t first = c > 0 || h > 0 ? 1u : 0u;
              if (q < nh) {
#pragma unroll
                for (int s = 0; s < kStep / 8; ++s) {
                  const uint32_t ao = a0 + (uint32_t)(c * (kChunk / 8) + h * (kStep / 8) + s) * 256u;
                  const uint32_t bo = b0 + (uint32_t)s * 256u;
                  const uint64_t ab = smem_desc(ao, 128, sbo), as = smem_desc(ao + fsz, 128, sbo);
                  const uint64_t bb = smem_desc(bo, 128, kStep * 32),
                                 bs = smem_desc(bo + (uint32_t)N * kStep * 4u, 128, kStep * 32);
                  tc_mma_tf32(big, as, bb, idesc, s > 0 ? 1u : first);
                  tc_mma_tf32(big, ab, bs, idesc, 1u);
                  tc_mma_tf32(big, ab, bb, idesc, 1u);
                }
              } else {
                uint64_t da[3], db[3];
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                  da[j] = smem_desc(a0 + j * asz + (uint32_t)(2 * c + h) * 256u, 128, sbo);
                  db[j] = smem_desc(b0 + j * (uint32_t)N * kStep * 2u, 128, kStep * 16);
                }
                tc_mma(small, da[2], db[0], idesc, first);
                tc_mma(small, da[0], db[2], idesc, 1u);
                tc_mma(small, da[1], db[1], idesc, 1u);
                tc_mma(small, da[1], db[0], idesc, 1u);
                tc_mma(small, da[0], db[1], idesc, 1u);
                tc_mma(big, da[0], db[0], idesc, first);
              }
              tc_commit(smem_u32(&bar_empty[st]));
            }
          }
          if (!failed) tc_commit(smem_u32(&bar_d[seq & 1]));
        }
      }
    }
  } else if (warp == kEpiThreads / 32 + 2) {
    // ---- the finished dz tiles to global memory ------------------------------------
    if (lane == 0) {
      const uint32_t bytes = kRows * 2u * (uint32_t)W;
      int k = 0;
      for (int it = 0; it < mine && !failed; ++it) {
        unsigned char* tile = p.tiles + ((size_t)blockIdx.x + (size_t)it * gridDim.x) * tile_bytes(W, nh);
        for (int l = nh - 1; l >= 0; --l, ++k) {
          if (!mbar_wait_bounded(smem_u32(&bar_z), k & 1)) {
            failed = 1;
            break;
          }
          unsigned char* dst = tile + dz_off(W, nh, l);
          for (int j = 0; j < 3; ++j) bulk_s2g(dst + (size_t)j * bytes, smem_u32(A) + j * asz, bytes);
          bulk_commit();
          bulk_wait_read();
          mbar_arrive(smem_u32(&bar_s));
        }
      }
      bulk_wait();
    }
  } else {
    // ---- inputs and epilogues -----------------------------------------------------
    const int wg = t >> 7, row = t & 127;
    const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const bool leaky = p.act == GS3_ACT_LEAKY_RELU;
    auto below = [&](float x) { return leaky ? 0.01f * x : 0.f; };  // act and its derivative's product where h <= 0
    auto hand_on = [&](int c) {  // this warp's part of activation chunk c is written
      fence_proxy_async();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bar_a[c]));
    };
    int seq = 0, stored = 0;
    bool ok = true;  // the same for a warp's lanes
    auto wait_product = [&] {  // the next product is in its accumulators; their address
      const int s = seq++;
      if (ok) ok = __all_sync(0xffffffffu, mbar_wait_bounded(smem_u32(&bar_d[s & 1]), (s >> 1) & 1));
      tc_fence_after();
      return lane_addr + (uint32_t)(s & 1) * 2u * (uint32_t)Wm;
    };
    auto wait_stored = [&] {  // the dz tile is copied out: it may be overwritten
      const int s = stored++;
      if (ok) ok = __all_sync(0xffffffffu, mbar_wait_bounded(smem_u32(&bar_s), s & 1));
    };
    // f(chunk, first column, 16 sums) over the chunks of the product at `big`
    auto for_chunks = [&](uint32_t big, int chunks, bool split, auto&& f) {
      for (int c = 0; c < chunks; ++c) {
        const int c0 = kChunk * c + 16 * wg;
        float v[16];
        if (split) {
          acc_load16(big + (uint32_t)c0, big + (uint32_t)(Wm + c0), v);
        } else {
          uint32_t b[16];
          tmem_issue16(big + (uint32_t)c0, b);
          tmem_wait16(b);
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(b[i]);
        }
        f(c, c0, v);
      }
    };
    float bacc[kOut];
#pragma unroll
    for (int o = 0; o < kOut; ++o) bacc[o] = 0.f;
    bool done = true;
    for (int it = 0; it < mine; ++it) {
      const int r = (p.tile0 + (int)blockIdx.x + it * (int)gridDim.x) * kRows + row, g = min(r, p.n - 1);
      unsigned char* tile = p.tiles + ((size_t)blockIdx.x + (size_t)it * gridDim.x) * tile_bytes(W, nh);
      // forward activations: to the next product, and for the weight gradients
      auto put_fwd = [&](int layer, int kdim, int k0, const float* x) {
        store_tf32x8(A, fsz, row, k0, kdim, x);
        store_split8(tile + h_off(W, layer), (uint32_t)(kRows * 2 * kdim), row, k0, kdim, x);
      };
      const auto put = [&](int k0, const float* x) { put_fwd(0, kK0, k0, x); };
      if (wg == 0) encode_half<WHICH, 0>(p.in, g, put);
      else encode_half<WHICH, 1>(p.in, g, put);
      hand_on(0);
      hand_on(1);
      float acc[kOut];
#pragma unroll
      for (int o = 0; o < kOut; ++o) acc[o] = 0.f;
      uint32_t big = 0;
      for (int l = 0; l < nh; ++l) {
        big = wait_product();
        if (!ok) continue;
        for_chunks(big, cn, false, [&](int c, int c0, float (&v)[16]) {
          uint32_t bits = 0;
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float h = v[i] + bsm[l * W + c0 + i];
            if (h > 0.f) bits |= 1u << i;
            v[i] = h > 0.f ? h : below(h);
          }
          if (l + 1 < nh) {
            sign[(l * cn + c) * kEpiThreads + t] = (uint16_t)bits;
            put_fwd(l + 1, W, c0, v);
            put_fwd(l + 1, W, c0 + 8, v + 8);
            hand_on(c);
          } else {
#pragma unroll
            for (int o = 0; o < kOut; ++o)
#pragma unroll
              for (int i = 0; i < 16; ++i) acc[o] = fmaf(v[i], wosm[o * W + c0 + i], acc[o]);
          }
        });
      }
      // the output layer: both halves' sums, in every thread of the row
#pragma unroll
      for (int o = 0; o < kOut; ++o) part[(wg * kRows + row) * kOut + o] = acc[o];
      if (epi_any(!ok)) {
        done = false;
        break;
      }
      float dzo[kOut];
#pragma unroll
      for (int o = 0; o < kOut; ++o) {
        const float s = part[row * kOut + o] + part[(kRows + row) * kOut + o];
        const float y = 1.f / (1.f + expf(-(s + bosm[o])));
        const float dy = r < p.n ? p.color[(size_t)kColorStride * g + (WHICH == 0 ? 3 : 4 + o)] : 0.f;
        dzo[o] = dy * y * (1.f - y);
        bacc[o] += dzo[o];
      }
      for_chunks(big, cn, false, [&](int c, int c0, float (&v)[16]) {
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const float h = v[i] + bsm[(nh - 1) * W + c0 + i];
          v[i] = h > 0.f ? h : below(h);
        }
#pragma unroll
        for (int o = 0; o < kOut; ++o) {
          float q[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) q[i] = dzo[o] * v[i];
          const float s = butterfly16(q, lane);
          if (!(lane & 1)) wsum[(warp * kOut + o) * (W / 2) + 16 * c + (lane >> 1)] += s;
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          float s = 0.f;
#pragma unroll
          for (int o = 0; o < kOut; ++o) s = fmaf(dzo[o], wosm[o * W + c0 + i], s);
          v[i] = v[i] > 0.f ? s : below(s);
        }
        store_split8(A, asz, row, c0, W, v);
        store_split8(A, asz, row, c0 + 8, W, v + 8);
        hand_on(c);
      });
      if (lane == 0) mbar_arrive(smem_u32(&bar_z));
      // data gradients of the layers below
      for (int l = nh - 2; l >= 0; --l) {
        big = wait_product();
        wait_stored();
        if (!ok) continue;
        for_chunks(big, cn, true, [&](int c, int c0, float (&v)[16]) {
          const uint32_t bits = sign[(l * cn + c) * kEpiThreads + t];
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = (bits >> i) & 1u ? v[i] : below(v[i]);
          store_split8(A, asz, row, c0, W, v);
          store_split8(A, asz, row, c0 + 8, W, v + 8);
          hand_on(c);
        });
        if (lane == 0) mbar_arrive(smem_u32(&bar_z));
      }
      // the inputs' gradients, [feature][row] where the activations were
      big = wait_product();
      wait_stored();
      float* D = reinterpret_cast<float*>(A);
      if (ok)
        for_chunks(big, kK0 / kChunk, true, [&](int, int c0, float (&v)[16]) {
#pragma unroll
          for (int i = 0; i < 16; ++i) D[(c0 + i) * kRows + row] = v[i];
        });
      if (epi_any(!ok)) {
        done = false;
        break;
      }
      if (r < p.n) {
        constexpr int b0 = WHICH == 0 ? 1 : 0;
        float* out = p.mlp_in + (size_t)kMlpInStride * g + 12 * WHICH;
        const float4 m = p.in.mean_op[g];
        float d[3];
        if (wg == 0) {
          const float dx = p.in.src.x - p.in.src.w * m.x, dy = p.in.src.y - p.in.src.w * m.y,
                      dz = p.in.src.z - p.in.src.w * m.z;
          const float il = rsqrtf(dx * dx + dy * dy + dz * dz);
          const float u[3] = {dx * il, dy * il, dz * il};
          pe_grad(D + b0 * kRows + row, u, d);
          out[3] = d[0]; out[4] = d[1]; out[5] = d[2];
          if (WHICH == 0) p.dT[g] = D[row];
        } else {
          const float u[3] = {m.x, m.y, m.z};
          pe_grad(D + (b0 + 27) * kRows + row, u, d);
          out[0] = d[0]; out[1] = d[1]; out[2] = d[2];
#pragma unroll
          for (int k = 0; k < 6; ++k) out[6 + k] = D[(b0 + 54 + k) * kRows + row];
        }
      }
      epi_sync();  // the next tile's inputs overwrite D
    }
    if (!done) failed = 1;
    if (done) {  // the CTA's dW_o and db_o, warps added in order
#pragma unroll
      for (int o = 0; o < kOut; ++o)
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) bacc[o] += __shfl_xor_sync(0xffffffffu, bacc[o], off);
      if (wg == 0 && lane == 0)
#pragma unroll
        for (int o = 0; o < kOut; ++o) part[warp * kOut + o] = bacc[o];
      epi_sync();
      float* out = p.opart + (size_t)blockIdx.x * (kOut * W + kOut);
      for (int i = t; i < kOut * W; i += kEpiThreads) {
        const int o = i / W, j = i - o * W, half = (j >> 4) & 1, idx = (j >> 5) * 16 + (j & 15);
        float s = 0.f;
        for (int w = 0; w < 4; ++w) s += wsum[((4 * half + w) * kOut + o) * (W / 2) + idx];
        out[i] = s;
      }
      if (t < kOut) {
        float s = 0.f;
        for (int w = 0; w < 4; ++w) s += part[w * kOut + t];
        out[kOut * W + t] = s;
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (t == 0 && failed) atomicCAS(p.status, 0u, (uint32_t)GS3_ERR_TIMEOUT);
  if (warp == 0) tmem_dealloc(tmem, ncols);
}

// ---- weight gradients ------------------------------------------------------------
constexpr int kWRows = 32;  // Gaussians per stage
constexpr int kWStages = 4;
constexpr int kWThreads = 128 + 64;  // output warps, then the copy and MMA warps

__host__ __device__ inline uint32_t wstage_bytes(int W) { return 3u * kWRows * 2u * (uint32_t)(W + wide(W)); }
__host__ __device__ inline uint32_t wcols(int W) { return W > kK0 ? 512u : 256u; }  // 2 max(W, 64) + 16 columns

struct WgradParams {
  int nh, width, in_dim, ntiles;
  const unsigned char* tiles;
  float* part;  // per CTA, layer after layer: [input, then 1][unit]
  uint32_t* status;
};

__global__ void __launch_bounds__(kWThreads, 1) k_mlp_x3_wgrad(WgradParams p) {
  after_previous();
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ __align__(16) __nv_bfloat16 ones[256];
  __shared__ __align__(8) uint64_t bar_full[kWStages], bar_empty[kWStages], bar_d, bar_o;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int failed;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int W = p.width, nh = p.nh, Wm = wide(W);
  const uint32_t sb = wstage_bytes(W);
  if (warp == 0) {
    tmem_alloc(smem_u32(&tmem_slot), wcols(W));
    tmem_relinquish();
  }
  for (int i = t; i < 256; i += kWThreads) ones[i] = __float2bfloat16_rn(1.f);
  if (t == 0) {
    for (int i = 0; i < kWStages; ++i) {
      mbar_init(smem_u32(&bar_full[i]), 1);
      mbar_init(smem_u32(&bar_empty[i]), 1);
    }
    mbar_init(smem_u32(&bar_d), 1);
    mbar_init(smem_u32(&bar_o), 4);
    fence_mbar_init();
    failed = 0;
  }
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  // the CTA's steps of 32 Gaussians, the same in every layer
  const long long steps = (long long)p.ntiles * (kRows / kWRows);
  const int u0 = (int)(steps * blockIdx.x / gridDim.x), u1 = (int)(steps * (blockIdx.x + 1) / gridDim.x);
  const int per_layer = u1 - u0, total = nh * per_layer;

  if (warp == 4) {
    if (lane == 0) {
      const size_t tb = tile_bytes(W, nh);
      int g = 0;
      for (; g < total && !failed; ++g) {
        const int st = g % kWStages, l = g / per_layer, u = u0 + g - l * per_layer;
        if (g >= kWStages && !mbar_wait_bounded(smem_u32(&bar_empty[st]), ((g / kWStages) & 1) ^ 1)) {
          failed = 1;
          break;
        }
        const int kd = l == 0 ? kK0 : W, q = u % (kRows / kWRows);
        const unsigned char* tile = p.tiles + (size_t)(u / (kRows / kWRows)) * tb;
        const unsigned char *dz = tile + dz_off(W, nh, l), *h = tile + h_off(W, l);
        const uint32_t zb = kWRows * 2u * (uint32_t)W, hb = kWRows * 2u * (uint32_t)kd;
        const uint32_t bar = smem_u32(&bar_full[st]), dst = smem_u32(sm + st * sb);
        mbar_expect_tx(bar, 3u * (zb + hb));
        for (int j = 0; j < 3; ++j) {
          bulk_g2s(dst + j * zb, dz + (size_t)(j * (kRows / kWRows) + q) * zb, zb, bar);
          bulk_g2s(dst + 3 * zb + j * hb, h + (size_t)(j * (kRows / kWRows) + q) * hb, hb, bar);
        }
      }
      if (failed)  // our own copies land before the CTA leaves
        for (int k = g > kWStages ? g - kWStages : 0; k < g; ++k)
          mbar_wait_bounded(smem_u32(&bar_full[k % kWStages]), (k / kWStages) & 1);
    }
  } else if (warp == 5) {
    if (lane == 0) {
      // A = dz (units x Gaussians), B = h (inputs x Gaussians), both MN-major.
      // Units past the width read what lies behind: rows of D that nobody reads.
      constexpr uint32_t kMn = (1u << 15) | (1u << 16);
      const uint32_t big = tmem, small = tmem + (uint32_t)Wm, sum = small + (uint32_t)Wm;
      const uint32_t idone = idesc_mma(2, kRows, 16) | kMn;
      const uint64_t dones = smem_desc(smem_u32(ones), 256, 128);
      int g = 0;
      for (int l = 0; l < nh && !failed; ++l) {
        const int kd = l == 0 ? kK0 : W;
        const uint32_t idesc = idesc_mma(2, kRows, kd) | kMn;
        const uint32_t zb = kWRows * 2u * (uint32_t)W, hb = kWRows * 2u * (uint32_t)kd;
        if (l > 0 && !mbar_wait_bounded(smem_u32(&bar_o), (l - 1) & 1)) {
          failed = 1;
          break;
        }
        for (int i = 0; i < per_layer; ++i, ++g) {
          const int st = g % kWStages;
          if (!mbar_wait_bounded(smem_u32(&bar_full[st]), (g / kWStages) & 1)) {
            failed = 1;
            break;
          }
          tc_fence_after();
          const uint32_t a0 = smem_u32(sm + st * sb), b0 = a0 + 3 * zb;
#pragma unroll
          for (int s = 0; s < kWRows / 16; ++s) {
            uint64_t da[3], db[3];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
              // 8 units: 128 bytes on; 8 Gaussians: one row group on
              da[j] = smem_desc(a0 + j * zb + (uint32_t)s * 32u * (uint32_t)W, 16u * (uint32_t)W, 128);
              db[j] = smem_desc(b0 + j * hb + (uint32_t)s * 32u * (uint32_t)kd, 16u * (uint32_t)kd, 128);
            }
            const uint32_t on = i > 0 || s > 0 ? 1u : 0u;
            tc_mma(small, da[2], db[0], idesc, on);
            tc_mma(small, da[0], db[2], idesc, 1u);
            tc_mma(small, da[1], db[1], idesc, 1u);
            tc_mma(small, da[1], db[0], idesc, 1u);
            tc_mma(small, da[0], db[1], idesc, 1u);
            tc_mma(big, da[0], db[0], idesc, on);
            tc_mma(sum, da[2], dones, idone, on);
            tc_mma(sum, da[1], dones, idone, 1u);
            tc_mma(sum, da[0], dones, idone, 1u);
          }
          tc_commit(smem_u32(&bar_empty[st]));
        }
        if (!failed) tc_commit(smem_u32(&bar_d));
      }
    }
  } else {
    // ---- layer by layer: thread t writes unit t's row --------------------------------
    size_t np = 0;
    for (int l = 0; l < nh; ++l) np += layer_params(W, p.in_dim, l);
    float* out = p.part + (size_t)blockIdx.x * np;
    const uint32_t lane_addr = tmem + ((uint32_t)(warp * 32) << 16);
    bool ok = true;
    for (int l = 0; l < nh; ++l) {
      if (ok) ok = __all_sync(0xffffffffu, mbar_wait_bounded(smem_u32(&bar_d), l & 1));
      if (!ok) break;
      tc_fence_after();
      const int nin = l == 0 ? p.in_dim : W;
      if (32 * warp < W) {
        for (int c0 = 0; c0 < nin; c0 += 16) {
          float v[16];
          acc_load16(lane_addr + (uint32_t)c0, lane_addr + (uint32_t)(Wm + c0), v);
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (c0 + i < nin) out[(size_t)(c0 + i) * W + t] = v[i];
        }
        uint32_t b[16];
        tmem_issue16(lane_addr + 2u * (uint32_t)Wm, b);
        tmem_wait16(b);
        out[(size_t)nin * W + t] = __uint_as_float(b[0]);
      }
      out += layer_params(W, p.in_dim, l);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bar_o));
    }
    if (!ok && lane == 0) failed = 1;
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (t == 0 && failed) atomicCAS(p.status, 0u, (uint32_t)GS3_ERR_TIMEOUT);
  if (warp == 0) tmem_dealloc(tmem, wcols(W));
}

// red = the CTAs' partials in the parameter order (per layer weights row-major,
// then biases): 32 parameters per block, warp w adds the partials w, w + 8, ...
constexpr int kSumWarps = 8;
struct SumParams {
  const float *wpart, *opart;
  int nw, no, np, op;  // partials and their lengths
  int W, in_dim;
  float* red;
};
__global__ void __launch_bounds__(kSumWarps * 32) k_mlp_x3_sum(SumParams p) {
  after_previous();
  __shared__ float acc[kSumWarps][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
  const bool hidden = i < p.np;
  const float* src = hidden ? p.wpart + i : p.opart + (i - p.np);
  const int count = i < p.np + p.op ? (hidden ? p.nw : p.no) : 0;
  const size_t stride = hidden ? p.np : p.op;
  float s = 0.f;
  for (int b = warp; b < count; b += kSumWarps) s += src[(size_t)b * stride];
  acc[warp][lane] = s;
  __syncthreads();
  if (warp != 0 || count == 0) return;
  float sum = 0.f;
  for (int w = 0; w < kSumWarps; ++w) sum += acc[w][lane];
  int dst = i;
  if (hidden) {
    const int first = layer_params(p.W, p.in_dim, 0), later = layer_params(p.W, p.in_dim, 1);
    const int base = i < first ? 0 : first + (i - first) / later * later, nin = i < first ? p.in_dim : p.W;
    const int k = (i - base) / p.W, j = (i - base) - k * p.W;
    dst = base + (k < nin ? j * nin + k : p.W * nin + j);
  }
  p.red[dst] = sum;
}

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

struct Plan {
  int ntiles, batches, np, op, grid;  // grid: partials per batch (at most)
  size_t blob, tiles, wpart, opart, total;
};
Plan plan(int n, const MlpDev& m) {
  Plan P;
  P.ntiles = (n + kRows - 1) / kRows;
  P.batches = (P.ntiles + kBatchTiles - 1) / kBatchTiles;
  P.np = 0;
  for (int l = 0; l < m.n_hidden; ++l) P.np += layer_params(m.width, m.in_dim, l);
  P.op = m.out_dim * m.width + m.out_dim;
  const int tb = P.ntiles < kBatchTiles ? P.ntiles : kBatchTiles;
  P.grid = tb * (kRows / kWRows) < kMaxCtas ? tb * (kRows / kWRows) : kMaxCtas;
  size_t c = 0;
  auto take = [&](size_t b) { const size_t o = c; c = align256(c + b); return o; };
  P.blob = take(Chunks(m.width, m.n_hidden).offset(m.width, Chunks(m.width, m.n_hidden).total()));
  P.tiles = take((size_t)tb * tile_bytes(m.width, m.n_hidden));
  P.wpart = take(4ull * P.batches * P.grid * P.np);
  P.opart = take(4ull * P.batches * P.grid * P.op);
  P.total = c;
  return P;
}

size_t rows_smem(const MlpDev& m) {
  const int W = m.width;
  return act_bytes(W) + (size_t)kStages * slot_bytes(W) +
         4 * ((size_t)m.n_hidden * W + m.out_dim * W + 4 + 2 * kRows * m.out_dim + 4 * m.out_dim * W) +
         2ull * m.n_hidden * (W / kChunk) * kEpiThreads;
}
// the CTAs that can share an SM never need more than its 512 tensor-memory columns
size_t smem_for_cols(size_t smem, uint32_t cols) {
  const size_t floor_bytes = 228 * 1024 / (size_t)(512 / cols + 1) + 1;
  return smem < floor_bytes ? floor_bytes : smem;
}

}  // namespace

size_t mlp_x3_bwd_scratch_bytes(int n, const MlpDev& m) { return plan(n, m).total; }

void run_mlp_x3_backward(const MlpArgs& a, void* scratch, float* wred, cudaStream_t s) {
  const MlpDev& m = a.net;
  const int W = m.width, nh = m.n_hidden;
  const Plan P = plan(a.n, m);
  unsigned char* base = static_cast<unsigned char*>(scratch);
  float* wpart = reinterpret_cast<float*>(base + P.wpart);
  float* opart = reinterpret_cast<float*>(base + P.opart);
  static DeviceOnce once;
  once.run([] {
    bool ok = true;
    for (const void* k : {(const void*)k_mlp_x3_rows<0>, (const void*)k_mlp_x3_rows<1>, (const void*)k_mlp_x3_wgrad})
      ok = ok && cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 225 * 1024) == cudaSuccess;
    return ok;
  });
  k_x3_pack_bwd<<<Chunks(W, nh).total(), 256, 0, s>>>(m.w, m.in_dim, W, nh, base + P.blob);
  RowsParams r;
  r.n = a.n; r.nh = nh; r.width = W; r.act = m.act;
  r.blob = base + P.blob;
  r.bias = m.b;
  r.wout = m.w + (size_t)W * m.in_dim + (size_t)(nh - 1) * W * W;
  r.bout = m.b + (size_t)nh * W;
  const float* src = a.which == 0 ? a.light_pos : a.cam_pos;
  r.in = {a.n, a.mean_op, a.latent, a.T, make_float4(src[0], src[1], src[2], a.which == 0 ? a.light_w : 1.f)};
  r.color = a.color;
  r.tiles = base + P.tiles;
  r.dT = a.dT;
  r.mlp_in = a.mlp_in;
  r.status = a.status;
  WgradParams w;
  w.nh = nh; w.width = W; w.in_dim = m.in_dim;
  w.tiles = r.tiles;
  w.status = a.status;
  const int nsm = device_sm_count() < kMaxCtas ? device_sm_count() : kMaxCtas;
  int nw = 0, no = 0;
  for (int b = 0; b < P.batches; ++b) {
    r.tile0 = b * kBatchTiles;
    r.tile1 = r.tile0 + kBatchTiles < P.ntiles ? r.tile0 + kBatchTiles : P.ntiles;
    w.ntiles = r.tile1 - r.tile0;
    const int gr = w.ntiles < nsm ? w.ntiles : nsm;
    const int gw = w.ntiles * (kRows / kWRows) < nsm ? w.ntiles * (kRows / kWRows) : nsm;
    r.opart = opart + (size_t)no * P.op;
    w.part = wpart + (size_t)nw * P.np;
    if (a.which == 0) launch_after(k_mlp_x3_rows<0>, gr, kThreads, smem_for_cols(rows_smem(m), 4u * wide(W)), s, r);
    else launch_after(k_mlp_x3_rows<1>, gr, kThreads, smem_for_cols(rows_smem(m), 4u * wide(W)), s, r);
    launch_after(k_mlp_x3_wgrad, gw, kWThreads, smem_for_cols((size_t)kWStages * wstage_bytes(W), wcols(W)), s, w);
    no += gr;
    nw += gw;
  }
  const SumParams q = {wpart, opart, nw, no, P.np, P.op, W, m.in_dim, wred};
  launch_after(k_mlp_x3_sum, (P.np + P.op + 31) / 32, kSumWarps * 32, 0, s, q);
  count_launch(2 + 2 * P.batches);
}

}  // namespace gs3
