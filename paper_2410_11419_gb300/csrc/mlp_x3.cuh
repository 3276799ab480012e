// Shared by the FP32 networks' forward and backward on the tensor cores
// (mlp_x3.cu, mlp_x3_bwd.cu): the split of an FP32 operand into three BF16
// values, activation tiles of 128 Gaussians in the K-major canonical layout (the
// three splits one after the other), weight chunks of 32 inputs, and the
// networks' inputs.
#pragma once
#include <cuda_bf16.h>

#include "gs3_internal.cuh"
#include "tc_ptx.cuh"

namespace gs3 {
namespace x3 {

using namespace tc;

constexpr int kRows = 128;        // Gaussians of a tile
constexpr int kEpiThreads = 256;  // two warpgroups run the inputs and epilogues
constexpr int kK0 = 64;           // padded input width (61 / 60 features)
constexpr int kChunk = 32;        // inputs of a layer per weight chunk
constexpr int kStages = 4;        // weight ring
constexpr int kMaxHidden = 4;

// a weight chunk of `rows` output units
__host__ __device__ inline uint32_t chunk_bytes(int rows) { return 3u * (uint32_t)rows * kChunk * 2u; }

__device__ __forceinline__ void split3(float x, __nv_bfloat16& h, __nv_bfloat16& m, __nv_bfloat16& l) {
  h = __float2bfloat16_rn(x);
  const float r = x - __bfloat162float(h);
  m = __float2bfloat16_rn(r);
  l = __float2bfloat16_rn(r - __bfloat162float(m));
}

// 16 columns of this thread's TMEM lane: the load, and the wait for it
__device__ __forceinline__ void tmem_issue16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
// (the registers pass through the statement: no use of them moves above it)
__device__ __forceinline__ void tmem_wait16(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}
// the sums of a product's two accumulators (loading the next columns under the
// arithmetic on these gained nothing)
__device__ __forceinline__ void acc_load16(uint32_t big, uint32_t small, float (&v)[16]) {
  uint32_t a[16], b[16];
  tmem_issue16(big, a);
  tmem_issue16(small, b);
  tmem_wait16(a);
  tmem_wait16(b);
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(a[i]) + __uint_as_float(b[i]);
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Whether x holds for any thread of the two warpgroups (a barrier of theirs)
__device__ __forceinline__ bool epi_any(bool x) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "barrier.cta.red.or.pred q, 1, %2, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r) : "r"((uint32_t)x), "n"(kEpiThreads) : "memory");
  return r != 0u;
}

// Eight values of row `row`, columns k0 .. k0 + 7, as three splits (16 bytes each)
__device__ __forceinline__ void store_split8(unsigned char* A, uint32_t split_bytes, int row, int k0, int kdim,
                                             const float* v) {
  __nv_bfloat162 h[4], m[4], l[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    h[i] = __float22bfloat162_rn(make_float2(v[2 * i], v[2 * i + 1]));
    const float2 hf = __bfloat1622float2(h[i]);
    const float2 r = make_float2(v[2 * i] - hf.x, v[2 * i + 1] - hf.y);
    m[i] = __float22bfloat162_rn(r);
    const float2 mf = __bfloat1622float2(m[i]);
    l[i] = __float22bfloat162_rn(make_float2(r.x - mf.x, r.y - mf.y));
  }
  unsigned char* p = A + canon_off(row, 2 * k0, 2 * kdim);
  *reinterpret_cast<uint4*>(p) = *reinterpret_cast<uint4*>(h);
  *reinterpret_cast<uint4*>(p + split_bytes) = *reinterpret_cast<uint4*>(m);
  *reinterpret_cast<uint4*>(p + 2 * split_bytes) = *reinterpret_cast<uint4*>(l);
}

// Features [base, base + 27) of x: [v, sin(2^q pi v), cos(2^q pi v)], q < bands
__device__ __forceinline__ void pe_bands(float* x, int base, const float (&v)[3], int bands) {
#pragma unroll
  for (int c = 0; c < 3; ++c) x[base + c] = v[c];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (q >= bands) break;
    const float f = (float)(1 << q);
#pragma unroll
    for (int c = 0; c < 3; ++c) sincospif(f * v[c], &x[base + 3 + 6 * q + c], &x[base + 6 + 6 * q + c]);
  }
}

struct X3Input {
  int n;
  const float4* mean_op;
  const float4* latent;
  const float* T;  // Phi
  float4 src;      // Phi: homogeneous light, Psi: camera position and 1
};

// Inputs 32 HALF .. 32 HALF + 31 of a row: Phi [T, PE(w_i), PE(mu), l], Psi
// [PE(w_o), PE(mu), l], padded to 64 with zeros; store(k, values) takes eight.
template <int WHICH, int HALF, typename F>
__device__ __forceinline__ void encode_half(const X3Input& in, int g, F&& store) {
  constexpr int b0 = WHICH == 0 ? 1 : 0;
  float x[kK0 + 8];
  const float4 m = in.mean_op[g];
  const float mu[3] = {m.x, m.y, m.z};
  if (HALF == 0) {
    const float dx = in.src.x - in.src.w * m.x, dy = in.src.y - in.src.w * m.y, dz = in.src.z - in.src.w * m.z;
    const float il = rsqrtf(dx * dx + dy * dy + dz * dz);
    const float d[3] = {dx * il, dy * il, dz * il};
    if (WHICH == 0) x[0] = in.T[g];
    pe_bands(x, b0, d, 4);
    pe_bands(x, b0 + 27, mu, 1);  // the first of them
  } else {
    pe_bands(x, b0 + 27, mu, 4);
    const float4 l0 = in.latent[g], l1 = in.latent[in.n + g];
    x[b0 + 54] = l0.x; x[b0 + 55] = l0.y; x[b0 + 56] = l0.z; x[b0 + 57] = l0.w;
    x[b0 + 58] = l1.x; x[b0 + 59] = l1.y;
#pragma unroll
    for (int k = b0 + 60; k < kK0; ++k) x[k] = 0.f;
  }
#pragma unroll
  for (int k0 = 32 * HALF; k0 < 32 * HALF + 32; k0 += 8) store(k0, x + k0);
}

}  // namespace x3
}  // namespace gs3
