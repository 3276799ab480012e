// K8 (FP32 form) on the tensor cores: Phi (Sec. 4.2) and Psi (Sec. 4.3) with
// hidden widths of 32, 64 or 128, to FP32 accuracy.
//
// Every FP32 operand x of a hidden layer is split into three BF16 values, hi =
// bf16(x), mid = bf16(x - hi), lo = bf16(x - hi - mid) (both differences are
// exact; the three hold x to 2^-27 of its size).  A product is formed as the
// six of its nine terms above 2^-27: hi hi' into one accumulator, and hi mid',
// mid hi', mid mid', hi lo', lo hi' into a second, whose rounding is then 2^-8
// of the first's; they are added in FP32.  Relative error of T' and the
// residual against float64: 5.7e-8 to 9.8e-8 (rms) over the networks of the
// object, paper, tiny and narrow scenes, where a chain of FP32 FMAs per output
// has 6.4e-8 to 9.8e-8.
//
// A CTA owns one 128-row tile of Gaussians at a time: two warpgroups, thread t
// of each row t, encode the inputs and run the epilogues, one 16-column half
// of every 32 columns each; one warp's lane issues the MMAs, another's copies
// the weights.  The weights, split and arranged per 32 inputs (x3_pack: they
// are read from the scene's arrays in every frame, which may train), do not
// fit beside the activations (96 KB as three splits), so they stream through a
// ring of four 24 KB chunks by bulk copies.  The accumulators are double
// buffered, and an epilogue hands its columns on 32 at a time, so that the
// next layer's MMAs on them run under the rest of the epilogue.
//
// Bound: the tensor pipe during a layer (six passes) and the epilogue's
// conversions between layers (a tile takes 11 us, its MMAs alone 4.3).  300k
// Gaussians, 3 x 128: 0.18 ms per network, against 0.68 ms for register-tiled
// FP32 FMAs (46 % of the FMA pipe).
#include "mlp_x3.cuh"

namespace gs3 {
namespace {

using namespace x3;

constexpr int kThreads = kEpiThreads + 64;  // and the MMA and copy warps

struct X3Params {
  int n, nh, width, act;
  const unsigned char* blob;  // packed hidden-layer weights
  const float* bias;          // nh x width
  const float* wout;          // out x width
  const float* bout;
  const float4* mean_op;
  const float4* latent;
  int nl;                          // Phi: lights of the batch (row l n + g); Psi: 1
  const float* T[kMaxBatch];       // Phi input T per light, by index
  float* out[kMaxBatch];           // Phi: T' per light; Psi: float4 residual at [0]
  const float4* shade[kMaxBatch];  // shading per light, by index (envcol only)
  float4 light[kMaxBatch];         // homogeneous light per light (light_h)
  float cam_pos[3];
  float4* ccol;    // camera colours by rank (nl = 1)
  float4* envcol;  // non-null (Phi): (shade_l, T'_l) at [r nl + l] instead of ccol
  const uint32_t* rank_of;
  uint32_t *status, *nonfinite;
};

// ---- packing -----------------------------------------------------------------
struct PackArgs {
  const float* w[2];  // Phi, Psi hidden weights
  int in_dim[2], width[2], nh[2];
  unsigned char* dst[2];
  int total[2];  // elements
};

// Element (layer, output row, input k) of a network's hidden layers into its
// chunk: chunk k / 32 of the layer holds the three splits one after the other,
// each [width rows][32 inputs] in the K-major canonical layout.
__global__ void __launch_bounds__(256) k_x3_pack(PackArgs a) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int net = i >= a.total[0] ? 1 : 0;
  if (net) i -= a.total[0];
  if (i >= a.total[net]) return;
  const int W = a.width[net];
  const float* w = a.w[net];
  unsigned char* dst = a.dst[net];
  int kdim = kK0, in = a.in_dim[net];
  if (i >= W * kK0) {  // a layer past the first
    i -= W * kK0;
    const int l = i / (W * W);
    i -= l * W * W;
    w += (size_t)W * in + (size_t)l * W * W;
    dst += (size_t)(kK0 / kChunk + l * (W / kChunk)) * chunk_bytes(W);
    kdim = in = W;
  }
  const int r = i / kdim, k = i - r * kdim;
  __nv_bfloat16 s[3];
  split3(k < in ? w[(size_t)r * in + k] : 0.f, s[0], s[1], s[2]);
  unsigned char* c = dst + (size_t)(k / kChunk) * chunk_bytes(W) + canon_off(r, 2 * (k % kChunk), 2 * kChunk);
#pragma unroll
  for (int j = 0; j < 3; ++j) *reinterpret_cast<__nv_bfloat16*>(c + j * W * kChunk * 2) = s[j];
}

int hidden_elems(const MlpDev& m) { return m.width * kK0 + (m.n_hidden - 1) * m.width * m.width; }

// ---- the networks -------------------------------------------------------------
__host__ __device__ inline uint32_t x3_cols(int W) {  // TMEM: two buffers of two accumulators
  return W < 32 ? 32u : 4u * (uint32_t)W;
}
__host__ __device__ inline uint32_t x3_act_bytes(int W) { return 3u * kRows * 2u * (uint32_t)(W > kK0 ? W : kK0); }

template <int WHICH>
__global__ void __launch_bounds__(kThreads, 1) k_mlp_x3(X3Params p) {
  after_previous();
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ __align__(8) uint64_t bar_full[kStages], bar_empty[kStages], bar_a[4], bar_d[2];
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int failed;
  constexpr int kOut = WHICH == 0 ? 1 : 3;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int W = p.width, nh = p.nh;
  const uint32_t cb = chunk_bytes(W), ncols = x3_cols(W);
  // [activations][weight ring][bias][wout][bout][partial outputs]
  unsigned char* A = sm;
  unsigned char* ring = sm + x3_act_bytes(W);
  float* bsm = reinterpret_cast<float*>(ring + kStages * cb);
  float* wosm = bsm + nh * W;
  float* bosm = wosm + kOut * W;
  float* part = bosm + 4;  // [128][kOut]
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
    fence_mbar_init();
    failed = 0;
  }
  for (int i = t; i < nh * W; i += kThreads) bsm[i] = p.bias[i];
  for (int i = t; i < kOut * W; i += kThreads) wosm[i] = p.wout[i];
  if (t < kOut) bosm[t] = p.bout[t];
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const int rows = p.n * p.nl, ntiles = (rows + kRows - 1) / kRows;
  const int mine = (ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;  // this CTA's tiles
  const int chunks0 = kK0 / kChunk, chunksN = W / kChunk, per_tile = chunks0 + (nh - 1) * chunksN;

  if (warp == kEpiThreads / 32 + 1) {
    // ---- weights: chunk after chunk, every tile anew --------------------------
    if (lane == 0) {
      const int total = mine * per_tile;
      int g = 0;
      for (; g < total && !failed; ++g) {
        const int st = g % kStages;
        if (g >= kStages && !mbar_wait_bounded(smem_u32(&bar_empty[st]), ((g / kStages) & 1) ^ 1)) {
          failed = 1;
          break;
        }
        mbar_expect_tx(smem_u32(&bar_full[st]), cb);
        bulk_g2s(smem_u32(ring + st * cb), p.blob + (size_t)(g % per_tile) * cb, cb, smem_u32(&bar_full[st]));
      }
      if (failed)  // our own copies land before the CTA leaves
        for (int k = g > kStages ? g - kStages : 0; k < g; ++k)
          mbar_wait_bounded(smem_u32(&bar_full[k % kStages]), (k / kStages) & 1);
    }
  } else if (warp == kEpiThreads / 32) {
    // ---- MMAs -------------------------------------------------------------------
    if (lane == 0) {
      const uint32_t idesc = idesc_mma(2, kRows, W), ring0 = smem_u32(ring), a0 = smem_u32(A);
      const uint32_t asz = x3_act_bytes(W) / 3, bsz = cb / 3;
      uint32_t a_phase = 0u;  // bit c: parity of chunk c's barrier
      int g = 0, layer = 0;
      for (int it = 0; it < mine && !failed; ++it) {
        for (int l = 0; l < nh && !failed; ++l, ++layer) {
          const int kdim = l == 0 ? kK0 : W, nk = l == 0 ? chunks0 : chunksN;
          const uint32_t sbo = (uint32_t)kdim * 16u;
          const uint32_t big = tmem + (uint32_t)(layer & 1) * 2u * (uint32_t)W, small = big + (uint32_t)W;
          for (int c = 0; c < nk; ++c, ++g) {
            const int st = g % kStages;
            if (!mbar_wait_bounded(smem_u32(&bar_a[c]), (a_phase >> c) & 1u) ||
                !mbar_wait_bounded(smem_u32(&bar_full[st]), (g / kStages) & 1)) {
              failed = 1;
              break;
            }
            a_phase ^= 1u << c;
            tc_fence_after();
            const uint32_t b0 = ring0 + (uint32_t)st * cb;
#pragma unroll
            for (int s = 0; s < kChunk / 16; ++s) {
              uint64_t da[3], db[3];
#pragma unroll
              for (int j = 0; j < 3; ++j) {
                da[j] = smem_desc(a0 + j * asz + (uint32_t)(2 * c + s) * 256u, 128, sbo);
                db[j] = smem_desc(b0 + j * bsz + (uint32_t)s * 256u, 128, kChunk * 16);
              }
              const uint32_t on = c > 0 || s > 0 ? 1u : 0u;
              tc_mma(small, da[2], db[0], idesc, on);
              tc_mma(small, da[0], db[2], idesc, 1u);
              tc_mma(small, da[1], db[1], idesc, 1u);
              tc_mma(small, da[1], db[0], idesc, 1u);
              tc_mma(small, da[0], db[1], idesc, 1u);
              tc_mma(big, da[0], db[0], idesc, on);
            }
            tc_commit(smem_u32(&bar_empty[st]));
          }
          if (!failed) tc_commit(smem_u32(&bar_d[layer & 1]));
        }
      }
    }
  } else {
    // ---- inputs and epilogues -----------------------------------------------------
    const int wg = t >> 7, row = t & 127;
    const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t split_bytes = x3_act_bytes(W) / 3;
    const bool leaky = p.act == GS3_ACT_LEAKY_RELU;
    auto hand_on = [&](int c) {  // this warp's part of activation chunk c is written
      fence_proxy_async();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bar_a[c]));
    };
    int layer = 0;
    for (int it = 0; it < mine; ++it) {
      bool ok = true;  // the same for a warp's lanes
      const int r = ((int)blockIdx.x + it * (int)gridDim.x) * kRows + row, rc = min(r, rows - 1);
      const int li = rc / p.n, g = rc - li * p.n;
      const X3Input in = {p.n, p.mean_op, p.latent, WHICH == 0 ? p.T[li] : nullptr,
                          WHICH == 0 ? p.light[li] : make_float4(p.cam_pos[0], p.cam_pos[1], p.cam_pos[2], 1.f)};
      const auto put = [&](int k0, const float* x) { store_split8(A, split_bytes, row, k0, kK0, x); };
      if (wg == 0) encode_half<WHICH, 0>(in, g, put);
      else encode_half<WHICH, 1>(in, g, put);
      hand_on(0);
      hand_on(1);
      float acc[kOut];
#pragma unroll
      for (int o = 0; o < kOut; ++o) acc[o] = 0.f;
      for (int l = 0; l < nh; ++l, ++layer) {
        if (ok) ok = __all_sync(0xffffffffu, mbar_wait_bounded(smem_u32(&bar_d[layer & 1]), (layer >> 1) & 1));
        if (!ok) continue;
        tc_fence_after();
        const uint32_t big = lane_addr + (uint32_t)(layer & 1) * 2u * (uint32_t)W;
        for (int c = 0; c < chunksN; ++c) {
          const int c0 = kChunk * c + 16 * wg;
          float v[16];
          acc_load16(big + (uint32_t)c0, big + (uint32_t)(W + c0), v);
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float h = v[i] + bsm[l * W + c0 + i];
            v[i] = h > 0.f ? h : (leaky ? 0.01f * h : 0.f);
          }
          if (l + 1 < nh) {
            store_split8(A, split_bytes, row, c0, W, v);
            store_split8(A, split_bytes, row, c0 + 8, W, v + 8);
            hand_on(c);
          } else {
#pragma unroll
            for (int o = 0; o < kOut; ++o)
#pragma unroll
              for (int i = 0; i < 16; ++i) acc[o] = fmaf(v[i], wosm[o * W + c0 + i], acc[o]);
          }
        }
      }
      // the second warpgroup's half of the output layer's sums, then the
      // outputs; all 256 threads leave together if a wait ran out
      if (wg == 1)
#pragma unroll
        for (int o = 0; o < kOut; ++o) part[row * kOut + o] = acc[o];
      if (epi_any(!ok)) {
        failed = 1;
        break;
      }
      if (wg == 0 && r < rows) {
        float y[kOut];
#pragma unroll
        for (int o = 0; o < kOut; ++o) y[o] = 1.f / (1.f + __expf(-((acc[o] + part[row * kOut + o]) + bosm[o])));
        const uint32_t rk = p.rank_of[g];
        if constexpr (WHICH == 0) {
          p.out[li][g] = y[0];
          if (p.envcol) {
            const float4 c = p.shade[li][g];
            p.envcol[(size_t)rk * p.nl + li] = make_float4(c.x, c.y, c.z, y[0]);
            if (non_finite(c.x + c.y + c.z + y[0])) *p.nonfinite = 1u;
          } else {
            p.ccol[2 * rk].w = y[0];
            if (non_finite(y[0])) *p.nonfinite = 1u;
          }
        } else {
          const float4 res = make_float4(y[0], y[1], y[2], 0.f);
          reinterpret_cast<float4*>(p.out[0])[g] = res;
          p.ccol[2 * rk + 1] = res;
          if (non_finite(y[0] + y[1] + y[2])) *p.nonfinite = 1u;
        }
      }
      // the next tile's partial sums wait for this read
      asm volatile("bar.sync 1, %0;" ::"r"(kEpiThreads) : "memory");
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (t == 0 && failed) atomicCAS(p.status, 0u, (uint32_t)GS3_ERR_TIMEOUT);
  if (warp == 0) tmem_dealloc(tmem, ncols);
}

size_t x3_smem(const MlpDev& m) {
  return x3_act_bytes(m.width) + (size_t)kStages * chunk_bytes(m.width) +
         4 * ((size_t)m.n_hidden * m.width + (size_t)m.out_dim * m.width + 4 + (size_t)kRows * m.out_dim);
}

unsigned char* net_blob(const FrameArgs& f, int which) {
  return f.ws + f.L->mlp_x3 + (which ? mlp_x3_bytes() / 2 : 0);
}

X3Params x3_params(const FrameArgs& f, int which) {
  const MlpDev& m = which == 0 ? f.sc.phi : f.sc.psi;
  X3Params p;
  p.n = f.sc.n;
  p.nh = m.n_hidden;
  p.width = m.width;
  p.act = m.act;
  p.blob = net_blob(f, which);
  p.bias = m.b;
  p.wout = m.w + (size_t)m.width * m.in_dim + (size_t)(m.n_hidden - 1) * m.width * m.width;
  p.bout = m.b + (size_t)m.n_hidden * m.width;
  p.mean_op = f.sc.mean_op;
  p.latent = f.sc.latent;
  p.nl = 1;
  p.T[0] = at<float>(f.ws, f.L->T);
  p.out[0] = at<float>(f.ws, which == 0 ? f.L->Tp : f.L->res);
  p.shade[0] = at<float4>(f.ws, f.L->shade);
  p.light[0] = light_h(f.light);
  for (int i = 0; i < 3; ++i) p.cam_pos[i] = f.cam.pos[i];
  p.ccol = at<float4>(f.ws, f.L->ccol);
  p.envcol = nullptr;
  p.rank_of = at<uint32_t>(f.ws, f.L->sp[0].rank_of);
  p.status = at<uint32_t>(f.ws, f.L->header) + H_STATUS;
  p.nonfinite = at<uint32_t>(f.ws, f.L->header) + H_NONFINITE;
  return p;
}

void launch_net(const X3Params& p, int which, const MlpDev& m, int sms, cudaStream_t s) {
  size_t smem = x3_smem(m);
  // the CTAs that can share an SM never need more than its 512 tensor-memory columns
  const size_t per_sm = 228 * 1024, reserve = 2048;
  const size_t floor_bytes = per_sm / (size_t)(512 / x3_cols(m.width) + 1) + 1;
  if (smem + reserve < floor_bytes) smem = floor_bytes - reserve;
  auto kern = which == 0 ? k_mlp_x3<0> : k_mlp_x3<1>;
  static DeviceOnce once;
  once.run([] {
    bool ok = true;
    for (const void* k : {(const void*)k_mlp_x3<0>, (const void*)k_mlp_x3<1>})
      ok = ok && cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024) == cudaSuccess;
    return ok;
  });
  const int ntiles = (p.n * p.nl + kRows - 1) / kRows, nsm = sms > 0 ? sms : device_sm_count();
  launch_after(kern, ntiles < nsm ? ntiles : nsm, kThreads, smem, s, p);
  count_launch();
}

}  // namespace

size_t mlp_x3_bytes() {
  const size_t net = (size_t)(kK0 / kChunk + (kMaxHidden - 1) * (128 / kChunk)) * chunk_bytes(128);
  return 2 * ((net + 255) & ~size_t(255));
}

bool mlp_x3_supported(const MlpDev& m) { return m.width == 32 || m.width == 64 || m.width == 128; }

void launch_mlp_x3(const FrameArgs& f, cudaStream_t s, int which_mask, int sms) {
  PackArgs a;
  int total = 0;
  for (int w = 0; w < 2; ++w) {
    const MlpDev& m = w == 0 ? f.sc.phi : f.sc.psi;
    a.w[w] = m.w;
    a.in_dim[w] = m.in_dim;
    a.width[w] = m.width;
    a.nh[w] = m.n_hidden;
    a.dst[w] = net_blob(f, w);
    a.total[w] = (which_mask & (1 << w)) ? hidden_elems(m) : 0;
    total += a.total[w];
  }
  if (total == 0) return;
  k_x3_pack<<<(total + 255) / 256, 256, 0, s>>>(a);
  count_launch();
  for (int w = 0; w < 2; ++w)
    if (which_mask & (1 << w)) launch_net(x3_params(f, w), w, w == 0 ? f.sc.phi : f.sc.psi, sms, s);
}

void launch_phi_lights_x3(const FrameArgs* const* f, int nl, float4* envcol, cudaStream_t s) {
  const MlpDev& m = f[0]->sc.phi;
  PackArgs a{};
  a.w[0] = m.w; a.in_dim[0] = m.in_dim; a.width[0] = m.width; a.nh[0] = m.n_hidden;
  a.dst[0] = net_blob(*f[0], 0);
  a.total[0] = hidden_elems(m);
  k_x3_pack<<<(a.total[0] + 255) / 256, 256, 0, s>>>(a);
  count_launch();
  X3Params p = x3_params(*f[0], 0);
  p.nl = nl;
  for (int l = 0; l < nl; ++l) {
    p.T[l] = at<float>(f[l]->ws, f[l]->L->T);
    p.out[l] = at<float>(f[l]->ws, f[l]->L->Tp);
    p.shade[l] = at<float4>(f[l]->ws, f[l]->L->shade);
    p.light[l] = light_h(f[l]->light);
  }
  p.ccol = nullptr;
  p.envcol = envcol;
  launch_net(p, 0, m, 0, s);
}

}  // namespace gs3
