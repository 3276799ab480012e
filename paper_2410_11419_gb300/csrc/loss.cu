// The training loss of Sec. 4.4 and its image gradient:
//   L = (1 - lambda) mean |I - I*| + lambda (1 - SSIM(I, I*))
// SSIM per pixel and channel with an 11x11 Gaussian window (sigma 1.5),
// C1 = 0.01^2, C2 = 0.03^2, zero padding, averaged over pixels and channels.
//
// Every window sum is a separable blur of planar maps.  With mu = G*I,
// Sxx = G*(I I), Sxy = G*(I I*) (and the same for the target) the SSIM map is
// m = (2 mu mu* + C1)(2 (Sxy - mu mu*) + C2) / ((mu^2 + mu*^2 + C1)(Sxx - mu^2 + Syy - mu*^2 + C2)),
// and dSSIM/dI = (G * dm/dmu) + I* (G * dm/dSxy) + 2 I (G * dm/dSxx), the
// blur being its own adjoint (symmetric kernel, zero padding).
//
// Two kernels, a block per 32 x 32 pixels and channel.  k_ssim reads its tile
// with a 5-pixel halo, blurs the five maps along the rows and then the
// columns in shared memory, and writes the three partial derivatives and the
// block's sums; k_ssim_grad blurs the derivatives the same way and writes
// the image gradient, and its first block adds up the sums in block order.
// What bounds them is the 206 FMAs per pixel and channel of the two blurs
// (the 9 planes between the kernels stay in the L2).  At 800 x 800 they take
// 46 + 22 us; the eight kernels before them (48 planes through memory, four
// blur passes over single maps, and the block sums added by one thread, which
// alone took 217 us) took 517 us.
#include "gs3_internal.cuh"

namespace gs3 {
namespace {

constexpr int kWin = 11, kHalf = 5;

__constant__ float c_gauss[kWin];

constexpr int kLT = 32;             // tile edge
constexpr int kLH = kLT + 2 * kHalf;  // with the halo
constexpr int kLRow = kLH + 1;      // padded row
constexpr int kLThreads = 256;
constexpr int kRun = 4;             // consecutive outputs a thread blurs together

// tile t of channel c: blocks run over the tiles of one channel, then the next
struct LossTile {
  int c, x0, y0;
};
__device__ __forceinline__ LossTile loss_tile(int W, int H) {
  const int tx = (W + kLT - 1) / kLT, ty = (H + kLT - 1) / kLT;
  const int nt = tx * ty, c = blockIdx.x / nt, t = blockIdx.x - c * nt;
  return {c, (t % tx) * kLT, (t / tx) * kLT};
}

// out[r] = sum_k gauss[k] v[r + k], taps in ascending order
__device__ __forceinline__ void blur_run(const float (&v)[kRun + 2 * kHalf], float (&out)[kRun]) {
#pragma unroll
  for (int r = 0; r < kRun; ++r) {
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < kWin; ++k) s = fmaf(c_gauss[k], v[r + k], s);
    out[r] = s;
  }
}

// SSIM map, its partial derivatives (3 planes per channel) and the block's
// sums of the map and of |I - I*|
__global__ void __launch_bounds__(kLThreads) k_ssim(const float* __restrict__ img, const float* __restrict__ tgt,
                                                    float* __restrict__ dmaps, double* __restrict__ part, int W, int H) {
  __shared__ float X[kLH][kLRow], Y[kLH][kLRow];
  __shared__ float B[5][kLH][kLT];
  __shared__ double red[2][kLThreads / 32];
  const LossTile T = loss_tile(W, H);
  const int t = threadIdx.x;
  for (int i = t; i < kLH * kLH; i += kLThreads) {
    const int r = i / kLH, q = i - r * kLH, y = T.y0 + r - kHalf, x = T.x0 + q - kHalf;
    const bool in = x >= 0 && x < W && y >= 0 && y < H;
    const size_t p = 3 * ((size_t)y * W + x) + T.c;
    X[r][q] = in ? img[p] : 0.f;
    Y[r][q] = in ? tgt[p] : 0.f;
  }
  __syncthreads();
  // rows: the products once per loaded pixel
  for (int i = t; i < kLH * (kLT / kRun); i += kLThreads) {
    const int r = i / (kLT / kRun), q = (i - r * (kLT / kRun)) * kRun;
    float x[kRun + 2 * kHalf], y[kRun + 2 * kHalf], v[kRun + 2 * kHalf], o[kRun];
#pragma unroll
    for (int k = 0; k < kRun + 2 * kHalf; ++k) {
      x[k] = X[r][q + k];
      y[k] = Y[r][q + k];
    }
#pragma unroll
    for (int m = 0; m < 5; ++m) {
#pragma unroll
      for (int k = 0; k < kRun + 2 * kHalf; ++k)
        v[k] = m == 0 ? x[k] : m == 1 ? y[k] : m == 2 ? x[k] * x[k] : m == 3 ? y[k] * y[k] : x[k] * y[k];
      blur_run(v, o);
#pragma unroll
      for (int k = 0; k < kRun; ++k) B[m][r][q + k] = o[k];
    }
  }
  __syncthreads();
  // columns: thread t takes column t & 31, rows 4 (t >> 5) .. + 3
  const int q = t & 31, r0 = (t >> 5) * kRun;
  float b[5][kRun];
#pragma unroll
  for (int m = 0; m < 5; ++m) {
    float v[kRun + 2 * kHalf];
#pragma unroll
    for (int k = 0; k < kRun + 2 * kHalf; ++k) v[k] = B[m][r0 + k][q];
    blur_run(v, b[m]);
  }
  const size_t plane = (size_t)W * H;
  float* d = dmaps + (size_t)T.c * 3 * plane;
  double sm = 0.0, sl = 0.0;
#pragma unroll
  for (int k = 0; k < kRun; ++k) {
    const int x = T.x0 + q, y = T.y0 + r0 + k;
    if (x >= W || y >= H) continue;
    const size_t p = (size_t)y * W + x;
    const float C1 = 1e-4f, C2 = 9e-4f;
    const float mx = b[0][k], my = b[1][k], sxx = b[2][k], syy = b[3][k], sxy = b[4][k];
    const float A1 = 2.f * mx * my + C1, A2 = 2.f * (sxy - mx * my) + C2;
    const float B1 = mx * mx + my * my + C1, B2 = (sxx - mx * mx) + (syy - my * my) + C2;
    const float iB = 1.f / (B1 * B2);
    const float m = A1 * A2 * iB;
    d[p] = (2.f * my * A2 - 2.f * my * A1) * iB - m * (2.f * mx / B1 - 2.f * mx / B2);  // dm/dmu
    d[plane + p] = 2.f * A1 * iB;                                                    // dm/dSxy
    d[2 * plane + p] = -m / B2;                                                      // dm/dSxx
    sm += m;
    sl += fabs((double)X[r0 + k + kHalf][q + kHalf] - (double)Y[r0 + k + kHalf][q + kHalf]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sm += __shfl_xor_sync(0xffffffffu, sm, o);
    sl += __shfl_xor_sync(0xffffffffu, sl, o);
  }
  if (q == 0) {
    red[0][t >> 5] = sm;
    red[1][t >> 5] = sl;
  }
  __syncthreads();
  if (t < 2) {
    double a = 0.0;
    for (int w = 0; w < kLThreads / 32; ++w) a += red[t][w];
    part[2 * (size_t)blockIdx.x + t] = a;
  }
}

// The image gradient from the derivative planes; the first block also adds
// up the loss (thread t takes partials t, t + 256, ..., then the threads'
// sums in a tree: a fixed order).
__global__ void __launch_bounds__(kLThreads) k_ssim_grad(const float* __restrict__ img, const float* __restrict__ tgt,
                                                         const float* __restrict__ dmaps,
                                                         const double* __restrict__ part, float* __restrict__ dimg,
                                                         float* __restrict__ loss, int W, int H, float lambda) {
  after_previous();
  __shared__ float D[3][kLH][kLRow];
  __shared__ float B[3][kLH][kLT];
  const LossTile T = loss_tile(W, H);
  const int t = threadIdx.x;
  const size_t plane = (size_t)W * H;
  const float* src = dmaps + (size_t)T.c * 3 * plane;
  for (int i = t; i < kLH * kLH; i += kLThreads) {
    const int r = i / kLH, q = i - r * kLH, y = T.y0 + r - kHalf, x = T.x0 + q - kHalf;
    const bool in = x >= 0 && x < W && y >= 0 && y < H;
    const size_t p = (size_t)y * W + x;
#pragma unroll
    for (int m = 0; m < 3; ++m) D[m][r][q] = in ? src[m * plane + p] : 0.f;
  }
  __syncthreads();
  for (int i = t; i < kLH * (kLT / kRun); i += kLThreads) {
    const int r = i / (kLT / kRun), q = (i - r * (kLT / kRun)) * kRun;
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      float v[kRun + 2 * kHalf], o[kRun];
#pragma unroll
      for (int k = 0; k < kRun + 2 * kHalf; ++k) v[k] = D[m][r][q + k];
      blur_run(v, o);
#pragma unroll
      for (int k = 0; k < kRun; ++k) B[m][r][q + k] = o[k];
    }
  }
  __syncthreads();
  const int q = t & 31, r0 = (t >> 5) * kRun;
  float d[3][kRun];
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    float v[kRun + 2 * kHalf];
#pragma unroll
    for (int k = 0; k < kRun + 2 * kHalf; ++k) v[k] = B[m][r0 + k][q];
    blur_run(v, d[m]);
  }
  const float inv = 1.f / (3.f * (float)plane);
#pragma unroll
  for (int k = 0; k < kRun; ++k) {
    const int px = T.x0 + q, py = T.y0 + r0 + k;
    if (px >= W || py >= H) continue;
    const size_t p = 3 * ((size_t)py * W + px) + T.c;
    const float x = img[p], y = tgt[p];
    const float dssim = (d[0][k] + y * d[1][k] + 2.f * x * d[2][k]) * inv;
    const float sgn = x > y ? 1.f : (x < y ? -1.f : 0.f);
    dimg[p] = (1.f - lambda) * sgn * inv - lambda * dssim;
  }
  if (blockIdx.x != 0) return;
  __syncthreads();
  double(*red)[kLThreads] = reinterpret_cast<double(*)[kLThreads]>(&D[0][0][0]);
  double sm = 0.0, sl = 0.0;
  for (unsigned i = t; i < gridDim.x; i += kLThreads) {
    sm += part[2 * (size_t)i];
    sl += part[2 * (size_t)i + 1];
  }
  red[0][t] = sm;
  red[1][t] = sl;
  __syncthreads();
  for (int o = kLThreads / 2; o > 0; o >>= 1) {
    if (t < o) {
      red[0][t] += red[0][t + o];
      red[1][t] += red[1][t + o];
    }
    __syncthreads();
  }
  const double count = 3.0 * (double)plane;
  if (t == 0) *loss = (float)((1.0 - lambda) * red[1][0] / count + lambda * (1.0 - red[0][0] / count));
}

size_t loss_tiles(int W, int H) { return (size_t)((W + kLT - 1) / kLT) * (size_t)((H + kLT - 1) / kLT); }

}  // namespace

// nine derivative planes, then the blocks' sums
size_t loss_scratch_bytes(int W, int H) { return 4 * 9 * (size_t)W * H + 48 * loss_tiles(W, H) + 256; }

gs3_status run_loss(const float* img, const float* tgt, int W, int H, float lambda, float* loss, float* dimg,
                    void* scratch, cudaStream_t s) {
  // the window lives in constant memory, one copy per device
  static DeviceOnce once;
  const bool ready = once.run([] {
    float g[kWin], sum = 0.f;
    for (int k = 0; k < kWin; ++k) {
      const float d = (float)(k - kHalf);
      g[k] = expf(-d * d / (2.f * 1.5f * 1.5f));
      sum += g[k];
    }
    for (int k = 0; k < kWin; ++k) g[k] /= sum;
    return cudaMemcpyToSymbol(c_gauss, g, sizeof(g)) == cudaSuccess;
  });
  if (!ready) return GS3_ERR_CUDA;
  float* dm = static_cast<float*>(scratch);
  // 8-byte aligned past the planes (the scratch may start at any float)
  double* part = reinterpret_cast<double*>((reinterpret_cast<uintptr_t>(dm + 9 * (size_t)W * H) + 7) & ~uintptr_t(7));
  const unsigned nb = (unsigned)(3 * loss_tiles(W, H));
  k_ssim<<<nb, kLThreads, 0, s>>>(img, tgt, dm, part, W, H);
  launch_after(k_ssim_grad, nb, kLThreads, 0, s, img, tgt, dm, part, dimg, loss, W, H, lambda);
  count_launch(2);
  return cudaGetLastError() == cudaSuccess ? GS3_OK : GS3_ERR_CUDA;
}

}  // namespace gs3
