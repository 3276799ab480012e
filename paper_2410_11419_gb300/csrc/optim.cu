// Adam (Kingma and Ba, 2015), the optimiser of the training in Sec. 4.4,
// applied in place to one parameter array in one pass:
//   m <- b1 m + (1 - b1) g,   v <- b2 v + (1 - b2) g^2,
//   p <- max(lo, p - lr (m / c1) / (sqrt(v / c2) + eps)),  c1 = 1 - b1^t, c2 = 1 - b2^t.
// `lo` keeps positive parameters (scales, lobe deviations) positive; -inf
// leaves a parameter unbounded.  Each element is independent, so the update
// is bandwidth-bound: 4 reads and 3 writes of 4 bytes per parameter.  Arrays
// that start on 16-byte boundaries go four elements per thread with 16-byte
// accesses, one group per thread, so that enough bytes are in flight: the
// 38.5 M parameters of a 300k-Gaussian scene (14 calls) take 186 us of kernel
// time, 5.8 TB/s; one element per thread over a grid-stride loop of 16 blocks
// per SM took 230 us.
#include "gs3_internal.cuh"

namespace gs3 {
namespace {

struct AdamArgs {
  float lr, b1, b2, eps, c1, c2, lo;
};

__device__ __forceinline__ void adam_one(const AdamArgs& a, float g, float& p, float& m, float& v) {
  m = fmaf(a.b1, m, (1.f - a.b1) * g);
  v = fmaf(a.b2, v, (1.f - a.b2) * g * g);
  const float step = a.lr * (m / a.c1) / (sqrtf(v / a.c2) + a.eps);
  p = fmaxf(a.lo, p - step);
}

// four consecutive elements per thread (16-byte aligned arrays); the thread past
// the whole groups takes the last n % 4
__global__ void __launch_bounds__(256) k_adam4(float4* __restrict__ p, const float4* __restrict__ g,
                                               float4* __restrict__ m, float4* __restrict__ v, size_t n4, int tail,
                                               AdamArgs a) {
  after_previous();
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n4) {
    if (i == n4)
      for (int k = 0; k < tail; ++k)
        adam_one(a, reinterpret_cast<const float*>(g + n4)[k], reinterpret_cast<float*>(p + n4)[k],
                 reinterpret_cast<float*>(m + n4)[k], reinterpret_cast<float*>(v + n4)[k]);
    return;
  }
  const float4 gi = __ldcs(g + i);
  float4 pi = p[i], mi = m[i], vi = v[i];
  adam_one(a, gi.x, pi.x, mi.x, vi.x);
  adam_one(a, gi.y, pi.y, mi.y, vi.y);
  adam_one(a, gi.z, pi.z, mi.z, vi.z);
  adam_one(a, gi.w, pi.w, mi.w, vi.w);
  m[i] = mi;
  v[i] = vi;
  p[i] = pi;
}

__global__ void __launch_bounds__(256) k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                                              float* __restrict__ v, size_t n, AdamArgs a) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    float pi = p[i], mi = m[i], vi = v[i];
    adam_one(a, g[i], pi, mi, vi);
    m[i] = mi;
    v[i] = vi;
    p[i] = pi;
  }
}

}  // namespace

void launch_adam(float* p, const float* g, float* m, float* v, size_t n, float lr, float b1, float b2, float eps,
                 int step, float lo, cudaStream_t s) {
  const double c1 = 1.0 - pow((double)b1, (double)step), c2 = 1.0 - pow((double)b2, (double)step);
  const AdamArgs a{lr, b1, b2, eps, (float)c1, (float)c2, lo};
  const uintptr_t addr = reinterpret_cast<uintptr_t>(p) | reinterpret_cast<uintptr_t>(g) |
                         reinterpret_cast<uintptr_t>(m) | reinterpret_cast<uintptr_t>(v);
  // groups of four with vector accesses; unaligned arrays and arrays past the
  // grid's limit one element at a time
  if ((addr & 15) == 0 && n / 4 < (size_t)0x7FFFFFFF * 256) {
    const size_t n4 = n / 4;
    const int tail = (int)(n - 4 * n4);
    auto f4 = [](float* x) { return reinterpret_cast<float4*>(x); };
    launch_after(k_adam4, (unsigned)((n4 + (tail ? 1 : 0) + 255) / 256), 256, 0, s, f4(p),
                 reinterpret_cast<const float4*>(g), f4(m), f4(v), n4, tail, a);
  } else {
    const size_t want = (n + 255) / 256, cap_blocks = (size_t)device_sm_count() * 16;
    k_adam<<<(int)(want < cap_blocks ? want : cap_blocks), 256, 0, s>>>(p, g, m, v, n, a);
  }
  count_launch();
}

}  // namespace gs3
