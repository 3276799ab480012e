// gs3_depth_order_static: the per-splat depth sort with its scratch memory in
// a file-scope device array instead of a caller workspace, for callers that
// may not allocate device memory.  It runs the frame's look-back passes: 300k
// keys take 50 us, against 123 us for a histogram, three scan kernels and a
// scatter per digit.  Their waits are bounded, so the array also holds a status
// word: cleared by every call, read by gs3_depth_order_static_status.
#include <mutex>
#include <string>

#include "gs3_internal.cuh"

namespace gs3 {
namespace {

constexpr uint32_t kStaticMaxKeys = GS3_STATIC_SORT_MAX_KEYS;
// ping-pong keys and values (3 of the 4 arrays; the caller's output is the
// 4th), the status and the look-back region
constexpr size_t kStaticWords = 3ull * kStaticMaxKeys + (kOrderFront + onesweep_bytes(kDepthOrderBlocks, 4) + 3) / 4;

static __device__ __align__(256) uint32_t g_static_scratch[kStaticWords];

// The array's device address per device, with the id of the CUDA context it
// was looked up in: a cudaDeviceReset destroys that context, and the module
// (with the array) may load at another address in the next one.
std::mutex g_mu;
uint32_t* g_scratch_addr[kMaxDevices] = {};
unsigned long long g_scratch_ctx[kMaxDevices] = {};

// Id of the calling thread's current CUDA context (0 when it cannot be read),
// through the driver entry points cuCtxGetCurrent and cuCtxGetId.
unsigned long long current_context_id() {
  typedef int (*get_current_fn)(void**);
  typedef int (*get_id_fn)(void*, unsigned long long*);
  struct Fns {
    get_current_fn cur = nullptr;
    get_id_fn id = nullptr;
  };
  static const Fns fns = [] {
    Fns f;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      f.cur = reinterpret_cast<get_current_fn>(p);
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      f.id = reinterpret_cast<get_id_fn>(p);
    return f;
  }();
  if (!fns.cur || !fns.id) return 0;
  void* ctx = nullptr;
  unsigned long long id = 0;
  if (fns.cur(&ctx) != 0 || !ctx || fns.id(ctx, &id) != 0) return 0;
  return id;
}

// The array's address on the current device, or null (with the error message set).
uint32_t* static_scratch(const char* who) {
  int dev = 0;
  // cudaSetDevice makes the device's primary context current on this thread,
  // so that its id can be compared with the one the address was found in
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices || cudaSetDevice(dev) != cudaSuccess) {
    set_last_error((std::string(who) + ": no usable current device").c_str());
    return nullptr;
  }
  uint32_t* base = nullptr;
  {
    // once per device and context, with that device current: the host-side
    // symbol is only a stand-in, the kernels need the array's device address
    std::lock_guard<std::mutex> lock(g_mu);
    const unsigned long long ctx = current_context_id();
    if (!g_scratch_addr[dev] || ctx == 0 || ctx != g_scratch_ctx[dev]) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || !p) {
        g_scratch_addr[dev] = nullptr;
        set_last_error((std::string(who) + ": cudaGetSymbolAddress of the scratch array failed").c_str());
        return nullptr;
      }
      g_scratch_addr[dev] = static_cast<uint32_t*>(p);
      g_scratch_ctx[dev] = current_context_id();
    }
    base = g_scratch_addr[dev];
  }
  return base;
}

void sort_static(uint32_t* base, const uint32_t* keys, uint32_t n, uint32_t* order_out, cudaStream_t s,
                 int first_ticket = 0) {
  // four 8-bit passes over the 32-bit keys; the odd passes write the values
  // into the caller's output, so the last pass leaves the order there
  depth_order(keys, n, base, base + kStaticMaxKeys, base + 2ull * kStaticMaxKeys, order_out,
              reinterpret_cast<unsigned char*>(base + 3ull * kStaticMaxKeys), s, first_ticket);  // counts its launches
}

}  // namespace
}  // namespace gs3

using namespace gs3;

extern "C" gs3_status gs3_depth_order_static(const uint32_t* keys, uint32_t n, uint32_t* order_out,
                                             void* stream) {
  static_assert(kDepthOrderBlocks * kSortThreads * 8 >= kStaticMaxKeys, "look-back region too small");
  if (n == 0) return GS3_OK;
  if (!keys || !order_out) {
    set_last_error("gs3_depth_order_static: null keys or order_out");
    return GS3_ERR_INVALID_ARG;
  }
  if (n > kStaticMaxKeys) {
    set_last_error("gs3_depth_order_static: n exceeds GS3_STATIC_SORT_MAX_KEYS (1048576)");
    return GS3_ERR_INVALID_ARG;
  }
  if (!device_range_ok(keys, (size_t)n * 4) || !device_range_ok(order_out, (size_t)n * 4)) {
    set_last_error("gs3_depth_order_static: keys or order_out is not device memory of n words");
    return GS3_ERR_INVALID_ARG;
  }
  uint32_t* base = static_scratch("gs3_depth_order_static");
  if (!base) return GS3_ERR_CUDA;
  // an error left by an earlier, unrelated call on this thread is not this
  // call's: clear it so that the check below sees only these launches
  (void)cudaGetLastError();
  sort_static(base, keys, n, order_out, reinterpret_cast<cudaStream_t>(stream));
  if (cudaGetLastError() != cudaSuccess) {
    set_last_error("gs3_depth_order_static: kernel launch failed");
    return GS3_ERR_CUDA;
  }
  return GS3_OK;
}

extern "C" gs3_status gs3_depth_order_static_status(uint32_t* status_out, void* stream) {
  if (!status_out) {
    set_last_error("gs3_depth_order_static_status: null status_out");
    return GS3_ERR_INVALID_ARG;
  }
  uint32_t* base = static_scratch("gs3_depth_order_static_status");
  if (!base) return GS3_ERR_CUDA;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  cudaError_t e = cudaMemcpyAsync(status_out, base + 3ull * kStaticMaxKeys, 4, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    set_last_error("gs3_depth_order_static_status: CUDA call failed");
    return GS3_ERR_CUDA;
  }
  return GS3_OK;
}

// The first pass's tickets start at 1, so every block's look-back reaches ticket
// 0's words, which no block writes, and gives up after kLookSpin polls; the
// passes behind it sort what it left.
extern "C" gs3_status gs3_selftest_depth_order_timeout(uint32_t n, uint32_t* status_out) {
  if (!status_out || n <= 4096 || n > kStaticMaxKeys) {
    set_last_error("gs3_selftest_depth_order_timeout: need status_out and 4096 < n <= GS3_STATIC_SORT_MAX_KEYS");
    return GS3_ERR_INVALID_ARG;
  }
  uint32_t* base = static_scratch("gs3_selftest_depth_order_timeout");
  if (!base) return GS3_ERR_CUDA;
  uint32_t* d = nullptr;
  if (cudaMalloc(&d, 8ull * n) != cudaSuccess) {
    set_last_error("gs3_selftest_depth_order_timeout: cudaMalloc failed");
    return GS3_ERR_OOM;
  }
  (void)cudaGetLastError();  // only this call's launches are checked below
  cudaError_t e = cudaMemset(d, 0, 8ull * n);
  if (e == cudaSuccess) {
    sort_static(base, d, n, d + n, 0, 1);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  cudaFree(d);
  if (e != cudaSuccess) {
    set_last_error("gs3_selftest_depth_order_timeout: CUDA call failed");
    return GS3_ERR_CUDA;
  }
  return gs3_depth_order_static_status(status_out, nullptr);
}
