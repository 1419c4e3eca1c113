// The projection op for callers that must not allocate device memory.
//
// Some callers cannot call cudaMalloc once they are running: a real-time robot controller
// that has finished start-up must not block on an allocation (cudaMalloc can take unbounded
// time and synchronize the device, stalling the control loop), and a host framework whose
// caching allocator has already reserved the GPU's memory would see a stray allocation fail
// or fragment its pool. uad_linear_static_scratch serves them: the projection combines its K splits
// on the chip, and the kernels' error words are in the library's device image.
#include <cstdio>
#include <mutex>

#include "../../include/uad.h"
#include "uad_internal.cuh"

namespace uad {
int launch_linear(const void* x, const void* w_tiled, const float* bias, float* out, int M, int N, int K, int* err,
                  bool stopped, cudaStream_t s);
int linear_tiles(int M, int N);
int static_err_words(int** err, bool look_up);
}  // namespace uad

namespace {

// The error words of the last calls, part of the library's device image.
static __device__ int g_linear_err[uad::kErrWords];

constexpr int kMaxDevices = 64;
std::mutex g_mu;
int* g_err_addr[kMaxDevices] = {};

}  // namespace

// Device address of g_linear_err on the current device. In host code the name only stands in for the
// symbol, so the address is looked up once per device, with that device current (look_up: now, if it has not
// been; else null until it has been).
int uad::static_err_words(int** err, bool look_up) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return UAD_ECUDA;
  if (dev < 0 || dev >= kMaxDevices) return UAD_EINVAL;
  std::lock_guard<std::mutex> lk(g_mu);
  if (!g_err_addr[dev] && look_up) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_linear_err);
    if (e != cudaSuccess) {
      fprintf(stderr, "uad_linear_static_scratch: cudaGetSymbolAddress failed: %s\n", cudaGetErrorString(e));
      return UAD_ECUDA;
    }
    g_err_addr[dev] = static_cast<int*>(p);
  }
  *err = g_err_addr[dev];
  return UAD_OK;
}

extern "C" int uad_linear_static_scratch(const void* x, const void* w_tiled, const float* bias, float* out,
                                         int32_t M, int32_t N, int32_t K, void* stream) {
  if (!x || !w_tiled || !out || M < 1 || N < 128 || N % 128 || K < 64 || K % 64) return UAD_EINVAL;
  const int tiles = uad::linear_tiles(M, N);
  if ((size_t)M * (size_t)N > (size_t)UAD_LINEAR_STATIC_MAX_ELEMS || tiles > UAD_LINEAR_STATIC_MAX_TILES) {
    fprintf(stderr, "uad_linear_static_scratch: M*N = %lld exceeds the limit of %d values and %d tiles\n",
            (long long)M * N, UAD_LINEAR_STATIC_MAX_ELEMS, UAD_LINEAR_STATIC_MAX_TILES);
    return UAD_ETOOBIG;
  }
  int* err = nullptr;
  const int rc = uad::static_err_words(&err, true);
  if (rc) return rc;
  return uad::launch_linear(x, w_tiled, bias, out, M, N, K, err, false, static_cast<cudaStream_t>(stream));
}
