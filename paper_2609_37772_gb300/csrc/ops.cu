// Kernel-level entry points: the step loop's tensor-core projection GEMM on caller buffers.
#include <cstring>
#include <algorithm>
#include <atomic>
#include <mutex>
#include <vector>

#include "../../include/uad.h"
#include "uad_internal.cuh"

using namespace uad;

namespace {

constexpr int kTileN = 128, kTileK = 64;

// On each device, allocated on first use: the error words of the last kErrWords calls, a word of its own for each
// (one that a wait set must end no other call's waits).
std::mutex g_mu;
std::vector<int*> g_err;
std::atomic<unsigned> g_call{0};

uint16_t f32_to_bf16_rne(float f) {
  uint32_t u;
  memcpy(&u, &f, 4);
  if ((u & 0x7f800000u) == 0x7f800000u && (u & 0x7fffffu)) return (uint16_t)((u >> 16) | 0x40);  // NaN
  const uint32_t lsb = (u >> 16) & 1u;
  return (uint16_t)((u + 0x7fffu + lsb) >> 16);
}

int check_linear_args(const void* x, const void* w, const float* out, int32_t M, int32_t N, int32_t K) {
  if (!x || !w || !out) return UAD_EINVAL;
  if (M < 1 || N < kTileN || N % kTileN || K < kTileK || K % kTileK) return UAD_EINVAL;
  return UAD_OK;
}

}  // namespace

namespace uad {

int static_err_words(int** err, bool look_up);   // ops_static.cu

// Shared by uad_linear and its static variant: launch the projection kernel with
// out[M][N] = x[M][K] w^T (+ bias), fp32 output. err: kErrWords words. stopped: as if a wait had run out.
int launch_linear(const void* x, const void* w_tiled, const float* bias, float* out, int M, int N, int K, int* err,
                  bool stopped, cudaStream_t s) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return UAD_ECUDA;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  CUtensorMap tm;
  if (encode_act_tmap(&tm, x, K, M, act_box_rows(M))) return UAD_ECUDA;
  TcGemmArgs a;
  a.w_tiled = w_tiled; a.M = M; a.N = N; a.K = K;
  gemm_tc_plan(M, N, K, sms, EPI_STORE, &a);   // the tile selection of the velocity network's projections
  a.epi = EPI_STORE; a.out = out; a.ldo = N; a.out_dtype = F32; a.bias = bias;
  a.err = err + g_call.fetch_add(1, std::memory_order_relaxed) % kErrWords;
  a.ordered = 1; a.own_err = !stopped;
  if (stopped && cudaMemsetAsync(a.err, 1, 4, s) != cudaSuccess) return UAD_ECUDA;
  if (gemm_tc_prepare()) return UAD_ECUDA;
  launch_gemm_tc(&tm, a, s);
  return cudaGetLastError() == cudaSuccess ? UAD_OK : UAD_ECUDA;
}

int linear_tiles(int M, int N) { return (N / kTileN) * ((M + 63) / 64); }

}  // namespace uad

extern "C" {

int uad_tile_weight(const float* w, int32_t K, int32_t N, uint16_t* out) {
  if (!w || !out || N < kTileN || N % kTileN || K < kTileK || K % kTileK) return UAD_EINVAL;
  const int KC = K / kTileK;
  for (int n = 0; n < N; ++n)
    for (int k = 0; k < K; ++k) {
      const int rr = n % kTileN, kk = k % kTileK;
      const size_t tile = (size_t)(n / kTileN) * KC + k / kTileK;
      const int gran = (kk >> 3) ^ (rr & 7);
      out[tile * kTileN * kTileK + rr * kTileK + gran * 8 + (kk & 7)] = f32_to_bf16_rne(w[(size_t)k * N + n]);
    }
  return UAD_OK;
}

static int linear(const void* x, const void* w_tiled, const float* bias, float* out, int32_t M, int32_t N, int32_t K,
                  bool stopped, void* stream) {
  int rc = check_linear_args(x, w_tiled, out, M, N, K);
  if (rc) return rc;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return UAD_ECUDA;
  std::lock_guard<std::mutex> lk(g_mu);
  if ((int)g_err.size() <= dev) g_err.resize(dev + 1, nullptr);
  if (!g_err[dev]) {
    int* e = nullptr;
    if (cudaMalloc(&e, kErrWords * 4) != cudaSuccess) return UAD_ENOMEM;
    if (cudaMemset(e, 0, kErrWords * 4) != cudaSuccess) {
      cudaFree(e);
      return UAD_ECUDA;
    }
    g_err[dev] = e;
  }
  return launch_linear(x, w_tiled, bias, out, M, N, K, g_err[dev], stopped, static_cast<cudaStream_t>(stream));
}

int uad_linear(const void* x, const void* w_tiled, const float* bias, float* out, int32_t M, int32_t N,
               int32_t K, void* stream) {
  return linear(x, w_tiled, bias, out, M, N, K, false, stream);
}

int uad_linear_check(const void* x, const void* w_tiled, const float* bias, float* out, int32_t M, int32_t N,
                     int32_t K, void* stream) {
  return linear(x, w_tiled, bias, out, M, N, K, true, stream);
}

int uad_linear_status(void) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return UAD_ECUDA;
  int* words[2] = {nullptr, nullptr};
  {
    std::lock_guard<std::mutex> lk(g_mu);
    if (dev < (int)g_err.size()) words[0] = g_err[dev];
  }
  static_err_words(&words[1], false);
  bool ran_out = false;
  for (int* w : words) {
    if (!w) continue;
    int codes[kErrWords];
    if (cudaMemcpy(codes, w, sizeof(codes), cudaMemcpyDeviceToHost) != cudaSuccess) return UAD_ECUDA;
    const bool any = std::any_of(codes, codes + kErrWords, [](int c) { return c != 0; });
    if (any && cudaMemset(w, 0, sizeof(codes)) != cudaSuccess) return UAD_ECUDA;
    ran_out |= any;
  }
  return ran_out ? UAD_ECUDA : UAD_OK;
}

}  // extern "C"
