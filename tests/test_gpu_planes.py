"""The planes of K splits that a residual projection of 129 to 511 tokens writes, summed as the next norm sums
them, against 64 bits: the projection's own plan and kernels, called from a program linked with the
library's objects (no public entry point returns these fp32 sums)."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu
PKG = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_37772_gb300")
SRC = r"""
#include "uad_internal.cuh"
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>
using namespace uad;
// positive products; x [M][K], w [K][N] and its tiled form, sums in 64 bits
__device__ float value(unsigned i, unsigned salt) {
  unsigned h = i * 2654435761u ^ salt;
  h ^= h >> 15; h *= 2246822519u; h ^= h >> 13;
  const float u = ((h & 0xffff) + 1) / 65536.f;
  return 2.f * u * u;   // over many powers of two, so that the products reach far below the sum's last bit
}
__global__ void fill(__nv_bfloat16* x, __nv_bfloat16* t, int M, int N, int K) {
  for (int i = blockIdx.x * 256 + threadIdx.x; i < M * K; i += gridDim.x * 256) x[i] = __float2bfloat16(value(i, 1));
  for (int i = blockIdx.x * 256 + threadIdx.x; i < N * K; i += gridDim.x * 256) {
    const int n = i % N, k = i / N, rr = n % 128, kk = k % 64;
    t[((size_t)(n / 128) * (K / 64) + k / 64) * 8192 + rr * 64 + (((kk >> 3) ^ (rr & 7)) * 8) + (kk & 7)] = __float2bfloat16(value(i, 2));
  }
}
__global__ void exact(const __nv_bfloat16* x, double* o, int M, int N, int K) {
  const int n = blockIdx.x * 128 + threadIdx.x, m = blockIdx.y;
  double s = 0;
  for (int k = 0; k < K; ++k)
    s += (double)__bfloat162float(x[(size_t)m * K + k]) * (double)__bfloat162float(__float2bfloat16(value(k * N + n, 2)));
  o[(size_t)m * N + n] = s;
}
int main(int, char** v) {
  const int M = atoi(v[1]), N = atoi(v[2]), K = atoi(v[3]);
  int dev = 0, sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  TcGemmArgs a;
  gemm_tc_plan(M, N, K, sms, EPI_PARTIAL, &a);
  if (!a.wide || gemm_tc_prepare()) return 2;
  __nv_bfloat16 *x, *t;
  double* ref;
  float* out;
  int* err;
  cudaMalloc(&x, (size_t)M * K * 2); cudaMalloc(&t, (size_t)N * K * 2); cudaMalloc(&ref, (size_t)M * N * 8);
  cudaMalloc(&out, (size_t)a.splits * M * N * 4); cudaMalloc(&err, 4); cudaMemset(err, 0, 4);
  fill<<<512, 256>>>(x, t, M, N, K);
  exact<<<dim3(N / 128, M), 128>>>(x, ref, M, N, K);
  CUtensorMap tm;
  if (encode_act_tmap(&tm, x, K, M, 64)) return 3;
  a.M = M; a.N = N; a.K = K; a.epi = EPI_PARTIAL; a.w_tiled = t; a.out = out; a.ldo = N; a.out_dtype = F32; a.err = err;
  launch_gemm_tc(&tm, a, 0);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    printf("%s\n", cudaGetErrorString(e));
    return 4;
  }
  std::vector<double> r((size_t)M * N);
  std::vector<float> p((size_t)a.splits * M * N);
  cudaMemcpy(r.data(), ref, r.size() * 8, cudaMemcpyDeviceToHost);
  cudaMemcpy(p.data(), out, p.size() * 4, cudaMemcpyDeviceToHost);
  double mean = 0, most = 0;
  for (size_t i = 0; i < r.size(); ++i) {
    float s = 0;
    for (int sp = 0; sp < a.splits; ++sp) s += p[sp * r.size() + i];
    const double e = (s - r[i]) / r[i];
    mean += e;
    most = fabs(e) > most ? fabs(e) : most;
  }
  printf("%.4e %.4e %d\n", mean / r.size(), most, sms);
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("planes")
    (d / "planes.cu").write_text(SRC)
    objs = [os.path.join(PKG, "_build", o) for o in ("gemm_tc.o", "gemm_cl.o", "kernels_simt.o", "ffma.o")]
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "--expt-relaxed-constexpr",
                    "-I", os.path.join(PKG, "csrc"), "-I", os.path.join(os.path.dirname(PKG), "include"), "-o", str(d / "planes"),
                    str(d / "planes.cu"), *objs, "-lcuda"], check=True)
    return str(d / "planes")


# the residual projections of the experts of width 1024 and 1536, from the first size of the persistent form to the last
# before it would be taken anyway; (129, 1024, 64), (130, 2048, 128): one and two k-blocks in all
@pytest.mark.parametrize("M,N,K", [(129, 1024, 2048), (180, 1024, 2048), (250, 1024, 4096), (500, 1024, 4096), (144, 1536, 1536),
                                   (200, 1536, 6144), (320, 1536, 6144), (129, 1024, 64), (130, 2048, 128), (333, 1280, 192)])
def test_residual_planes_sum_short_runs(program, M, N, K):
    """Positive products: a truncating accumulation loses up to an ulp of the sum so far with every step of 16
    products, half of one on average, so 2 x 2^-24 of the sum a k-block of 64. The bound is that of the run which
    one 128 x 64 tile per SM would make of K, or two tiles an SM where that is more than four k-blocks."""
    r = subprocess.run([program, str(M), str(N), str(K)], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout)
    mean, most, sms = (float(s) for s in r.stdout.split())
    tiles, blocks = N // 128 * ((M + 63) // 64), K // 64
    run = -(-blocks // max(1, int(sms) // tiles))
    if run > 4:
        run = max(4, -(-blocks // max(1, 2 * int(sms) // tiles)))
    print(f"{M} x {K} x {N}: mean {mean:.2e}, largest {most:.2e}, runs of {run}")
    assert abs(mean) <= (2 * run + 2) * 2.0 ** -24   # and the roundings of the planes' sum
    assert most <= (8 * run + 16) * 2.0 ** -24
