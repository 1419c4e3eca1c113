"""The few-query attention (bf16, head dim 64) against 64 bits, its kernel called from a program linked with the
library's objects: values and probabilities chosen so that its bf16 outputs show the error of its sums."""
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
// Zero queries: every key has the same probability, exactly 1 before the division. A head dim's values are positive
// but for those of the last six keys, which make their sum exactly zero: what comes out is the rounding of the
// sums alone (size: the sum of the values' sizes).
int main(int, char** v) {
  const int H = 16, P = atoi(v[1]), heads = atoi(v[2]), B = atoi(v[3]), dh = 64, w = heads * dh;
  std::vector<__nv_bfloat16> q((size_t)B * H * w, __float2bfloat16(0.f)), k((size_t)B * P * w, __float2bfloat16(0.f)), x(k.size());
  std::vector<double> size((size_t)B * w);
  srand(3);
  for (int b = 0; b < B; ++b)
    for (int c = 0; c < w; ++c) {
      double s = 0, a = 0;
      for (int p = 0; p < P; ++p) {
        const float u = 0.03125f + 0.96875f * (rand() % 65536) / 65536.f;   // values down to 2^-20, their bits to 2^-28
        const __nv_bfloat16 e = __float2bfloat16(p + 6 < P ? u * u * u * u : (float)-s);   // the last ones: what is left of -s
        x[((size_t)b * P + p) * w + c] = e;
        s += __bfloat162float(e);
        a += fabs(__bfloat162float(e));
      }
      if (s != 0) return 5;
      size[(size_t)b * w + c] = a / P;
    }
  __nv_bfloat16 *dq, *dk, *dx, *out;
  cudaMalloc(&dq, q.size() * 2); cudaMalloc(&dk, k.size() * 2); cudaMalloc(&dx, x.size() * 2); cudaMalloc(&out, q.size() * 2);
  cudaMemcpy(dq, q.data(), q.size() * 2, cudaMemcpyHostToDevice);
  cudaMemcpy(dk, k.data(), k.size() * 2, cudaMemcpyHostToDevice);
  cudaMemcpy(dx, x.data(), x.size() * 2, cudaMemcpyHostToDevice);
  cudaMemset(out, 0xff, q.size() * 2);
  AttnArgs a;
  a.n_heads = a.n_kv_heads = heads; a.head_dim = dh; a.H = H; a.B = B; a.q = dq; a.q_ld = w; a.kp = dk; a.vp = dx; a.P = P;
  a.kp_bstride = (long long)P * w; a.kp_ld = w; a.kc_ld = w; a.out = out; a.out_ld = w; a.dtype = BF16; a.scale = 0.125f;
  launch_attention_prepare();
  launch_attention(a, 0);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    printf("%s\n", cudaGetErrorString(e));
    return 4;
  }
  std::vector<__nv_bfloat16> o(q.size());
  cudaMemcpy(o.data(), out, o.size() * 2, cudaMemcpyDeviceToHost);
  double d2 = 0, most = 0;
  for (int b = 0; b < B; ++b)
    for (int i = 0; i < H; ++i)
      for (int c = 0; c < w; ++c) {
        const double d = fabs(__bfloat162float(o[((size_t)b * H + i) * w + c])) / size[(size_t)b * w + c];
        d2 += d * d;
        most = fmax(most, d);
      }
  printf("%.4e %.4e\n", sqrt(d2 / o.size()), most);
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("few")
    (d / "few.cu").write_text(SRC)
    objs = [os.path.join(PKG, "_build", o) for o in ("kernels_simt.o", "ffma.o")]
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "--expt-relaxed-constexpr",
                    "-I", os.path.join(PKG, "csrc"), "-I", os.path.join(os.path.dirname(PKG), "include"), "-o", str(d / "few"),
                    str(d / "few.cu"), *objs, "-lcuda"], check=True)
    return str(d / "few")


# 24 heads: one CTA a key tile (one robot), a CTA that walks all tiles alone (eight robots); one tile and many
@pytest.mark.parametrize("prefix,heads,robots", [(64, 24, 1), (320, 24, 1), (320, 24, 8), (1000, 24, 8), (300, 6, 1), (1000, 6, 2)])
def test_few_query_attention_sums(program, prefix, heads, robots):
    """In units of u = 2^-24 of the sum of the values' sizes, half of which is the largest running sum. A tile's four
    steps of 16 products lose half an ulp, at most u, of the tile's own sum so far on average: 2 u of it, u of the sizes.
    The tile sums are added with a rounding of at most u / 2 each, either way. (One accumulator over all tiles
    loses each step's half ulp of the whole sum so far: 1.8e-7 at 320 keys, 7.2e-7 at 1000.)"""
    r = subprocess.run([program, str(prefix), str(heads), str(robots)], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout)
    rms, most = (float(s) for s in r.stdout.split())
    tiles = -(-prefix // 64)
    print(f"{prefix} keys, {heads} heads, {robots} robots: rms {rms:.2e}, largest {most:.2e}")
    assert rms <= (1 + tiles ** 0.5 / 4) * 2.0 ** -24
