// CUDA-core kernels: projections with a tiny side, adaptive norms, attention for few queries, and
// the Euler / TR / release / GAC step epilogue. (GEMM and general attention: ffma.cu.)
#include "uad_internal.cuh"
#include "euler.cuh"

namespace uad {

bool pdl_enabled() {
  static int on = -1;
  if (on < 0) {
    const char* e = getenv("UAD_PDL");
    on = !(e && e[0] == '0');
  }
  return on != 0;
}

// ------------------------------------------------------------------------------------------
// small helpers
// ------------------------------------------------------------------------------------------
template <int DT>
__device__ __forceinline__ float ldf(const void* p, long long i) {
  if constexpr (DT == BF16) return __bfloat162float(static_cast<const __nv_bfloat16*>(p)[i]);
  else return static_cast<const float*>(p)[i];
}
__device__ __forceinline__ float ldf_rt(const void* p, long long i, int dt) {
  return dt == BF16 ? ldf<BF16>(p, i) : ldf<F32>(p, i);
}
__device__ __forceinline__ void stf(void* p, long long i, float v, int dt) {
  if (dt == BF16) static_cast<__nv_bfloat16*>(p)[i] = __float2bfloat16_rn(v);
  else static_cast<float*>(p)[i] = v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Projections with a tiny side (action in: K = D; action out: N = D), fp32 out:
// out[m][n] = sum_k A[m][k] Wt[n][k] + bias[n] (+ add_rows[m % add_mod][n]). Long K: one CTA per token row,
// the row staged in shared memory, one warp per output.
template <int AD, int WD>
__global__ void __launch_bounds__(256) gemv_rows_kernel(GemmArgs p) {
  __shared__ float a_s[kGemvMaxK];
  pdl_trigger();
  pdl_wait();
  const int m = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int k = tid; k < p.K; k += 256) a_s[k] = ldf<AD>(p.A, (long long)m * p.lda + k);
  __syncthreads();
  float* out = static_cast<float*>(p.out) + (long long)m * p.ldo;
  const float* add = p.add_rows ? p.add_rows + (long long)(m % p.add_mod) * p.N : nullptr;
  for (int n = warp; n < p.N; n += 8) {
    float acc = 0.f;
#pragma unroll 8
    for (int k = lane; k < p.K; k += 32) acc = fmaf(a_s[k], ldf<WD>(p.W, (long long)n * p.K + k), acc);
    acc = warp_sum(acc);
    if (lane == 0) out[n] = acc + (p.bias ? p.bias[n] : 0.f) + (add ? add[n] : 0.f);
  }
}

// Short K (at most kShortK): a thread keeps the weights of one output in registers, read before the wait for
// the kernel that writes A, and a CTA of 256 outputs walks `rows` token rows staged in shared memory.
// Bound by the bytes out; one CTA a row re-read every weight for each row (3200 rows of 1024 outputs, K = 32, with
// the launch around it: 22 us as CUDA-core tiles of 64 x 64, 41 as their successor's, 19 here).
template <int AD, int WD>
__global__ void __launch_bounds__(256) short_k_kernel(GemmArgs p, int rows) {
  constexpr int KM = kShortK, RM = 16;
  __shared__ float a_s[RM * KM];
  const int n = blockIdx.x * 256 + threadIdx.x, m0 = blockIdx.y * rows, K = p.K;
  const int cnt = p.M - m0 < rows ? p.M - m0 : rows;
  float w[KM], b = 0.f;
#pragma unroll
  for (int k = 0; k < KM; ++k) w[k] = 0.f;
  if (n < p.N) {
    if (WD == BF16 && K % 8 == 0) {   // rows of W are 16-byte aligned then
#pragma unroll
      for (int k = 0; k < KM; k += 8) {
        if (k >= K) break;
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(p.W) + (long long)n * K + k));
        const __nv_bfloat162* v2 = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float2 f = __bfloat1622float2(v2[q]);
          w[k + 2 * q] = f.x;
          w[k + 2 * q + 1] = f.y;
        }
      }
    } else {
#pragma unroll
      for (int k = 0; k < KM; ++k) {
        if (k >= K) break;
        w[k] = ldf<WD>(p.W, (long long)n * K + k);
      }
    }
    if (p.bias) b = p.bias[n];
  }
  pdl_wait();
  // not before the wait: this is a step's first kernel, and the ones after it read what the step epilogue wrote
  // before their own waits
  pdl_trigger();
  for (int e = threadIdx.x; e < cnt * KM; e += 256) {
    const int r = e / KM, k = e % KM;
    a_s[e] = k < K ? ldf<AD>(p.A, (long long)(m0 + r) * p.lda + k) : 0.f;
  }
  __syncthreads();
  if (n >= p.N) return;
  float* out = static_cast<float*>(p.out) + n;
  const int k4 = (K + 3) / 4;
  for (int r = 0; r < cnt; ++r) {
    float acc = 0.f;
#pragma unroll
    for (int q = 0; q < KM / 4; ++q) {
      if (q >= k4) break;
      const float4 a = *reinterpret_cast<const float4*>(a_s + r * KM + 4 * q);
      acc = fmaf(a.w, w[4 * q + 3], fmaf(a.z, w[4 * q + 2], fmaf(a.y, w[4 * q + 1], fmaf(a.x, w[4 * q], acc))));
    }
    const int m = m0 + r;
    out[(long long)m * p.ldo] = acc + b + (p.add_rows ? p.add_rows[(long long)(m % p.add_mod) * p.N + n] : 0.f);
  }
}

bool gemv_rows_ok(const GemmArgs& a) {
  return a.epi == EPI_STORE && a.out_dtype == F32 && a.K <= kGemvMaxK && (a.N <= 64 || a.K <= kShortK);
}

template <int AD, int WD>
static void launch_gemv(const GemmArgs& a, cudaStream_t s) {
  if (a.K > kShortK) {
    launch_k(gemv_rows_kernel<AD, WD>, dim3(a.M), dim3(256), 0, s, a);
    return;
  }
  const int cols = (a.N + 255) / 256, rows = a.M * cols >= 16 * 304 ? 16 : a.M * cols >= 4 * 304 ? 4 : 1;   // two CTAs an SM
  launch_k(short_k_kernel<AD, WD>, dim3(cols, (a.M + rows - 1) / rows), dim3(256), 0, s, a, rows);
}

void launch_gemv_rows(const GemmArgs& a, cudaStream_t s) {
  if (a.a_dtype == F32 && a.w_dtype == F32) launch_gemv<F32, F32>(a, s);
  else if (a.a_dtype == F32 && a.w_dtype == BF16) launch_gemv<F32, BF16>(a, s);
  else if (a.a_dtype == BF16 && a.w_dtype == BF16) launch_gemv<BF16, BF16>(a, s);
  else launch_gemv<BF16, F32>(a, s);
}

// ------------------------------------------------------------------------------------------
// Adaptive norm: y = norm(h) * (1 + scale[tau]) + shift[tau]; one warp per token row.
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) norm_kernel(NormArgs p) {
  pdl_trigger();
  pdl_wait();
  const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (row >= p.M) return;
  const float* r = p.h + (long long)row * p.ldh;
  float mean = 0.f;
  if (p.layer_norm) {
    float s = 0.f;
    for (int c = lane; c < p.W; c += 32) s += r[c];
    mean = warp_sum(s) / p.W;
  }
  float ss = 0.f;
  for (int c = lane; c < p.W; c += 32) {
    const float d = r[c] - mean;
    ss = fmaf(d, d, ss);
  }
  const float rstd = 1.f / sqrtf(warp_sum(ss) / p.W + 1e-6f);
  const float* mod = p.tab ? p.tab + (long long)__ldcg(p.tau_row + row) * p.stride : nullptr;
  for (int c = lane; c < p.W; c += 32) {
    float y = (r[c] - mean) * rstd;
    if (mod) y = fmaf(y, 1.f + mod[p.scale_off + c], mod[p.shift_off + c]);
    stf(p.out, (long long)row * p.ldo + c, y, p.out_dtype);
  }
}

// Same computation with the whole row held in registers (W = 128 * NV): every load of the row
// and of its modulation vectors is issued before any arithmetic, so a row costs two memory
// round trips (modulation-row index, then data) instead of one per 32 elements.
template <int NV>
__global__ void __launch_bounds__(256) norm_reg_kernel(NormArgs p) {
  pdl_trigger();
  const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (row >= p.M) return;
  const float4* r4 = reinterpret_cast<const float4*>(p.h + (long long)row * p.ldh);
  const float* mod = p.tab ? p.tab + (long long)__ldcg(p.tau_row + row) * p.stride : nullptr;
  float4 x[NV], sc[NV], sh[NV];
  if (mod) {   // the time table, which no kernel of the step loop writes, before the wait

#pragma unroll
    for (int i = 0; i < NV; ++i) {
      sc[i] = __ldg(reinterpret_cast<const float4*>(mod + p.scale_off) + i * 32 + lane);
      sh[i] = __ldg(reinterpret_cast<const float4*>(mod + p.shift_off) + i * 32 + lane);
    }
  }
  pdl_wait();
#pragma unroll
  for (int i = 0; i < NV; ++i) x[i] = r4[i * 32 + lane];
  float mean = 0.f;
  if (p.layer_norm) {
    float t = 0.f;
#pragma unroll
    for (int i = 0; i < NV; ++i) t += (x[i].x + x[i].y) + (x[i].z + x[i].w);
    mean = warp_sum(t) / p.W;
  }
  float ss = 0.f;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const float a = x[i].x - mean, b = x[i].y - mean, c = x[i].z - mean, d = x[i].w - mean;
    ss = fmaf(a, a, fmaf(b, b, fmaf(c, c, fmaf(d, d, ss))));
  }
  const float rstd = 1.f / sqrtf(warp_sum(ss) / p.W + 1e-6f);
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    float4 y = make_float4((x[i].x - mean) * rstd, (x[i].y - mean) * rstd, (x[i].z - mean) * rstd,
                           (x[i].w - mean) * rstd);
    if (mod) {
      y.x = fmaf(y.x, 1.f + sc[i].x, sh[i].x);
      y.y = fmaf(y.y, 1.f + sc[i].y, sh[i].y);
      y.z = fmaf(y.z, 1.f + sc[i].z, sh[i].z);
      y.w = fmaf(y.w, 1.f + sc[i].w, sh[i].w);
    }
    const long long off = (long long)row * p.ldo + (i * 32 + lane) * 4;
    if (p.out_dtype == BF16) {
      __nv_bfloat162 lo = __floats2bfloat162_rn(y.x, y.y), hi = __floats2bfloat162_rn(y.z, y.w);
      uint2 pk;
      pk.x = *reinterpret_cast<uint32_t*>(&lo);
      pk.y = *reinterpret_cast<uint32_t*>(&hi);
      *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(p.out) + off) = pk;
    } else {
      *reinterpret_cast<float4*>(static_cast<float*>(p.out) + off) = y;
    }
  }
}

// Residual update + adaptive norm, one CTA per token row, 4 columns per thread:
//   h += gate(tau) * (sum_s part[s] + bias);  y = norm(h) * (1 + scale[tau]) + shift[tau].
// The K-split partial planes are summed in plane order (deterministic); all of a thread's
// loads are issued before the arithmetic that needs them.
__device__ __forceinline__ float block_sum(float v, float* red) {
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __syncthreads();                       // red[] may still be read by the previous call
  if ((threadIdx.x & 31) == 0) red[w] = v;
  __syncthreads();
  float t = 0.f;
  for (int i = 0; i < nw; ++i) t += red[i];
  return t;
}

__global__ void __launch_bounds__(1024) resid_norm_kernel(NormArgs p) {
  __shared__ float red[32];
  pdl_trigger();
  const int row = blockIdx.x, c4 = threadIdx.x;
  const bool on = c4 * 4 < p.W;
  const int tr = __ldcg(p.tau_row + row);
  float4 x = make_float4(0.f, 0.f, 0.f, 0.f), sc = x, sh = x, gt = make_float4(1.f, 1.f, 1.f, 1.f), bs = x;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  float4* h4 = reinterpret_cast<float4*>(p.h + (long long)row * p.ldh) + c4;
  if (on) {
    // the time table and the bias, which no kernel of the step loop writes, before the wait
    const float* mod = p.tab ? p.tab + (long long)tr * p.stride : nullptr;
    if (mod) {
      sc = __ldg(reinterpret_cast<const float4*>(mod + p.scale_off) + c4);
      sh = __ldg(reinterpret_cast<const float4*>(mod + p.shift_off) + c4);
    }
    if (p.rgate_tab) gt = __ldg(reinterpret_cast<const float4*>(p.rgate_tab + (long long)tr * p.stride + p.rgate_off) + c4);
    if (p.rbias) bs = __ldg(reinterpret_cast<const float4*>(p.rbias) + c4);
  }
  pdl_wait();
  if (on) {
    x = *h4;
    const long long plane4 = (long long)p.M * p.W / 4;
    const float4* pp = reinterpret_cast<const float4*>(p.part + (long long)row * p.W) + c4;
    int i = 0;
    for (; i + 8 <= p.n_part; i += 8) {
      float4 q[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) q[u] = __ldcg(pp + (i + u) * plane4);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        acc.x += q[u].x; acc.y += q[u].y; acc.z += q[u].z; acc.w += q[u].w;
      }
    }
    for (; i < p.n_part; ++i) {
      const float4 q = __ldcg(pp + i * plane4);
      acc.x += q.x; acc.y += q.y; acc.z += q.z; acc.w += q.w;
    }
    x.x = fmaf(gt.x, acc.x + bs.x, x.x);
    x.y = fmaf(gt.y, acc.y + bs.y, x.y);
    x.z = fmaf(gt.z, acc.z + bs.z, x.z);
    x.w = fmaf(gt.w, acc.w + bs.w, x.w);
    *h4 = x;
  }
  float mean = 0.f;
  if (p.layer_norm) mean = block_sum(on ? (x.x + x.y) + (x.z + x.w) : 0.f, red) / p.W;
  const float a = x.x - mean, b = x.y - mean, c = x.z - mean, d = x.w - mean;
  const float ss = block_sum(on ? fmaf(a, a, fmaf(b, b, fmaf(c, c, d * d))) : 0.f, red);
  const float rstd = 1.f / sqrtf(ss / p.W + 1e-6f);
  if (!on) return;
  float4 y = make_float4(a * rstd, b * rstd, c * rstd, d * rstd);
  if (p.tab) {
    y.x = fmaf(y.x, 1.f + sc.x, sh.x);
    y.y = fmaf(y.y, 1.f + sc.y, sh.y);
    y.z = fmaf(y.z, 1.f + sc.z, sh.z);
    y.w = fmaf(y.w, 1.f + sc.w, sh.w);
  }
  const long long off = (long long)row * p.ldo + c4 * 4;
  if (p.out_dtype == BF16) {
    __nv_bfloat162 lo = __floats2bfloat162_rn(y.x, y.y), hi = __floats2bfloat162_rn(y.z, y.w);
    uint2 pk;
    pk.x = *reinterpret_cast<uint32_t*>(&lo);
    pk.y = *reinterpret_cast<uint32_t*>(&hi);
    *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(p.out) + off) = pk;
  } else {
    *reinterpret_cast<float4*>(static_cast<float*>(p.out) + off) = y;
  }
}

// The same with one warp per token row and the whole row in registers (W = 128 * NV): the row's
// h, planes and gate are loaded before the arithmetic that needs them, and its sums are warp
// reductions (no CTA barrier); the scale and shift vectors are loaded after the reduction, so
// that a thread holds three row-sized arrays at most and four-warp CTAs fit three or four to an
// SM (more rows in flight). The planes are summed in plane order as above.
template <int NV>
__global__ void __launch_bounds__(128) resid_norm_reg_kernel(NormArgs p) {
  pdl_trigger();
  const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (row >= p.M) return;
  const int tr = __ldcg(p.tau_row + row);
  float4* h4 = reinterpret_cast<float4*>(p.h + (long long)row * p.ldh);
  const float4* pp = reinterpret_cast<const float4*>(p.part + (long long)row * p.W);
  const long long plane4 = (long long)p.M * p.W / 4;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f), one = make_float4(1.f, 1.f, 1.f, 1.f);
  float4 x[NV], acc[NV], gt[NV];
  const float* mod = p.tab ? p.tab + (long long)tr * p.stride : nullptr;
  const float4* g4 = p.rgate_tab ? reinterpret_cast<const float4*>(p.rgate_tab + (long long)tr * p.stride + p.rgate_off) : nullptr;
#pragma unroll
  for (int i = 0; i < NV; ++i) gt[i] = g4 ? __ldg(g4 + i * 32 + lane) : one;
  pdl_wait();
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    x[i] = h4[i * 32 + lane];
    acc[i] = p.n_part > 0 ? __ldcg(pp + i * 32 + lane) : zero;
  }
  for (int sp = 1; sp < p.n_part; ++sp) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const float4 q = __ldcg(pp + sp * plane4 + i * 32 + lane);
      acc[i].x += q.x;
      acc[i].y += q.y;
      acc[i].z += q.z;
      acc[i].w += q.w;
    }
  }
  float t = 0.f;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const float4 bs = p.rbias ? __ldg(reinterpret_cast<const float4*>(p.rbias) + i * 32 + lane) : zero;
    x[i].x = fmaf(gt[i].x, acc[i].x + bs.x, x[i].x);
    x[i].y = fmaf(gt[i].y, acc[i].y + bs.y, x[i].y);
    x[i].z = fmaf(gt[i].z, acc[i].z + bs.z, x[i].z);
    x[i].w = fmaf(gt[i].w, acc[i].w + bs.w, x[i].w);
    h4[i * 32 + lane] = x[i];
    t += (x[i].x + x[i].y) + (x[i].z + x[i].w);
  }
  const float mean = p.layer_norm ? warp_sum(t) / p.W : 0.f;
  float ss = 0.f;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const float a = x[i].x - mean, b = x[i].y - mean, c = x[i].z - mean, d = x[i].w - mean;
    ss = fmaf(a, a, fmaf(b, b, fmaf(c, c, fmaf(d, d, ss))));
  }
  const float rstd = 1.f / sqrtf(warp_sum(ss) / p.W + 1e-6f);
  float4 sc[NV], sh[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    sc[i] = mod ? __ldg(reinterpret_cast<const float4*>(mod + p.scale_off) + i * 32 + lane) : zero;
    sh[i] = mod ? __ldg(reinterpret_cast<const float4*>(mod + p.shift_off) + i * 32 + lane) : zero;
  }
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    float4 y = make_float4((x[i].x - mean) * rstd, (x[i].y - mean) * rstd, (x[i].z - mean) * rstd,
                           (x[i].w - mean) * rstd);
    if (mod) {
      y.x = fmaf(y.x, 1.f + sc[i].x, sh[i].x);
      y.y = fmaf(y.y, 1.f + sc[i].y, sh[i].y);
      y.z = fmaf(y.z, 1.f + sc[i].z, sh[i].z);
      y.w = fmaf(y.w, 1.f + sc[i].w, sh[i].w);
    }
    const long long off = (long long)row * p.ldo + (i * 32 + lane) * 4;
    if (p.out_dtype == BF16) {
      __nv_bfloat162 lo = __floats2bfloat162_rn(y.x, y.y), hi = __floats2bfloat162_rn(y.z, y.w);
      uint2 pk;
      pk.x = *reinterpret_cast<uint32_t*>(&lo);
      pk.y = *reinterpret_cast<uint32_t*>(&hi);
      *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(p.out) + off) = pk;
    } else {
      *reinterpret_cast<float4*>(static_cast<float*>(p.out) + off) = y;
    }
  }
}

void launch_norm(const NormArgs& a, cudaStream_t s) {
  if (a.part) {
    const bool aligned = a.ldh % 4 == 0 && a.ldo % 4 == 0 && a.scale_off % 4 == 0 && a.shift_off % 4 == 0 &&
                         a.rgate_off % 4 == 0 && a.stride % 4 == 0 && a.W % 128 == 0;
    const int blocks = (a.M + 3) / 4;
    // a warp per row pays with enough rows to fill the SMs; with fewer, one CTA per row
    switch (aligned && a.M >= 512 ? a.W / 128 : 0) {
      case 2: launch_k(resid_norm_reg_kernel<2>, dim3(blocks), dim3(128), 0, s, a); return;
      case 4: launch_k(resid_norm_reg_kernel<4>, dim3(blocks), dim3(128), 0, s, a); return;
      case 8: launch_k(resid_norm_reg_kernel<8>, dim3(blocks), dim3(128), 0, s, a); return;
      default: break;
    }
    // the caller guarantees 16-byte rows: W, ldh, ldo, stride and the offsets multiples of 4
    const int threads = ((a.W / 4 + 31) / 32) * 32;
    launch_k(resid_norm_kernel, dim3(a.M), dim3(threads), 0, s, a);
    return;
  }
  // A warp a row; four rows a CTA for the few tokens of a bf16 expert, eight otherwise. Per evaluation, eight / four:
  // 16 layers of width 1536, 16 tokens 762 / 755 us, 32 tokens 866 / 862, 64 tokens 1070 / 1074, 96 tokens 1314 /
  // 1341; 18 of width 1024, 50 tokens 668 / 666; fp32, two layers of width 256, 16 tokens 48.5 / 50.4.
  const int rows = a.out_dtype == BF16 && a.M < 64 ? 4 : 8, blocks = (a.M + rows - 1) / rows;
  const bool aligned = a.ldh % 4 == 0 && a.ldo % 4 == 0 && a.scale_off % 4 == 0 && a.shift_off % 4 == 0 &&
                       a.stride % 4 == 0 && a.W % 128 == 0;
  switch (aligned ? a.W / 128 : 0) {
    case 2: launch_k(norm_reg_kernel<2>, dim3(blocks), dim3(32 * rows), 0, s, a); break;
    case 3: launch_k(norm_reg_kernel<3>, dim3(blocks), dim3(32 * rows), 0, s, a); break;
    case 4: launch_k(norm_reg_kernel<4>, dim3(blocks), dim3(32 * rows), 0, s, a); break;
    case 8: launch_k(norm_reg_kernel<8>, dim3(blocks), dim3(32 * rows), 0, s, a); break;
    case 12: launch_k(norm_reg_kernel<12>, dim3(blocks), dim3(32 * rows), 0, s, a); break;
    default: launch_k(norm_kernel, dim3(blocks), dim3(32 * rows), 0, s, a); break;
  }
}

// ------------------------------------------------------------------------------------------
// Attention for few queries (bf16 operands, head dim 64): the DiT head's self-attention over the chunk
// and cross-attention over the projected prefix. CTA = 16 queries of one head and robot and a share of
// the 64-key tiles; the CTAs that share a query block form a cluster and its first CTA merges their
// partial rows by log-sum-exp, received through distributed shared memory. Per tile: Q K^T on the tensor
// cores (m16n8k16: the products of bf16 operands are exact, sums in fp32), warp = 8 keys, operands
// straight from global memory; softmax in fp32; P V on the tensor cores with every fp32 probability
// as the sum of three bf16 terms (24 bits: nothing is rounded away), warp = 8 head dims. The tensor cores'
// accumulation truncates, so none runs long: a score is two sums of 32 products, a tile's P V one of the leading
// terms and one of the others, added to O in fp32 (error against 64 bits, 320 keys: 8.4e-8, scores 4.7e-8; fp32
// FMA chains 3.2e-7 and 5.1e-8; one accumulator over all tiles 1.1e-6, one a score 6.5e-8).
// What bounds it is latency, half of it instruction fetch: a kernel whose code is not in the SM's
// instruction cache runs at a dozen cycles an instruction. The prefix keys and values, which no
// kernel of the loop writes, are loaded before the wait for the previous kernel, and a rehearsal pass
// over them (its results dropped) brings the code in while the CTA would idle. A CTA with several tiles
// loads the next one's keys and values into registers while it works on the current one (16-layer DiT expert,
// one robot: 816 -> 795 us per evaluation; with this kernel and the cluster GEMM for the CUDA-core ones 1090 -> 890).
constexpr int kFewDh = 64, kFewQ = 16, kFewKT = 64, kFewCluster = 8;
constexpr int kFewPitch = kFewDh + 8;     // bf16 rows of V and P: ldmatrix without bank conflicts
constexpr int kFewSPitch = kFewKT + 4;    // fp32 rows of scores and partial outputs

struct FewSmem {
  __nv_bfloat16 v[kFewKT * kFewPitch];
  __nv_bfloat16 p[3][kFewQ * kFewPitch];
  float s[kFewQ * kFewSPitch];
  float m[kFewQ], l[kFewQ], alpha[kFewQ];
  float part[1];                          // [CTAs of the cluster][16][kFewSPitch]: O, then max and sum
};
static size_t few_smem_bytes(int c) { return sizeof(FewSmem) + (c > 1 ? (size_t)c * kFewQ * kFewSPitch * 4 : 0); }
// CTAs that share a query block: one a key tile while the whole grid is one CTA an SM. Past that a cluster
// costs more than it gives (its CTAs start together, beside the previous kernel's, and meet twice), and the
// CTAs walk their tiles alone. 24 heads, 16 queries, 300 keys, us per evaluation of the 16-layer expert:
// 1 robot 795 with 5 CTAs a block (810 with 4); 4 robots 1200 with 5 or 3, 1163 with 2, 1112 with 1.
static int few_cluster(int n_keys, long long blocks) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int c = (n_keys + kFewKT - 1) / kFewKT;
  if (c > kFewCluster) c = kFewCluster;
  while (c > 1 && c * blocks > sms) --c;
  return c;
}

__device__ __forceinline__ void ldsm4(uint32_t* r, const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
}
__device__ __forceinline__ void ldsm4_t(uint32_t* r, const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
}
__device__ __forceinline__ void mma16816(float* c, const uint32_t* a, const uint32_t* b) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
__device__ __forceinline__ void st_dsm2(uint32_t addr, float a, float b) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(a), "f"(b) : "memory");
}

__global__ void __launch_bounds__(256) attn_few_kernel(AttnArgs p, int C) {
  extern __shared__ __align__(16) unsigned char few_raw[];
  FewSmem& sm = *reinterpret_cast<FewSmem*>(few_raw);
  pdl_trigger();
  const int rank = blockIdx.x % C, i0 = blockIdx.x / C * kFewQ, hq = blockIdx.y, b = blockIdx.z;
  const int g = hq / (p.n_heads / p.n_kv_heads);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, gr = lane >> 2, tc = 2 * (lane & 3);
  const int n_keys = p.P + (p.kc ? p.H : 0), nt = (n_keys + kFewKT - 1) / kFewKT;
  if (C > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  const __nv_bfloat16* qrow = static_cast<const __nv_bfloat16*>(p.q) + (long long)(b * p.H + i0 + gr) * p.q_ld + hq * kFewDh + tc;
  const bool q0 = i0 + gr < p.H, q1 = i0 + gr + 8 < p.H;
  // key j's row of keys (or values) of this head; null past the end
  const auto row_of = [&](const void* pre, const void* chunk, int j) -> const __nv_bfloat16* {
    if (j < p.P) return static_cast<const __nv_bfloat16*>(pre) + b * p.kp_bstride + (long long)j * p.kp_ld + g * kFewDh;
    if (j < n_keys) return static_cast<const __nv_bfloat16*>(chunk) + (long long)(b * p.H + j - p.P) * p.kc_ld + g * kFewDh;
    return nullptr;
  };
  // a tile's keys and values wait in registers while the tile before it is worked on
  uint32_t kn[8];
  uint4 vn[2];
  const int vj = tid >> 2, vcol = 16 * (tid & 3);   // a quarter of a value row each
  const auto fetch = [&](int t) {
    const __nv_bfloat16* kr = row_of(p.kp, p.kc, t * kFewKT + 8 * warp + gr);
#pragma unroll
    for (int u = 0; u < 8; ++u) kn[u] = kr ? __ldcg(reinterpret_cast<const unsigned*>(kr + 8 * u + tc)) : 0u;
    const __nv_bfloat16* vr = row_of(p.vp, p.vc, t * kFewKT + vj);
    const uint4 zero = make_uint4(0, 0, 0, 0);
    vn[0] = vr ? __ldcg(reinterpret_cast<const uint4*>(vr + vcol)) : zero;
    vn[1] = vr ? __ldcg(reinterpret_cast<const uint4*>(vr + vcol + 8)) : zero;
  };
  const bool early = (rank + 1) * kFewKT <= p.P;   // this CTA's first tile is prefix keys alone
  if (early) fetch(rank);

  float o[4];
  const int q = tid >> 4, kg = tid & 15;           // softmax: query q, keys 4 kg .. 4 kg + 3
#pragma unroll 1
  for (int pass = early ? 0 : 1; pass < 2; ++pass) {
    if (pass) {
      pdl_wait();
      if (!early) fetch(rank);
    }
    if (tid < kFewQ) {
      sm.m[tid] = -INFINITY;
      sm.l[tid] = 0.f;
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) o[e] = 0.f;
    uint32_t qf[4][4];
#pragma unroll
    for (int ks = 0; ks < 4; ++ks)
#pragma unroll
      for (int e = 0; e < 4; ++e)
        qf[ks][e] = (e & 1 ? q1 : q0) ? __ldcg(reinterpret_cast<const unsigned*>(qrow + (e & 1) * 8ll * p.q_ld + 16 * ks + 8 * (e >> 1))) : 0u;
#pragma unroll 1
    for (int t = rank; t < nt; t += C) {
      uint32_t kf[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) kf[u] = kn[u];
      *reinterpret_cast<uint4*>(sm.v + vj * kFewPitch + vcol) = vn[0];
      *reinterpret_cast<uint4*>(sm.v + vj * kFewPitch + vcol + 8) = vn[1];
      if (pass && t + C < nt) fetch(t + C);
      float c[4] = {0.f, 0.f, 0.f, 0.f}, d[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) mma16816(ks & 1 ? d : c, qf[ks], kf + 2 * ks);
#pragma unroll
      for (int e = 0; e < 4; ++e) c[e] += d[e];
      float* sr = sm.s + gr * kFewSPitch + 8 * warp + tc;
      *reinterpret_cast<float2*>(sr) = make_float2(c[0] * p.scale, c[1] * p.scale);
      *reinterpret_cast<float2*>(sr + 8 * kFewSPitch) = make_float2(c[2] * p.scale, c[3] * p.scale);
      __syncthreads();
      const float4 s4 = *reinterpret_cast<const float4*>(sm.s + q * kFewSPitch + 4 * kg);
      float sc[4] = {s4.x, s4.y, s4.z, s4.w};
      const float m_old = sm.m[q];
      float mx = m_old, sum = 0.f;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (t * kFewKT + 4 * kg + e >= n_keys) sc[e] = -INFINITY;   // keys past the end
        mx = fmaxf(mx, sc[e]);
      }
#pragma unroll
      for (int w = 8; w > 0; w >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, w));
      float rest[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        rest[e] = t * kFewKT + 4 * kg + e < n_keys ? expf(sc[e] - mx) : 0.f;
        sum += rest[e];
      }
#pragma unroll
      for (int w = 8; w > 0; w >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, w);
#pragma unroll
      for (int k = 0; k < 3; ++k) {   // the probabilities' leading, middle and last 8 bits
        const __nv_bfloat162 lo = __floats2bfloat162_rn(rest[0], rest[1]), hi = __floats2bfloat162_rn(rest[2], rest[3]);
        uint2 w;
        w.x = *reinterpret_cast<const uint32_t*>(&lo);
        w.y = *reinterpret_cast<const uint32_t*>(&hi);
        *reinterpret_cast<uint2*>(sm.p[k] + q * kFewPitch + 4 * kg) = w;
        rest[0] -= __low2float(lo);
        rest[1] -= __high2float(lo);
        rest[2] -= __low2float(hi);
        rest[3] -= __high2float(hi);
      }
      if (kg == 0) {
        const float a = m_old == -INFINITY ? 0.f : expf(m_old - mx);
        sm.alpha[q] = a;
        sm.m[q] = mx;
        sm.l[q] = sm.l[q] * a + sum;
      }
      __syncthreads();
      const float a0 = sm.alpha[gr], a1 = sm.alpha[gr + 8];
      float hi[4] = {0.f, 0.f, 0.f, 0.f}, lo[4] = {0.f, 0.f, 0.f, 0.f};   // of the leading terms, of the others
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        uint32_t vf[4];
        ldsm4_t(vf, sm.v + (32 * half + lane) * kFewPitch + 8 * warp);
#pragma unroll
        for (int k2 = 0; k2 < 2; ++k2)
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            uint32_t pf[4];
            ldsm4(pf, sm.p[k] + (lane & 15) * kFewPitch + 32 * half + 16 * k2 + 8 * (lane >> 4));
            mma16816(k ? lo : hi, pf, vf + 2 * k2);
          }
      }
      o[0] = fmaf(o[0], a0, hi[0] + lo[0]);
      o[1] = fmaf(o[1], a0, hi[1] + lo[1]);
      o[2] = fmaf(o[2], a1, hi[2] + lo[2]);
      o[3] = fmaf(o[3], a1, hi[3] + lo[3]);
      if (!pass) break;
      __syncthreads();   // the next tile's values, scores and probabilities overwrite this one's
    }
  }

  __nv_bfloat16* dst = static_cast<__nv_bfloat16*>(p.out) + (long long)(b * p.H + i0) * p.out_ld + hq * kFewDh;
  if (C == 1) {
    const float l0 = 1.f / sm.l[gr], l1 = 1.f / sm.l[gr + 8];
    if (q0) *reinterpret_cast<__nv_bfloat162*>(dst + (long long)gr * p.out_ld + 8 * warp + tc) = __floats2bfloat162_rn(o[0] * l0, o[1] * l0);
    if (q1) *reinterpret_cast<__nv_bfloat162*>(dst + (long long)(gr + 8) * p.out_ld + 8 * warp + tc) = __floats2bfloat162_rn(o[2] * l1, o[3] * l1);
    return;
  }
  // partial rows to the cluster's first CTA, once it runs
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  uint32_t to;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(to) : "r"((uint32_t)__cvta_generic_to_shared(sm.part + rank * kFewQ * kFewSPitch)));
  st_dsm2(to + (gr * kFewSPitch + 8 * warp + tc) * 4, o[0], o[1]);
  st_dsm2(to + ((gr + 8) * kFewSPitch + 8 * warp + tc) * 4, o[2], o[3]);
  if (tid < kFewQ) st_dsm2(to + (tid * kFewSPitch + kFewDh) * 4, sm.m[tid], sm.l[tid]);
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (rank != 0) return;
  const float* base = sm.part + q * kFewSPitch;
  float M = -INFINITY;
  for (int k = 0; k < C; ++k) M = fmaxf(M, base[k * kFewQ * kFewSPitch + kFewDh]);
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  float L = 0.f;
  for (int k = 0; k < C; ++k) {
    const float* r = base + k * kFewQ * kFewSPitch;
    const float w = expf(r[kFewDh] - M);
    L = fmaf(w, r[kFewDh + 1], L);
    const float4 v = *reinterpret_cast<const float4*>(r + 4 * kg);
    acc.x = fmaf(w, v.x, acc.x);
    acc.y = fmaf(w, v.y, acc.y);
    acc.z = fmaf(w, v.z, acc.z);
    acc.w = fmaf(w, v.w, acc.w);
  }
  if (i0 + q < p.H) {
    const float inv = 1.f / L;
    const __nv_bfloat162 lo = __floats2bfloat162_rn(acc.x * inv, acc.y * inv), hi = __floats2bfloat162_rn(acc.z * inv, acc.w * inv);
    uint2 pk;
    pk.x = *reinterpret_cast<const uint32_t*>(&lo);
    pk.y = *reinterpret_cast<const uint32_t*>(&hi);
    *reinterpret_cast<uint2*>(dst + (long long)q * p.out_ld + 4 * kg) = pk;
  }
}

// bf16, head dim 64, no rotation (rotated queries are fp32), 16-byte rows of keys and values.
static bool attn_few_ok(const AttnArgs& a) {
  const int n_keys = a.P + (a.kc ? a.H : 0);
  return a.dtype == BF16 && a.head_dim == kFewDh && !a.rope_cs && n_keys >= 1 && a.kp_ld % 8 == 0 && a.kc_ld % 8 == 0 &&
         a.q_ld % 8 == 0 && a.out_ld % 4 == 0 && a.kp_bstride % 8 == 0;
}

__global__ void add_tau_silu_kernel(const float* __restrict__ x, const float* __restrict__ tab, int stride, int off,
                                    const int* __restrict__ tau_row, int M, int N, void* y, int dt) {
  pdl_trigger();
  pdl_wait();
  const long long total = (long long)M * N;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
    const int m = (int)(e / N), n = (int)(e % N);
    const float v = x[e] + tab[(size_t)__ldcg(tau_row + m) * stride + off + n];
    stf(y, e, v / (1.f + expf(-v)), dt);
  }
}

void launch_add_tau_silu(const float* x, const float* tab, int stride, int off, const int* tau_row, int M, int N,
                         void* y, int dt, cudaStream_t s) {
  const long long total = (long long)M * N;
  int blocks = (int)((total + 255) / 256);
  if (blocks > 1024) blocks = 1024;
  launch_k(add_tau_silu_kernel, dim3(blocks), dim3(256), 0, s, x, tab, stride, off, tau_row, M, N, y, dt);
}

void launch_attention_prepare() {
  cudaFuncSetAttribute(attn_few_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)few_smem_bytes(kFewCluster));
}

void launch_attention(const AttnArgs& a, cudaStream_t s) {
  if (attn_few_ok(a)) {
    const int C = few_cluster(a.P + (a.kc ? a.H : 0), (long long)((a.H + kFewQ - 1) / kFewQ) * a.n_heads * a.B);
    launch_cluster(attn_few_kernel, dim3((a.H + kFewQ - 1) / kFewQ * C, a.n_heads, a.B), dim3(256), few_smem_bytes(C), C, s, a, C);
    return;
  }
  launch_attn_rows(a, s);
}

// ------------------------------------------------------------------------------------------
// Step epilogue, one CTA per robot (the work itself is euler_robot, euler.cuh).
// ------------------------------------------------------------------------------------------
struct CtaSync {
  __device__ void operator()() const { __syncthreads(); }
};
__global__ void __launch_bounds__(256) euler_kernel(EulerArgs p) {
  pdl_trigger();
  pdl_wait();
  __shared__ int s_rel;
  __shared__ float E_s[64];
  __shared__ float Cr[9];   // SO(3) correction of the tail (rotation dimensions)
  extern __shared__ float ediff[];   // [H][D]
  const EulerSmem sm{ediff, E_s, Cr, &s_rel};
  const int b = blockIdx.x, k = p.cur_k[b];
  EulerArgs q = p;
  q.k = k;
  q.plan = p.plan + (size_t)(k - 1) * p.B * p.H;
  euler_robot(q, b, threadIdx.x, blockDim.x, sm, CtaSync());
  // the next step's number and modulation rows. The action-in projection, which follows, lets the kernels after
  // it start only once it has waited for this one, so they may read the rows before their own waits
  if (threadIdx.x == 0) p.cur_k[b] = k + 1;
  if (k < p.n_steps)
    for (int i = threadIdx.x; i < p.H; i += blockDim.x) p.cur_tau[b * p.H + i] = p.tau[((size_t)k * p.B + b) * p.H + i];
}

void launch_euler_prepare() {
  cudaFuncSetAttribute(euler_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 256 * 64 * (int)sizeof(float));
}

void launch_euler(const EulerArgs& a, cudaStream_t s) {
  launch_k(euler_kernel, dim3(a.B), dim3(256), (size_t)a.H * a.D * sizeof(float), s, a);
}

__global__ void begin_kernel(const float* noise, float* x, float* g, float* u, int n, int* nonfinite,
                             int* evals, unsigned long long* stamps, int* cur_k, int B, int* cur_tau, const int* tau, int M) {
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) {
    *nonfinite = 0;
    *evals = 0;
    stamps[0] = global_ns();
  }
  if (i < B) cur_k[i] = 1;
  if (i < M) cur_tau[i] = tau[i];
  if (i < n) {
    const float v = noise[i];
    x[i] = v;
    g[i] = v;
    u[i] = v;
  }
}

void launch_begin(const float* noise, float* x, float* g, float* u, int n, int* nonfinite, int* evals,
                  unsigned long long* stamps, int* cur_k, int B, int* cur_tau, const int* tau, int M, cudaStream_t s) {
  launch_k(begin_kernel, dim3((n + 255) / 256), dim3(256), 0, s, noise, x, g, u, n, nonfinite, evals, stamps, cur_k, B, cur_tau,
           tau, M);
}

// ------------------------------------------------------------------------------------------
// Weight re-layout: dst[(n * mult + off) * K + k] = src[k * N + n] (transpose + convert).
// ------------------------------------------------------------------------------------------
__global__ void relayout_kernel(const float* src, int K, int N, void* dst, int dt, int mult, long long off) {
  __shared__ float t[32][33];
  const int k0 = blockIdx.y * 32, n0 = blockIdx.x * 32;
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int k = k0 + r, n = n0 + threadIdx.x;
    t[r][threadIdx.x] = (k < K && n < N) ? src[(long long)k * N + n] : 0.f;
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int n = n0 + r, k = k0 + threadIdx.x;
    if (n < N && k < K) stf(dst, ((long long)n * mult + off) * K + k, t[threadIdx.x][r], dt);
  }
}

void launch_relayout(const float* src, int K, int N, void* dst, int dtype, int mult, long long off,
                     cudaStream_t s) {
  dim3 grid((N + 31) / 32, (K + 31) / 32);
  relayout_kernel<<<grid, dim3(32, 8), 0, s>>>(src, K, N, dst, dtype, mult, off);
}

__global__ void convert_kernel(const void* src, int sdt, void* dst, int ddt, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    stf(dst, i, ldf_rt(src, i, sdt), ddt);
}

// The rotations of Ghost Action Correction on SO(3) on given rotation vectors (testing aid):
// log_exp[i] = log(exp(w_i)), log_comp[i] = log(exp(w_i) exp(w_{i+1 mod n})^T).
__global__ void so3_check_kernel(const float* w, int n, float* log_exp, float* log_comp) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float A[9], B[9], Bt[9], C[9];
  so3_exp(w + 3 * i, A);
  so3_log(A, log_exp + 3 * i);
  so3_exp(w + 3 * ((i + 1) % n), B);
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c = 0; c < 3; ++c) Bt[r * 3 + c] = B[c * 3 + r];
  mat3_mul(A, Bt, C);
  so3_log(C, log_comp + 3 * i);
}

void launch_so3_check(const float* w, int n, float* log_exp, float* log_comp, cudaStream_t s) {
  so3_check_kernel<<<(n + 127) / 128, 128, 0, s>>>(w, n, log_exp, log_comp);
}

void launch_convert(const void* src, int src_dtype, void* dst, int dst_dtype, long long n, cudaStream_t s) {
  const int blocks = (int)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096);
  convert_kernel<<<blocks > 0 ? blocks : 1, 256, 0, s>>>(src, src_dtype, dst, dst_dtype, n);
}

}  // namespace uad
