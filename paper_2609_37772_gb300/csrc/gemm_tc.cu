// Tensor-core projection GEMM for sm_103a: out[m][n] = epi(sum_k X[m][k] * Wt[n][k]).
//
// Swap-AB tiling for few tokens: 128 weight rows form the MMA's M side, 64 tokens its N
// side, so one CTA computes a 128 x 64 fp32 tile in tensor memory (TMEM). Weights are
// pre-tiled at init into 128 x 64 bf16 blocks already in the 128-byte-swizzled K-major
// shared-memory layout, so each block arrives with one 16 KB bulk copy (cp.async.bulk);
// activation tiles come through a 2-D TMA tensor map (cp.async.bulk.tensor) with the same
// swizzle and zero fill past the last row. One thread issues tcgen05.mma, one thread feeds
// the TMA ring, four warps drain TMEM with tcgen05.ld.
//
// Projections with so few tiles that the SMs need K splits take the cluster form (gemm_cl.cu).
// Many tokens (a batch of robots) take the persistent wide form instead: one CTA per SM walks
// units of up to 256 tokens x 128 weight rows with two tensor-memory accumulators, so that the
// epilogue of one unit overlaps the main loop of the next.
// Every wait is bounded: on timeout the kernel records an error code and winds down.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <array>
#include <cstdlib>
#include <map>

#include "uad_internal.cuh"
#include "ptx.cuh"
#include "once_per_device.h"

namespace uad {

using namespace ptx;

namespace {

constexpr int kBM = 128, kBN = 64, kBK = 64;
constexpr int kStageA = kBM * kBK * 2;  // 16 KB
constexpr int kStageB = kBN * kBK * 2;  // 8 KB
constexpr unsigned long long kWaitNs = 2000000000ull;  // 2 s bound on any wait
// persistent form: tokens per epilogue slice, epilogue groups (four warps each), staging pitch
// in floats (132: a float4 column read across 8 tokens touches all 32 banks once), threads
constexpr int kPersSlice = 16, kPersGroups = 4, kPersPitch = kBM + 4;
constexpr int kPersThreads = 64 + kPersGroups * 128;

__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, int* err, int code) {
  return ptx::mbar_wait(b, parity, err, code, kWaitNs);
}

__device__ __forceinline__ float gelu_tanh_f(float x) {
  const float k0 = 0.7978845608028654f;
  return 0.5f * x * (1.f + tanhf(k0 * (x + 0.044715f * x * x * x)));
}
// The same with the hardware tanh (MUFU), for outputs rounded to bf16 next: its error is far
// below bf16's.
__device__ __forceinline__ float gelu_tanh_fast(float x) {
  const float k0 = 0.7978845608028654f;
  float t;
  asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(k0 * (x + 0.044715f * x * x * x)));
  return 0.5f * x * (1.f + t);
}

__device__ __forceinline__ void store_out(void* out, long long i, float v, int dt) {
  if (dt == BF16) static_cast<__nv_bfloat16*>(out)[i] = __float2bfloat16_rn(v);
  else static_cast<float*>(out)[i] = v;
}


// Shared-memory plan of the narrow form: [pipeline stages, at least 32 KB (reused as the staged tile)]
// [mbarriers, TMEM slot].
__host__ __device__ __forceinline__ int tc_stages(int nch) {
  return nch < kTcMaxStages ? nch : kTcMaxStages;
}
__host__ __device__ __forceinline__ size_t tc_pipe_bytes(int stages) {
  const size_t b = (size_t)stages * (kStageA + kStageB);
  return b < 32768 ? 32768 : b;
}


// Epilogue of one tile slice: T[j * pitch + row] holds the fp32 accumulator of token m0 + j
// (j < mcount) for output row n = this thread's row (row = 32 w + lane over the four warps w of
// the slice's group). Partial-plane epilogues (EPI_PARTIAL) are written by the kernels themselves
// as whole-row 16-byte stores. Small rolled loops keep the code compact.
__device__ __forceinline__ void tile_epilogue(const TcGemmArgs& p, const float* T, int pitch, int m0,
                                              int mcount, int n, int row, int lane) {
  const float b = p.bias && (p.n_store <= 0 || n < p.n_store) ? p.bias[n] : 0.f;
  const float* Tr = T + row;
  switch (p.epi) {
    case EPI_GEGLU: {
      // rows 2i (gate) and 2i + 1 (up) give output i: tokens over the warps, lane owns rows
      // 4 lane .. 4 lane + 3 (outputs 2 lane, 2 lane + 1 of the tile), so that a warp writes one
      // token's 64 outputs as one contiguous run
      const int o0 = (n - row) / 2 + 2 * lane;
      const bool fast = p.out_dtype == BF16;
      for (int j = row >> 5; j < mcount; j += kBM / 32) {
        const float4 v = *reinterpret_cast<const float4*>(T + j * pitch + 4 * lane);
        const size_t off = (size_t)(m0 + j) * p.ldo + o0;
        if (fast) {
          *reinterpret_cast<__nv_bfloat162*>(static_cast<__nv_bfloat16*>(p.out) + off) =
              __floats2bfloat162_rn(gelu_tanh_fast(v.x) * v.y, gelu_tanh_fast(v.z) * v.w);
        } else {
          store_out(p.out, off, gelu_tanh_f(v.x) * v.y, p.out_dtype);
          store_out(p.out, off + 1, gelu_tanh_f(v.z) * v.w, p.out_dtype);
        }
      }
      break;
    }
    case EPI_BIAS_GELU:
#pragma unroll 4
      for (int j = 0; j < mcount; ++j)
        store_out(p.out, (size_t)(m0 + j) * p.ldo + n, gelu_tanh_f(Tr[j * pitch] + b), p.out_dtype);
      break;
    case EPI_QKV_TC: {
      const QkvTcOut& o = p.qkv;
      const int n0 = n - row;   // the tile's first output row; q, k and v each span whole tiles
      if (n0 < o.qd + o.kvd) {
        // q or k rows: tokens over the warps, lane owns 4 consecutive rows (two RoPE pairs, with
        // rows 2j, 2j + 1 of a head holding dims j and j + dh/2), so that each token's features
        // go out as contiguous runs; (cos, sin) of the token's position from the table
        const bool isq = n0 < o.qd;
        const int sn = (isq ? n0 : n0 - o.qd) + 4 * lane;
        const int h = sn / o.dh, r = sn % o.dh, half = o.dh / 2;
        __nv_bfloat16* base = isq ? o.q + ((size_t)(h / o.G) * o.G + (h % o.G)) * o.H * o.dh
                                  : o.kcache + (((size_t)o.layer * o.Hkv + h) * o.NK + o.P) * o.dh;
        const size_t sb = isq ? (size_t)o.Hkv * o.G * o.H * o.dh : (size_t)o.L * o.Hkv * o.NK * o.dh;
        // four tokens at a time (a warp's tokens j, j + 4, ...): every (cos, sin) load of the four
        // is issued before the first use, so that the table's L2 round trips overlap
        constexpr int kStep = kBM / 32, kU = 4;
        for (int j0 = row >> 5; j0 < mcount; j0 += kStep * kU) {
          float4 v[kU], cs[kU];
          int ii[kU];
          __nv_bfloat16* dst[kU];
#pragma unroll
          for (int u = 0; u < kU; ++u) {
            const int j = j0 + kStep * u;
            if (j >= mcount) continue;
            const int m = m0 + j, bi = m / o.H;
            ii[u] = m - bi * o.H;
            dst[u] = base + bi * sb + (size_t)ii[u] * o.dh;
            v[u] = *reinterpret_cast<const float4*>(T + j * pitch + 4 * lane);
            if (o.rope) cs[u] = __ldg(reinterpret_cast<const float4*>(o.rope + (size_t)ii[u] * o.dh + r));
          }
#pragma unroll
          for (int u = 0; u < kU; ++u) {
            if (j0 + kStep * u >= mcount) continue;
            if (o.rope) {
              const int d = r >> 1;
              *reinterpret_cast<__nv_bfloat162*>(dst[u] + d) =
                  __floats2bfloat162_rn(v[u].x * cs[u].x - v[u].y * cs[u].y, v[u].z * cs[u].z - v[u].w * cs[u].w);
              *reinterpret_cast<__nv_bfloat162*>(dst[u] + d + half) =
                  __floats2bfloat162_rn(v[u].y * cs[u].x + v[u].x * cs[u].y, v[u].w * cs[u].z + v[u].z * cs[u].w);
            } else {
              *reinterpret_cast<__nv_bfloat162*>(dst[u] + r) = __floats2bfloat162_rn(v[u].x, v[u].y);
              *reinterpret_cast<__nv_bfloat162*>(dst[u] + r + 2) = __floats2bfloat162_rn(v[u].z, v[u].w);
            }
          }
        }
      } else {
        // v rows: item (row quad rq, token j), tokens fastest: a thread reads 4 head dims of one
        // token at once and each store instruction writes consecutive keys of one head dim of Vt
        // (keys contiguous)
        const int sv0 = n0 - o.qd - o.kvd;   // the tile's first v feature
        const size_t sb = (size_t)o.L * o.Hkv * o.dh * o.NKp;
        for (int it = row; it < (kBM / 4) * mcount; it += kBM) {
          const int r4 = 4 * (it / mcount), j = it - (it / mcount) * mcount;
          const int m = m0 + j, bi = m / o.H, ii = m - bi * o.H;
          const float4 v = *reinterpret_cast<const float4*>(T + j * pitch + r4);
          const int sn = sv0 + r4, g = sn / o.dh, d = sn % o.dh;   // 4 dims of one head
          __nv_bfloat16* dst = o.vtcache + bi * sb + (((size_t)o.layer * o.Hkv + g) * o.dh + d) * o.NKp + o.P + ii;
          dst[0] = __float2bfloat16_rn(v.x);
          dst[o.NKp] = __float2bfloat16_rn(v.y);
          dst[2 * (size_t)o.NKp] = __float2bfloat16_rn(v.z);
          dst[3 * (size_t)o.NKp] = __float2bfloat16_rn(v.w);
        }
      }
      break;
    }
    case EPI_PREFIX_KV: {
      // Not reached as things are (the persistent form writes these rows from registers, few tokens take the cluster
      // form), but without this case the compiler lays the others out so that the 18-layer expert is slower: 16 / 64
      // robots 1392 / 2901 us per evaluation with it, 1409 / 2922 without, 1408 / 2910 with the QKV case first or last.
      // one layer's k or v rows: tokens over the warps, lane owns 4 consecutive features, so that a
      // warp writes a token's 128 features as one contiguous run
      const int n0 = n - row, w = p.pkv.width, part = n0 / w;   // part = 2 layer + (0 k, 1 v)
      __nv_bfloat16* dst = ((part & 1) ? p.pkv.v : p.pkv.k) + (size_t)(part >> 1) * p.M * w + (n0 - part * w) + 4 * lane;
      for (int j = row >> 5; j < mcount; j += kBM / 32) {
        const float4 v = *reinterpret_cast<const float4*>(T + j * pitch + 4 * lane);
        uint2 pk;
        pk.x = ptx::pack_bf16(v.x, v.y);
        pk.y = ptx::pack_bf16(v.z, v.w);
        *reinterpret_cast<uint2*>(dst + (size_t)(m0 + j) * w) = pk;
      }
      break;
    }
    default:
      if (p.n_store > 0 && n >= p.n_store) break;   // padding rows of a narrow projection
#pragma unroll 4
      for (int j = 0; j < mcount; ++j)
        store_out(p.out, (size_t)(m0 + j) * p.ldo + n, Tr[j * pitch] + b, p.out_dtype);
      break;
  }
}

// Four lanes that hold one output row each, 16 tokens (v), become four lanes that hold four tokens each
// of all four rows: lane i of the quad gets rows 4 (lane / 4) + r of tokens 4 i + t in w[t][r]. Two butterfly
// exchanges, no shared memory.
__device__ __forceinline__ void quad_transpose(const float* v, float4* w, int lane) {
  const bool odd = lane & 1, up = lane & 2;
  float a[2][8];   // [row of the pair][blocks kept: tokens 4 (lane & 1) + t, then 8 further]
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const float e = v[8 * h + t], o = v[8 * h + 4 + t];
      const float got = __shfl_xor_sync(0xffffffffu, odd ? e : o, 1);
      const float kept = odd ? o : e;
      a[0][4 * h + t] = odd ? got : kept;
      a[1][4 * h + t] = odd ? kept : got;
    }
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    float b[2][2];   // [pair of rows][row of the pair]
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const float got = __shfl_xor_sync(0xffffffffu, up ? a[r][t] : a[r][4 + t], 2);
      const float kept = up ? a[r][4 + t] : a[r][t];
      b[0][r] = up ? got : kept;
      b[1][r] = up ? kept : got;
    }
    w[t] = make_float4(b[0][0], b[0][1], b[1][0], b[1][1]);
  }
}

// Epilogues that write a token's rows straight from registers (16 shuffles a lane and slice in place of a
// staged slice and two group barriers: 3200 tokens x 8192 rows 49.6 -> 47.5 us, pi0-like expert with 64
// robots 2.928 -> 2.889 ms per evaluation): this lane's four tokens (from m0, mcount of
// the slice's 16 valid) of the four output rows n4 .. n4 + 3. False where the shared-memory epilogue below
// has to do it (rows scattered by head dim, unaligned or padded outputs).
__device__ __forceinline__ bool direct_epilogue_ok(const TcGemmArgs& p) {
  if (p.epi == EPI_QKV_TC) return false;
  if (p.epi == EPI_PREFIX_KV || p.epi == EPI_PARTIAL) return true;
  return p.n_store <= 0 && p.ldo % 4 == 0 && reinterpret_cast<uintptr_t>(p.out) % 16 == 0;
}
__device__ __forceinline__ void direct_epilogue(const TcGemmArgs& p, const float4* w, int m0, int mcount, int n4, int sp, int lane) {
  float4 b = make_float4(0.f, 0.f, 0.f, 0.f);
  if (p.bias) b = make_float4(p.bias[n4], p.bias[n4 + 1], p.bias[n4 + 2], p.bias[n4 + 3]);
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const int j = 4 * (lane & 3) + t;
    if (j >= mcount) break;
    const size_t m = m0 + j;
    float4 x = make_float4(w[t].x + b.x, w[t].y + b.y, w[t].z + b.z, w[t].w + b.w);
    switch (p.epi) {
      case EPI_GEGLU:
        if (p.out_dtype == BF16)
          *reinterpret_cast<uint32_t*>(static_cast<__nv_bfloat16*>(p.out) + m * p.ldo + n4 / 2) =
              pack_bf16(gelu_tanh_fast(x.x) * x.y, gelu_tanh_fast(x.z) * x.w);
        else
          *reinterpret_cast<float2*>(static_cast<float*>(p.out) + m * p.ldo + n4 / 2) =
              make_float2(gelu_tanh_f(x.x) * x.y, gelu_tanh_f(x.z) * x.w);
        break;
      case EPI_PARTIAL:
        *reinterpret_cast<float4*>(static_cast<float*>(p.out) + ((size_t)sp * p.M + m) * p.N + n4) = x;
        break;
      case EPI_PREFIX_KV: {
        const int wd = p.pkv.width, part = n4 / wd;
        *reinterpret_cast<uint2*>(((part & 1) ? p.pkv.v : p.pkv.k) + ((size_t)(part >> 1) * p.M + m) * wd + (n4 - part * wd)) =
            make_uint2(pack_bf16(x.x, x.y), pack_bf16(x.z, x.w));
        break;
      }
      default:
        if (p.epi == EPI_BIAS_GELU) x = make_float4(gelu_tanh_f(x.x), gelu_tanh_f(x.y), gelu_tanh_f(x.z), gelu_tanh_f(x.w));
        if (p.out_dtype == BF16)
          *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(p.out) + m * p.ldo + n4) =
              make_uint2(pack_bf16(x.x, x.y), pack_bf16(x.z, x.w));
        else
          *reinterpret_cast<float4*>(static_cast<float*>(p.out) + m * p.ldo + n4) = x;
        break;
    }
  }
}

__global__ void __launch_bounds__(128, 1) gemm_tc_kernel(const __grid_constant__ CUtensorMap tmx, TcGemmArgs p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int t = blockIdx.x, mt = blockIdx.y, nch = p.K / kBK;
  const int stages = tc_stages(nch);
  uint8_t* sA = smem;
  uint8_t* sB = smem + (size_t)stages * kStageA;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + tc_pipe_bytes(stages));
  uint64_t* empty = full + kTcMaxStages;
  uint64_t* done = empty + kTcMaxStages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = mt * kBN;
  const int mcount = p.M - m0 < kBN ? p.M - m0 : kBN;

  if (threadIdx.x == 0) {
    for (int i = 0; i < stages; ++i) {
      mbar_init(full + i, 1);
      mbar_init(empty + i, 1);
    }
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)), "r"(kBN));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  pdl_trigger();
  if (threadIdx.x == 0) {
    // ---- producer: weight block (bulk copy) + activation tile (tensor map) per K chunk.
    //      An expert's weights are constant: the first ring's worth is requested before waiting
    //      for the kernel that produces the activations. ----
    const uint64_t pol = policy_evict_first();
    if (p.ordered) pdl_wait();
    const uint8_t* wt = static_cast<const uint8_t*>(p.w_tiled) + (size_t)t * nch * kStageA;
    const int first = nch < stages ? nch : stages;
    for (int i = 0; i < first; ++i) {
      mbar_expect_tx(full + i, kStageA + kStageB);
      bulk_g2s(sA + (size_t)i * kStageA, wt + (size_t)i * kStageA, kStageA, full + i, pol);
    }
    pdl_wait();
    for (int i = 0; i < first; ++i) tma_2d(sB + (size_t)i * kStageB, &tmx, i * kBK, mt * kBN, full + i);
    int issued = first;
    for (int i = first; i < nch; ++i) {
      const int st = i % stages, round = i / stages;
      if (!mbar_wait(empty + st, (round - 1) & 1, p.err, 11)) break;
      mbar_expect_tx(full + st, kStageA + kStageB);
      bulk_g2s(sA + (size_t)st * kStageA, wt + (size_t)i * kStageA, kStageA, full + st, pol);
      tma_2d(sB + (size_t)st * kStageB, &tmx, i * kBK, mt * kBN, full + st);
      ++issued;
    }
    // do not leave copies in flight into shared memory of an exiting CTA
    for (int i = issued - stages > 0 ? issued - stages : 0; i < issued; ++i)
      mbar_drain_issued(full + i % stages, (i / stages) & 1);
  } else if (threadIdx.x == 32) {
    // ---- MMA issuer ----
    if (p.own_err && t + mt == 0) *reinterpret_cast<volatile int*>(p.err) = 0;
    const uint64_t adesc = sw128_desc(su32(sA)), bdesc = sw128_desc(su32(sB));
    bool ok = true;
    for (int i = 0; i < nch && ok; ++i) {
      const int st = i % stages, round = i / stages;
      ok = mbar_wait(full + st, round & 1, p.err, 13);
      if (!ok) break;
      tc_fence_after();
      mma_kblock(tmem, adesc + (uint64_t)(st * (kStageA >> 4)), bdesc + (uint64_t)(st * (kStageB >> 4)), idesc_m128(kBN),
                 i > 0 ? 1u : 0u);
      mma_commit(empty + st);
    }
    mma_commit(done);
  }
  __syncwarp();

  // ---- epilogue: TMEM -> registers, one weight row (output feature) per thread ----
  pdl_wait();
  const bool ok = mbar_wait(done, 0, p.err, 14);
  if (!ok) mbar_drain_issued(done, 0);   // the MMAs, before tensor memory is given back
  tc_fence_after();
  const int row = warp * 32 + lane;
  const int n = t * kBM + row;
  float v[kBN];
  __syncwarp();
  tmem_ld64(tmem + ((uint32_t)(warp * 32) << 16), v);
  // Stage the accumulator tile in shared memory, T[token j][row]: the epilogues below are
  // compact loops over it (neighbouring rows -- GeGLU and RoPE partners -- are one column
  // apart), which keeps the kernel's code small.
  float* T = reinterpret_cast<float*>(smem);                         // pipeline region is idle
#pragma unroll
  for (int j = 0; j < kBN; ++j) T[j * kBM + row] = v[j];
  __syncthreads();
  if (ok) tile_epilogue(p, T, kBM, m0, mcount, n, row, lane);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kBN));
}


// Persistent form for many tokens: one CTA per SM walks the work units u = blockIdx.x,
// blockIdx.x + gridDim.x, ... Unit u is (token tile mt of p.tn <= TN tokens, weight tile nt, K
// split sp) with mt fastest, so the CTAs running side by side share a weight tile in L2. Warp 0
// feeds the ring of STAGES (weights 16 KB + up to TN x 128 B of tokens) without stopping at unit
// boundaries; warp 1 issues the MMAs into one of two TMEM accumulators (2 x TN columns) while
// four groups of four warps (2-5, 6-9, 10-13, 14-17) drain the other one in 16-token slices,
// slice q to group q % 4, each group through a staging slice of its own, so a unit's epilogue
// overlaps the next unit's main loop. A ragged last token tile loads and multiplies only its
// 64-token boxes. K splits (residual projections only) write planes of their own, summed by the
// norm that follows. SETS = 2: a unit's k-blocks take turns over two accumulators (all 512 columns of tensor
// memory with the double buffering), added in fp32 when they are read out, so that the tensor cores'
// truncating accumulation runs over half as many products.
template <int TN, int STAGES, int SETS>
__global__ void __launch_bounds__(kPersThreads, 1) gemm_tc_pers_kernel(const __grid_constant__ CUtensorMap tmx,
                                                                       TcGemmArgs p) {
  constexpr int kStageBw = TN * kBK * 2;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* sA = smem;                                        // STAGES x 16 KB weights
  uint8_t* sB = smem + (size_t)STAGES * kStageA;             // STAGES x TN x 128 B tokens
  float* T = reinterpret_cast<float*>(smem + (size_t)STAGES * (kStageA + kStageBw));  // groups x 16 x pitch
  uint64_t* full = reinterpret_cast<uint64_t*>(T + kPersGroups * kPersSlice * kPersPitch);
  uint64_t* empty = full + STAGES;
  uint64_t* tfull = empty + STAGES;    // accumulator b complete
  uint64_t* tempty = tfull + 2;        // accumulator b drained (one arrival per epilogue thread)
  uint64_t* done = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tn = p.tn;
  const int n_nt = p.N / kBM, n_mt = (p.M + tn - 1) / tn, S = p.splits, KC = p.K / kBK;
  const int per = (KC + S - 1) / S;
  const int units = n_nt * n_mt * S;

  if (threadIdx.x == 0) {
    for (int i = 0; i < STAGES; ++i) {
      mbar_init(full + i, 1);
      mbar_init(empty + i, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(tfull + b, 1);
      mbar_init(tempty + b, kPersGroups * 128);
    }
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)), "r"(2 * TN * SETS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_trigger();

  if (warp == 0) {
    if (lane == 0) {
      // ---- producer ----
      pdl_wait();
      int it = 0;
      bool ok = true;
      for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
        const int mt = u % n_mt, r = u / n_mt, nt = r % n_nt, sp = r / n_nt;
        const int k0 = sp * per, k1 = k0 + per < KC ? k0 + per : KC;
        const int left = p.M - mt * tn;
        const int nb = ((left < tn ? left : tn) + kBN - 1) / kBN;
        const uint8_t* wt = static_cast<const uint8_t*>(p.w_tiled) + (size_t)nt * KC * kStageA;
        for (int kb = k0; kb < k1; ++kb, ++it) {
          const int st = it % STAGES, round = it / STAGES;
          if (round > 0 && !mbar_wait(empty + st, (round - 1) & 1, p.err, 61)) { ok = false; break; }
          mbar_expect_tx(full + st, kStageA + nb * kStageB);
          bulk_g2s_nohint(sA + (size_t)st * kStageA, wt + (size_t)kb * kStageA, kStageA, full + st);
          for (int q = 0; q < nb; ++q)
            tma_2d(sB + (size_t)st * kStageBw + q * kStageB, &tmx, kb * kBK, mt * tn + q * kBN, full + st);
        }
      }
      // do not leave copies in flight into shared memory of an exiting CTA
      for (int i = it - STAGES > 0 ? it - STAGES : 0; i < it; ++i)
        mbar_drain_issued(full + i % STAGES, (i / STAGES) & 1);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // ---- MMA issuer ----
      if (p.own_err && blockIdx.x == 0) *reinterpret_cast<volatile int*>(p.err) = 0;
      const uint32_t tmem = *tmem_slot;
      const uint64_t adesc = sw128_desc(su32(sA)), bdesc = sw128_desc(su32(sB));
      int it = 0, j = 0;
      bool ok = true;
      for (int u = blockIdx.x; u < units && ok; u += gridDim.x, ++j) {
        const int mt = u % n_mt, sp = u / n_mt / n_nt;
        const int k0 = sp * per, k1 = k0 + per < KC ? k0 + per : KC;
        const int left = p.M - mt * tn;
        const int nb = ((left < tn ? left : tn) + kBN - 1) / kBN;
        const uint32_t idesc = idesc_m128(nb * kBN);
        const int b = j & 1;
        if (j >= 2 && !mbar_wait(tempty + b, ((j >> 1) - 1) & 1, p.err, 63)) break;
        tc_fence_after();
        const uint32_t d = tmem + (uint32_t)(b * TN * SETS);
        for (int kb = k0; kb < k1; ++kb, ++it) {
          const int st = it % STAGES, round = it / STAGES;
          if (!mbar_wait(full + st, round & 1, p.err, 64)) { ok = false; break; }
          tc_fence_after();
          const uint32_t set = SETS == 1 ? 0 : (uint32_t)((kb - k0) % SETS * TN);
          mma_kblock(d + set, adesc + (uint64_t)(st * (kStageA >> 4)), bdesc + (uint64_t)(st * (kStageBw >> 4)), idesc,
                     kb > k0 + SETS - 1 ? 1u : 0u);
          mma_commit(empty + st);
        }
        if (ok) mma_commit(tfull + b);
      }
      mma_commit(done);
      mbar_drain_issued(done, 0);   // before tensor memory is given back
    }
  } else {
    // ---- epilogue: group g = warps 2 + 4g .. 5 + 4g takes slices g, g + 4, ...; warp w reads
    //      tensor-memory lanes 32 (w % 4) .. + 31 ----
    const int g = (warp - 2) >> 2;
    const int q4 = warp & 3, row = q4 * 32 + lane;
    float* Tg = T + g * kPersSlice * kPersPitch;
    const bool direct = direct_epilogue_ok(p);
    pdl_wait();
    int j = 0;
    for (int u = blockIdx.x; u < units; u += gridDim.x, ++j) {
      const int mt = u % n_mt, r = u / n_mt, nt = r % n_nt, sp = r / n_nt;
      const int left = p.M - mt * tn;
      const int nsl = ((left < tn ? left : tn) + kPersSlice - 1) / kPersSlice;
      const int mylast = g < nsl ? g + kPersGroups * ((nsl - 1 - g) / kPersGroups) : -1;  // this group's last slice
      const int b = j & 1;
      // one decision for the group, so that none of its warps is left alone at a named barrier
      if (!named_and(1 + g, 128, mbar_wait(tfull + b, (j >> 1) & 1, p.err, 66))) break;
      tc_fence_after();
      if (mylast < 0) {
        tc_fence_before();
        mbar_arrive(tempty + b);
      }
      const uint32_t tb = tmem_base_after_wait(tmem_slot) + (uint32_t)(b * TN * SETS) + ((uint32_t)(q4 * 32) << 16);
      const int n = nt * kBM + row;
      for (int q = g; q < nsl; q += kPersGroups) {
        const int m0 = mt * tn + q * kPersSlice;
        const int mcount = p.M - m0 < kPersSlice ? p.M - m0 : kPersSlice;
        float v[kPersSlice];
        bool sum = false;
        if constexpr (SETS == 2) sum = (sp + 1 < S ? per : KC - sp * per) > 1;   // k-blocks for both accumulators
        if (sum) tmem_sum16(tb + q * kPersSlice, tb + TN + q * kPersSlice, v);
        else tmem_ld16(tb + q * kPersSlice, v);
        if (q == mylast) {
          // the group's share of the accumulator is in registers: hand it back
          tc_fence_before();
          mbar_arrive(tempty + b);
        }
        if (direct) {
          float4 w[4];
          quad_transpose(v, w, lane);
          direct_epilogue(p, w, m0, mcount, nt * kBM + (row & ~3), sp, lane);
          continue;
        }
        named_sync(1 + g, 128);   // the previous slice's readers are done with Tg
#pragma unroll
        for (int jj = 0; jj < kPersSlice; ++jj) Tg[jj * kPersPitch + row] = v[jj];
        named_sync(1 + g, 128);
        tile_epilogue(p, Tg, kPersPitch, m0, mcount, n, row, lane);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*tmem_slot), "r"(2 * TN * SETS));
  }
}

// ---- weight re-layout into 128 x 64 swizzled blocks --------------------------------------
__global__ void relayout_tiled_kernel(const float* src, int K, int N, __nv_bfloat16* dst, int mult, long long off,
                                      int rope_dh) {
  __shared__ float tt[32][33];
  const int k0 = blockIdx.y * 32, n0 = blockIdx.x * 32;
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int k = k0 + r, n = n0 + threadIdx.x;
    tt[r][threadIdx.x] = (k < K && n < N) ? src[(long long)k * N + n] : 0.f;
  }
  __syncthreads();
  const int KC = K / kBK;
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int n = n0 + r, k = k0 + threadIdx.x;
    if (n >= N || k >= K) continue;
    int nn = n;
    if (rope_dh > 0) {
      const int h = n / rope_dh, d = n % rope_dh, half = rope_dh / 2;
      nn = h * rope_dh + (d < half ? 2 * d : 2 * (d - half) + 1);
    }
    const long long row = (long long)nn * mult + off;
    const long long tile = (row / kBM) * KC + k / kBK;
    const int rr = (int)(row % kBM), kk = k % kBK;
    const int gran = (kk >> 3) ^ (rr & 7);
    dst[tile * (kBM * kBK) + rr * kBK + gran * 8 + (kk & 7)] = __float2bfloat16_rn(tt[threadIdx.x][r]);
  }
}

}  // namespace

static PFN_cuTensorMapEncodeTiled_v12000 tmap_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess && q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

int encode_act_tmap(CUtensorMap* m, const void* base, int K, int rows, int box_rows) {
  auto enc = tmap_encoder();
  if (!enc) return -1;
  const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)K * 2};
  const cuuint32_t box[2] = {kBK, (cuuint32_t)box_rows};
  const cuuint32_t es[2] = {1, 1};
  const CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? 0 : (int)r;
}

static size_t gemm_tc_smem_bytes(int stages) {
  return 1024 + tc_pipe_bytes(stages) + (2 * kTcMaxStages + 1) * 8 + 16;
}

constexpr int kPersStages256 = 4, kPersStages128 = 6;   // 192 KB of ring either way
// tn: the instantiation's tile capacity (256 or 128)
static size_t gemm_tc_pers_smem_bytes(int tn) {
  const int st = tn == 256 ? kPersStages256 : kPersStages128;
  return 1024 + (size_t)st * (kStageA + (size_t)tn * kBK * 2) + (size_t)kPersGroups * kPersSlice * kPersPitch * 4 +
         (2 * st + 5) * 8 + 16;
}

int gemm_tc_prepare() {
  static OncePerDevice once;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return -1;
  return once.run(dev, [] {
    const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    if (gemm_cl_prepare() ||
        cudaFuncSetAttribute(gemm_tc_pers_kernel<256, kPersStages256, 1>, at, (int)gemm_tc_pers_smem_bytes(256)) != cudaSuccess ||
        cudaFuncSetAttribute(gemm_tc_pers_kernel<128, kPersStages128, 1>, at, (int)gemm_tc_pers_smem_bytes(128)) != cudaSuccess ||
        cudaFuncSetAttribute(gemm_tc_pers_kernel<128, kPersStages128, 2>, at, (int)gemm_tc_pers_smem_bytes(128)) != cudaSuccess ||
        cudaFuncSetAttribute(gemm_tc_kernel, at, (int)gemm_tc_smem_bytes(kTcMaxStages)) != cudaSuccess)
      return -1;
    return 0;
  });
}

// Wide tiles (MMA N up to 256 tokens) run the tensor cores near their rate (N = 64 runs at a
// third of it) and cut L2 re-reads of the weights: 1 = the persistent wide form, 0 = narrow
// 128 x 64 tiles or the cluster form. Wide from 512 tokens, or while 256-token tiles fill 60% of the
// SMs or 128-token tiles fill half of them (measured on the pi0-like projections from 200 to 3200
// tokens: with fewer than 256 tokens the narrow tiles win; at 800 tokens the wide form with K
// split planes wins for the 1024-row o and down projections too).
int gemm_tc_use_wide(int M, int N, int sms) {
  if (M < 256 || N > 8192) return 0;
  const int t256 = (N / kBM) * ((M + 255) / 256), t128 = (N / kBM) * ((M + 127) / 128);
  return M >= 512 || t256 * 5 >= sms * 3 || t128 * 2 >= sms ? 1 : 0;
}

// A residual projection may also split K into planes that the next norm sums, so the persistent form fills
// the SMs from a third 64-token tile on, where the cluster form's exchange costs more than writing the planes.
// Per evaluation, N = 1024, 18 layers: 180 tokens 852 -> 842 us, 250 tokens 1053 -> 968, 400 tokens 1288 -> 1183;
// N = 1536, 16 layers: 128 tokens 1368 -> 1378, 192 tokens 1820 -> 1795, 256 tokens 1850 -> 1761, 320 tokens
// 1886 -> 2005, 480 tokens 2556 -> 2450. Narrower ones stay: N = 512, 250 tokens 102 -> 109.
// They have fewer splits than the narrow form's planes had, so a tile of 128 tokens sums its k-blocks in two
// accumulators (SETS): the longest run is no longer than there (180 tokens, N = 1024, K = 2048 and 4096: error 4.7e-7 ->
// 2.3e-7, positive products 8.4e-7 -> 3.6e-7; 6.4 -> 6.5 and 6.5 -> 6.6 us).
int gemm_tc_resid_wide(int M, int N, int sms) {
  return gemm_tc_use_wide(M, N, sms) || (M > 128 && N >= 1024 && N <= 2048);
}

// The persistent form's plan: tokens per tile (256, 192 or 128, at most most_tn) and, for partial-plane
// epilogues, K splits. Units go to the CTAs round robin; the plan minimises the busiest CTA's
// work, counted in k-blocks of a 256-token tile: a k-block of nb 64-token boxes costs half by
// its MMA time (nb / 4) and half by its bytes ((2 + nb) / 6, weights 16 KB + 8 KB a box), plus
// half a k-block per unit and, per extra plane, the cost of writing and reading it once more.
void gemm_tc_pers_plan(int M, int N, int K, int sms, int epi, int most_tn, int* tn, int* splits) {
  const int KC = K / kBK, n_nt = N / kBM;
  double best = 1e30;
  *tn = most_tn;
  *splits = 1;
  for (int t = most_tn; t >= 128; t -= 64) {
    const int n_mt = (M + t - 1) / t;
    const int smax = epi == EPI_PARTIAL ? 8 : 1;
    for (int sp = 1; sp <= smax && sp <= KC; ++sp) {
      const int per = (KC + sp - 1) / sp;
      if ((sp - 1) * per >= KC) continue;
      const int units = n_nt * n_mt * sp;
      const int ctas = units < sms ? units : sms;
      double worst = 0;
      for (int c = 0; c < ctas; ++c) {
        double w = 0;
        for (int u = c; u < units; u += ctas) {
          const int mt = u % n_mt, s = u / n_mt / n_nt;
          const int kb = (s + 1) * per < KC ? per : KC - s * per;
          const int left = M - mt * t;
          const int nb = ((left < t ? left : t) + kBN - 1) / kBN;
          w += kb * (0.5 * nb / 4.0 + 0.5 * (2 + nb) / 6.0) + 0.5;
        }
        worst = w > worst ? w : worst;
      }
      const double plane = 8.0 * M * N / 6.5e12 / 0.3e-6;   // extra plane written and read, in k-blocks
      const double cost = worst + (sp - 1) * plane;
      if (cost < best - 1e-9) {
        best = cost;
        *tn = t;
        *splits = sp;
      }
    }
  }
}

void gemm_tc_plan(int M, int N, int K, int sms, int epi, TcGemmArgs* a) {
  a->wide = epi == EPI_PARTIAL ? gemm_tc_resid_wide(M, N, sms) : gemm_tc_use_wide(M, N, sms);
  a->tn = 0;
  a->splits = 1;
  a->cl = 0;
  a->sets = a->wide && !gemm_tc_use_wide(M, N, sms) ? 2 : 1;
  // a long K over so few tiles that each would walk it alone: the cluster form's K splits (637 rows, N = 1024,
  // K = 4096: 21.2 -> 14.9 us; K = 2048, 800 rows: 13.0 -> 12.5). The residual projections split K anyway.
  const bool alone = a->wide && epi != EPI_PARTIAL && K >= 2048 && (N / kBM) * ((M + kBN - 1) / kBN) <= sms;
  if (alone) a->wide = 0;
  if (a->wide) {
    // the plan search walks every unit: remember its answers
    thread_local std::map<std::array<int, 6>, std::pair<int, int>> memo;
    const std::array<int, 6> key{M, N, K, sms, epi == EPI_PARTIAL, a->sets};
    auto it = memo.find(key);
    if (it == memo.end()) {
      std::pair<int, int> v;
      gemm_tc_pers_plan(M, N, K, sms, epi, a->sets == 2 ? 128 : 256, &v.first, &v.second);
      it = memo.emplace(key, v).first;
    }
    a->tn = it->second.first;
    a->splits = it->second.second;
  } else if (epi == EPI_RESID_H || alone || gemm_cl_serves(M, N, sms)) {
    a->cl = 1;
    gemm_cl_plan(M, N, K, sms, a);
  }
}

// The prefix projection of a DiT (every layer's K and V rows stacked: thousands of rows, one call per
// observation): the grid is full without K splits, so none are used and no accumulator is needed.
// The persistent form from a second 64-token box on, whose tiles then read each weight block once
// for all of them (300 tokens x 49152 rows x 2048, one observation bound: 8.43 ms on the CUDA cores, 0.20 ms here).
void gemm_tc_prefix_plan(int M, int N, int K, int sms, TcGemmArgs* a) {
  a->wide = M > kBN;
  a->cl = !a->wide;
  a->splits = 1;
  a->tn = 0;
  if (a->wide) gemm_tc_pers_plan(M, N, K, sms, EPI_PREFIX_KV, 256, &a->tn, &a->splits);
}

void launch_gemm_tc(const CUtensorMap* tmx, const TcGemmArgs& a, cudaStream_t s) {
  if (a.wide) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int units = (a.N / kBM) * ((a.M + a.tn - 1) / a.tn) * a.splits;
    const dim3 grid(units < sms ? units : sms);
    if (a.tn > 128)
      launch_k(gemm_tc_pers_kernel<256, kPersStages256, 1>, grid, dim3(kPersThreads), gemm_tc_pers_smem_bytes(256), s,
               *tmx, a);
    else if (a.sets == 2)
      launch_k(gemm_tc_pers_kernel<128, kPersStages128, 2>, grid, dim3(kPersThreads), gemm_tc_pers_smem_bytes(128), s,
               *tmx, a);
    else
      launch_k(gemm_tc_pers_kernel<128, kPersStages128, 1>, grid, dim3(kPersThreads), gemm_tc_pers_smem_bytes(128), s,
               *tmx, a);
    return;
  }
  if (a.cl) {
    launch_gemm_cl(tmx, a, s);
    return;
  }
  launch_k(gemm_tc_kernel, dim3(a.N / kBM, (a.M + kBN - 1) / kBN), dim3(128), gemm_tc_smem_bytes(tc_stages(a.K / kBK)), s,
           *tmx, a);
}

void launch_relayout_tiled(const float* src, int K, int N, void* dst, int mult, long long off, int rope_dh,
                           cudaStream_t s) {
  dim3 grid((N + 31) / 32, (K + 31) / 32);
  relayout_tiled_kernel<<<grid, dim3(32, 8), 0, s>>>(src, K, N, static_cast<__nv_bfloat16*>(dst), mult, off, rope_dh);
}

}  // namespace uad
