// Few-token tensor-core projection: the K range of an output tile split over a thread-block cluster.
//
// out[m][n] = epi(sum_k X[m][k] * Wt[n][k]) for tiles of 128 or 64 weight rows x up to 64 tokens. With few
// tokens a projection is a short chain of dependent steps (operands, MMAs, the sum over the K splits,
// the epilogue), so the kernel keeps that sum out of global memory: the S CTAs of a cluster each
// multiply their share of K into tensor memory, stage the fp32 tile in shared memory and send every
// other CTA the token rows it owns with one bulk copy through distributed shared memory; each CTA adds
// the S partial rows of its tokens in rank order (the result does not depend on timing) and applies
// the epilogue to them. The receive area lies apart from the operand ring, so that rows arrive while other
// CTAs' MMAs still run (aliased on the ring: DiT head 916 us per evaluation, apart 840; four robots 1246 and
// 1214). The exchange is slow (10-13 B a cycle and SM): it pays while a CTA's share is a few KB. An expert's
// weights are requested before the wait for the kernel that produces the activations (a caller's after it:
// TcGemmArgs::ordered). Every wait is bounded; the cluster barriers are reached on every path, and no CTA leaves with
// copies in flight into its shared memory.
#include <cuda.h>
#include <cudaTypedefs.h>

#include "uad_internal.cuh"
#include "ptx.cuh"

namespace uad {

using namespace ptx;

namespace {

constexpr int kTileM = 128, kBN = 64, kBK = 64;
constexpr int kTileBytes = kTileM * kBK * 2;     // a k-block of the tiled weights: 16 KB, its rows 0-63 first
// A k-block's activations come in one box, of 64 token rows or, for up to 16 tokens, 16: 8 KB or 2 KB a slot, so
// that a fifth slot of weights fits (16-layer DiT expert, 16 tokens: 772 -> 762 us per evaluation; two boxes of 16
// for up to 32 tokens lost 1%).
constexpr int kConsWarps = 8, kCons = 32 * kConsWarps;
// The tensor cores' accumulation truncates, so its error grows with the run of products: a CTA's k-blocks take turns
// over one, two or four accumulators, which are added in fp32, rounded to nearest, when the tile is read out.
// Products of positive numbers, mean error of 16 x 6144 x 1536 1.5e-6 with one accumulator, 2.7e-7 with four; DiT
// expert, one / four robots 755 / 1070 -> 759 / 1084 us per evaluation, 18-layer expert at one robot 672 -> 677.
constexpr int kTmCols = 256;                     // tensor memory of a CTA, half an SM's: four accumulators of 64 tokens
constexpr int kThreads = kCons + 64;             // + producer warp, + MMA warp
constexpr unsigned long long kWaitNs = 2000000000ull;

__device__ __forceinline__ bool wait_bar(uint64_t* b, uint32_t parity, int* err, int code) {
  return ptx::mbar_wait(b, parity, err, code, kWaitNs);
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// Shared memory -> another CTA's shared memory; completes on that CTA's barrier.
__device__ __forceinline__ void bulk_s2dsm(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "r"(su32(src)), "r"(bytes), "r"(bar) : "memory");
}

__device__ __forceinline__ float gelu_tanh_f(float x) {
  const float k0 = 0.7978845608028654f;
  return 0.5f * x * (1.f + tanhf(k0 * (x + 0.044715f * x * x * x)));
}
__device__ __forceinline__ uint2 pack4(float a, float b, float c, float d) { return make_uint2(pack_bf16(a, b), pack_bf16(c, d)); }

// Where a CTA's shared memory goes: the ring of k-block slots, reused after the MMAs as the staged tile
// T[token][bm]; then the partial rows received from the other CTAs, [rank][owned token][bm], apart from
// the ring, so that they may arrive while this CTA's MMAs still run. `rows`: tokens of the largest
// tile, bm: weight rows of a tile.
__host__ __device__ __forceinline__ size_t cl_ring_bytes(int ring, int rows, int bm) {
  const size_t pipe = (size_t)ring * (bm + act_box_rows(rows)) * kBK * 2, tile = (size_t)((rows + 15) / 16 * 16) * bm * 4;
  return pipe > tile ? pipe : tile;
}
__host__ __device__ __forceinline__ size_t cl_recv_bytes(int rows, int splits, int bm) {
  return splits > 1 ? (size_t)((rows + splits - 1) / splits) * splits * bm * 4 : 0;
}

// E: the epilogue this instantiation is for, or, read from the arguments, kAny: any; kPlain: any but EPI_QKV_TC
// and EPI_GEGLU. A kernel whose code is not in the SM's instruction cache runs at a dozen cycles an instruction,
// so it matters which projections share code (TcGemmArgs::cl_code).
constexpr int kAny = -2, kPlain = -1;
template <int E, int kBM, int kBox>
__global__ void __launch_bounds__(kThreads, 2) gemm_cl_kernel(const __grid_constant__ CUtensorMap tmx, TcGemmArgs p, int ring_sets) {
  // in one word: a field of its own, further on in the arguments, cost 1% (a cold line of constant memory)
  const int ring = ring_sets & 255, sets = ring_sets >> 8;   // ring slots, accumulators
  extern __shared__ uint8_t smem_raw[];
  constexpr int kSlotA = kBM * kBK * 2, kSlot = kSlotA + kBox * kBK * 2;
  constexpr int kLanes = kBM / 4, TP = 32 / kLanes;   // lanes that share a token row, rows a warp takes at once
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int S = p.splits, rank = blockIdx.x, nt = blockIdx.y, mt = blockIdx.z;
  const int KC = p.K / kBK, c0 = rank * KC / S, nkb = (rank + 1) * KC / S - c0;
  const int m0 = mt * kBN, mcount = p.M - m0 < kBN ? p.M - m0 : kBN;
  const int per = (mcount + S - 1) / S, t0 = rank * per;            // token rows this CTA finishes
  const int cnt = mcount - t0 < 0 ? 0 : mcount - t0 < per ? mcount - t0 : per;
  const int width = (mcount + 15) / 16 * 16;   // columns of an accumulator
  float* T = reinterpret_cast<float*>(smem);
  const int rows = p.M < kBN ? p.M : kBN;
  float* recv = reinterpret_cast<float*>(smem + cl_ring_bytes(ring, rows, kBM));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + cl_ring_bytes(ring, rows, kBM) + cl_recv_bytes(rows, S, kBM));
  uint64_t* empty = full + ring;
  uint64_t* done = empty + ring;
  uint64_t* got = done + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(got + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int i = 0; i < ring; ++i) {
      mbar_init(full + i, 1);
      mbar_init(empty + i, 1);
    }
    mbar_init(done, 1);
    mbar_init(got, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (S > 1 && cnt > 0) mbar_expect_tx(got, (uint32_t)((S - 1) * cnt * kBM * 4));
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)), "r"(kTmCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (S > 1) cluster_arrive();   // this CTA's barriers are set up and its receive area is free
  pdl_trigger();

  if (warp == kConsWarps) {
    // ---- producer ----
    if (lane == 0) {
      const uint64_t pol = policy_evict_first();
      const uint8_t* wt = static_cast<const uint8_t*>(p.w_tiled) + ((size_t)(nt * kBM / kTileM) * KC + c0) * kTileBytes + nt * kBM % kTileM * kBK * 2;
      const int first = nkb < ring ? nkb : ring;
      if (p.ordered) pdl_wait();
      for (int i = 0; i < first; ++i) {
        mbar_expect_tx(full + i, kSlot);
        bulk_g2s(smem + (size_t)i * kSlot, wt + (size_t)i * kTileBytes, kSlotA, full + i, pol);
      }
      pdl_wait();
      for (int i = 0; i < first; ++i) tma_2d(smem + (size_t)i * kSlot + kSlotA, &tmx, (c0 + i) * kBK, m0, full + i);
      int issued = first;
      for (int i = first; i < nkb; ++i, ++issued) {
        const int st = i % ring;
        if (!wait_bar(empty + st, (i / ring - 1) & 1, p.err, 71)) break;
        mbar_expect_tx(full + st, kSlot);
        bulk_g2s(smem + (size_t)st * kSlot, wt + (size_t)i * kTileBytes, kSlotA, full + st, pol);
        tma_2d(smem + (size_t)st * kSlot + kSlotA, &tmx, (c0 + i) * kBK, m0, full + st);
      }
      // no copies in flight into shared memory that is reused, or of a CTA that exits
      for (int i = issued - ring > 0 ? issued - ring : 0; i < issued; ++i) mbar_drain_issued(full + i % ring, (i / ring) & 1);
    }
    __syncwarp();
    if (S > 1) {
      cluster_wait();
      cluster_arrive();
    }
  } else if (warp == kConsWarps + 1) {
    // ---- MMA issuer ----
    if (lane == 0) {
      if (p.own_err && rank + nt + mt == 0) *reinterpret_cast<volatile int*>(p.err) = 0;
      const uint32_t tmem = *tmem_slot;
      const uint32_t idesc = idesc_rows(kBM, width), last = tmem + (sets - 1) * width;
      uint32_t d = tmem;
      const uint64_t ring0 = sw128_desc(su32(smem));
      for (int i = 0; i < nkb; ++i) {
        const int st = i % ring;
        if (!wait_bar(full + st, (i / ring) & 1, p.err, 73)) break;
        tc_fence_after();
        const uint64_t a = ring0 + (uint64_t)(st * (kSlot >> 4));
        mma_kblock(d, a, a + (kSlotA >> 4), idesc, i >= sets ? 1u : 0u);
        d = d == last ? tmem : d + width;
        if (i + ring < nkb) mma_commit(empty + st);
      }
      mma_commit(done);
    }
    __syncwarp();
    if (S > 1) {
      cluster_wait();
      cluster_arrive();
    }
  } else {
    // ---- epilogue warps ----
    // residual update: this warp's first tokens' gates and residual rows are requested before the
    // MMAs are waited for
    constexpr int U = 4;
    const int fl = lane % kLanes, sub = lane / kLanes, n = nt * kBM + 4 * fl;   // this lane's four output features
    const int epi = E >= 0 ? E : p.epi;
    const bool resid = epi == EPI_RESID_H;
    const bool vec = reinterpret_cast<uintptr_t>(p.out) % 16 == 0 && p.ldo % 4 == 0;   // a caller's pointer may not be
    float4 hv[U], gv[U], bias = make_float4(0.f, 0.f, 0.f, 0.f);
    if (p.ordered) pdl_wait();
    if (p.bias) {
      const int nb = p.n_store > 0 ? p.n_store : p.N;
      if (n < nb) bias.x = __ldg(p.bias + n);
      if (n + 1 < nb) bias.y = __ldg(p.bias + n + 1);
      if (n + 2 < nb) bias.z = __ldg(p.bias + n + 2);
      if (n + 3 < nb) bias.w = __ldg(p.bias + n + 3);
    }
    const auto load_gates = [&](int t) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int tt = (t + kConsWarps * u) * TP + sub;
        gv[u] = make_float4(1.f, 1.f, 1.f, 1.f);
        if (tt < cnt && p.gate_tab)
          gv[u] = __ldg(reinterpret_cast<const float4*>(p.gate_tab + (size_t)__ldcg(p.tau_row + m0 + t0 + tt) * p.gate_stride + n));
      }
    };
    const auto load_h = [&](int t) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int tt = (t + kConsWarps * u) * TP + sub;
        if (tt < cnt) hv[u] = __ldcg(reinterpret_cast<const float4*>(p.resid + (size_t)(m0 + t0 + tt) * p.N + n));
      }
    };
    // RoPE: likewise the (cos, sin) of this warp's first tokens (constant), kept where the residual rows would be
    const bool qkv = E == EPI_QKV_TC || (E == kAny && p.epi == EPI_QKV_TC);
    const bool qk = qkv && p.qkv.rope && nt * kBM < p.qkv.qd + p.qkv.kvd;
    const auto load_cs = [&](int t) {
      const int sn = n < p.qkv.qd ? n : n - p.qkv.qd, r = sn % p.qkv.dh;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int tt = (t + kConsWarps * u) * TP + sub;
        if (tt < cnt) hv[u] = __ldg(reinterpret_cast<const float4*>(p.qkv.rope + (size_t)((m0 + t0 + tt) % p.qkv.H) * p.qkv.dh + r));
      }
    };
    if (resid) load_gates(warp);
    if (qk) load_cs(warp);
    // 64 rows: 16 in each warp's quarter of tensor memory
    const int row = kBM == 128 ? (warp & 3) * 32 + lane : (warp & 3) * 16 + (lane & 15);
    pdl_wait();
    if (resid) load_h(warp);
    const bool ok = wait_bar(done, 0, p.err, 74);
    if (!ok) mbar_drain_issued(done, 0);   // the MMAs, before tensor memory is given back
    tc_fence_after();
    const uint32_t tm = tmem_base_after_wait(tmem_slot) + ((uint32_t)((warp & 3) * 32) << 16);
    __syncwarp();
    if (sets <= 2) {
      for (int q = 16 * (warp >> 2); q < mcount; q += 32) {   // warps 4-7 take the odd 16-token slices
        float v[16];
        if (sets == 2) tmem_sum16(tm + q, tm + width + q, v);
        else tmem_ld16(tm + q, v);
#pragma unroll
        for (int e = 0; e < 16; ++e)
          if (kBM == 128 || lane < 16) T[(q + e) * kBM + row] = v[e];
      }
    } else {
      for (int q = 8 * (warp >> 2); q < width; q += 16) {
        float v[8];
        tmem_sum8x4(tm + q, width, v);
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if (kBM == 128 || lane < 16) T[(q + e) * kBM + row] = v[e];
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    named_sync(1, kCons);
    if (S > 1) {
      cluster_wait();   // every CTA has started
      if (threadIdx.x < S && (int)threadIdx.x != rank) {
        const int r = threadIdx.x, first = r * per, rc = mcount - first < per ? mcount - first : per;
        if (rc > 0)
          bulk_s2dsm(mapa(su32(recv + (size_t)rank * per * kBM), r), T + (size_t)first * kBM, (uint32_t)(rc * kBM * 4),
                     mapa(su32(got), r));
      }
    }
    const bool all = S == 1 || cnt == 0 || wait_bar(got, 0, p.err, 75);
    if (!all) mbar_drain(got, 0, 2 * kWaitNs);   // the others' rows, which they send also if a wait of theirs gave up
    __syncwarp();
    if (S > 1) cluster_arrive();   // this CTA's rows are here: once every CTA says so, none reads another's memory
    if (ok && all) {
      for (int t = warp; t * TP < cnt; t += kConsWarps * U) {
        if (resid && t != warp) {
          load_gates(t);
          load_h(t);
        }
        if (qk && t != warp) load_cs(t);
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int tt = (t + kConsWarps * u) * TP + sub;
          if (tt >= cnt) break;
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
          for (int r = 0; r < S; ++r) {
            const float* src = r == rank ? T + (size_t)(t0 + tt) * kBM : recv + ((size_t)r * per + tt) * kBM;
            const float4 q = *reinterpret_cast<const float4*>(src + 4 * fl);
            v.x += q.x;
            v.y += q.y;
            v.z += q.z;
            v.w += q.w;
          }
          const int m = m0 + t0 + tt;
          v.x += bias.x;
          v.y += bias.y;
          v.z += bias.z;
          v.w += bias.w;
          switch (epi) {
            case EPI_RESID_H: {
              float4 h = hv[u];
              h.x = fmaf(gv[u].x, v.x, h.x);
              h.y = fmaf(gv[u].y, v.y, h.y);
              h.z = fmaf(gv[u].z, v.z, h.z);
              h.w = fmaf(gv[u].w, v.w, h.w);
              *reinterpret_cast<float4*>(p.resid + (size_t)m * p.N + n) = h;
              break;
            }
            case EPI_GEGLU: if constexpr (E == EPI_GEGLU || E == kAny) {
              // rows 2i (gate) and 2i + 1 (up) give output i
              const size_t off = (size_t)m * p.ldo + n / 2;
              const uint32_t pk = pack_bf16(gelu_tanh_approx(v.x) * v.y, gelu_tanh_approx(v.z) * v.w);
              if (p.out_dtype == BF16)
                *reinterpret_cast<uint32_t*>(static_cast<__nv_bfloat16*>(p.out) + off) = pk;
              else
                *reinterpret_cast<float2*>(static_cast<float*>(p.out) + off) = make_float2(gelu_tanh_f(v.x) * v.y, gelu_tanh_f(v.z) * v.w);
            }
            break;
            case EPI_QKV_TC: if constexpr (E == EPI_QKV_TC || E == kAny) {
              const QkvTcOut& o = p.qkv;
              const int b = m / o.H, i = m - b * o.H;
              if (nt * kBM < o.qd + o.kvd) {
                // q or k: two RoPE pairs (rows 2j, 2j + 1 of a head hold dims j and j + dh/2)
                const bool isq = nt * kBM < o.qd;
                const int sn = isq ? n : n - o.qd, h = sn / o.dh, r = sn % o.dh, half = o.dh / 2;
                __nv_bfloat16* dst = isq ? o.q + (((size_t)b * o.Hkv * o.G + h) * o.H + i) * o.dh
                                         : o.kcache + ((((size_t)b * o.L + o.layer) * o.Hkv + h) * o.NK + o.P + i) * o.dh;
                if (o.rope) {
                  const float4 cs = hv[u];
                  const int d = r >> 1;
                  const uint32_t w0 = pack_bf16(v.x * cs.x - v.y * cs.y, v.z * cs.z - v.w * cs.w);
                  const uint32_t w1 = pack_bf16(v.y * cs.x + v.x * cs.y, v.w * cs.z + v.z * cs.w);
                  *reinterpret_cast<uint32_t*>(dst + d) = w0;
                  *reinterpret_cast<uint32_t*>(dst + d + half) = w1;
                } else {
                  *reinterpret_cast<uint2*>(dst + r) = pack4(v.x, v.y, v.z, v.w);
                }
              } else {
                // v: into this token's staged row (16-byte pieces swizzled by token), for the writes below, once every
                // lane of the row has read its own piece of it
                __syncwarp(kLanes == 32 ? 0xffffffffu : 0xffffu << (16 * sub));
                *reinterpret_cast<float4*>(T + (size_t)(t0 + tt) * kBM + 4 * (fl ^ (tt & (kLanes - 1)))) = v;
              }
            }
            break;
            case EPI_PREFIX_KV: {
              const int w = p.pkv.width, part = nt * kBM / w;   // part = 2 layer + (0 k, 1 v)
              *reinterpret_cast<uint2*>(((part & 1) ? p.pkv.v : p.pkv.k) + ((size_t)(part >> 1) * p.M + m) * w + (n - part * w)) =
                  pack4(v.x, v.y, v.z, v.w);
              break;
            }
            default: {
              if (epi == EPI_BIAS_GELU) v = make_float4(gelu_tanh_f(v.x), gelu_tanh_f(v.y), gelu_tanh_f(v.z), gelu_tanh_f(v.w));
              const size_t off = (size_t)m * p.ldo + n;
              const int ns = p.n_store > 0 ? p.n_store : p.N;   // a narrow projection's padding rows are not stored
              if (!vec || n + 3 >= ns) {
                const float e[4] = {v.x, v.y, v.z, v.w};
                for (int k = 0; k < 4 && n + k < ns; ++k) {
                  if (p.out_dtype == BF16) static_cast<__nv_bfloat16*>(p.out)[off + k] = __float2bfloat16_rn(e[k]);
                  else static_cast<float*>(p.out)[off + k] = e[k];
                }
              } else if (p.out_dtype == BF16) {
                *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(p.out) + off) = pack4(v.x, v.y, v.z, v.w);
              } else {
                *reinterpret_cast<float4*>(static_cast<float*>(p.out) + off) = v;
              }
              break;
            }
          }
        }
      }
    }
    if (qkv && nt * kBM >= p.qkv.qd + p.qkv.kvd) {
      // the CTA's v values, tokens fastest over the lanes: Vt holds a head dim's keys contiguously (a 2-byte
      // store a key and dim straight from the sums: 897 us per evaluation of 18 layers at 200 tokens, so 870)
      const QkvTcOut& o = p.qkv;
      named_sync(1, kCons);   // reached by every epilogue warp, also by one whose wait ran out
      for (int tt = lane; ok && all && tt < cnt; tt += 32) {
        const int m = m0 + t0 + tt, b = m / o.H;
        __nv_bfloat16* dst = o.vtcache + (((size_t)b * o.L + o.layer) * o.kvd + (nt * kBM - o.qd - o.kvd)) * o.NKp + o.P + (m - b * o.H);
        for (int r = warp; r < kBM; r += kConsWarps)
          dst[(size_t)r * o.NKp] = __float2bfloat16_rn(T[(size_t)(t0 + tt) * kBM + ((r & ~3) ^ (4 * (tt & (kLanes - 1)))) + (r & 3)]);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  // a CTA leaves once every CTA has received its rows: until then its own are still being read
  if (S > 1) cluster_wait();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*tmem_slot), "r"(kTmCols));
  }
}

}  // namespace

// Rows of a tile and K splits (= CTAs of a cluster, at most eight).
// Rows: 64 for one tile of more than 32 tokens of a narrow projection, where eight splits of 128 rows would leave
// SMs idle: half as much to exchange, and most or all of a CTA's weights fit its ring, requested before the wait
// (18-layer expert, 50 tokens, N = 1024 and 2560: 694 -> 675 us per evaluation; two-layer time-concatenating
// one 84 -> 81). With 16 tokens the activation boxes weigh as much as the weights (16-layer DiT expert 772 with
// 128 rows, 817 with 64), with a second token tile every weight is read twice (18 layers, 100 tokens: 770, 799).
// Splits: up to 32 tokens, where a CTA's work is shorter than its start, one CTA an SM unless a split would
// sum more than 768 products (the tensor cores' accumulation truncates, so the error grows with the run); else as
// many as keep the grid near one and a half CTAs an SM, so that the next kernel's CTAs find room beside them
// and fetch their first weights early. Per evaluation, 1 / 1.5 / 1.75 CTAs an SM: DiT expert 805 / 838 / 887 us,
// its four robots 1227 / 1212 / 1321, 18-layer expert at one robot 717 / 706 / 706, four robots 957 / 900 / 897.
// With so few tiles that one CTA an SM is five splits or more, further ones pay only until a CTA's share
// fits four slots (DiT expert, N = 1536, K = 1536: six robots 1530 us with eight splits, 1312 with six; 18-layer
// expert, N = 1024, K = 2048 and 4096, four robots: 863 with eight, 878 with six); with four, none do (DiT
// expert, N = 4608, K = 1536, 64 tokens: 1089 us with six splits, 1073 with four; 144 tokens: 1770 and 1498).
void gemm_cl_plan(int M, int N, int K, int sms, TcGemmArgs* a) {
  const int mt = (M + kBN - 1) / kBN, KC = K / kBK;
  a->cl_bm = M > 32 && mt == 1 && 6 * (N / kTileM) <= sms ? 64 : 128;
  const int tiles = (N / a->cl_bm) * mt;
  const int one = (sms + tiles / 2) / tiles, half = (3 * sms + tiles) / (2 * tiles), fit = (KC + 3) / 4;
  int s = half;
  if (M <= 32 || (one == 4 && a->cl_bm == 128)) s = one;
  else if (one >= 5) s = fit < one ? one : fit < half ? fit : half;
  while (s < half && K > 768 * s) ++s;
  s = s < 1 ? 1 : s > kClMaxSplits ? kClMaxSplits : s;
  a->splits = s < KC ? s : KC;
  // Accumulators: as many as keep a run to the k-blocks that a CTA would sum if K were cut until the grid had one CTA
  // an SM (two, where that is more than four k-blocks), however few splits a cluster can have
  const int t64 = N / kTileM * mt, nkb = KC / a->splits, most = (KC + a->splits - 1) / a->splits;
  const auto run_of = [&](int ctas) { return (KC * t64 + ctas / 2) / ctas > 1 ? (KC * t64 + ctas / 2) / ctas : 1; };
  const int run = run_of(sms) <= 4 ? run_of(sms) : run_of(2 * sms) > 4 ? run_of(2 * sms) : 4;
  a->sets = most <= run || nkb < 2 ? 1 : most <= 2 * run || nkb < 4 ? 2 : 4;
}

// The cluster form serves every projection of one 64-token tile, and with more tokens those with so
// few tiles that the SMs need K splits; a projection with more tiles takes one CTA a tile (narrow form,
// gemm_tc.cu), whose epilogue it shares with nobody.
bool gemm_cl_serves(int M, int N, int sms) {
  return M <= kBN || 2 * (N / kTileM) * ((M + kBN - 1) / kBN) <= sms;
}

static size_t gemm_cl_smem_bytes(int ring, int rows, int splits, int bm) {
  return 1024 + cl_ring_bytes(ring, rows, bm) + cl_recv_bytes(rows, splits, bm) + (2 * ring + 2) * 8 + 16;
}
constexpr int kClMaxStages = 12;
constexpr size_t kClSmem = 112 * 1024;   // two CTAs fit an SM

namespace {
using ClKernel = void (*)(CUtensorMap, TcGemmArgs, int);

// One CTA's rows of the output features: BM; token rows of an activation box: BOX.
template <int BM, int BOX>
ClKernel cl_kernel(const TcGemmArgs& a) {
  const bool own = a.cl_code == kClOwn, gated = a.epi == EPI_QKV_TC || a.epi == EPI_GEGLU;
  return own && a.epi == EPI_QKV_TC ? gemm_cl_kernel<EPI_QKV_TC, BM, BOX>
         : own && a.epi == EPI_GEGLU ? gemm_cl_kernel<EPI_GEGLU, BM, BOX>
         : own && a.epi == EPI_RESID_H ? gemm_cl_kernel<EPI_RESID_H, BM, BOX>
         : a.cl_code == kClPlain && !gated ? gemm_cl_kernel<kPlain, BM, BOX> : gemm_cl_kernel<kAny, BM, BOX>;
}
template <int BM, int BOX>
int cl_prepare() {
  for (const auto k : {gemm_cl_kernel<kAny, BM, BOX>, gemm_cl_kernel<kPlain, BM, BOX>, gemm_cl_kernel<EPI_QKV_TC, BM, BOX>,
                       gemm_cl_kernel<EPI_GEGLU, BM, BOX>, gemm_cl_kernel<EPI_RESID_H, BM, BOX>})
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClSmem) != cudaSuccess) return -1;
  return 0;
}
}  // namespace

int gemm_cl_prepare() { return cl_prepare<128, 64>() || cl_prepare<128, 16>() || cl_prepare<64, 64>() ? -1 : 0; }

void launch_gemm_cl(const CUtensorMap* tmx, const TcGemmArgs& a, cudaStream_t s) {
  const int KC = a.K / kBK, per = (KC + a.splits - 1) / a.splits, rows = a.M < kBN ? a.M : kBN;
  int ring = per < kClMaxStages ? per : kClMaxStages;
  while (gemm_cl_smem_bytes(ring, rows, a.splits, a.cl_bm) > kClSmem) --ring;   // three slots at least
  launch_cluster(a.cl_bm == 64 ? cl_kernel<64, 64>(a) : act_box_rows(a.M) == 16 ? cl_kernel<128, 16>(a) : cl_kernel<128, 64>(a), dim3(a.splits, a.N / a.cl_bm, (a.M + kBN - 1) / kBN),
                 dim3(kThreads), gemm_cl_smem_bytes(ring, rows, a.splits, a.cl_bm), a.splits, s, *tmx, a, ring | a.sets << 8);
}

}  // namespace uad
