// Tensor-core attention of chunk queries over [prefix keys ; chunk keys] (grouped KV heads),
// for bf16 experts with joint attention over the observation prefix.
//
// Layouts (written by the QKV projection epilogue and, for the prefix, by set_prefix):
//   Q  [B][Hkv][G][H][dh]       queries of one KV group are the R = G*H rows of one matrix
//   K  [B][L][Hkv][NK][dh]      keys: P prefix rows then H chunk rows (NK = P + H)
//   Vt [B][L][Hkv][dh][NKp]     values transposed (keys contiguous), NKp = NK rounded up to 8
// Few query tiles (split-KV): one CTA = one 128-row query tile x one 128-key chunk of one
//   (robot, group): TMA loads Q, K, Vt tiles (128-byte swizzle); S = Q K^T on tcgen05 into TMEM;
//   four warps read S rows, apply the 1/sqrt(dh) scale and key mask, write P = exp(S - rowmax) in
//   bf16 into shared memory in the K-major swizzled layout; O = P Vt^T on tcgen05; O rows
//   (unnormalised) and per-row (max, sum) go to a workspace. attn_combine merges the key chunks
//   (the usual log-sum-exp rescaling) and writes o [B*H][Hq*dh] in bf16 for the O projection.
// Many query tiles (attn_tc2_kernel): one CTA per query tile walks all key chunks in one pass,
//   O accumulating in TMEM, and writes o itself; with at most half as many tiles as SMs, two CTAs
//   per tile, one per half of the head dims.
#include <cuda.h>
#include <cudaTypedefs.h>

#include "uad_internal.cuh"
#include "attn_ring.cuh"
#include "ptx.cuh"

namespace uad {

using namespace ptx;

namespace {

constexpr int kQT = 128, kKT = 128;
constexpr int kMaxKeyChunks = 16;   // keys per (robot, layer) <= 2048
constexpr uint32_t kTmemCols = 256; // S (128 columns) then O (dh <= 256 columns) in the same columns
constexpr unsigned long long kWaitNs = 2000000000ull;

__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, int* err, int code) {
  return ptx::mbar_wait(b, parity, err, code, kWaitNs);
}
__device__ __forceinline__ float ex2_fast(float x) { return ptx::ex2_approx(x); }


// smem plan for head dim dh: Q tiles (dh/64 blocks of 128 x 64), K tiles (same), Vt tiles
// (2 blocks of dh x 64 keys), P (2 blocks of 128 x 64, aliased on Q when Q is >= 32 KB).
__host__ __device__ __forceinline__ size_t attn_q_bytes(int dh) { return (size_t)dh * kQT * 2; }
__host__ __device__ __forceinline__ size_t attn_p_extra(int dh) { return attn_q_bytes(dh) >= 32768 ? 0 : 32768; }

// DV = head dims of O per CTA: DH, or a half or a quarter of it while the grid stays within the SMs (each CTA
// computes S and P in full, and P V and its partial rows for its dims only): the loads of V, the readout of O
// and the partial rows written shrink with it, the scores are computed by CTAs that would be idle.
template <int DH, int DV>
__global__ void __launch_bounds__(128, 1) attn_tc_kernel(const __grid_constant__ CUtensorMap tq,
                                                         const __grid_constant__ CUtensorMap tk,
                                                         const __grid_constant__ CUtensorMap tv, AttnTcArgs p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  constexpr int NC = DH / 64;
  constexpr uint32_t QB = DH * kQT * 2, KB = DH * kKT * 2, VB = DV * kKT * 2, VBLK = DV * 128;
  uint8_t* sQ = smem;
  uint8_t* sK = sQ + QB;
  uint8_t* sV = sK + KB;
  uint8_t* sP = attn_p_extra(DH) ? sV + VB : sQ;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sV + VB + attn_p_extra(DH));
  uint64_t *bar_qk = bars, *bar_v = bars + 1, *bar_s = bars + 2, *bar_o = bars + 3;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 4);

  constexpr int SP = DH / DV;
  const int qt = blockIdx.x / SP, d0 = blockIdx.x % SP * DV, kc = blockIdx.y, bg = blockIdx.z;   // bg = b * Hkv + g
  const int b = bg / p.n_kv_heads, g = bg % p.n_kv_heads;
  const int kvz = (b * p.n_layers + p.layer) * p.n_kv_heads + g;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int i = 0; i < 4; ++i) mbar_init(bars + i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)), "r"(kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // S occupies columns [0, 128); O = P V reuses columns [0, DH) once every thread has read S
  const uint32_t tS = tmem, tO = tmem;
  pdl_trigger();

  if (threadIdx.x == 0) {
    // a chunk of prefix keys alone, which no kernel of the step loop writes, is loaded before the wait for the
    // kernel that writes Q and the chunk's keys
    const uint64_t pol = policy_evict_last();
    const bool early = (kc + 1) * kKT <= p.prefix;
    if (!early) pdl_wait();
    mbar_expect_tx(bar_qk, QB + KB);
#pragma unroll
    for (int c = 0; c < NC; ++c) tma_3d(sK + c * (kKT * 128), &tk, c * 64, kc * kKT, kvz, bar_qk, pol);
    mbar_expect_tx(bar_v, VB);
#pragma unroll
    for (int u = 0; u < kKT / 64; ++u) tma_3d(sV + u * VBLK, &tv, kc * kKT + u * 64, d0, kvz, bar_v, pol);
    if (early) pdl_wait();
#pragma unroll
    for (int c = 0; c < NC; ++c) tma_3d(sQ + c * (kQT * 128), &tq, c * 64, qt * kQT, bg, bar_qk, pol);
  } else if (threadIdx.x == 32) {
    if (mbar_wait(bar_qk, 0, p.err, 21)) {
      tc_fence_after();
      const uint64_t qd = sw128_desc(su32(sQ)), kd = sw128_desc(su32(sK));
#pragma unroll
      for (int c = 0; c < NC; ++c)
        mma_kblock(tS, qd + c * (kQT * 128 >> 4), kd + c * (kKT * 128 >> 4), idesc_m128(kKT), c ? 1u : 0u);
    } else {
      mbar_drain_issued(bar_qk, 0);   // no copies in flight into shared memory of an exiting CTA
    }
    mma_commit(bar_s);
  }
  __syncwarp();

  // ---- softmax over this key chunk: one query row per thread. Warps 2 and 3, which have nothing to do until
  //      the scores are there, first go through it once (on whatever tensor memory holds, storing nothing): that
  //      brings its code, run once a CTA, into the SM's instruction cache. 18 layers, 180 tokens: 862 -> 854 us per
  //      evaluation ----
  const int row = warp * 32 + lane;
  const uint32_t lane_base = (uint32_t)(warp * 32) << 16;
  const float c2 = p.scale_log2;             // log2(e) / sqrt(dh)
  const int key0 = kc * kKT;
  const int nv = p.n_keys - key0;            // valid keys of the chunk (all of them but in the last)
  const int r8 = row & 7;
  float sv[kKT];                             // the chunk's scores of this row, one wait for all
  float mx, l;
  bool ok_s = false;
#pragma unroll 1
  for (int pass = warp >= 2 ? 0 : 1; pass < 2; ++pass) {
    if (pass) {
      pdl_wait();
      ok_s = mbar_wait(bar_s, 0, p.err, 22);
      tc_fence_after();
    }
    __syncwarp();
    tmem_ld128(tS + lane_base, sv);
    if (nv < kKT) {   // keys past the end (last chunk): excluded from the maximum, P = 2^-inf = 0
#pragma unroll
      for (int i = 0; i < kKT; ++i)
        if (i >= nv) sv[i] = -INFINITY;
    }
    mx = -INFINITY;
#pragma unroll
    for (int i = 0; i < kKT; ++i) mx = fmaxf(mx, sv[i]);
    const float ms = mx * c2;
    l = 0.f;
#pragma unroll
    for (int cc = 0; cc < kKT / 32; ++cc) {
      uint32_t pk[16];
#pragma unroll
      for (int i = 0; i < 32; i += 2) {
        const int k = cc * 32 + i;
        const float e0 = ex2_fast(fmaf(sv[k], c2, -ms)), e1 = ex2_fast(fmaf(sv[k + 1], c2, -ms));
        const __nv_bfloat162 h = __floats2bfloat162_rn(e0, e1);
        const float2 hf = __bfloat1622float2(h);
        l += hf.x + hf.y;   // normalise by what the MMA actually sums
        pk[i / 2] = *reinterpret_cast<const uint32_t*>(&h);
      }
      // 32 keys = four 16-byte granules of row `row` in P block (cc / 2), granules (cc % 2) * 4 + q
      uint8_t* prow = sP + (cc / 2) * (kQT * 128) + row * 128;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int gidx = (cc % 2) * 4 + q;
        if (pass) *reinterpret_cast<uint4*>(prow + ((gidx ^ r8) * 16)) = make_uint4(pk[4 * q], pk[4 * q + 1], pk[4 * q + 2], pk[4 * q + 3]);
      }
    }
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  tc_fence_before();
  __syncthreads();

  if (threadIdx.x == 32) {
    tc_fence_after();
    if (ok_s && mbar_wait(bar_v, 0, p.err, 23)) {
      const uint64_t pd = sw128_desc(su32(sP)), vd = sw128_desc(su32(sV));
#pragma unroll
      for (int u = 0; u < kKT / 64; ++u)
        mma_kblock(tO, pd + u * (kQT * 128 >> 4), vd + u * (VBLK >> 4), idesc_m128(DV), u ? 1u : 0u);
    } else {
      mbar_drain_issued(bar_v, 0);
    }
    mma_commit(bar_o);
  }
  __syncwarp();
  const bool ok_o = mbar_wait(bar_o, 0, p.err, 24);
  if (!ok_o) mbar_drain_issued(bar_o, 0);   // nor MMAs, once tensor memory is given back
  tc_fence_after();

  // ---- partial output row (unnormalised) + (max, sum): the row is staged in shared memory (all
  //      operand tiles are free once O is complete; rows padded by 16 bytes against bank
  //      conflicts) and written with one 1-KB bulk copy per row ----
  const int qrow = qt * kQT + row;
  const size_t prow_idx = ((size_t)bg * gridDim.y + kc) * p.r_pad + qrow;
  constexpr uint32_t pitch = DV * 4 + 16;
  uint8_t* srow = smem + (size_t)row * pitch;
  __syncwarp();
#pragma unroll 1
  for (int cc = 0; cc < DV / 32; ++cc) {
    tmem_ld32(tO + lane_base + cc * 32, sv);
#pragma unroll
    for (int i = 0; i < 32; i += 4)
      *reinterpret_cast<float4*>(srow + (cc * 32 + i) * 4) = make_float4(sv[i], sv[i + 1], sv[i + 2], sv[i + 3]);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (ok_o && qrow < p.rows) {
    bulk_s2g(p.part_o + prow_idx * DH + d0, srow, DV * 4);
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    if (d0 == 0) {
      p.part_ml[prow_idx * 2] = mx;
      p.part_ml[prow_idx * 2 + 1] = l;
    }
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
}

// ---- one-pass attention for many query tiles: no partials, no combine ---------------------
// One CTA per (128-row query tile, robot-group), keys in chunks of 128 (S = Q K^T with MMA
// N = 128). Shared memory: Q and a ring of five operand slots that take, in the order the MMAs
// read them, each chunk's K in head-dim pieces and its Vt in two 64-key halves; a slot is refilled
// as soon as the MMAs that read it are done, so the next chunk's operands load while S and P V of
// this one run. Per chunk: S on tcgen05 (double-buffered in TMEM), then each softmax thread (one
// query row) forms P = exp(S - M) in bf16 against its running maximum M and writes it into tensor
// memory over the S it came from, and O += P V accumulates in TMEM with P as the MMA's A operand
// from tensor memory (P is double-buffered with S). The issuer issues S of chunk c + 1 before
// P V of chunk c, so that it runs while the softmax of chunk c does. M is raised only when the
// chunk's maximum exceeds it by more than 2^8 in the exponent; the O row and the row sum are then
// rescaled in place (after the previous P V has completed). Otherwise the stale M stays: every P
// is at most 2^8, and O and the row sum share the same reference, so O / sum is unchanged. O / l
// is written in bf16.
constexpr int kKC2 = kRingChunk;                // keys per chunk
constexpr uint32_t kTmem2 = 512;                // S buffers at columns [0,128) and [128,256), O at [256, 256 + DV)
constexpr float kRescaleLog2 = 8.f;             // raise M only past this many powers of two
constexpr int kSlots2 = 5;                      // operand ring slots
constexpr int kBars2 = 9 + 2 * kSlots2;         // mbarriers of the kernel
__host__ __device__ constexpr int attn2_kpieces(int dh) { return dh >= 128 ? 2 : 1; }
// ring slot bytes: a K piece (128 keys x dh / pieces) or a Vt half (dh x 64 keys), the larger
__host__ __device__ constexpr uint32_t attn2_slot_bytes(int dh) {
  return (uint32_t)(dh / attn2_kpieces(dh)) * kKC2 * 2 > (uint32_t)dh * 128 ? (uint32_t)(dh / attn2_kpieces(dh)) * kKC2 * 2
                                                                           : (uint32_t)dh * 128;
}

// Warps 0-3: softmax and output (they own the four TMEM lane quadrants); warp 4: TMA producer;
// warp 5: MMA issuer. The producer and issuer wait on the softmax warps' progress, so they must
// not share a warp with them. DV = head dims of O per CTA: DH, or DH / 2 when the query tiles are
// at most half as many as the SMs (two CTAs per tile, blockIdx.z = which half of the head dims;
// each computes S and P in full, and P V and the output for its half only).
template <int DH, int DV>
__global__ void __launch_bounds__(192, 1) attn_tc2_kernel(const __grid_constant__ CUtensorMap tq,
                                                          const __grid_constant__ CUtensorMap tk,
                                                          const __grid_constant__ CUtensorMap tv, AttnTcArgs p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  constexpr int NC = DH / 64;
  constexpr int KP = attn2_kpieces(DH);          // K pieces per chunk
  constexpr int NCP = NC / KP;                   // 64-dim blocks of 128 keys per piece
  constexpr uint32_t QB = DH * kQT * 2;          // Q: NC blocks of 128 rows x 64
  constexpr uint32_t PB = NCP * kKC2 * 128;      // one K piece
  constexpr uint32_t VBLK = DV * 128;            // one Vt half: DV rows x 64 keys
  constexpr uint32_t SLOT = attn2_slot_bytes(DH);
  uint8_t* sQ = smem;
  uint8_t* sR = sQ + QB;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sR + kSlots2 * SLOT);
  uint64_t* q_full = bars;          // Q landed
  uint64_t* s_full = bars + 1;      // [2] S buffer written
  uint64_t* s_empty = bars + 3;     // [2] S / P buffer free (the P V that read its P is done)
  uint64_t* p_full = bars + 5;      // [2] P of the S buffer written (and O rescaled) by the 4 warps
  uint64_t* p_empty = bars + 7;     // P V done: O complete up to this chunk
  uint64_t* o_done = bars + 8;
  uint64_t* r_full = bars + 9;            // [kSlots2] ring slot loaded
  uint64_t* r_empty = r_full + kSlots2;   // [kSlots2] ring slot free (the MMAs that read it are done)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kBars2);

  const int qt = blockIdx.x, bg = blockIdx.y, d0 = blockIdx.z * DV;
  const int b = bg / p.n_kv_heads, g = bg % p.n_kv_heads;
  const int kvz = (b * p.n_layers + p.layer) * p.n_kv_heads + g;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nck = (p.n_keys + kKC2 - 1) / kKC2;

  if (threadIdx.x == 0) {
    mbar_init(q_full, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(s_full + i, 1);
      mbar_init(s_empty + i, 1);
      mbar_init(p_full + i, 4);
    }
    for (int i = 0; i < kSlots2; ++i) {
      mbar_init(r_full + i, 1);
      mbar_init(r_empty + i, 1);
    }
    mbar_init(p_empty, 1);
    mbar_init(o_done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)), "r"(kTmem2));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t tO = tmem + 2 * kKC2;
  pdl_trigger();

  const AttnRing ring{KP, nck};   // its entries, in the order the MMAs read them

  if (threadIdx.x == 128) {
    // producer: ring entry e into slot e % kSlots2 once entry e - kSlots2 has been read. The first entries that
    // hold prefix keys alone, which no kernel of the step loop writes, are requested before the wait for the
    // kernel that writes Q and the chunk's keys (not always the whole ring: with one K piece a chunk, head
    // dim 64, its fifth entry is K of chunk 2)
    const uint64_t pol = policy_evict_last();
    const int total = ring.total();
    const auto load = [&](int e) {
      const int t = e % kSlots2;
      const AttnRing::Entry x = ring.at(e);
      if (x.k) {
        mbar_expect_tx(r_full + t, PB);
#pragma unroll
        for (int cc = 0; cc < NCP; ++cc)
          tma_3d(sR + t * SLOT + cc * (kKC2 * 128), &tk, (x.part * NCP + cc) * 64, x.chunk * kKC2, kvz, r_full + t, pol);
      } else {
        mbar_expect_tx(r_full + t, VBLK);
        tma_3d(sR + t * SLOT, &tv, x.chunk * kKC2 + x.part * 64, d0, kvz, r_full + t, pol);
      }
    };
    int e = 0;
    for (const int n = ring.early(kSlots2, p.prefix); e < n; ++e) load(e);
    pdl_wait();
    mbar_expect_tx(q_full, QB);
#pragma unroll
    for (int c = 0; c < NC; ++c) tma_3d(sQ + c * (kQT * 128), &tq, c * 64, qt * kQT, bg, q_full, pol);
    for (; e < total; ++e) {
      if (e >= kSlots2 && !mbar_wait(r_empty + e % kSlots2, (e / kSlots2 - 1) & 1, p.err, 41)) break;
      load(e);
    }
    // do not leave copies in flight into shared memory of an exiting CTA
    mbar_drain_issued(q_full, 0);
    for (int i = e - kSlots2 > 0 ? e - kSlots2 : 0; i < e; ++i) mbar_drain_issued(r_full + i % kSlots2, (i / kSlots2) & 1);
  } else if (threadIdx.x == 160) {
    // issuer: S(0); per chunk c: S(c + 1), then P V(c) once the softmax warps have written P(c)
    bool ok = mbar_wait(q_full, 0, p.err, 42);
    const uint64_t qdesc = sw128_desc(su32(sQ)), rdesc = sw128_desc(su32(sR));
    const auto issue_s = [&](int c) {
      const int sb = c & 1;
      if (c >= 2) ok = mbar_wait(s_empty + sb, ((c >> 1) - 1) & 1, p.err, 44);
      for (int j = 0; j < KP && ok; ++j) {
        const int e = ring.k_entry(c, j), t = e % kSlots2;
        ok = mbar_wait(r_full + t, (e / kSlots2) & 1, p.err, 43);
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int cc = 0; cc < NCP; ++cc)
          mma_kblock(tmem + sb * kKC2, qdesc + (uint64_t)((j * NCP + cc) * (kQT * 128 >> 4)),
                     rdesc + (uint64_t)(t * (SLOT >> 4) + cc * (kKC2 * 128 >> 4)), idesc_m128(kKC2), (j | cc) ? 1u : 0u);
        mma_commit(r_empty + t);
      }
      if (ok) mma_commit(s_full + sb);
    };
    if (ok) issue_s(0);
    for (int ch = 0; ch < nck && ok; ++ch) {
      const int sb = ch & 1;
      if (ch + 1 < nck) issue_s(ch + 1);
      ok = ok && mbar_wait(p_full + sb, (ch >> 1) & 1, p.err, 45);
      for (int h = 0; h < 2 && ok; ++h) {
        const int e = ring.v_entry(ch, h), t = e % kSlots2;
        ok = mbar_wait(r_full + t, (e / kSlots2) & 1, p.err, 46);
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int k = 0; k < 4; ++k)
          mma_bf16_ts(tO, tmem + sb * kKC2 + 8 * (4 * h + k), rdesc + (uint64_t)(t * (SLOT >> 4) + 2 * k), idesc_m128(DV),
                      (ch | h | k) ? 1u : 0u);
        mma_commit(r_empty + t);
      }
      if (!ok) break;
      mma_commit(p_empty);
      mma_commit(s_empty + sb);
    }
    mma_commit(o_done);
    mbar_drain_issued(o_done, 0);   // before tensor memory is given back
  }
  if (warp >= 4) {
    // producer / issuer warps: done issuing; wait for the output stage before releasing TMEM
    __syncthreads();
    return;
  }

  // ---- softmax warps: one query row per thread ----
  pdl_wait();
  const int row = warp * 32 + lane;
  const uint32_t lane_base = (uint32_t)(warp * 32) << 16;
  const float c2s = p.scale_log2;
  float sv[kKC2];                    // the chunk's scores of this row
  float mref = -INFINITY, l = 0.f;   // the row's reference maximum and sum of P
  bool ok = true;
  for (int ch = 0; ch < nck; ++ch) {
    const int sb = ch & 1;
    const int key0 = ch * kKC2;
    const int nv = p.n_keys - key0;   // valid keys of the chunk (all of them but in the last)
    ok = ok && mbar_wait(s_full + sb, (ch >> 1) & 1, p.err, 47);
    tc_fence_after();
    __syncwarp();
    tmem_ld128(tmem + sb * kKC2 + lane_base, sv);
    if (nv < kKC2) {   // keys past the end (last chunk): excluded from the maximum, P = 2^-inf = 0
#pragma unroll
      for (int i = 0; i < kKC2; ++i)
        if (i >= nv) sv[i] = -INFINITY;
    }
    float mx[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) mx[j] = sv[j];
#pragma unroll
    for (int i = 8; i < kKC2; ++i) mx[i & 7] = fmaxf(mx[i & 7], sv[i]);
    const float mc = fmaxf(fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])), fmaxf(fmaxf(mx[4], mx[5]), fmaxf(mx[6], mx[7])));
    // raise the reference past 2^8 (and at the first chunk); the previous P V must have completed
    // before O is touched (P goes to this chunk's own buffer, free since S landed in it)
    const bool raise = ch == 0 ? true : (mc - mref) * c2s > kRescaleLog2;
    const float factor = ch == 0 ? 1.f : (raise ? exp2f((mref - mc) * c2s) : 1.f);
    if (__any_sync(0xffffffffu, ch > 0 && raise)) {
      ok = ok && mbar_wait(p_empty, (ch - 1) & 1, p.err, 48);
      tc_fence_after();
      float ov[32];
#pragma unroll 1
      for (int cc = 0; cc < DV / 32; ++cc) {
        tmem_ld32(tO + lane_base + cc * 32, ov);
#pragma unroll
        for (int i = 0; i < 32; ++i) ov[i] *= factor;
        tmem_st32(tO + lane_base + cc * 32, ov);
      }
    }
    if (raise) {
      l *= factor;
      mref = mc;
    }
    const float ms = mref * c2s;
    float la = 0.f, lb = 0.f;
#pragma unroll
    for (int cc = 0; cc < kKC2 / 32; ++cc) {
      uint32_t pk[16];
#pragma unroll
      for (int i = 0; i < 32; i += 2) {
        const int k = cc * 32 + i;
        const float e0 = ex2_fast(fmaf(sv[k], c2s, -ms)), e1 = ex2_fast(fmaf(sv[k + 1], c2s, -ms));
        const __nv_bfloat162 h = __floats2bfloat162_rn(e0, e1);
        const float2 hf = __bfloat1622float2(h);
        la += hf.x;   // normalise by what the MMA sums
        lb += hf.y;
        pk[i / 2] = *reinterpret_cast<const uint32_t*>(&h);
      }
      // keys 32 cc .. 32 cc + 31 -> columns 16 cc .. + 15 of the chunk's S buffer (its scores are
      // in registers)
      tmem_st16_nowait(tmem + sb * kKC2 + lane_base + 16 * cc, pk);
    }
    l += la + lb;
    tmem_wait_st();
    // (p_full of this S buffer completes again only after S of chunk ch + 2, which the issuer
    // issues after its wait for this phase)
    tc_fence_before();
    __syncwarp();
    if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(p_full + sb)) : "memory");
  }
  float sv32[32];
  ok = ok && mbar_wait(o_done, 0, p.err, 49);
  tc_fence_after();
  __syncwarp();

  // ---- o = O / l in bf16, row (j, i) of this tile -> o[(b*H + i)][(g*G + j)*dh + d] ----
  const int qrow = qt * kQT + row;
  const float inv = 1.f / l;
  const int jj = qrow / p.H, ii = qrow % p.H;
  __nv_bfloat16* orow = p.out + ((size_t)b * p.H + ii) * p.out_ld + (size_t)(g * p.group + jj) * DH + d0;
#pragma unroll
  for (int cc = 0; cc < DV / 32; ++cc) {
    tmem_ld32(tO + lane_base + cc * 32, sv32);
    if (ok && qrow < p.rows) {
#pragma unroll
      for (int i = 0; i < 32; i += 8) {
        uint4 w;
        w.x = pack_bf16(sv32[i] * inv, sv32[i + 1] * inv);
        w.y = pack_bf16(sv32[i + 2] * inv, sv32[i + 3] * inv);
        w.z = pack_bf16(sv32[i + 4] * inv, sv32[i + 5] * inv);
        w.w = pack_bf16(sv32[i + 6] * inv, sv32[i + 7] * inv);
        *reinterpret_cast<uint4*>(orow + cc * 32 + i) = w;
      }
    }
  }
  tc_fence_before();
  __syncthreads();   // pairs with the producer / issuer warps' final barrier
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmem2));
}

// Merge the key chunks of every query row: o = sum_c w_c O_c / sum_c w_c l_c, w_c = 2^((m_c - M) c2).
// A thread owns four head dims of one row, a CTA of 256 threads 1024 / DH rows, so that the whole grid starts
// at once and the next kernel's CTAs can come in beside it (one row a CTA of 128 threads held them back);
// every partial is loaded before any arithmetic. 18 layers, 400 rows of 256, 7 chunks: 717 -> 703 us per evaluation.
// Writes o [(b*H + i)][(g*G + j)*dh + d] in bf16.
__global__ void __launch_bounds__(256) attn_combine_kernel(AttnTcArgs p, int n_chunks) {
  constexpr int MAXC = kMaxKeyChunks;
  pdl_trigger();
  const int DH = p.head_dim, tpr = DH / 4, r = blockIdx.x * (256 / tpr) + threadIdx.x / tpr, bg = blockIdx.y;
  const int d = 4 * (threadIdx.x % tpr);
  if (r >= p.rows) return;
  const int b = bg / p.n_kv_heads, g = bg % p.n_kv_heads;
  pdl_wait();
  float m[MAXC], l[MAXC];
  float4 o[MAXC];
#pragma unroll
  for (int c = 0; c < MAXC; ++c) {
    if (c < n_chunks) {
      const size_t idx = ((size_t)bg * n_chunks + c) * p.r_pad + r;
      m[c] = p.part_ml[idx * 2];
      l[c] = p.part_ml[idx * 2 + 1];
      o[c] = *reinterpret_cast<const float4*>(p.part_o + idx * DH + d);
    }
  }
  float M = -INFINITY;
#pragma unroll
  for (int c = 0; c < MAXC; ++c)
    if (c < n_chunks) M = fmaxf(M, m[c]);
  float L = 0.f;
  float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int c = 0; c < MAXC; ++c) {
    if (c < n_chunks) {
      const float w = exp2f((m[c] - M) * p.scale_log2);
      L = fmaf(w, l[c], L);
      a.x = fmaf(w, o[c].x, a.x);
      a.y = fmaf(w, o[c].y, a.y);
      a.z = fmaf(w, o[c].z, a.z);
      a.w = fmaf(w, o[c].w, a.w);
    }
  }
  const int j = r / p.H, i = r % p.H;
  *reinterpret_cast<uint2*>(p.out + ((size_t)b * p.H + i) * p.out_ld + (size_t)(g * p.group + j) * DH + d) =
      make_uint2(pack_bf16(a.x / L, a.y / L), pack_bf16(a.z / L, a.w / L));
}

// Prefix K/V of one robot (fp32 or bf16 source [L][P][Hkv][dh], 16-byte aligned) into the K and Vt
// caches. CTA = 64 positions x 64 head dims of one (layer, KV head): 16-byte loads and K stores, the
// V tile transposed in shared memory so that Vt goes out as 16-byte runs of eight keys. Bound by the
// bytes in and out (pi0-like, bf16: 15 MB each way); writing Vt element by element instead put every
// 2 bytes of a warp into a row of its own. With the caller's device buffer read in place and no
// allocation in the call, binding a pi0-like observation went from 278 to 31 us.
constexpr int kPfTile = 64, kPfPitch = kPfTile + 2;   // pitch 33 words: both sides of the transposition spread over the banks
template <int SRC>
__global__ void __launch_bounds__(256) kv_prefix_kernel(const void* __restrict__ k, const void* __restrict__ v,
                                                        AttnTcArgs p, int robot) {
  __shared__ __align__(4) __nv_bfloat16 t[kPfTile * kPfPitch];
  const int l = blockIdx.x / p.n_kv_heads, g = blockIdx.x % p.n_kv_heads, d0 = blockIdx.y * kPfTile, p0 = blockIdx.z * kPfTile;
  const int dh = p.head_dim, tid = threadIdx.x, a = tid >> 3, o = tid & 7;
  const size_t z = ((size_t)robot * p.n_layers + l) * p.n_kv_heads + g;
#pragma unroll
  for (int i = 0; i < kPfTile / 32; ++i) {
    const int pos = a + 32 * i, pp = p0 + pos;
    if (pp >= p.prefix) break;
    const size_t e = (((size_t)l * p.prefix + pp) * p.n_kv_heads + g) * dh + d0 + 8 * o;
    uint4 kk, vv;
    if constexpr (SRC == BF16) {
      kk = *reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(k) + e);
      vv = *reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(v) + e);
    } else {
      const float4* kf = reinterpret_cast<const float4*>(static_cast<const float*>(k) + e);
      const float4* vf = reinterpret_cast<const float4*>(static_cast<const float*>(v) + e);
      const float4 k0 = kf[0], k1 = kf[1], v0 = vf[0], v1 = vf[1];
      kk = make_uint4(pack_bf16(k0.x, k0.y), pack_bf16(k0.z, k0.w), pack_bf16(k1.x, k1.y), pack_bf16(k1.z, k1.w));
      vv = make_uint4(pack_bf16(v0.x, v0.y), pack_bf16(v0.z, v0.w), pack_bf16(v1.x, v1.y), pack_bf16(v1.z, v1.w));
    }
    *reinterpret_cast<uint4*>(p.kcache + (z * p.n_keys + pp) * dh + d0 + 8 * o) = kk;
    const __nv_bfloat16* ve = reinterpret_cast<const __nv_bfloat16*>(&vv);
#pragma unroll
    for (int q = 0; q < 8; ++q) t[(8 * o + q) * kPfPitch + pos] = ve[q];
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kPfTile / 32; ++i) {
    const int d = a + 32 * i, pp = p0 + 8 * o;
    __nv_bfloat16* dst = p.vtcache + (z * dh + d0 + d) * p.nk_pad + pp;
    const __nv_bfloat16* src = t + d * kPfPitch + 8 * o;
    if (pp + 8 <= p.prefix) {
      const uint32_t* w = reinterpret_cast<const uint32_t*>(src);
      *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
    } else {
      for (int q = 0; pp + q < p.prefix; ++q) dst[q] = src[q];   // the chunk's keys follow
    }
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* q = nullptr;
    cudaDriverEntryPointQueryResult r;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &q, 12000, cudaEnableDefault, &r) ==
            cudaSuccess && r == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(q);
  }
  return fn;
}

int tmap3(CUtensorMap* m, const void* base, uint64_t d0, uint64_t d1, uint64_t d2, uint64_t s1, uint64_t s2,
          uint32_t b0, uint32_t b1) {
  auto enc = encoder();
  if (!enc) return -1;
  const cuuint64_t dims[3] = {d0, d1, d2};
  const cuuint64_t strides[2] = {s1, s2};
  const cuuint32_t box[3] = {b0, b1, 1};
  const cuuint32_t es[3] = {1, 1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS ? 0 : -2;
}

}  // namespace

size_t attn_tc2_smem_bytes(int dh) {
  return 1024 + (size_t)dh * kQT * 2 + (size_t)kSlots2 * attn2_slot_bytes(dh) + (kBars2 + 1) * 8;
}

bool attn_tc_use_two_pass(const AttnTcArgs& a) {
  const int tiles = (a.rows + kQT - 1) / kQT * a.batch * a.n_kv_heads;
  return tiles >= 64;
}

size_t attn_tc_smem_bytes(int dh) {
  const size_t tiles = 3 * attn_q_bytes(dh) + attn_p_extra(dh);
  const size_t ostage = (size_t)kQT * (dh * 4 + 16);   // O rows staged over the free operand tiles
  return 1024 + (tiles > ostage ? tiles : ostage) + 4 * 8 + 16;
}

int attn_tc_prepare(AttnTcMaps* maps, const AttnTcArgs& a, int batch_max) {
  const int dh = a.head_dim;
  const uint64_t R = a.rows, NK = a.n_keys, NKp = a.nk_pad;
  if (tmap3(&maps->q, a.q, dh, R, (uint64_t)batch_max * a.n_kv_heads, (uint64_t)dh * 2, R * dh * 2, 64, kQT)) return -1;
  if (tmap3(&maps->k, a.kcache, dh, NK, (uint64_t)batch_max * a.n_layers * a.n_kv_heads, (uint64_t)dh * 2,
            NK * dh * 2, 64, kKT)) return -1;
  if (tmap3(&maps->vt, a.vtcache, NK, dh, (uint64_t)batch_max * a.n_layers * a.n_kv_heads, NKp * 2,
            (uint64_t)dh * NKp * 2, 64, (uint32_t)dh)) return -1;
  // 64-key K boxes for the persistent step kernel's attention items; the one-pass kernel loads
  // 128-key K chunks through `k` and Vt in 64-key boxes
  if (tmap3(&maps->k2, a.kcache, dh, NK, (uint64_t)batch_max * a.n_layers * a.n_kv_heads, (uint64_t)dh * 2,
            NK * dh * 2, 64, 64)) return -1;
  // Vt boxes of half the head dims (the kernels' split forms) and of a quarter
  maps->vt4 = maps->vt;
  if (dh == 256 && tmap3(&maps->vt4, a.vtcache, NK, dh, (uint64_t)batch_max * a.n_layers * a.n_kv_heads, NKp * 2,
                         (uint64_t)dh * NKp * 2, 64, (uint32_t)dh / 4)) return -1;
  if (dh >= 128) {
    if (tmap3(&maps->vt2, a.vtcache, NK, dh, (uint64_t)batch_max * a.n_layers * a.n_kv_heads, NKp * 2,
              (uint64_t)dh * NKp * 2, 64, (uint32_t)dh / 2)) return -1;
  } else {
    maps->vt2 = maps->vt;
  }
  const int smem2 = (int)attn_tc2_smem_bytes(dh);
  if (dh == 64) cudaFuncSetAttribute(attn_tc2_kernel<64, 64>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem2);
  if (dh == 128) {
    cudaFuncSetAttribute(attn_tc2_kernel<128, 128>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem2);
    cudaFuncSetAttribute(attn_tc2_kernel<128, 64>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem2);
  }
  if (dh == 256) {
    cudaFuncSetAttribute(attn_tc2_kernel<256, 256>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem2);
    cudaFuncSetAttribute(attn_tc2_kernel<256, 128>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem2);
  }
  const int smem = (int)attn_tc_smem_bytes(dh);
  const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
  if (dh == 64) cudaFuncSetAttribute(attn_tc_kernel<64, 64>, at, smem);
  if (dh == 128) {
    cudaFuncSetAttribute(attn_tc_kernel<128, 128>, at, smem);
    cudaFuncSetAttribute(attn_tc_kernel<128, 64>, at, smem);
  }
  if (dh == 256) {
    cudaFuncSetAttribute(attn_tc_kernel<256, 256>, at, smem);
    cudaFuncSetAttribute(attn_tc_kernel<256, 128>, at, smem);
    cudaFuncSetAttribute(attn_tc_kernel<256, 64>, at, smem);
  }
  return 0;
}

int attn_tc_chunks(int n_keys) { return (n_keys + kKT - 1) / kKT; }
int attn_tc_max_keys() { return kMaxKeyChunks * kKT; }
int attn_tc_rpad(int rows) { return (rows + kQT - 1) / kQT * kQT; }

void launch_attn_tc(const AttnTcMaps& maps, const AttnTcArgs& a, cudaStream_t s) {
  if (attn_tc_use_two_pass(a)) {
    const int tiles = (a.rows + kQT - 1) / kQT * a.batch * a.n_kv_heads;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const bool split = a.head_dim >= 128 && 2 * tiles <= sms;
    dim3 grid2((a.rows + kQT - 1) / kQT, a.batch * a.n_kv_heads, split ? 2 : 1);
    const size_t smem2 = attn_tc2_smem_bytes(a.head_dim);
    if (a.head_dim == 64) launch_k(attn_tc2_kernel<64, 64>, grid2, dim3(192), smem2, s, maps.q, maps.k, maps.vt, a);
    if (a.head_dim == 128) {
      if (split) launch_k(attn_tc2_kernel<128, 64>, grid2, dim3(192), smem2, s, maps.q, maps.k, maps.vt2, a);
      else launch_k(attn_tc2_kernel<128, 128>, grid2, dim3(192), smem2, s, maps.q, maps.k, maps.vt, a);
    }
    if (a.head_dim == 256) {
      if (split) launch_k(attn_tc2_kernel<256, 128>, grid2, dim3(192), smem2, s, maps.q, maps.k, maps.vt2, a);
      else launch_k(attn_tc2_kernel<256, 256>, grid2, dim3(192), smem2, s, maps.q, maps.k, maps.vt, a);
    }
    return;
  }
  const int qt = (a.rows + kQT - 1) / kQT, kc = attn_tc_chunks(a.n_keys), bg = a.batch * a.n_kv_heads;
  int sp = 1;
  {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    while (a.head_dim / (2 * sp) >= 64 && 2 * sp * qt * kc * bg <= sms) sp *= 2;
  }
  const dim3 grid(qt * sp, kc, bg);
  const size_t smem = attn_tc_smem_bytes(a.head_dim);
  const CUtensorMap& vt = sp == 1 ? maps.vt : sp == 2 ? maps.vt2 : maps.vt4;
  if (a.head_dim == 64) launch_k(attn_tc_kernel<64, 64>, grid, dim3(128), smem, s, maps.q, maps.k, vt, a);
  if (a.head_dim == 128) {
    if (sp == 1) launch_k(attn_tc_kernel<128, 128>, grid, dim3(128), smem, s, maps.q, maps.k, vt, a);
    else launch_k(attn_tc_kernel<128, 64>, grid, dim3(128), smem, s, maps.q, maps.k, vt, a);
  }
  if (a.head_dim == 256) {
    if (sp == 1) launch_k(attn_tc_kernel<256, 256>, grid, dim3(128), smem, s, maps.q, maps.k, vt, a);
    else if (sp == 2) launch_k(attn_tc_kernel<256, 128>, grid, dim3(128), smem, s, maps.q, maps.k, vt, a);
    else launch_k(attn_tc_kernel<256, 64>, grid, dim3(128), smem, s, maps.q, maps.k, vt, a);
  }
  const int rows = 1024 / a.head_dim;
  launch_k(attn_combine_kernel, dim3((a.rows + rows - 1) / rows, bg), dim3(256), 0, s, a, kc);
}

void launch_kv_prefix(const void* k, const void* v, int src_dtype, const AttnTcArgs& a, int robot, cudaStream_t s) {
  if (a.prefix < 1 || a.n_layers < 1) return;
  const dim3 grid(a.n_layers * a.n_kv_heads, a.head_dim / kPfTile, (a.prefix + kPfTile - 1) / kPfTile);
  if (src_dtype == BF16) kv_prefix_kernel<BF16><<<grid, 256, 0, s>>>(k, v, a, robot);
  else kv_prefix_kernel<F32><<<grid, 256, 0, s>>>(k, v, a, robot);
}

}  // namespace uad
