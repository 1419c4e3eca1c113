// CUDA-core projection GEMM and attention: the fp32 experts (every projection and their attention),
// bf16 weights whose shape the tensor-core layout does not take, and the time-conditioning table.
// fp32 products and sums throughout (packed two to an instruction, each rounded as fmaf rounds).
#include "uad_internal.cuh"
#include "ptx.cuh"

namespace uad {

using namespace ptx;

namespace {

__device__ __forceinline__ float gelu_tanh_f(float x) {
  const float k0 = 0.7978845608028654f;  // sqrt(2/pi)
  return 0.5f * x * (1.f + tanhf(k0 * (x + 0.044715f * x * x * x)));
}
__device__ __forceinline__ float silu(float x) { return x / (1.f + expf(-x)); }
__device__ __forceinline__ void store_as(void* p, long long i, float v, int dt) {
  if (dt == BF16) static_cast<__nv_bfloat16*>(p)[i] = __float2bfloat16_rn(v);
  else static_cast<float*>(p)[i] = v;
}
template <int DT>
__device__ __forceinline__ float load_as(const void* p, long long i) {
  if constexpr (DT == BF16) return __bfloat162float(static_cast<const __nv_bfloat16*>(p)[i]);
  else return static_cast<const float*>(p)[i];
}
__device__ __forceinline__ void commit_copies() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void wait_copies() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Two fp32 products accumulated at once (both rounded to nearest).
__device__ __forceinline__ void fma2(unsigned long long& d, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

__device__ __forceinline__ float lo_word(unsigned long long v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float hi_word(unsigned long long v) { return __uint_as_float((unsigned)(v >> 32)); }

// Four consecutive values of a row into shared memory as fp32; `vec`: rows are 16-byte (fp32) or
// 8-byte (bf16) aligned and a multiple of 4 long. fp32 vectors are asynchronous copies.
template <int DT>
__device__ __forceinline__ void load4(float* dst, const void* base, long long off, int left, bool vec) {
  if (vec) {
    if constexpr (DT == F32) {
      cp16(dst, static_cast<const float*>(base) + off);
    } else {
      const uint2 v = *reinterpret_cast<const uint2*>(static_cast<const __nv_bfloat16*>(base) + off);
      const float2 lo = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.x));
      const float2 hi = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.y));
      *reinterpret_cast<float4*>(dst) = make_float4(lo.x, lo.y, hi.x, hi.y);
    }
    return;
  }
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (left > 0) v.x = load_as<DT>(base, off);
  if (left > 1) v.y = load_as<DT>(base, off + 1);
  if (left > 2) v.z = load_as<DT>(base, off + 2);
  if (left > 3) v.w = load_as<DT>(base, off + 3);
  *reinterpret_cast<float4*>(dst) = v;
}

// ------------------------------------------------------------------------------------------
// GEMM: out[m][n] = epi(sum_k A[m][k] * Wt[n][k]). A CTA of eight warps (16 for the larger tiles, whose grids
// leave an SM one CTA) owns a BM x BN tile; WM x WN
// warps cover it and KS groups of them each own a share of every K chunk, so that a tile of 16
// tokens still keeps them all busy; the groups' sums are added in group order (deterministic).
// A lane owns BM / WM / 8 rows x BN / WN / 4 columns and reads four k at a time from rows that lie
// K-contiguous in shared memory (pitch KC + 4: no bank conflicts), as the copies bring them. The
// first chunks of the weights, which no kernel of the loop writes, are requested before the wait for
// the kernel that writes A. Bound by the latency of its chain with few rows and by FFMA issue with
// many. Against one 64 x 64 tile per CTA with K in series (4 CTAs for 16 rows x 256 outputs): tiny
// fp32 expert, down projection (K = 1024) of 16 rows 75 -> 11 us, of 512 rows 93 -> 17 us (20 us with eight
// warps: two a scheduler do not hide the shared-memory loads).
// ------------------------------------------------------------------------------------------
template <int THREADS_, int BM_, int BN_, int WM_, int WN_, int KC_, int ST_, bool SERIAL_ = false>
struct FfTile {
  static constexpr bool SERIAL = SERIAL_;   // every output one fp32 sum over ascending k
  static constexpr int THREADS = THREADS_, BM = BM_, BN = BN_, WM = WM_, WN = WN_, KC = KC_, ST = ST_;
  static constexpr int KS = THREADS / 32 / (WM * WN), RM = BM / WM / 8, RN = BN / WN / 4, PITCH = KC + 4;
  static constexpr int STAGE = (BM + BN) * PITCH;          // floats
  static constexpr int RPITCH = BN + 4;                    // reduction rows
  // shared memory of a K that takes `chunks` chunks: no more than it uses, so that the next kernel's
  // CTAs find room on the SM and fetch their first weights while this one runs
  static constexpr size_t smem(int chunks) {
    const size_t pipe = (size_t)(chunks < ST ? chunks : ST) * STAGE, red = (size_t)KS * BM * RPITCH;
    return (pipe > red ? pipe : red) * sizeof(float);
  }
};
using FfSmall = FfTile<256, 16, 16, 1, 1, 256, 4>;
using FfMid = FfTile<512, 32, 32, 1, 1, 256, 2>;
using FfWide = FfTile<512, 64, 64, 2, 2, 64, 3>;
// The time table's: one sum per output over ascending k, so that a row has the same bits whichever tile made it
// and however many rows are filled at once. Every modulation of every step goes through these rows: a
// last bit of theirs moves bf16 roundings of every layer (18-layer expert, 16 and 64 robots: with sums
// in groups the actions differed by 6.9e-4, at the same distance from 64 bits, 5.2e-4).
using FfTabSmall = FfTile<64, 16, 16, 1, 2, 256, 4, true>;
using FfTabWide = FfTile<256, 64, 64, 4, 2, 64, 3, true>;

template <int AD, int WD, class T>
__global__ void __launch_bounds__(T::THREADS) gemm_ffma_kernel(GemmArgs p) {
  extern __shared__ __align__(16) float fsm[];
  constexpr int KC = T::KC, PITCH = T::PITCH, ST = T::ST, RM = T::RM, RN = T::RN;
  const int m0 = blockIdx.y * T::BM, n0 = blockIdx.x * T::BN, K = p.K;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nch = (K + KC - 1) / KC;
  const bool va = K % 4 == 0 && p.lda % 4 == 0 && reinterpret_cast<uintptr_t>(p.A) % 16 == 0;
  const bool vw = K % 4 == 0 && reinterpret_cast<uintptr_t>(p.W) % 16 == 0;
  pdl_trigger();

  const auto load_w = [&](int c) {
    float* dst = fsm + (c % ST) * T::STAGE + T::BM * PITCH;
#pragma unroll 4
    for (int e = tid; e < T::BN * (KC / 4); e += T::THREADS) {
      const int r = e / (KC / 4), c4 = e % (KC / 4), n = n0 + r, k = c * KC + 4 * c4;
      if (n < p.N && k < K) load4<WD>(dst + r * PITCH + 4 * c4, p.W, (long long)n * K + k, K - k, vw);
      else *reinterpret_cast<float4*>(dst + r * PITCH + 4 * c4) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  const auto load_a = [&](int c) {
    float* dst = fsm + (c % ST) * T::STAGE;
#pragma unroll 4
    for (int e = tid; e < T::BM * (KC / 4); e += T::THREADS) {
      const int r = e / (KC / 4), c4 = e % (KC / 4), m = m0 + r, k = c * KC + 4 * c4;
      if (m < p.M && k < K) load4<AD>(dst + r * PITCH + 4 * c4, p.A, (long long)m * p.lda + k, K - k, va);
      else *reinterpret_cast<float4*>(dst + r * PITCH + 4 * c4) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  for (int c = 0; c < ST && c < nch; ++c) load_w(c);
  // residual update: this thread's first outputs' gates before the wait, their residual values right after
  // it, so that neither is fetched at the end
  constexpr int EP = T::BM * T::BN / T::THREADS < 4 ? (T::BM * T::BN + T::THREADS - 1) / T::THREADS : 4;
  float gate[EP], res[EP];
  const auto out_of = [&](int u, int& m, int& n) {
    const int e = tid + T::THREADS * u;
    m = m0 + e / T::BN;
    n = n0 + e % T::BN;
    return m < p.M && n < p.N;
  };
  if (p.epi == EPI_RESID_GATE) {
#pragma unroll
    for (int u = 0; u < EP; ++u) {
      int m, n;
      gate[u] = out_of(u, m, n) && p.gate_tab ? p.gate_tab[(long long)__ldcg(p.tau_row + m) * p.gate_stride + n] : 1.f;
    }
  }
  pdl_wait();
  if (p.epi == EPI_RESID_GATE) {
#pragma unroll
    for (int u = 0; u < EP; ++u) {
      int m, n;
      res[u] = out_of(u, m, n) ? p.resid[(long long)m * p.ldr + n] : 0.f;
    }
  }
#pragma unroll 1
  for (int c = 0; c < ST; ++c) {
    if (c < nch) load_a(c);
    commit_copies();
  }

  constexpr int WT = T::WM * T::WN, KW = KC / T::KS;   // warps over the tile; k of a chunk per group
  const int ks = warp / WT, wm = (warp % WT) / T::WN, wn = warp % T::WN;
  const int lr = lane >> 2, lc = lane & 3;
  static_assert(!T::SERIAL || T::KS == 1, "one group of warps walks the whole K");
  unsigned long long acc[RM][RN];   // the sums of even and odd k; SERIAL: one sum, in the low word
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j) acc[i][j] = 0ull;
  for (int c = 0; c < nch; ++c) {
    wait_copies<ST - 1>();
    __syncthreads();
    const float* a = fsm + (c % ST) * T::STAGE + (wm * (T::BM / T::WM) + lr) * PITCH + ks * KW;
    const float* w = fsm + (c % ST) * T::STAGE + (T::BM + wn * (T::BN / T::WN) + lc) * PITCH + ks * KW;
#pragma unroll 4
    for (int k = 0; k < KW; k += 4) {
      ulonglong2 av[RM], wv[RN];
#pragma unroll
      for (int i = 0; i < RM; ++i) av[i] = *reinterpret_cast<const ulonglong2*>(a + 8 * i * PITCH + k);
#pragma unroll
      for (int j = 0; j < RN; ++j) wv[j] = *reinterpret_cast<const ulonglong2*>(w + 4 * j * PITCH + k);
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j) {
          if constexpr (T::SERIAL) {
            float r = lo_word(acc[i][j]);
            r = fmaf(lo_word(av[i].x), lo_word(wv[j].x), r);
            r = fmaf(hi_word(av[i].x), hi_word(wv[j].x), r);
            r = fmaf(lo_word(av[i].y), lo_word(wv[j].y), r);
            r = fmaf(hi_word(av[i].y), hi_word(wv[j].y), r);
            acc[i][j] = __float_as_uint(r);
          } else {
            fma2(acc[i][j], av[i].x, wv[j].x);
            fma2(acc[i][j], av[i].y, wv[j].y);
          }
        }
    }
    __syncthreads();
    if (c + ST < nch) {
      load_w(c + ST);
      load_a(c + ST);
    }
    commit_copies();
  }

  // the K groups' sums, in group order
  float* red = fsm;
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j) {
      const float lo = lo_word(acc[i][j]), hi = hi_word(acc[i][j]);
      red[((size_t)ks * T::BM + wm * (T::BM / T::WM) + lr + 8 * i) * T::RPITCH + wn * (T::BN / T::WN) + lc + 4 * j] = T::SERIAL ? lo : lo + hi;
    }
  __syncthreads();
  const auto total = [&](int m, int n) {
    float s = red[m * T::RPITCH + n];
#pragma unroll
    for (int g = 1; g < T::KS; ++g) s += red[(g * T::BM + m) * T::RPITCH + n];
    return s;
  };
  if (p.epi == EPI_GEGLU) {
    for (int e = tid; e < T::BM * T::BN / 2; e += T::THREADS) {
      const int ml = e / (T::BN / 2), nl = 2 * (e % (T::BN / 2)), m = m0 + ml, n = n0 + nl;
      if (m < p.M && n + 1 < p.N)
        store_as(p.out, (long long)m * p.ldo + n / 2, gelu_tanh_f(total(ml, nl)) * total(ml, nl + 1), p.out_dtype);
    }
    return;
  }
  if (p.epi == EPI_RESID_GATE) {
#pragma unroll
    for (int u = 0; u < EP; ++u) {
      int m, n;
      if (out_of(u, m, n)) p.resid[(long long)m * p.ldr + n] = fmaf(gate[u], total(m - m0, n - n0) + (p.bias ? p.bias[n] : 0.f), res[u]);
    }
  }
  for (int e = tid + (p.epi == EPI_RESID_GATE ? T::THREADS * EP : 0); e < T::BM * T::BN; e += T::THREADS) {
    const int ml = e / T::BN, nl = e % T::BN, m = m0 + ml, n = n0 + nl;
    if (m >= p.M || n >= p.N) continue;
    float r = total(ml, nl) + (p.bias ? p.bias[n] : 0.f);
    switch (p.epi) {
      case EPI_STORE:
        if (p.add_rows) r += p.add_rows[(long long)(m % p.add_mod) * p.N + n];
        store_as(p.out, (long long)m * p.ldo + n, r, p.out_dtype);
        break;
      case EPI_BIAS_SILU: store_as(p.out, (long long)m * p.ldo + n, silu(r), p.out_dtype); break;
      case EPI_BIAS_GELU: store_as(p.out, (long long)m * p.ldo + n, gelu_tanh_f(r), p.out_dtype); break;
      case EPI_RESID_GATE: {
        const float gt = p.gate_tab ? p.gate_tab[(long long)__ldcg(p.tau_row + m) * p.gate_stride + n] : 1.f;
        float* dst = p.resid + (long long)m * p.ldr + n;
        *dst = fmaf(gt, r, *dst);
        break;
      }
      default: break;
    }
  }
}

template <int AD, int WD, class T>
void launch_tile(const GemmArgs& a, cudaStream_t s) {
  launch_k(gemm_ffma_kernel<AD, WD, T>, dim3((a.N + T::BN - 1) / T::BN, (a.M + T::BM - 1) / T::BM), dim3(T::THREADS),
           T::smem((a.K + T::KC - 1) / T::KC), s, a);
}

// The largest tile whose grid still fills the SMs (two thirds of them for the middle one): a larger
// tile reads less per product, a smaller one keeps a short projection from running on a few SMs. On
// the tiny expert 16 rows x 2048 outputs take 128 small tiles, 512 x 256 take 128 middle ones.
template <int AD, int WD>
void launch_types(const GemmArgs& a, int sms, cudaStream_t s) {
  const auto tiles = [&](int t) { return (long long)((a.M + t - 1) / t) * ((a.N + t - 1) / t); };
  if (tiles(64) >= sms) launch_tile<AD, WD, FfWide>(a, s);
  else if (tiles(32) * 3 >= 2 * sms) launch_tile<AD, WD, FfMid>(a, s);
  else launch_tile<AD, WD, FfSmall>(a, s);
}

// ------------------------------------------------------------------------------------------
// Attention of chunk queries over [prefix keys ; chunk keys] with grouped KV heads, online softmax in
// fp32. CTA = eight warps of QW queries each of one head and robot; tiles of KT keys come in by
// asynchronous copies, double-buffered. Scores: lane = keys lane, lane + 32, ... of the tile, four
// head dims a load (pitch DH + 4: no bank conflicts); output: lane owns DH / 32 consecutive dims.
// ------------------------------------------------------------------------------------------
template <int DH>
struct AttnTile {
  static constexpr int KT = DH == 64 ? 64 : 32;
  static constexpr int KP = DH + 4;
  static size_t smem(int qw) { return sizeof(float) * (2 * KT * (KP + DH) + 8 * qw * (DH + KT)); }
};

template <int DT>
__device__ __forceinline__ float rope_dim(const void* base, long long off, int d, int half, const float* cs) {
  const float x = load_as<DT>(base, off + d);
  const int j = d < half ? d : d - half;
  const float c = cs[2 * j], s = cs[2 * j + 1];
  const float o = load_as<DT>(base, off + (d < half ? d + half : d - half));
  return d < half ? x * c - o * s : x * c + o * s;
}

template <int DT, int DH, int QW>
__global__ void __launch_bounds__(256) attn_rows_kernel(AttnArgs p) {
  using T = AttnTile<DH>;
  constexpr int KT = T::KT, KP = T::KP, KL = KT / 32, DPL = DH / 32, half = DH / 2;
  extern __shared__ __align__(16) float asm_[];
  float* ks = asm_;                      // [2][KT][KP]
  float* vs = ks + 2 * KT * KP;          // [2][KT][DH]
  float* qs = vs + 2 * KT * DH;          // [8 QW][DH]
  float* ps = qs + 8 * QW * DH;          // [8 QW][KT]
  const int b = blockIdx.z, hq = blockIdx.y, i0 = blockIdx.x * 8 * QW;
  const int g = hq / (p.n_heads / p.n_kv_heads);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n_keys = p.P + (p.kc ? p.H : 0), nt = (n_keys + KT - 1) / KT;
  pdl_trigger();

  const auto load_tile = [&](int t) {
    float* kd = ks + (t & 1) * KT * KP;
    float* vd = vs + (t & 1) * KT * DH;
    for (int e = tid; e < KT * (DH / 4); e += 256) {
      const int jj = e / (DH / 4), d = 4 * (e % (DH / 4)), j = t * KT + jj;
      float* kr = kd + jj * KP + d;
      float* vr = vd + jj * DH + d;
      if (j < p.P) {
        const long long off = b * p.kp_bstride + (long long)j * p.kp_ld + g * DH + d;
        load4<DT>(kr, p.kp, off, 4, true);
        load4<DT>(vr, p.vp, off, 4, true);
      } else if (j < n_keys) {
        const int i = j - p.P;
        const long long row = (long long)(b * p.H + i) * p.kc_ld + g * DH;
        if (p.rope_cs) {
          const float* cs = p.rope_cs + (long long)i * DH;
#pragma unroll
          for (int q = 0; q < 4; ++q) kr[q] = rope_dim<DT>(p.kc, row, d + q, half, cs);
        } else {
          load4<DT>(kr, p.kc, row + d, 4, true);
        }
        load4<DT>(vr, p.vc, row + d, 4, true);
      } else {
        *reinterpret_cast<float4*>(kr) = make_float4(0.f, 0.f, 0.f, 0.f);
        *reinterpret_cast<float4*>(vr) = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
  };
  // a first tile of prefix keys alone, which no kernel of the loop writes, is requested early
  const bool early = KT <= p.P;
  if (early) load_tile(0);
  pdl_wait();
  if (!early && nt > 0) load_tile(0);
  commit_copies();
  for (int e = tid; e < 8 * QW * DH; e += 256) {
    const int qi = e / DH, d = e % DH, i = i0 + qi;
    float val = 0.f;
    if (i < p.H) {
      const long long off = (long long)(b * p.H + i) * p.q_ld + hq * DH;
      val = p.rope_cs ? rope_dim<DT>(p.q, off, d, half, p.rope_cs + (long long)i * DH) : load_as<DT>(p.q, off + d);
    }
    qs[qi * DH + d] = val * p.scale;
  }

  float m_run[QW], l_run[QW], o[QW][DPL];
#pragma unroll
  for (int q = 0; q < QW; ++q) {
    m_run[q] = -INFINITY;
    l_run[q] = 0.f;
#pragma unroll
    for (int t = 0; t < DPL; ++t) o[q][t] = 0.f;
  }
  const float* qw = qs + warp * QW * DH;
  float* pw = ps + warp * QW * KT;
  for (int t = 0; t < nt; ++t) {
    if (t + 1 < nt) load_tile(t + 1);
    commit_copies();
    wait_copies<1>();
    __syncthreads();
    const float* kd = ks + (t & 1) * KT * KP + lane * KP;
    const float* vd = vs + (t & 1) * KT * DH + lane * DPL;
    float s[QW][KL];
#pragma unroll
    for (int q = 0; q < QW; ++q)
#pragma unroll
      for (int u = 0; u < KL; ++u) s[q][u] = 0.f;
#pragma unroll 4
    for (int d = 0; d < DH; d += 4) {
      float4 kv[KL];
#pragma unroll
      for (int u = 0; u < KL; ++u) kv[u] = *reinterpret_cast<const float4*>(kd + 32 * u * KP + d);
#pragma unroll
      for (int q = 0; q < QW; ++q) {
        const float4 qv = *reinterpret_cast<const float4*>(qw + q * DH + d);
#pragma unroll
        for (int u = 0; u < KL; ++u)
          s[q][u] = fmaf(qv.w, kv[u].w, fmaf(qv.z, kv[u].z, fmaf(qv.y, kv[u].y, fmaf(qv.x, kv[u].x, s[q][u]))));
      }
    }
#pragma unroll
    for (int q = 0; q < QW; ++q) {
      float mx = -INFINITY;
#pragma unroll
      for (int u = 0; u < KL; ++u) {
        if (t * KT + lane + 32 * u >= n_keys) s[q][u] = -INFINITY;
        mx = fmaxf(mx, s[q][u]);
      }
      const float m_new = fmaxf(m_run[q], warp_max(mx));
      const float alpha = m_run[q] == -INFINITY ? 0.f : expf(m_run[q] - m_new);
      float sum = 0.f;
#pragma unroll
      for (int u = 0; u < KL; ++u) {
        const float pe = t * KT + lane + 32 * u < n_keys ? expf(s[q][u] - m_new) : 0.f;
        pw[q * KT + lane + 32 * u] = pe;
        sum += pe;
      }
      l_run[q] = l_run[q] * alpha + warp_sum(sum);
      m_run[q] = m_new;
#pragma unroll
      for (int e = 0; e < DPL; ++e) o[q][e] *= alpha;
    }
    __syncwarp();
#pragma unroll 2
    for (int j = 0; j < KT; j += 4) {
      float4 pj[QW];
#pragma unroll
      for (int q = 0; q < QW; ++q) pj[q] = *reinterpret_cast<const float4*>(pw + q * KT + j);
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) {
        float v[DPL];
#pragma unroll
        for (int e = 0; e < DPL; e += 2) {
          const float2 f = *reinterpret_cast<const float2*>(vd + (j + jj) * DH + e);
          v[e] = f.x;
          v[e + 1] = f.y;
        }
#pragma unroll
        for (int q = 0; q < QW; ++q) {
          const float pq = jj == 0 ? pj[q].x : jj == 1 ? pj[q].y : jj == 2 ? pj[q].z : pj[q].w;
#pragma unroll
          for (int e = 0; e < DPL; ++e) o[q][e] = fmaf(pq, v[e], o[q][e]);
        }
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < QW; ++q) {
    const int i = i0 + warp * QW + q;
    if (i >= p.H) continue;
    const float inv = 1.f / l_run[q];
    const long long off = (long long)(b * p.H + i) * p.out_ld + hq * DH + lane * DPL;
#pragma unroll
    for (int e = 0; e < DPL; ++e) store_as(p.out, off + e, o[q][e] * inv, DT);
  }
}

template <int DT, int DH, int QW>
void launch_rows(const AttnArgs& a, cudaStream_t s) {
  launch_k(attn_rows_kernel<DT, DH, QW>, dim3((a.H + 8 * QW - 1) / (8 * QW), a.n_heads, a.B), dim3(256), AttnTile<DH>::smem(QW), s, a);
}
template <int DT, int DH>
void launch_rows_qw(const AttnArgs& a, int sms, cudaStream_t s) {
  // two queries a warp halve the key and value reads, once the grid is full without them
  if ((long long)((a.H + 15) / 16) * a.n_heads * a.B >= sms) launch_rows<DT, DH, 2>(a, s);
  else launch_rows<DT, DH, 1>(a, s);
}
template <int DT, int DH>
void prepare_rows() {
  const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaFuncSetAttribute(attn_rows_kernel<DT, DH, 1>, at, (int)AttnTile<DH>::smem(1));
  cudaFuncSetAttribute(attn_rows_kernel<DT, DH, 2>, at, (int)AttnTile<DH>::smem(2));
}

template <int AD, int WD>
void prepare_tiles() {
  const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaFuncSetAttribute(gemm_ffma_kernel<AD, WD, FfSmall>, at, (int)FfSmall::smem(FfSmall::ST));
  cudaFuncSetAttribute(gemm_ffma_kernel<AD, WD, FfMid>, at, (int)FfMid::smem(FfMid::ST));
  cudaFuncSetAttribute(gemm_ffma_kernel<AD, WD, FfWide>, at, (int)FfWide::smem(FfWide::ST));
}
template <int WD>
void prepare_table_tiles() {
  const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaFuncSetAttribute(gemm_ffma_kernel<F32, WD, FfTabSmall>, at, (int)FfTabSmall::smem(FfTabSmall::ST));
  cudaFuncSetAttribute(gemm_ffma_kernel<F32, WD, FfTabWide>, at, (int)FfTabWide::smem(FfTabWide::ST));
}

int device_sms() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

}  // namespace

void launch_gemm_ffma(const GemmArgs& a, cudaStream_t s) {
  const int sms = device_sms();
  if (a.a_dtype == F32 && a.w_dtype == F32) launch_types<F32, F32>(a, sms, s);
  else if (a.a_dtype == F32 && a.w_dtype == BF16) launch_types<F32, BF16>(a, sms, s);
  else if (a.a_dtype == BF16 && a.w_dtype == BF16) launch_types<BF16, BF16>(a, sms, s);
  else launch_types<BF16, F32>(a, sms, s);
}

// The time table's projections (fp32 activations): the wide tile once its grid covers the SMs.
void launch_gemm_table(const GemmArgs& a, cudaStream_t s) {
  const bool wide = (long long)((a.M + 63) / 64) * ((a.N + 63) / 64) >= device_sms();
  if (a.w_dtype == F32) {
    if (wide) launch_tile<F32, F32, FfTabWide>(a, s);
    else launch_tile<F32, F32, FfTabSmall>(a, s);
  } else {
    if (wide) launch_tile<F32, BF16, FfTabWide>(a, s);
    else launch_tile<F32, BF16, FfTabSmall>(a, s);
  }
}

void ffma_prepare(int dh) {
  prepare_table_tiles<F32>();
  prepare_table_tiles<BF16>();
  prepare_tiles<F32, F32>();
  prepare_tiles<F32, BF16>();
  prepare_tiles<BF16, BF16>();
  prepare_tiles<BF16, F32>();
  if (dh == 64) { prepare_rows<F32, 64>(); prepare_rows<BF16, 64>(); }
  if (dh == 128) { prepare_rows<F32, 128>(); prepare_rows<BF16, 128>(); }
  if (dh == 256) { prepare_rows<F32, 256>(); prepare_rows<BF16, 256>(); }
}

void launch_attn_rows(const AttnArgs& a, cudaStream_t s) {
  const int sms = device_sms();
  if (a.dtype == F32) {
    if (a.head_dim == 64) launch_rows_qw<F32, 64>(a, sms, s);
    if (a.head_dim == 128) launch_rows_qw<F32, 128>(a, sms, s);
    if (a.head_dim == 256) launch_rows_qw<F32, 256>(a, sms, s);
  } else {
    if (a.head_dim == 64) launch_rows_qw<BF16, 64>(a, sms, s);
    if (a.head_dim == 128) launch_rows_qw<BF16, 128>(a, sms, s);
    if (a.head_dim == 256) launch_rows_qw<BF16, 256>(a, sms, s);
  }
}

}  // namespace uad
