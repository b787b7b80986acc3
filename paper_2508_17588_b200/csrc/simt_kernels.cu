// CUDA-core GEMM and attention for the fp32 run mode (fp32 parity at ~1e-5 against the float64 oracle rules out
// tensor-core input rounding).  Same epilogue contract as the tensor-core path: bias, optional GELU-tanh / gate, and
// the merge of Eq. 3 done by writing rows straight into their cache slots.
//
// Both kernels form dot products of K-contiguous rows from shared memory: operands are copied row by row with
// cp.async (no transposition), rows are padded to 4 floats more than a multiple of 32 so that eight neighbouring rows
// read 16 bytes each without a bank conflict, and the products are accumulated in packed pairs of even and odd k
// (fma.rn.f32x2: the same roundings as two FMAs, half the issue slots).
#include "hero_internal.h"
#include "tc_common.cuh"

namespace hero {
namespace {

__device__ __forceinline__ float gelu_tanh(float t) {
  const float kAlpha = 0.7978845608028654f;   // sqrt(2/pi)
  return 0.5f * t * (1.0f + tanhf(kAlpha * (t + 0.044715f * t * t * t)));
}

// 16 bytes from global to shared memory; zeros when the source does not exist.
__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool exists) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(tc::smem_u32(dst)), "l"(src), "r"(exists ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ void dot4(float2& acc, const float4& a, const float4& b) {
  acc = __ffma2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y), acc);
  acc = __ffma2_rn(make_float2(a.z, a.w), make_float2(b.z, b.w), acc);
}

// ---------------------------------------------------------------------------------------------------------------
// C[M, Nout] = A[M, K] W[Nout, K]^T + bias.  Tile BM x BN per CTA of 256 threads in KG groups: group g multiplies the
// g-th 32 of every KG * 32 k (so that a problem of few tiles still keeps all four schedulers of an SM busy), each
// thread TM x TN outputs, rows ty + i * (BM / TM) and columns tx + j * (BN / TN).  The groups' sums are added in group
// order.  Three chunks of k in the ring; two CTAs share an SM (eight warps alone keep its FMA pipe 46 % busy): 240 tiles of
// 64 x 64 x 512 in 42 us, 50 with the registers of one CTA a SM.
// ---------------------------------------------------------------------------------------------------------------
constexpr int kGemmPitch = 36;           // floats per staged row of 32
template <int BM, int BN, int TM, int TN>
struct SimtCfg {
  static constexpr int kGroupThreads = (BM / TM) * (BN / TN);
  static constexpr int kGroups = 256 / kGroupThreads;
  static constexpr int kStages = 3;
  static constexpr int kStageFloats = kGroups * (BM + BN) * kGemmPitch;
  static constexpr size_t kSmem = (size_t)kStages * kStageFloats * sizeof(float) + BN * sizeof(float) + BM * sizeof(long long);
  static_assert((size_t)(kGroups - 1) * BM * BN <= (size_t)kStages * kStageFloats, "the sums of the groups fit in the ring");
};

template <int BM, int BN, int TM, int TN>
__global__ void __launch_bounds__(256, 2) simt_gemm_kernel(const float* __restrict__ A, const float* __restrict__ W,
                                                        const float* __restrict__ bias, int M, int Nout, int K,
                                                        const GemmOut out) {
  using Cfg = SimtCfg<BM, BN, TM, TN>;
  constexpr int TX = BN / TN, TY = BM / TM, KG = Cfg::kGroups, kChunk = KG * 32;
  extern __shared__ __align__(16) float ring[];
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int group = threadIdx.x / Cfg::kGroupThreads, lt = threadIdx.x % Cfg::kGroupThreads;
  const int tx = lt % TX, ty = lt / TX;
  const int chunks = (K + kChunk - 1) / kChunk;

  float* s_bias = ring + Cfg::kStages * Cfg::kStageFloats;
  long long* s_scat = reinterpret_cast<long long*>(s_bias + BN);
  auto load_rows = [&](int chunk, int first, int rows) {       // of the BM rows of A and, behind them, the BN rows of W
    float* st = ring + (chunk % Cfg::kStages) * Cfg::kStageFloats;
    // 16-byte packets: (row, group, packet of 8)
    for (int e = threadIdx.x; e < rows * KG * 8; e += 256) {
      const int p = e & 7, g = (e >> 3) % KG, r = first + (e >> 3) / KG;
      const int k = chunk * kChunk + g * 32 + p * 4;
      const bool is_a = r < BM;
      const int row = is_a ? m0 + r : n0 + r - BM;
      const bool exists = k < K && row < (is_a ? M : Nout);
      const float* src = (is_a ? A : W) + (exists ? (long long)row * K + k : 0);
      cp_async16(st + (g * (BM + BN) + r) * kGemmPitch + p * 4, src, exists);
    }
  };
  // What no kernel in front has a hand in, first: the first chunks' weights, the bias and where the rows go (the lists are
  // as settled as the weights).  Fetched after the wait, and the latter two in the epilogue, they made the eight GEMMs of a
  // step of width 128 1.5 us longer each (101.8 -> 89.5 us the step; width 512, 620 rows: 587 -> 564).
  auto fetch_ahead = [&]() {
#pragma unroll
    for (int c = 0; c < Cfg::kStages - 1; ++c)
      if (c < chunks) load_rows(c, BM, BN);
    if (threadIdx.x < BN) {
      const int n = n0 + threadIdx.x;
      s_bias[threadIdx.x] = n < Nout ? __ldg(bias + n) : 0.f;
    } else if (threadIdx.x < BN + BM) {
      const int m = m0 + threadIdx.x - BN;
      if (m < M) {
        const int b = m / out.n_sel, li = m - b * out.n_sel;
        s_scat[threadIdx.x - BN] = (long long)b * out.n_rows + (out.idx ? __ldg(out.idx + li) : li);
      }
    }
  };
  if (out.weights_settled) fetch_ahead();
  stream_order();
  if (!out.weights_settled) fetch_ahead();
  float2 acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = make_float2(0.f, 0.f);
#pragma unroll
  for (int c = 0; c < Cfg::kStages - 1; ++c) {
    if (c < chunks) load_rows(c, 0, BM);
    cp_async_commit();
  }
  for (int c = 0; c < chunks; ++c) {
    cp_async_wait<Cfg::kStages - 2>();
    __syncthreads();                       // chunk c is there for everybody, and nobody reads chunk c - 1 any more
    if (c + Cfg::kStages - 1 < chunks) load_rows(c + Cfg::kStages - 1, 0, BM + BN);
    cp_async_commit();
    const float* sa = ring + (c % Cfg::kStages) * Cfg::kStageFloats + group * (BM + BN) * kGemmPitch;
    const float* sw = sa + BM * kGemmPitch;
#pragma unroll
    for (int k = 0; k < 32; k += 4) {
      float4 a[TM], w[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = *reinterpret_cast<const float4*>(sa + (ty + i * TY) * kGemmPitch + k);
#pragma unroll
      for (int j = 0; j < TN; ++j) w[j] = *reinterpret_cast<const float4*>(sw + (tx + j * TX) * kGemmPitch + k);
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) dot4(acc[i][j], a[i], w[j]);
    }
  }
  cp_async_wait<0>();
  __syncthreads();                         // the ring is free: the other groups hand their sums to group 0
  if (KG > 1 && group > 0) {
    float* dst = ring + (group - 1) * BM * BN + lt;
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) dst[(i * TN + j) * Cfg::kGroupThreads] = acc[i][j].x + acc[i][j].y;
  }
  if (KG > 1) __syncthreads();
  if (group > 0) return;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int m = m0 + ty + i * TY;
    if (m >= M) continue;
    const long long scat = s_scat[ty + i * TY];
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int n = n0 + tx + j * TX;
      if (n >= Nout) continue;
      float v = acc[i][j].x + acc[i][j].y;
#pragma unroll
      for (int g = 1; g < KG; ++g) v += ring[(g - 1) * BM * BN + (i * TN + j) * Cfg::kGroupThreads + lt];
      const bool s1 = n >= out.seg_cols, s2 = n >= 2 * out.seg_cols;
      const int col = n - (s2 ? 2 * out.seg_cols : (s1 ? out.seg_cols : 0));
      v += s_bias[tx + j * TX];
      if (out.act == 1) v = gelu_tanh(v);
      if (out.gate) v *= out.gate[(long long)(m / out.n_sel) * out.gate_ld + col];
      void* const base = s2 ? out.ptr[2] : (s1 ? out.ptr[1] : out.ptr[0]);
      const long long ld = s2 ? out.ld[2] : (s1 ? out.ld[1] : out.ld[0]);
      const int scatter = s2 ? out.scatter[2] : (s1 ? out.scatter[1] : out.scatter[0]);
      static_cast<float*>(base)[(scatter ? scat : (long long)m) * ld + col] = v;
    }
  }
}

// ---------------------------------------------------------------------------------------------------------------
// Flash attention in fp32.  A CTA of 128 threads takes 32 queries of one (batch, head) over a run of keys, 64 at a
// time (the next K tile and this tile's V in flight: three CTAs then share an SM); a thread owns four query rows (8 row groups) and, of a score tile, the keys tx + 16 j, of
// the output, HD / 16 features.  Online softmax with a running maximum: no score matrix is stored, P of a warp's own
// rows passes through shared memory.  Where the grid would leave SMs idle the keys are split over a cluster of
// `split` CTAs, which then merge their (maximum, sum, output) rows through distributed shared memory, in rank order.
// ---------------------------------------------------------------------------------------------------------------
constexpr int kAttQ = 32, kAttK = 64, kAttRows = 4;
template <int HD>
struct SimtAttCfg {
  static constexpr int kPitch = HD + 4, kPPitch = kAttK + 4;
  static constexpr int kTileFloats = kAttK * kPitch;
  static constexpr int kFloats = kAttQ * kPitch + kAttQ * kPPitch + 3 * kTileFloats + 2 * kAttQ;
  static constexpr size_t kSmem = (size_t)kFloats * sizeof(float);
};

__device__ __forceinline__ float ld_cluster(uint32_t cluster_addr) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(cluster_addr) : "memory");
  return v;
}

template <int HD>
__global__ void __launch_bounds__(128) simt_attention_kernel(const float* __restrict__ Q, const float* __restrict__ Kc,
                                                             const float* __restrict__ Vc, float* __restrict__ O,
                                                             int n_q, int N, int heads, int split) {
  stream_order();
  using Cfg = SimtAttCfg<HD>;
  constexpr int kPitch = Cfg::kPitch, CPT = HD / 16;       // output features per thread
  extern __shared__ __align__(16) float smem[];
  float* s_q = smem;
  float* s_p = s_q + kAttQ * kPitch;
  float* s_kv = s_p + kAttQ * Cfg::kPPitch;                // two K tiles, one V tile
  float* s_v = s_kv + 2 * Cfg::kTileFloats;
  float* s_ml = s_v + Cfg::kTileFloats;                    // [kAttQ] maxima, [kAttQ] sums
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int rank = blockIdx.x % split;
  const int q_tiles = (n_q + kAttQ - 1) / kAttQ;
  int rest = blockIdx.x / split;
  const int q0 = (rest % q_tiles) * kAttQ;
  rest /= q_tiles;
  const int h = rest % heads, b = rest / heads;
  const int D = heads * HD;
  const float* qb = Q + (long long)b * n_q * D + h * HD;
  const float* kb = Kc + (long long)b * N * D + h * HD;
  const float* vb = Vc + (long long)b * N * D + h * HD;
  const int tiles = (N + kAttK - 1) / kAttK;
  const int t0 = tiles * rank / split, t1 = tiles * (rank + 1) / split;

  auto load_rows = [&](float* dst, const float* src, int first, int rows, int limit) {
    for (int e = threadIdx.x; e < rows * (HD / 4); e += 128) {
      const int r = e / (HD / 4), p = e % (HD / 4);
      const bool exists = first + r < limit;
      cp_async16(dst + r * kPitch + p * 4, src + (exists ? (long long)(first + r) * D + p * 4 : 0), exists);
    }
  };
  load_rows(s_q, qb, q0, kAttQ, n_q);
  if (t0 < t1) load_rows(s_kv, kb, t0 * kAttK, kAttK, N);
  cp_async_commit();

  const float scale = rsqrtf((float)HD);
  float m_run[kAttRows], l_run[kAttRows], o[kAttRows][CPT];
#pragma unroll
  for (int i = 0; i < kAttRows; ++i) {
    m_run[i] = -INFINITY; l_run[i] = 0.f;
#pragma unroll
    for (int c = 0; c < CPT; ++c) o[i][c] = 0.f;
  }
  for (int t = t0; t < t1; ++t) {
    const int buf = (t - t0) & 1;
    const float* s_k = s_kv + buf * Cfg::kTileFloats;
    cp_async_wait<0>();
    __syncthreads();                       // K of tile t is there; nobody reads the other K buffer or V any more
    load_rows(s_v, vb, t * kAttK, kAttK, N);                     // (there by the time the scores are)
    cp_async_commit();
    if (t + 1 < t1) load_rows(s_kv + (buf ^ 1) * Cfg::kTileFloats, kb, (t + 1) * kAttK, kAttK, N);
    cp_async_commit();
    float2 s2[kAttRows][4];
#pragma unroll
    for (int i = 0; i < kAttRows; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) s2[i][j] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int c = 0; c < HD; c += 4) {
      float4 q[kAttRows], k[4];
#pragma unroll
      for (int i = 0; i < kAttRows; ++i) q[i] = *reinterpret_cast<const float4*>(s_q + (ty * kAttRows + i) * kPitch + c);
#pragma unroll
      for (int j = 0; j < 4; ++j) k[j] = *reinterpret_cast<const float4*>(s_k + (tx + 16 * j) * kPitch + c);
#pragma unroll
      for (int i = 0; i < kAttRows; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) dot4(s2[i][j], q[i], k[j]);
    }
#pragma unroll
    for (int i = 0; i < kAttRows; ++i) {
      float s[4], m = m_run[i];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        s[j] = t * kAttK + tx + 16 * j < N ? (s2[i][j].x + s2[i][j].y) * scale : -INFINITY;
        m = fmaxf(m, s[j]);
      }
#pragma unroll
      for (int d = 1; d < 16; d <<= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, d));
      const float alpha = expf(m_run[i] - m);          // (m is finite: a tile has at least one key)
      m_run[i] = m;
      l_run[i] *= alpha;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float p = expf(s[j] - m);
        l_run[i] += p;
        s_p[(ty * kAttRows + i) * Cfg::kPPitch + tx + 16 * j] = p;
      }
#pragma unroll
      for (int c = 0; c < CPT; ++c) o[i][c] *= alpha;
    }
    cp_async_wait<1>();
    __syncthreads();                       // V of tile t is there (and a warp's own P rows)
#pragma unroll 4
    for (int k = 0; k < kAttK; k += 4) {
      float4 p[kAttRows];
#pragma unroll
      for (int i = 0; i < kAttRows; ++i)
        p[i] = *reinterpret_cast<const float4*>(s_p + (ty * kAttRows + i) * Cfg::kPPitch + k);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        float v[CPT];
#pragma unroll
        for (int c = 0; c < CPT; c += (CPT < 4 ? 2 : 4)) {
          const float* src = s_v + (k + kk) * kPitch + (CPT < 4 ? tx * 2 : tx * 4 + 16 * c);
          if constexpr (CPT < 4) {
            const float2 w = *reinterpret_cast<const float2*>(src);
            v[0] = w.x; v[1] = w.y;
          } else {
            const float4 w = *reinterpret_cast<const float4*>(src);
            v[c] = w.x; v[c + 1] = w.y; v[c + 2] = w.z; v[c + 3] = w.w;
          }
        }
#pragma unroll
        for (int i = 0; i < kAttRows; ++i) {
          const float pk = kk == 0 ? p[i].x : (kk == 1 ? p[i].y : (kk == 2 ? p[i].z : p[i].w));
#pragma unroll
          for (int c = 0; c < CPT; ++c) o[i][c] = fmaf(pk, v[c], o[i][c]);
        }
      }
    }
    __syncwarp();
  }
#pragma unroll
  for (int i = 0; i < kAttRows; ++i)
#pragma unroll
    for (int d = 1; d < 16; d <<= 1) l_run[i] += __shfl_xor_sync(0xFFFFFFFFu, l_run[i], d);
  auto feature = [&](int c) { return CPT < 4 ? tx * 2 + c : tx * 4 + (c & 3) + 16 * (c & ~3); };

  if (split == 1) {
#pragma unroll
    for (int i = 0; i < kAttRows; ++i) {
      const int row = q0 + ty * kAttRows + i;
      if (row >= n_q) continue;
      float* dst = O + ((long long)b * n_q + row) * D + h * HD;
#pragma unroll
      for (int c = 0; c < CPT; ++c) dst[feature(c)] = o[i][c] / l_run[i];
    }
    return;
  }
  // Merge: every CTA lays its rows out over its (now idle) key and value tiles, then finishes kAttQ / split rows of all.
  cp_async_wait<0>();
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kAttRows; ++i) {
    const int row = ty * kAttRows + i;
#pragma unroll
    for (int c = 0; c < CPT; ++c) s_kv[row * HD + feature(c)] = o[i][c];
    if (tx == 0) { s_ml[row] = m_run[i]; s_ml[kAttQ + row] = l_run[i]; }
  }
  tc::cluster_sync();
  for (int e = threadIdx.x; e < kAttQ / split * HD; e += 128) {
    const int row = rank * (kAttQ / split) + e / HD, col = e % HD;
    float m = -INFINITY;
    for (int r = 0; r < split; ++r) m = fmaxf(m, ld_cluster(tc::cluster_map(tc::smem_u32(s_ml + row), r)));
    float l = 0.f, acc = 0.f;
    for (int r = 0; r < split; ++r) {
      const float w = expf(ld_cluster(tc::cluster_map(tc::smem_u32(s_ml + row), r)) - m);
      l = fmaf(w, ld_cluster(tc::cluster_map(tc::smem_u32(s_ml + kAttQ + row), r)), l);
      acc = fmaf(w, ld_cluster(tc::cluster_map(tc::smem_u32(s_kv + row * HD + col), r)), acc);
    }
    if (q0 + row < n_q) O[((long long)b * n_q + q0 + row) * D + h * HD + col] = acc / l;
  }
  tc::cluster_sync();                      // nobody leaves while its rows are being read
}

template <int BM, int BN, int TM, int TN>
int gemm_launch(const float* a, const float* w, const float* bias, int M, int Nout, int K, const GemmOut& out,
                cudaStream_t s) {
  using Cfg = SimtCfg<BM, BN, TM, TN>;
  static PerDeviceOnce once;
  HERO_TRY(per_device_once(once, [](int) {
    HERO_CUDA_TRY(cudaFuncSetAttribute(simt_gemm_kernel<BM, BN, TM, TN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)Cfg::kSmem));
    return HERO_OK;
  }));
  const dim3 grid((Nout + BN - 1) / BN, (M + BM - 1) / BM);
  HERO_TRY(launch_kernel(simt_gemm_kernel<BM, BN, TM, TN>, grid, 256, Cfg::kSmem, s, 1, a, w, bias, M, Nout, K, out));
  return HERO_OK;
}

template <int HD>
int attention_launch(const float* q, const float* k, const float* v, float* o, int B, int n_q, int N, int heads,
                     cudaStream_t s) {
  using Cfg = SimtAttCfg<HD>;
  static PerDeviceOnce once;
  HERO_TRY(per_device_once(once, [](int) {
    HERO_CUDA_TRY(cudaFuncSetAttribute(simt_attention_kernel<HD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::kSmem));
    return HERO_OK;
  }));
  const long long groups = (long long)B * heads * ((n_q + kAttQ - 1) / kAttQ);
  const int tiles = (N + kAttK - 1) / kAttK;
  // Keys over a cluster while that shortens the longest run of tiles (a CTA may go without: 144 keys are three tiles, over
  // four CTAs 8.2 us, over two 12.8) and leaves the grid within what the chip holds at once: a CTA of four
  // warps alone keeps an SM's FMA pipe 40 % busy, two 80 % (310 queries, 1319 keys, 16 heads: 160 CTAs 102 us, 320 83 us).
  const int resident = HD > 64 ? 1 : 3;
  int split = 1;
  while (split < 8 && split < tiles && groups * split * 2 <= (long long)num_sms() * resident * 3 / 4) split *= 2;
  if (groups * split > 0x7FFFFFFFll) return HERO_ERR_ARG;
  return launch_kernel(simt_attention_kernel<HD>, (unsigned)(groups * split), 128, Cfg::kSmem, s, (unsigned)split, q, k,
                       v, o, n_q, N, heads, split);
}

}  // namespace

int launch_simt_gemm(const float* a, const float* w, const float* bias, int M, int Nout, int K, const GemmOut& out,
                     cudaStream_t s) {
  if (M <= 0) return HERO_OK;
  // 64 x 64 tiles (8 x 4 outputs a thread, two groups) where they give every SM work of its own, else 32 x 32 (4 x 4
  // outputs, four groups)
  const long long tiles = (long long)((M + 63) / 64) * ((Nout + 63) / 64);
  if (tiles >= num_sms()) return gemm_launch<64, 64, 8, 4>(a, w, bias, M, Nout, K, out, s);
  return gemm_launch<32, 32, 4, 4>(a, w, bias, M, Nout, K, out, s);
}

int launch_simt_attention(const float* q, const float* k, const float* v, float* o, int B, int n_q, int N, int heads,
                          int head_dim, cudaStream_t s) {
  if (B <= 0 || n_q <= 0) return HERO_OK;
  switch (head_dim) {
    case 32: return attention_launch<32>(q, k, v, o, B, n_q, N, heads, s);
    case 64: return attention_launch<64>(q, k, v, o, B, n_q, N, heads, s);
    case 128: return attention_launch<128>(q, k, v, o, B, n_q, N, heads, s);
    default: return HERO_ERR_ARG;
  }
}

}  // namespace hero
