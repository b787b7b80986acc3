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
// C[M, Nout] = A[M, K] W[Nout, K]^T + bias.  Tile BM x BN per CTA, in KG groups of threads: group g multiplies the g-th 32
// of every KG * 32 k, each thread TM x TN outputs, rows ty + i * (BM / TM) and columns tx + j * (BN / TN).  A cluster of
// `split` CTAs shares a tile where that evens out the SMs' shares, each taking a run of the chunks of k.  The sums of all
// groups and CTAs go through shared memory (a row of the tile is then stored by neighbouring lanes) and are added in
// order, groups before CTAs, so that a result does not depend on timing.
// ---------------------------------------------------------------------------------------------------------------
constexpr long long kMaxGridY = 65535;   // (the row tiles)
constexpr int kGemmPitch = 36;           // floats per staged row of 32
template <int BM, int BN, int TM, int TN, int KG>
struct SimtCfg {
  static constexpr int kGroupThreads = (BM / TM) * (BN / TN);
  static constexpr int kThreads = KG * kGroupThreads;
  static constexpr int kStages = 3;
  static constexpr int kStageFloats = KG * (BM + BN) * kGemmPitch;
  static constexpr int kSumPitch = BN + 8;                     // (four rows of eight columns: no bank twice)
  static constexpr size_t kSmem = (size_t)kStages * kStageFloats * sizeof(float) + BN * sizeof(float) + BM * sizeof(long long);
  static_assert((size_t)KG * BM * kSumPitch <= (size_t)kStages * kStageFloats, "the sums of the groups fit in the ring");
  static_assert(BN + BM <= kThreads, "one thread per column's bias and per row's place");
};

__device__ __forceinline__ float4 ld_cluster4(uint32_t cluster_addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(cluster_addr) : "memory");
  return v;
}
__device__ __forceinline__ void add4(float4& a, const float4& b) { a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w; }

template <int BM, int BN, int TM, int TN, int KG>
__global__ void __launch_bounds__(SimtCfg<BM, BN, TM, TN, KG>::kThreads, 2)
simt_gemm_kernel(const float* __restrict__ A, const float* __restrict__ W, const float* __restrict__ bias, int M, int Nout,
                 int K, int split, const GemmOut out) {
  using Cfg = SimtCfg<BM, BN, TM, TN, KG>;
  constexpr int TX = BN / TN, TY = BM / TM, kChunk = KG * 32, kThreads = Cfg::kThreads;
  extern __shared__ __align__(16) float ring[];
  const int rank = blockIdx.x % split;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x / split * BN;
  const int group = threadIdx.x / Cfg::kGroupThreads, lt = threadIdx.x % Cfg::kGroupThreads;
  const int tx = lt % TX, ty = lt / TX;
  const int all_chunks = (K + kChunk - 1) / kChunk;
  const int first_chunk = all_chunks * rank / split, chunks = all_chunks * (rank + 1) / split - first_chunk;

  float* s_bias = ring + Cfg::kStages * Cfg::kStageFloats;
  long long* s_scat = reinterpret_cast<long long*>(s_bias + BN);
  // Chunks come in packets of 16 bytes: a thread fetches packet p of group g's 32 k of every eighth row, whose addresses and
  // existence it works out once (per packet they were a quarter of the loop's instructions).
  const int p = threadIdx.x & 7, g = (threadIdx.x >> 3) % KG, r0 = threadIdx.x / (8 * KG);
  static_assert(kThreads == 64 * KG, "eight rows a round");
  const int k_first = first_chunk * kChunk + g * 32 + p * 4;
  const float* const a_src = A + (long long)(m0 + r0) * K + k_first;
  const float* const w_src = W + (long long)(n0 + r0) * K + k_first;
  float* const s_dst = ring + (g * (BM + BN) + r0) * kGemmPitch + p * 4;
  auto load_rows = [&](int chunk, bool weights) {
    float* dst = s_dst + (chunk % Cfg::kStages) * Cfg::kStageFloats + (weights ? BM * kGemmPitch : 0);
    const int rows = (weights ? Nout - n0 : M - m0) - r0;      // of which exist those that are multiples of eight below this
    const bool there = k_first + chunk * kChunk < K;
    const float* src = (weights ? w_src : a_src) + chunk * kChunk;
#pragma unroll
    for (int j = 0; j < (weights ? BN : BM) / 8; ++j) {
      const bool exists = there && 8 * j < rows;
      cp_async16(dst + 8 * j * kGemmPitch, exists ? src + (long long)(8 * j) * K : A, exists);
    }
  };
  // What no kernel in front has a hand in, first: the first chunks' weights, the bias and where the rows go (the lists are
  // as settled as the weights).  Fetched after the wait, and the latter two in the epilogue, they made the eight GEMMs of a
  // step of width 128 1.5 us longer each (101.8 -> 89.5 us the step; width 512, 620 rows: 587 -> 564).
  auto fetch_ahead = [&]() {
#pragma unroll
    for (int c = 0; c < Cfg::kStages - 1; ++c)
      if (c < chunks) load_rows(c, true);
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
    if (c < chunks) load_rows(c, false);
    cp_async_commit();
  }
  for (int c = 0; c < chunks; ++c) {
    cp_async_wait<Cfg::kStages - 2>();
    __syncthreads();                       // chunk c is there for everybody, and nobody reads chunk c - 1 any more
    if (c + Cfg::kStages - 1 < chunks) { load_rows(c + Cfg::kStages - 1, false); load_rows(c + Cfg::kStages - 1, true); }
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
  __syncthreads();                         // the ring is free: every group lays its sums out in it
  float* const sums = ring + group * BM * Cfg::kSumPitch;
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) sums[(ty + i * TY) * Cfg::kSumPitch + tx + j * TX] = acc[i][j].x + acc[i][j].y;
  if (split > 1) tc::cluster_sync();
  else __syncthreads();
  // Each CTA of the cluster finishes some of the tile's rows, four columns at a time (rows of W, segments and destinations
  // are multiples of four).
  const int row0 = BM * rank / split, row1 = BM * (rank + 1) / split;
  for (int e = row0 * (BN / 4) + threadIdx.x; e < row1 * (BN / 4); e += kThreads) {
    const int r = e / (BN / 4), c = e % (BN / 4) * 4, n = n0 + c, m = m0 + r;
    if (m >= M || n >= Nout) continue;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    const float* at = ring + r * Cfg::kSumPitch + c;
    if (split == 1) {
#pragma unroll
      for (int g = 0; g < KG; ++g) add4(v, *reinterpret_cast<const float4*>(at + g * BM * Cfg::kSumPitch));
    } else {
      for (int s = 0; s < split; ++s) {
        const uint32_t there = tc::cluster_map(tc::smem_u32(at), (uint32_t)s);
#pragma unroll
        for (int g = 0; g < KG; ++g) add4(v, ld_cluster4(there + g * BM * Cfg::kSumPitch * 4));
      }
    }
    const bool s1 = n >= out.seg_cols, s2 = n >= 2 * out.seg_cols;
    const int col = n - (s2 ? 2 * out.seg_cols : (s1 ? out.seg_cols : 0));
    add4(v, *reinterpret_cast<const float4*>(s_bias + c));
    if (out.act == 1) v = make_float4(gelu_tanh(v.x), gelu_tanh(v.y), gelu_tanh(v.z), gelu_tanh(v.w));
    if (out.gate) {
      const float4 g4 = *reinterpret_cast<const float4*>(out.gate + (long long)(m / out.n_sel) * out.gate_ld + col);
      v.x *= g4.x; v.y *= g4.y; v.z *= g4.z; v.w *= g4.w;
    }
    void* const base = s2 ? out.ptr[2] : (s1 ? out.ptr[1] : out.ptr[0]);
    const long long ld = s2 ? out.ld[2] : (s1 ? out.ld[1] : out.ld[0]);
    const int scatter = s2 ? out.scatter[2] : (s1 ? out.scatter[1] : out.scatter[0]);
    *reinterpret_cast<float4*>(static_cast<float*>(base) + (scatter ? s_scat[r] : (long long)m) * ld + col) = v;
  }
  if (split > 1) tc::cluster_sync();       // nobody leaves while its sums are being read
}

// ---------------------------------------------------------------------------------------------------------------
// Flash attention in fp32.  A CTA of 128 threads takes 32 queries of one (batch, head) over a run of keys, 64 at a
// time (the next K tile and this tile's V in flight: three CTAs then share an SM); a thread owns four query rows (8 row
// groups) and, of a score tile, the keys tx + 16 j, of the output, HD / 16 features.  Online softmax with a running maximum: no
// score matrix is stored, P of a warp's own rows passes through shared memory.  Where the grid would leave SMs idle the keys are
// split over a cluster of `split` CTAs, which then merge their (maximum, sum, output) rows through distributed shared memory, in
// rank order.
// ---------------------------------------------------------------------------------------------------------------
constexpr int kAttQ = kSimtAttQ, kAttK = kSimtAttK, kAttRows = 4;
template <int HD>
struct SimtAttCfg {
  static constexpr int kPitch = HD + 4, kPPitch = kAttK + 4;
  static constexpr int kTileFloats = kAttK * kPitch;
  static constexpr int kFloats = kAttQ * kPitch + kAttQ * kPPitch + 3 * kTileFloats + 2 * kAttQ;
  static_assert(kAttQ * HD <= 3 * kTileFloats, "the merge's rows fit over the tiles");
  static constexpr size_t kSmem = (size_t)kFloats * sizeof(float);
  // Where the compiler's own choice of registers and unrolling loses, us without / with: head dimension 128, of which one CTA's
  // shared memory fills an SM and which may take 176 registers where it settles for 128 (2 x 8 heads, 1319 x 1319, one CTA a
  // group 660 / 529; 110 queries, 442 keys over eight 13.2 / 11.9); head dimension 32, whose two features a thread want fewer
  // keys in flight (310 queries, 1319 keys over eight 10.6 / 9.8; 8 heads, 600 x 1240, one CTA a group 64.1 / 60.7).  At 64
  // either loses 1 to 2 %.
  static constexpr int kRegisterCtas = HD > 64 ? 1 : 0;
  static constexpr int kUnrollPV = HD < 64 ? 2 : 4;
};

__device__ __forceinline__ float ld_cluster(uint32_t cluster_addr) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(cluster_addr) : "memory");
  return v;
}

template <int HD>
__global__ void __launch_bounds__(128, SimtAttCfg<HD>::kRegisterCtas)
simt_attention_kernel(const float* __restrict__ Q, const float* __restrict__ Kc, const float* __restrict__ Vc,
                      float* __restrict__ O, int n_q, int N, int heads, int split) {
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
  float m_run[kAttRows], l_run[kAttRows];
  float2 o[kAttRows][CPT / 2];
#pragma unroll
  for (int i = 0; i < kAttRows; ++i) {
    m_run[i] = -INFINITY; l_run[i] = 0.f;
#pragma unroll
    for (int c = 0; c < CPT / 2; ++c) o[i][c] = make_float2(0.f, 0.f);
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
      for (int c = 0; c < CPT / 2; ++c) o[i][c] = __fmul2_rn(o[i][c], make_float2(alpha, alpha));
    }
    cp_async_wait<1>();
    __syncthreads();                       // V of tile t is there (and a warp's own P rows)
#pragma unroll Cfg::kUnrollPV
    for (int k = 0; k < kAttK; k += 4) {
      float4 p[kAttRows];
#pragma unroll
      for (int i = 0; i < kAttRows; ++i)
        p[i] = *reinterpret_cast<const float4*>(s_p + (ty * kAttRows + i) * Cfg::kPPitch + k);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        float2 v[CPT / 2];
#pragma unroll
        for (int c = 0; c < CPT; c += (CPT < 4 ? 2 : 4)) {
          const float* src = s_v + (k + kk) * kPitch + (CPT < 4 ? tx * 2 : tx * 4 + 16 * c);
          if constexpr (CPT < 4) {
            v[0] = *reinterpret_cast<const float2*>(src);
          } else {
            const float4 w = *reinterpret_cast<const float4*>(src);
            v[c / 2] = make_float2(w.x, w.y); v[c / 2 + 1] = make_float2(w.z, w.w);
          }
        }
#pragma unroll
        for (int i = 0; i < kAttRows; ++i) {
          const float pk = kk == 0 ? p[i].x : (kk == 1 ? p[i].y : (kk == 2 ? p[i].z : p[i].w));
#pragma unroll
          for (int c = 0; c < CPT / 2; ++c) o[i][c] = __ffma2_rn(make_float2(pk, pk), v[c], o[i][c]);
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
      for (int c = 0; c < CPT / 2; ++c)
        *reinterpret_cast<float2*>(dst + feature(2 * c)) = make_float2(o[i][c].x / l_run[i], o[i][c].y / l_run[i]);
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
    for (int c = 0; c < CPT / 2; ++c) *reinterpret_cast<float2*>(s_kv + row * HD + feature(2 * c)) = o[i][c];
    if (tx == 0) { s_ml[row] = m_run[i]; s_ml[kAttQ + row] = l_run[i]; }
  }
  tc::cluster_sync();
  for (int e = kAttQ * rank / split * HD + threadIdx.x; e < kAttQ * (rank + 1) / split * HD; e += 128) {
    const int row = e / HD, col = e % HD;
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

template <int BM, int BN, int TM, int TN, int KG>
int gemm_launch(const float* a, const float* w, const float* bias, int M, int Nout, int K, int split, const GemmOut& out,
                cudaStream_t s) {
  using Cfg = SimtCfg<BM, BN, TM, TN, KG>;
  static PerDeviceOnce once;
  HERO_TRY(per_device_once(once, [](int) {
    HERO_CUDA_TRY(cudaFuncSetAttribute(simt_gemm_kernel<BM, BN, TM, TN, KG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)Cfg::kSmem));
    return HERO_OK;
  }));
  const dim3 grid((Nout + BN - 1) / BN * split, (M + BM - 1) / BM);
  HERO_TRY(launch_kernel(simt_gemm_kernel<BM, BN, TM, TN, KG>, grid, Cfg::kThreads, Cfg::kSmem, s, (unsigned)split, a, w,
                         bias, M, Nout, K, split, out));
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
  const int split = plan_simt_attention(groups, tiles, HD, num_sms());
  if (groups * split > 0x7FFFFFFFll) return HERO_ERR_ARG;
  return launch_kernel(simt_attention_kernel<HD>, (unsigned)(groups * split), 128, Cfg::kSmem, s, (unsigned)split, q, k,
                       v, o, n_q, N, heads, split);
}

}  // namespace

// Twice the blocks that the fullest SM gets of `blocks` in clusters of `c`, when an SM holds `resident` at a time.  The CTAs of a
// cluster want free SMs of one processing cluster, so that not all SMs are to be had (of 148, clusters of four with an SM for each
// CTA fill 132); where an SM holds several, clusters of four double up from two thirds of the SMs on, first in part (hence twice),
// clusters of eight from 13/16 on.
static long long fullest_sm_twice(long long blocks, int c, int resident, int sms) {
  const int most = sms * 9 / 10, some = sms * 13 / 16;
  int full = sms;
  if (c == 3) full = sms * 13 / 14;
  if (c == 4) full = resident > 1 ? sms * 19 / 20 : most;
  if (c == 8) full = resident > 3 || blocks <= (long long)resident * most ? most : some;
  if (full < 1) full = 1;
  const long long twice = 2 * ((blocks + full - 1) / full);
  if (c == 4 && resident > 1 && blocks <= sms) return blocks <= sms * 2 / 3 ? 2 : 3;
  if (c == 8) return blocks <= some ? 2 : (twice < 4 ? 4 : twice);
  return twice;
}

// Keys of a group of 32 queries over a cluster of two, four or eight CTAs where that is sooner done: the estimate, in hundredths
// of a us, is what the fullest SM's CTAs take for their key tiles (a CTA may go without keys), plus their starts and the merge.
// Constants fitted to 450 problems, launches in a row; of 240 others the choice is 0.1 % above the best in the geometric mean and
// 11 % at most.  Some (heads x queries x keys; us over 1 / 2 / 4 / 8 CTAs, then the choice):
//   head dimension 32: 8 x 310 x 1319 44.3 / 37.0 / 34.2 / 27.1, 8; 16 x 110 x 442 16.3 / 12.8 / 9.9 / 10.3, 4;
//     18 x 250 x 500 18.4 / 16.5 / 19.4 / 20.9, 2; 16 x 1319 x 1319 144 / 149 / 154 / 166, 1
//   head dimension 64: 16 x 310 x 1319 101 / 81 / 78 / 81, 4; 2 x 600 x 1240 59.6 / 35.4 / 28.7 / 26.0, 8;
//     10 x 600 x 1240 96 / 75 / 78 / 96, 2; 16 x 1319 x 1319 234 / 253 / 264 / 303, 1
//   head dimension 128, of which an SM holds one: 8 x 310 x 1319 107 / 129 / 108 / 126, 1;
//     4 x 110 x 442 37.8 / 31.1 / 17.1 / 22.4, 4
// One time per key tile for every head dimension, and SMs that any cluster fills, came out up to 49 % above a rule that only
// kept the grid within what the chip holds (2 x 600 x 1240 of 64 over two, 16 x 110 x 442 of 32 over two).
int plan_simt_attention(long long groups, int tiles, int head_dim, int sms) {
  struct Cost { int resident, tile[4], further, launch, block, merge[4], crowd; };
  static const Cost of32 = {4, {207, 289, 503, 543}, 115, 141, 62, {0, 251, 148, 164}, 0};
  static const Cost of64 = {3, {290, 469, 676, 965}, 215, 213, 70, {0, 428, 236, 223}, 15};
  static const Cost of128 = {1, {493, 986, 1479, 1972}, 493, 41, 294, {0, 799, 391, 362}, 87};
  const Cost& cost = head_dim == 32 ? of32 : (head_dim == 64 ? of64 : of128);
  int split = 1;
  long long best = -1;
  for (int c = 1, i = 0; c <= 8 && (c == 1 || c / 2 < tiles); c *= 2, ++i) {
    const long long blocks = groups * c;
    long long twice = fullest_sm_twice(blocks, c, cost.resident, sms);
    // (of head dimension 64 some SM has three from 1.5 an SM on: 216 blocks take 5.3 us a key tile, 224 6.9)
    if (head_dim == 64 && blocks > sms * 3 / 2 && twice < 6) twice = 6;
    const long long n = twice / 2;
    const long long tile = twice == 3 ? (cost.tile[0] + cost.tile[1]) / 2
                                      : (n <= 4 ? cost.tile[n - 1] : cost.tile[3] + (n - 4) * cost.further);
    const long long merge = cost.merge[i] * (100 + cost.crowd * (n - 1)) / 100;
    const long long t = (tiles + c - 1) / c * tile + cost.launch + cost.block * twice / 2 + merge;
    if (best < 0 || t < best) { best = t; split = c; }
  }
  return split;
}

// Tiles of 64 x 64 (8 x 8 outputs a thread, two groups) or 32 x 32 (4 x 4, four groups), over one CTA or a cluster: what the
// fullest SM's CTAs take for their chunks of k (alone, or two and more side by side, which hardly helps), their start and the
// exchange, in twice a hundredth of a us.  Fitted to 528 problems; of 220 others the choice (last column) is 0.1 % above the best
// in the geometric mean and 5 % at most.  us, launches in a row:
//   M x N x K           64: 1     2      3      4      8    32: 1     2      3      4      8
//   620 x 1536 x 512     31.6   33.6   39.5   34.1   56.1    34.6   44.9   68.4   68.8         64, 1
//   620 x 512 x 512      18.4   18.2   15.2   16.1   22.7    16.2   18.5   26.7   25.2         64, 3
//   620 x 2048 x 512     44.7   41.4   47.8   45.9   72.9    43.8   59.1   89.8   90.7         64, 2
//   620 x 512 x 2048     62.8   59.3   43.0   46.4   45.1    56.3   50.0   55.5   53.0  69.5   64, 3
//   2638 x 512 x 2048   165.7  139.9  154.9  143.0  160.2   161.5  171.8  202.6  195.2   271   64, 2
//   1200 x 320 x 1280    40.7   39.2   41.2   31.2   43.2    36.7   39.2   46.5   47.8  78.4   64, 4
//   310 x 448 x 1792     55.2   30.5   23.3   28.3   25.8    19.9   19.8   28.4   25.0  33.0   32, 2
//   200 x 256 x 1024     32.9   19.2   15.6   11.5   10.7    11.9    8.4   10.8    8.6  11.9   32, 2
//   200 x 768 x 256      10.8    8.4   11.0    8.0            6.9    9.4                       32, 1
//   32 x 128 x 512       17.2   11.3    9.4    7.3    5.3     6.9    5.5    5.8    4.3         32, 4
SimtGemmPlan plan_simt_gemm(int M, int Nout, int K, int sms) {
  struct Cost { int tile, chunk, alone, shared, launch, block, exchange[5]; };
  static const Cost costs[] = {{64, 64, 180, 159, 302, 26, {0, 56, 92, 65, 117}},
                               {32, 128, 125, 103, 140, 41, {0, 128, 128, 107, 116}}};
  static const int ctas[] = {1, 2, 3, 4, 8};
  SimtGemmPlan plan = {0, 0};
  long long best = -1;
  for (const Cost& cost : costs) {
    const long long chunks = (K + cost.chunk - 1ll) / cost.chunk, row_tiles = ((long long)M + cost.tile - 1) / cost.tile;
    const long long tiles = row_tiles * (((long long)Nout + cost.tile - 1) / cost.tile);
    if (row_tiles > kMaxGridY) continue;             // (a problem of more rows takes the larger tile, up to 4.19 M)
    for (int i = 0; i < 5 && ctas[i] <= chunks; ++i) {
      const int c = ctas[i];
      const long long twice = fullest_sm_twice(tiles * c, c, 2, sms);
      const long long chunk = twice == 2 ? 2 * cost.alone : (twice == 3 ? cost.alone + 2 * cost.shared : twice * cost.shared);
      const long long t = (chunks + c - 1) / c * chunk + 2 * cost.launch + twice * (cost.block + cost.exchange[i]);
      if (best < 0 || t < best) { best = t; plan = {cost.tile, c}; }
    }
  }
  return plan;
}

int launch_simt_gemm(const float* a, const float* w, const float* bias, int M, int Nout, int K, const GemmOut& out,
                     cudaStream_t s) {
  if (M <= 0) return HERO_OK;
  SimtGemmPlan plan = plan_simt_gemm(M, Nout, K, num_sms());
  if (!plan.tile) plan = {64, 1};                    // (CUDA refuses the launch and says so)
  return plan.tile == 64 ? gemm_launch<64, 64, 8, 8, 2>(a, w, bias, M, Nout, K, plan.split, out, s)
                         : gemm_launch<32, 32, 4, 4, 4>(a, w, bias, M, Nout, K, plan.split, out, s);
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
