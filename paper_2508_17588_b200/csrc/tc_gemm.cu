// bf16 GEMM of the refresh path on the 5th-generation tensor cores:
//   C[M, Nout] = A[M, K] * W[Nout, K]^T + bias   (fp32 accumulation in TMEM)
// followed by the epilogue of Eq. 2 / Eq. 3: optional GELU-tanh or gate, bf16 rounding, and
// rows written either compactly or straight into their slots of a [B, N, D] cache.
//
// Two kernels (launch_tc_gemm says which runs when):
//  * tc_gemm_pair_kernel for problems that fill the chip: persistent CTA pairs on 256-row tiles (cta_group::2);
//  * tc_gemm_split_kernel for the others: one 128-row tile per CTA, the K loop cut over the CTAs of a cluster.
#include <cuda.h>

#include <mutex>

#include "hero_internal.h"
#include "tc_common.cuh"

namespace hero {

// ---------------------------------------------------------------------------
// Driver entry point for tensor-map encoding (resolved at run time: no -lcuda needed)
// ---------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn g_encode = nullptr;
static std::once_flag g_encode_once;

int tc_init_driver_api() {
  std::call_once(g_encode_once, [] {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      g_encode = reinterpret_cast<EncodeTiledFn>(fn);
  });
  if (!g_encode) {
    set_cuda_error(cudaErrorUnknown, "cuTensorMapEncodeTiled not available");
    return HERO_ERR_CUDA;
  }
  return HERO_OK;
}

// bf16 tensor [.., rows, cols] with cols contiguous; box = box_rows x 64 columns (128 bytes), 128B swizzle,
// out-of-range elements read as zero.
int make_tmap_bf16(CUtensorMap* m, const void* base, int rank, const uint64_t* dims, const uint64_t* strides_bytes,
                   const uint32_t* box) {
  HERO_TRY(tc_init_driver_api());
  cuuint64_t gdim[3];
  cuuint64_t gstr[2];
  cuuint32_t bx[3], es[3];
  for (int i = 0; i < rank; ++i) { gdim[i] = dims[i]; bx[i] = box[i]; es[i] = 1; }
  for (int i = 0; i + 1 < rank; ++i) gstr[i] = strides_bytes[i];
  CUresult r = g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(base), gdim, gstr,
                        bx, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    set_cuda_error(cudaErrorInvalidValue, "cuTensorMapEncodeTiled");
    return HERO_ERR_CUDA;
  }
  return HERO_OK;
}

namespace {
using namespace tc;

constexpr int kBM = 128, kBK = 64;                     // rows of A per CTA; K step (one 128-byte swizzle row)
constexpr int kABytes = kBM * kBK * 2;                 // 16 KB
constexpr int kGemmThreads = 320;                      // producer, issuer, eight epilogue warps
constexpr int kEpiWarps = 8;                           // two per TMEM lane quadrant, each with half of a tile's columns
constexpr size_t kAlignSlack = 1024, kBarrierBytes = 512;

__device__ __forceinline__ float gelu_tanh_f(float t) {
  // 0.5 t (1 + tanh(sqrt(2/pi) (t + 0.044715 t^3))) with the hardware tanh (one special-function
  // instruction, relative error 2^-11: below the bf16 rounding of the result).  The epilogue shares the
  // SM's power budget with the tensor core, so every instruction saved here is tensor clock gained.
  const float t2 = t * t;
  const float u = t * fmaf(0.0356774081f, t2, 0.7978845608f);
  float th;
  asm("tanh.approx.f32 %0, %1;" : "=f"(th) : "f"(u));
  const float h = 0.5f * t;
  return fmaf(h, th, h);
}

// Where one accumulator row goes.
struct RowOut {
  bool ok;                 // the row exists
  int m, b;                // row of the compact operand, its batch item
  long long scat;          // its row in a [B, n_rows] destination
};
__device__ __forceinline__ RowOut row_out(const GemmOut& out, int m, int M) {
  RowOut r;
  r.ok = m < M;
  r.m = m; r.b = 0; r.scat = 0;
  if (r.ok) {
    r.b = m / out.n_sel;
    const int li = m - r.b * out.n_sel;
    r.scat = (long long)r.b * out.n_rows + (out.idx ? __ldg(out.idx + li) : li);
  }
  return r;
}

// Finish NC accumulator columns [n0, n0 + NC) of one row, all of one segment: bias (fp32, staged in shared memory),
// activation, scale or gate, bf16, full 32-byte sectors per lane (16-byte stores where the destination is not 32-byte
// aligned or ends inside the columns).
template <int NC>
__device__ __forceinline__ void emit(const uint32_t (&acc)[NC], const float* s_bias, int n0, int Nout, const GemmOut& out,
                                     const RowOut& row) {
  float2 f[NC / 2];
#pragma unroll
  for (int v = 0; v < NC / 4; ++v) {
    const float4 b4 = *reinterpret_cast<const float4*>(s_bias + v * 4);
    f[2 * v] = __fadd2_rn(make_float2(__uint_as_float(acc[4 * v]), __uint_as_float(acc[4 * v + 1])), make_float2(b4.x, b4.y));
    f[2 * v + 1] = __fadd2_rn(make_float2(__uint_as_float(acc[4 * v + 2]), __uint_as_float(acc[4 * v + 3])), make_float2(b4.z, b4.w));
  }
  // (segments are selected, not indexed or divided for: at most three, and a parameter indexed at run time would be
  // copied to local memory)
  const bool s1 = n0 >= out.seg_cols, s2 = n0 >= 2 * out.seg_cols;        // warp-uniform
  const int col0 = n0 - (s2 ? 2 * out.seg_cols : (s1 ? out.seg_cols : 0));
  if (out.act == 1) {
#pragma unroll
    for (int i = 0; i < NC / 2; ++i) f[i] = make_float2(gelu_tanh_f(f[i].x), gelu_tanh_f(f[i].y));
  }
  if (out.seg0_scale != 0.f && !s1) {
#pragma unroll
    for (int i = 0; i < NC / 2; ++i) f[i] = __fmul2_rn(f[i], make_float2(out.seg0_scale, out.seg0_scale));
  }
  if (!row.ok) return;
  if (out.gate) {
    const float* gate = out.gate + (long long)row.b * out.gate_ld + col0;
#pragma unroll
    for (int i = 0; i < NC / 2; ++i)
      if (n0 + 2 * i < Nout) f[i] = __fmul2_rn(f[i], __ldg(reinterpret_cast<const float2*>(gate + 2 * i)));
  }
  uint32_t packed[NC / 2];
#pragma unroll
  for (int i = 0; i < NC / 2; ++i) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(f[i].x, f[i].y);
    packed[i] = *reinterpret_cast<const uint32_t*>(&p);
  }
  void* const base = s2 ? out.ptr[2] : (s1 ? out.ptr[1] : out.ptr[0]);
  const long long ld = s2 ? out.ld[2] : (s1 ? out.ld[1] : out.ld[0]);
  const int scatter = s2 ? out.scatter[2] : (s1 ? out.scatter[1] : out.scatter[0]);
  __nv_bfloat16* dst = static_cast<__nv_bfloat16*>(base) + (scatter ? row.scat : (long long)row.m) * ld + col0;
  if (n0 + NC <= Nout && (reinterpret_cast<uintptr_t>(dst) & 31) == 0) {
#pragma unroll
    for (int v = 0; v < NC / 16; ++v) st_global_v8(dst + v * 16, &packed[v * 8]);
  } else {
#pragma unroll
    for (int v = 0; v < NC / 8; ++v)
      if (n0 + v * 8 < Nout)
        *reinterpret_cast<uint4*>(dst + v * 8) = make_uint4(packed[4 * v], packed[4 * v + 1], packed[4 * v + 2], packed[4 * v + 3]);
  }
}

// (a kernel without this treatment has no use for the parameter)
template <bool QK> struct QkParam {};
template <> struct QkParam<true> : QkEpilogue {};

// What the q and k columns of a row go through besides (QkEpilogue): where its angles stand in the table, worked out
// while the MMAs run.  Pairs 0..7 of a head turn with the frame, 8..19 with the grid row, 20..31 with the grid column.
struct RowAngles { int t, h, w; };           // entry of the axis' first pair; t < 0: the row is not turned
constexpr int kPairsT = 8, kPairsH = 12;
__device__ __forceinline__ RowAngles row_angles(const QkEpilogue& qk, const RowOut& row, int n_rows) {
  RowAngles a = {-1, 0, 0};
  const int token = (int)(row.scat - (long long)row.b * n_rows) - qk.n_text;
  if (row.ok && qk.rope != nullptr && token >= 0) {
    const int per_frame = qk.grid_h * qk.grid_w;
    const int ft = token / per_frame, in_frame = token - ft * per_frame;
    const int gh = in_frame / qk.grid_w, gw = in_frame - gh * qk.grid_w;
    a.t = ft * kPairsT;
    a.h = qk.frames * kPairsT + gh * kPairsH;
    a.w = qk.frames * kPairsT + qk.grid_h * kPairsH + gw * kPairsH;
  }
  return a;
}
// Finish one head (64 columns from n0 on) of one row of the QKV projection: bias, for q and k the LayerNorm over the
// head's features and the turn by the row's position, for q the softmax scale; bf16; stored as in emit.  The row never
// leaves the thread's registers between the projection and its final form: a pass of its own over q and the fresh rows of
// the K cache read and wrote them once more (77 us in a block of 5940 rows x 3072: that cached step of 6 blocks 10.08 ->
// 9.84 ms; of 4 blocks of 371 x 768 228 -> 222 us).
__device__ __forceinline__ void emit_head(const uint32_t (&acc)[2][32], const float* s_bias, int n0, const GemmOut& out,
                                          const RowOut& row, const QkEpilogue& qk, const RowAngles& ang) {
  float2 f[32];
#pragma unroll
  for (int v = 0; v < 16; ++v) {
    const float4 b4 = *reinterpret_cast<const float4*>(s_bias + v * 4);
    const uint32_t* a = &acc[v / 8][(v % 8) * 4];
    f[2 * v] = __fadd2_rn(make_float2(__uint_as_float(a[0]), __uint_as_float(a[1])), make_float2(b4.x, b4.y));
    f[2 * v + 1] = __fadd2_rn(make_float2(__uint_as_float(a[2]), __uint_as_float(a[3])), make_float2(b4.z, b4.w));
  }
  const int seg = n0 >= 2 * out.seg_cols ? 2 : (n0 >= out.seg_cols ? 1 : 0);            // warp-uniform
  if (seg < 2 && qk.qn_w != nullptr) {
    float2 s2 = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < 32; ++i) s2 = __fadd2_rn(s2, f[i]);
    const float mu = (s2.x + s2.y) * (1.0f / 64.0f);
    float2 q2 = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      f[i] = __fadd2_rn(f[i], make_float2(-mu, -mu));
      q2 = __ffma2_rn(f[i], f[i], q2);
    }
    const float rstd = rsqrtf((q2.x + q2.y) * (1.0f / 64.0f) + qk.eps);
    const uint4* gw = static_cast<const uint4*>(seg ? qk.kn_w : qk.qn_w);
    const uint4* gb = static_cast<const uint4*>(seg ? qk.kn_b : qk.qn_b);
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      const uint4 w4 = __ldg(gw + v), b4 = __ldg(gb + v);
      const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int q = 0; q < 4; ++q)
        f[4 * v + q] = __ffma2_rn(__fmul2_rn(f[4 * v + q], make_float2(rstd, rstd)),
                                  make_float2(__uint_as_float(w[q] << 16), __uint_as_float(w[q] & 0xFFFF0000u)),
                                  make_float2(__uint_as_float(b[q] << 16), __uint_as_float(b[q] & 0xFFFF0000u)));
    }
  }
  if (seg < 2 && ang.t >= 0) {
#pragma unroll
    for (int i = 0; i < 32; i += 2) {
      const int entry = i < kPairsT ? ang.t + i : (i < kPairsT + kPairsH ? ang.h + i - kPairsT : ang.w + i - kPairsT - kPairsH);
      const float4 cs = __ldg(reinterpret_cast<const float4*>(qk.rope + entry));         // two (cos, sin)
      const float2 x = f[i], y = f[i + 1];
      f[i] = make_float2(x.x * cs.x - x.y * cs.y, x.x * cs.y + x.y * cs.x);
      f[i + 1] = make_float2(y.x * cs.z - y.y * cs.w, y.x * cs.w + y.y * cs.z);
    }
  }
  if (seg == 0) {
#pragma unroll
    for (int i = 0; i < 32; ++i) f[i] = __fmul2_rn(f[i], make_float2(qk.q_scale, qk.q_scale));
  }
  if (!row.ok) return;
  void* const base = seg == 2 ? out.ptr[2] : (seg == 1 ? out.ptr[1] : out.ptr[0]);
  const long long ld = seg == 2 ? out.ld[2] : (seg == 1 ? out.ld[1] : out.ld[0]);
  const int scatter = seg == 2 ? out.scatter[2] : (seg == 1 ? out.scatter[1] : out.scatter[0]);
  __nv_bfloat16* dst = static_cast<__nv_bfloat16*>(base) + (scatter ? row.scat : (long long)row.m) * ld + n0 - seg * out.seg_cols;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    uint32_t packed[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const __nv_bfloat162 p = __floats2bfloat162_rn(f[8 * v + i].x, f[8 * v + i].y);
      packed[i] = *reinterpret_cast<const uint32_t*>(&p);
    }
    if ((reinterpret_cast<uintptr_t>(dst) & 31) == 0) {
      st_global_v8(dst + v * 16, packed);
    } else {
      *reinterpret_cast<uint4*>(dst + v * 16) = make_uint4(packed[0], packed[1], packed[2], packed[3]);
      *reinterpret_cast<uint4*>(dst + v * 16 + 8) = make_uint4(packed[4], packed[5], packed[6], packed[7]);
    }
  }
}

// A warp puts NC bias values from column n_base on into its own piece of shared memory, in fp32 (values past the end
// of the row are not read by anybody).
template <int NC>
__device__ __forceinline__ void stage_bias(float* s_bias, const __nv_bfloat16* bias, int n_base, int Nout, int lane) {
  for (int v = lane; v < NC / 8; v += 32)
    if (n_base + v * 8 < Nout) {
      const uint4 raw = __ldg(reinterpret_cast<const uint4*>(bias + n_base + v * 8));
      const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
      for (int q = 0; q < 2; ++q)
        *reinterpret_cast<float4*>(s_bias + v * 8 + 4 * q) =
            make_float4(__uint_as_float(w[2 * q] << 16), __uint_as_float(w[2 * q] & 0xFFFF0000u),
                        __uint_as_float(w[2 * q + 1] << 16), __uint_as_float(w[2 * q + 1] & 0xFFFF0000u));
    }
  __syncwarp();
}

// ---------------------------------------------------------------------------------------------------------------
// Problems that fill the chip.  Persistent clusters of two CTAs, one per pair of SMs, on tiles of 256 x BN: each
// CTA fetches its own 128 rows of A and half of the tile's rows of W, so a K step of 64 costs an SM 32 KB from L2
// (BN = 256) for the 4.2 MFLOP it computes, two thirds of what a 128 x 256 tile per CTA costs, and the tensor core
// reads each operand half from its own SM's shared memory once.
//   warp 0      TMA producer (both CTAs, each its own operand rows; all bytes reported to the even CTA's barrier)
//   warp 1      MMA issuer (even CTA only): 4 x tcgen05.mma M256 N=BN K16 per stage; the commit frees both CTAs' stage
//   warps 2..9  epilogue (both CTAs, each its own 128 rows; two warps share 32 rows, half of the columns each)
// Two accumulators in TMEM let the epilogue of tile i overlap the MMAs of tile i + 1.
// Bound: at BN = 256 the tensor core (512 clocks a K step) and what an SM can fetch from L2 (64 bytes a clock, 512
// clocks for 32 KB) meet; at large sizes the 1 kW cap lowers the clock of both.  Measured, 8774 x 9216 x 3072: 325 us,
// 1530 TFLOP/s (one CTA per 128 x 256 tile, 48 KB a step: 352 us, bound by the fetch); 8774 x 3072 x 12288: 443 us
// (481); 3510 x 3072 x 12288: 188 us on 256 x 224 (the narrower tile leaves the last of three rounds fuller: 200 on
// 256 x 256).
// ---------------------------------------------------------------------------------------------------------------
template <int BN>
struct PairCfg {
  static constexpr int kBBytes = BN / 2 * kBK * 2;
  static constexpr int kStageBytes = kABytes + kBBytes;
  static constexpr int kStages = 196608 / kStageBytes;         // 192 KB: 6 (BN = 256) to 8 (BN = 128)
  static constexpr int kTmemCols = 2 * BN > 256 ? 512 : 256;   // (a power of two)
  static constexpr size_t kBiasBytes = kEpiWarps * 2 * (BN / 2) * 4;   // a warp's columns of two tiles
  static constexpr size_t kSmem = kAlignSlack + (size_t)kStages * kStageBytes + kBiasBytes + kBarrierBytes;
};

// Tile order of the persistent pairs.  Consecutive tile numbers run down kGroupM row tiles (of 256) before moving to
// the next column tile, and only then to the next band of rows: the 74 tiles in flight at any time then cover about
// 12 x 6 tiles, whose operands stay in L2 and are shared by the pairs working on them, instead of every pair
// streaming its own panel of A from DRAM.
constexpr int kGroupM = 12;
__device__ __forceinline__ void tile_coords(int tile, int m_tiles, int n_tiles, int& mt, int& nt) {
  const int per_group = kGroupM * n_tiles;
  const int group = tile / per_group;
  const int first_m = group * kGroupM;
  const int rows = min(kGroupM, m_tiles - first_m);
  const int r = tile - group * per_group;
  mt = first_m + r % rows;
  nt = r / rows;
}

template <int BN, bool QK>
__global__ void __launch_bounds__(kGemmThreads, 1)
tc_gemm_pair_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_w,
                    const __nv_bfloat16* __restrict__ bias, const GemmOut out, const QkParam<QK> qk, int M, int Nout, int K,
                    int* __restrict__ status) {
  static_assert(!QK || BN % 128 == 0, "an epilogue warp's columns are whole heads");
  using Cfg = PairCfg<BN>;
  constexpr int kStages = Cfg::kStages;
  extern __shared__ uint8_t smem_raw[];
  // The dynamic shared memory starts at the same offset in both CTAs, and so does everything carved from it: a
  // descriptor or a barrier offset means the same place in either.
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  float* s_bias_all = reinterpret_cast<float*>(smem + (size_t)kStages * Cfg::kStageBytes);
  uint64_t* bars = reinterpret_cast<uint64_t*>(reinterpret_cast<uint8_t*>(s_bias_all) + Cfg::kBiasBytes);
  uint64_t* full = bars;                    // [kStages] both CTAs' TMA -> MMA (the even CTA's is the one in use)
  uint64_t* empty = bars + kStages;         // [kStages] MMA -> TMA (each CTA its own)
  uint64_t* acc_full = bars + 2 * kStages;  // [2] MMA -> epilogue (each CTA its own)
  uint64_t* acc_empty = acc_full + 2;       // [2] both CTAs' epilogues -> MMA (the even CTA's)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const int m_tiles = (M - 1) / (2 * kBM) + 1, n_tiles = (Nout + BN - 1) / BN;
  const int n_tiles_total = m_tiles * n_tiles;
  const int k_blocks = (K + kBK - 1) / kBK;

  if (threadIdx.x == 0) {
    for (int i = 0; i < kStages; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], 2 * kEpiWarps); }
    *abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == 0 && lane == 0) { tma_prefetch_desc(&tm_a); tma_prefetch_desc(&tm_w); }
  if (warp == 1) tmem_alloc_pair(tmem_slot, Cfg::kTmemCols);
  tc_fence_before();
  __syncwarp();
  cluster_sync();                           // both CTAs' barriers exist before anybody signals across
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      int stage = 0; uint32_t phase = 0;
      bool ok = true;
      auto load = [&](int kb, int row, bool weights) {
        const uint32_t sa = smem_u32(smem + (size_t)stage * Cfg::kStageBytes), bar = cluster_map(smem_u32(&full[stage]), 0);
        if (weights) tma_load_2d_pair(sa + kABytes, &tm_w, bar, kb * kBK, row);
        else tma_load_2d_pair(sa, &tm_a, bar, kb * kBK, row);
      };
      // The even CTA's barrier counts the bytes of both CTAs.  The odd CTA's may land before it is armed: its
      // phase cannot complete before the arrival that arms it.
      int ahead = 0;                         // stages whose weights were fetched before the wait for the kernel before
      for (int tile = pair; tile < n_tiles_total && ok; tile += n_pairs) {
        int mt, nt;
        tile_coords(tile, m_tiles, n_tiles, mt, nt);
        const int row_a = (2 * mt + (int)rank) * kBM, row_w = nt * BN + (int)rank * (BN / 2);
        if (tile == pair) {
          if (out.weights_settled) {
            for (; ahead < kStages && ahead < k_blocks; ++ahead) {
              stage = ahead;
              if (rank == 0) mbar_expect_tx(&full[stage], 2 * Cfg::kStageBytes);
              load(ahead, row_w, true);
            }
            stage = 0;
          }
          stream_order();
        }
        for (int kb = 0; kb < k_blocks; ++kb) {
          if (ahead > 0) {
            --ahead;
          } else {
            if (!(ok = mbar_wait(&empty[stage], phase ^ 1, abort_flag))) break;
            if (rank == 0) mbar_expect_tx(&full[stage], 2 * Cfg::kStageBytes);
            load(kb, row_w, true);
          }
          load(kb, row_a, false);
          if (++stage == kStages) { stage = 0; phase ^= 1; }
        }
      }
      // On the way out make sure every stage that was armed has been consumed (bounded): the CTA must
      // not retire with bulk copies still writing its shared memory.
      for (int i = 0; i < kStages; ++i) {
        if (!mbar_wait(&empty[stage], phase ^ 1, abort_flag)) break;
        if (++stage == kStages) { stage = 0; phase ^= 1; }
      }
    } else {
      stream_order();
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (even CTA)
    // All 32 lanes run the loop and one elected lane issues: tile counters, stage addresses and descriptors
    // then stay warp-uniform values instead of one diverged lane's private registers, which is what the
    // tensor-core instructions are fed from.
    stream_order();
    if (rank == 0) {
      const bool leader = elect_one();
      constexpr uint32_t idesc = idesc_bf16(2 * kBM, BN, 0);
      int stage = 0; uint32_t phase = 0;
      bool ok = true;
      int t = 0;
      for (int tile = pair; tile < n_tiles_total && ok; tile += n_pairs, ++t) {
        const int acc = t & 1;
        if (!(ok = mbar_wait_warp(&acc_empty[acc], ((t >> 1) & 1) ^ 1, abort_flag))) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)acc * BN;
        for (int kb = 0; kb < k_blocks; ++kb) {
          if (!(ok = mbar_wait_warp(&full[stage], phase, abort_flag))) break;
          tc_fence_after();
          const uint32_t sa = smem_u32(smem + (size_t)stage * Cfg::kStageBytes);
          const uint64_t da = smem_desc_sw128(sa, 1024), db = smem_desc_sw128(sa + kABytes, 1024);
          if (leader) {
#pragma unroll
            for (int k = 0; k < kBK / 16; ++k)   // +32 bytes (encoded >>4) per K step of 16 inside the swizzle atom
              mma_ss_pair(d_tmem, da + 2 * k, db + 2 * k, idesc, (kb | k) != 0);
            mma_commit_pair(&empty[stage]);
          }
          if (++stage == kStages) { stage = 0; phase ^= 1; }
        }
        if (ok && leader) mma_commit_pair(&acc_full[acc]);
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue (warps 2..9)
    stream_order();
    const int quad = warp & 3;                 // TMEM lane quadrant this warp may read
    const int half = (warp - 2) >> 2;          // which half of the tile's columns it finishes
    float* s_bias_warp = s_bias_all + (size_t)(warp - 2) * BN;
    bool ok = true;
    int t = 0;
    for (int tile = pair; tile < n_tiles_total && ok; tile += n_pairs, ++t) {
      int mt, nt;
      tile_coords(tile, m_tiles, n_tiles, mt, nt);
      const int acc = t & 1;
      const int n_first = nt * BN + half * (BN / 2);
      // bias and destination of this tile are fetched while its MMAs still run
      const float* s_bias = s_bias_warp + acc * (BN / 2);
      stage_bias<BN / 2>(s_bias_warp + acc * (BN / 2), bias, n_first, Nout, lane);
      const RowOut row = row_out(out, (2 * mt + (int)rank) * kBM + quad * 32 + lane, M);
      RowAngles ang = {};
      if constexpr (QK) ang = row_angles(qk, row, out.n_rows);
      ok = mbar_wait_warp(&acc_full[acc], (t >> 1) & 1, abort_flag);
      if (!ok) break;
      tc_fence_after();
      const uint32_t t_row = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc * BN + half * (BN / 2));
      if constexpr (QK) {
#pragma unroll 1
        for (int c = 0; c < BN / 2; c += 64) {
          uint32_t r[2][32];
          tmem_ld32(t_row + c, r[0]);
          tmem_ld32(t_row + c + 32, r[1]);
          tmem_ld_wait();
          if (n_first + c < Nout) emit_head(r, s_bias + c, n_first + c, out, row, qk, ang);          // warp-uniform
        }
      } else {
        constexpr int kCh = BN % 64 == 0 ? 32 : 16;      // columns per TMEM read: a divisor of the half tile, and of
        constexpr int kChunks = BN / 2 / kCh;            // its offset, so that no read straddles two segments
        uint32_t r[2][kCh];
        tmem_ld(t_row, r[0]);
#pragma unroll
        for (int c = 0; c < kChunks; ++c) {
          const int n0 = n_first + c * kCh;
          tmem_ld_wait();
          if (c + 1 < kChunks) tmem_ld(t_row + (c + 1) * kCh, r[(c + 1) & 1]);
          if (n0 < Nout) emit<kCh>(r[c & 1], s_bias + c * kCh, n0, Nout, out, row);      // warp-uniform
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(cluster_map(smem_u32(&acc_empty[acc]), 0));
    }
  }

  // ---------------------------------------------------------------- teardown
  tc_fence_before();
  __syncwarp();
  cluster_sync();                            // neither CTA leaves while the other may still reach into it
  if (threadIdx.x == 0 && *abort_flag) atomicExch(status, 1);
  if (warp == 1) { tc_fence_after(); tmem_dealloc_pair(tmem_base, Cfg::kTmemCols); }
}

// ---------------------------------------------------------------------------------------------------------------
// Problems that do not: one tile of 128 x BN per CTA, one launch wave, everything about latency.  A cluster of
// `split` CTAs shares a tile, each taking a run of its K steps; they then trade partial sums through distributed
// shared memory, each finishing BN / split of the tile's columns (the partial sums of the other CTAs are added in
// rank order, so a result does not depend on timing).  Warp roles as above; the epilogue warps fetch bias and
// destination rows while the MMAs run, and the producer fetches the first weights while the kernel before still runs.
// Bound by latency: of 3.4 us at 148 x 768 x 256 (4.0 without the early weights, 14.0 with one CTA per 128 x 256 tile and
// the bias fetched between accumulator reads) 1.1 us are the K loop, the rest is launch, first fetch and epilogue.
// 614 x 256 x 768 over two CTAs a tile: 4.2 us (4.6 over one), 371 x 768 x 3072 over four: 8.1 (13.2 over one).
// ---------------------------------------------------------------------------------------------------------------
template <int BN>
struct SplitCfg {
  static constexpr int kBBytes = BN * kBK * 2;
  static constexpr int kStageBytes = kABytes + kBBytes;
  static constexpr int kStages = BN == 128 ? 4 : 6;
  static constexpr int kBiasCols = 64;                         // a warp's columns at most
  static constexpr size_t kBiasBytes = kEpiWarps * kBiasCols * 4;
  static constexpr int kMaxSplit = 4;                          // a CTA finishes at least 16 columns
  static constexpr size_t part_bytes(int split) { return (size_t)(split - 1) * (BN / split) * kBM * 4; }
  static constexpr size_t smem(int split) {
    return kAlignSlack + (size_t)kStages * kStageBytes + part_bytes(split) + kBiasBytes + kBarrierBytes;
  }
};

template <int BN, bool QK>
__global__ void __launch_bounds__(kGemmThreads)
tc_gemm_split_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_w,
                     const __nv_bfloat16* __restrict__ bias, const GemmOut out, const QkParam<QK> qk, int M, int Nout, int K,
                     int split, int* __restrict__ status) {
  using Cfg = SplitCfg<BN>;
  constexpr int kStages = Cfg::kStages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  float* s_bias_all = reinterpret_cast<float*>(smem + (size_t)kStages * Cfg::kStageBytes);
  uint64_t* bars = reinterpret_cast<uint64_t*>(reinterpret_cast<uint8_t*>(s_bias_all) + Cfg::kBiasBytes);
  uint64_t* full = bars;                    // [kStages] TMA -> MMA
  uint64_t* empty = bars + kStages;         // [kStages] MMA -> TMA
  uint64_t* acc_full = bars + 2 * kStages;  // MMA -> epilogue
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_full + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float4* s_part = reinterpret_cast<float4*>(reinterpret_cast<uint8_t*>(bars) + kBarrierBytes);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = split > 1 ? (int)cluster_rank() : 0;
  const int tile = blockIdx.x / split;
  const int m_tiles = (M + kBM - 1) / kBM;
  const int mt = tile % m_tiles, nt = tile / m_tiles;
  const int k_blocks = (K + kBK - 1) / kBK;
  const int kb0 = k_blocks * rank / split, kb1 = k_blocks * (rank + 1) / split;

  if (threadIdx.x == 0) {
    for (int i = 0; i < kStages; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    mbar_init(acc_full, 1);
    *abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == 0 && lane == 0) { tma_prefetch_desc(&tm_a); tma_prefetch_desc(&tm_w); }
  if (warp == 1) { tmem_alloc(tmem_slot, BN); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (split > 1) cluster_arrive();           // waited for before anything is sent to another CTA
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      int stage = 0; uint32_t phase = 0;
      int ahead = kb0;                         // K steps whose weights were fetched before the wait for the kernel before
      if (out.weights_settled) {
        for (; ahead < kb1 && ahead < kb0 + kStages; ++ahead) {
          mbar_expect_tx(&full[ahead - kb0], Cfg::kStageBytes);
          tma_load_2d(smem + (size_t)(ahead - kb0) * Cfg::kStageBytes + kABytes, &tm_w, &full[ahead - kb0], ahead * kBK, nt * BN);
        }
      }
      stream_order();
      for (int kb = kb0; kb < kb1; ++kb) {
        uint8_t* sa = smem + (size_t)stage * Cfg::kStageBytes;
        if (kb >= ahead) {
          if (!mbar_wait(&empty[stage], phase ^ 1, abort_flag)) break;
          mbar_expect_tx(&full[stage], Cfg::kStageBytes);
          tma_load_2d(sa + kABytes, &tm_w, &full[stage], kb * kBK, nt * BN);
        }
        tma_load_2d(sa, &tm_a, &full[stage], kb * kBK, mt * kBM);
        if (++stage == kStages) { stage = 0; phase ^= 1; }
      }
      for (int i = 0; i < kStages; ++i) {      // all armed stages consumed before the CTA retires
        if (!mbar_wait(&empty[stage], phase ^ 1, abort_flag)) break;
        if (++stage == kStages) { stage = 0; phase ^= 1; }
      }
    } else {
      stream_order();
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    stream_order();
    const bool leader = elect_one();
    constexpr uint32_t idesc = idesc_bf16(kBM, BN, 0);
    int stage = 0; uint32_t phase = 0;
    bool ok = true;
    for (int kb = kb0; kb < kb1; ++kb) {
      if (!(ok = mbar_wait_warp(&full[stage], phase, abort_flag))) break;
      tc_fence_after();
      const uint32_t sa = smem_u32(smem + (size_t)stage * Cfg::kStageBytes);
      const uint64_t da = smem_desc_sw128(sa, 1024), db = smem_desc_sw128(sa + kABytes, 1024);
      if (leader) {
#pragma unroll
        for (int k = 0; k < kBK / 16; ++k) mma_ss(tmem_base, da + 2 * k, db + 2 * k, idesc, (kb > kb0) || k != 0);
        mma_commit(&empty[stage]);
      }
      if (++stage == kStages) { stage = 0; phase ^= 1; }
    }
    if (ok && leader) mma_commit(acc_full);
  }

  // ------------------------------------------------------------ epilogue (warps 2..9)
  const int quad = warp & 3;                 // TMEM lane quadrant this warp may read
  const int half = (warp - 2) >> 2;
  const int tile_row = quad * 32 + lane;
  const uint32_t t_row = tmem_base + ((uint32_t)(quad * 32) << 16);
  // This CTA finishes columns [rank * width, (rank + 1) * width) and this warp `mine` of them: half, or, where halves would
  // be less than a piece of 16 columns or than a head, the first warp of two all of them.
  const int width = BN / split;
  const bool alone = QK ? BN == 64 : width < 32;
  const int mine = alone ? (half == 0 ? width : 0) : width / 2;
  const int c_first = rank * width + (alone ? 0 : half * (width / 2));
  constexpr int kBiasCols = Cfg::kBiasCols;
  float* s_bias = s_bias_all + (size_t)(warp - 2) * kBiasCols;
  RowOut row = {};
  bool ok = true;
  if (warp >= 2) {
    stream_order();
    stage_bias<kBiasCols>(s_bias, bias, nt * BN + c_first, Nout, lane);
    row = row_out(out, mt * kBM + tile_row, M);
    ok = mbar_wait_warp(acc_full, 0, abort_flag);
    if (ok) tc_fence_after();
  }
  if (split > 1) {
    __syncwarp();
    cluster_wait();                          // the other CTAs have started (long since)
    if (warp >= 2 && ok) {
      // everybody else's columns go to them: slot of the sender, four columns per 16-byte word, row by row
      for (int c = half * 16; c < BN; c += 32) {
        const int owner = c / width;
        if (owner == rank) continue;         // warp-uniform
        uint32_t r[16];
        tmem_ld16(t_row + c, r);
        tmem_ld_wait();
        const int slot = rank < owner ? rank : rank - 1;
        const uint32_t base =
            cluster_map(smem_u32(s_part + ((size_t)slot * (width / 4) + (c - owner * width) / 4) * kBM + tile_row), (uint32_t)owner);
#pragma unroll
        for (int q = 0; q < 4; ++q)
          st_cluster_v4(base + q * kBM * 16, __uint_as_float(r[4 * q]), __uint_as_float(r[4 * q + 1]),
                        __uint_as_float(r[4 * q + 2]), __uint_as_float(r[4 * q + 3]));
      }
    }
    __syncwarp();
    cluster_sync();                          // every wait above is bounded, so everybody gets here
  }
  if constexpr (QK) {                        // (split is 1: the warp's 64 columns are one head)
    if (warp >= 2 && ok && mine > 0 && nt * BN + c_first < Nout) {
      uint32_t r[2][32];
      tmem_ld32(t_row + c_first, r[0]);
      tmem_ld32(t_row + c_first + 32, r[1]);
      tmem_ld_wait();
      emit_head(r, s_bias, nt * BN + c_first, out, row, qk, row_angles(qk, row, out.n_rows));
    }
  } else if (warp >= 2 && ok) {
    for (int c = c_first; c < c_first + mine; c += 16) {
      const int n0 = nt * BN + c;
      if (n0 >= Nout) break;                 // warp-uniform
      uint32_t r[16];
      tmem_ld16(t_row + c, r);
      tmem_ld_wait();
      for (int s = 0; s < split - 1; ++s) {
        const float4* part = s_part + ((size_t)s * (width / 4) + (c - rank * width) / 4) * kBM + tile_row;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float4 v = part[q * kBM];
          r[4 * q] = __float_as_uint(__uint_as_float(r[4 * q]) + v.x);
          r[4 * q + 1] = __float_as_uint(__uint_as_float(r[4 * q + 1]) + v.y);
          r[4 * q + 2] = __float_as_uint(__uint_as_float(r[4 * q + 2]) + v.z);
          r[4 * q + 3] = __float_as_uint(__uint_as_float(r[4 * q + 3]) + v.w);
        }
      }
      emit<16>(r, s_bias + (c - c_first), n0, Nout, out, row);
    }
  }

  // ---------------------------------------------------------------- teardown
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) atomicExch(status, 1);
  if (warp == 1) { tc_fence_after(); tmem_dealloc(tmem_base, BN); }
}

// Self-test of the bounded wait: the barrier below is initialised for one arrival that never comes.
__global__ void wait_timeout_selftest_kernel(int* __restrict__ status, unsigned long long budget_ns) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) { mbar_init(&bar, 1); abort_flag = 0; mbar_fence_init(); }
  __syncthreads();
  const bool ok = mbar_wait_warp(&bar, 0, &abort_flag, budget_ns);
  __syncthreads();
  if (threadIdx.x == 0 && (!ok || abort_flag)) atomicExch(status, 1);
}

}  // namespace

int launch_wait_timeout_selftest(int* d_status, int budget_us, cudaStream_t s) {
  wait_timeout_selftest_kernel<<<1, 64, 0, s>>>(d_status, (unsigned long long)budget_us * 1000ull);
  HERO_CUDA_TRY(cudaGetLastError());
  return HERO_OK;
}

// ---------------------------------------------------------------------------------------------------------------
// Which kernel, which tile, how many CTAs per tile.  The estimate is in SM clocks: rounds of tiles times K steps times
// the clocks of a step (bound by what an SM can fetch from L2, about 64 bytes per clock at best: 24 / 32 KB for a tile of
// 128 x 64 / 128 x 128 in a CTA, 24 to 32 KB per CTA of a pair), plus what a launch costs outside its K loop, which is as
// much again for a small problem: start, epilogue, and for a split tile the exchange.  Fitted to launches in a row (us):
//   M x N x K            pair 256  pair 224  pair 192  pair 128  CTA 128  over 2  over 4   CTA 64  over 2
//   148 x 768 x 256                                        4.9      4.2     4.7     5.0      3.4     3.7
//   148 x 256 x 768                                        5.5      5.4     5.2     5.1      4.6     4.2
//   371 x 3072 x 768                                       7.2      6.2     6.7    18.4      5.8    11.0
//   371 x 768 x 3072                                      13.6     13.2     9.5     8.1     12.1     8.1
//   1394 x 1024 x 1024      9.9       9.2       8.3       7.4      7.2    12.7              11.6
//   1394 x 3072 x 1024     11.4      13.2      12.3      12.2     14.4    27.1              23.8
//   1394 x 1024 x 4096     23.4      21.2      19.6      19.0     20.4    25.4              32.5
//   5254 x 1152 x 1152     15.9      15.1      14.2      17.0     21.9    40.8              37.4
//   5254 x 3456 x 1152     32.2      33.7      35.2      41.7     62.5
//   3510 x 3072 x 3072     51.8      49.5      54.3      64.7     86.3
// Launches in a row of problems that were not used for the fit; the rule takes the best entry of the first four and is 4 %
// above it in the last (it takes 224).
//   640 x 1920 x 640        8.2       7.7       7.1       6.4      6.2     11.5    18.0      9.5    14.8
//   820 x 640 x 2560       16.5      15.0      14.0      12.6     14.1     10.2    15.5     11.3     8.6
//   200 x 1280 x 5120      27.5      24.6      23.0      21.8     25.1     15.4    11.4     19.6    12.6
//   2300 x 2048 x 2048     16.6      21.8      20.6      20.1     25.9     38.4    72.2     39.3    60.7
//   7000 x 1536 x 6144     99.1     103.4     125.7     143.8    168.9    181.1   259.5    220.0   315.1
// 64 columns over four CTAs, where K is long and the tiles are few (CTA 64 over 1 / 2 / 4): 250 x 384 x 1536 7.6 / 5.9 / 4.9,
// 500 x 512 x 2048 9.4 / 6.9 / 6.1, 60 x 704 x 2112 9.2 / 6.9 / 5.3; 371 x 768 x 3072, whose 36 clusters of four do not all
// fit, 12.8 / 8.8 / 12.7.  The more clusters, the longer the exchange, which short K does not pay for: 25 x 2048 x 512 4.7 / 4.7 / 5.2,
// 60 x 1920 x 640 5.0 / 5.0 / 5.5, but 148 x 512 x 512 4.8 / 4.8 / 4.4.  With q/k treatment (pair 256 / pair 128 / CTA 128 /
// CTA 64): 371 x 2304 x 768 10.4 / 7.3 / 7.3 / 6.2, 614 x 768 x 256 8.0 / 5.9 / 5.3 / 4.3, 700 x 1536 x 512 9.4 / 6.8 / 6.7 / 5.3,
// 1394 x 3072 x 1024 12.8 / 13.7 / 15.6 / 25.4.
// ---------------------------------------------------------------------------------------------------------------
TcGemmPlan plan_tc_gemm(int M, int Nout, int K, bool qk, int sms) {
  const long long kb = ((long long)K + kBK - 1) / kBK;
  auto ceil_div = [](long long a, long long b) { return (a + b - 1) / b; };
  TcGemmPlan best = {256, 0};
  long long best_t = -1;
  auto consider = [&](int bn, int split, long long t) {
    if (best_t < 0 || t < best_t) { best_t = t; best = {bn, split}; }
  };
  struct { int bn, step, fixed; } const pair[] = {{256, 560, 11500}, {224, 510, 10100}, {192, 500, 8000}, {128, 460, 7400}};
  for (const auto& p : pair) {
    if (qk && p.bn % 128 != 0) continue;             // (only what gives an epilogue warp whole heads)
    const long long tiles = ceil_div(M, 2 * kBM) * ceil_div(Nout, p.bn);
    consider(p.bn, 0, ceil_div(tiles, sms < 2 ? 1 : sms / 2) * kb * p.step + p.fixed);
  }
  for (int bn : {128, 64}) {
    const long long tiles = ceil_div(M, kBM) * ceil_div(Nout, bn);
    const int max_split = qk ? 1 : SplitCfg<128>::kMaxSplit;
    for (int split = 1; split <= max_split && split <= kb; split *= 2) {
      const long long ctas = tiles * split;
      if (ctas > 0x7FFFFFFFll) continue;
      // (clusters of four do not fill the chip: they need four free SMs of one processing cluster)
      const long long fours = sms < 2 ? 1 : sms * 7 / 8, waves = ceil_div(ctas, split == 4 ? fours : sms);
      const long long step = bn == 64 ? 390 : 400 + (ctas < 100 ? ctas : 100);
      long long exchange = split == 1 ? 0 : (bn == 64 ? 1700 : (split == 2 ? 2000 : 3500));
      if (bn == 64 && split == 4) exchange += 100 + (ctas > 60 ? 15 * (ctas - 60) : 0);
      consider(bn, split, waves * (ceil_div(kb, split) * step + (bn == 64 ? 4500 : 6300) + exchange));
    }
  }
  return best;
}

namespace {

template <int BN, bool QK = false>
int launch_pair(const CUtensorMap& tm_a, const CUtensorMap& tm_w, const void* bias, const GemmOut& out, const QkEpilogue& qk,
                int M, int Nout, int K, int* d_status, cudaStream_t s) {
  static PerDeviceOnce attr_once;            // the opt-in is a property of the kernel ON a device
  HERO_TRY(per_device_once(attr_once, [](int) {
    HERO_CUDA_TRY(cudaFuncSetAttribute(tc_gemm_pair_kernel<BN, QK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)PairCfg<BN>::kSmem));
    return HERO_OK;
  }));
  const int tiles = ((M - 1) / (2 * kBM) + 1) * ((Nout + BN - 1) / BN);
  const int pairs = tiles < num_sms() / 2 ? tiles : num_sms() / 2;
  QkParam<QK> param;
  if constexpr (QK) static_cast<QkEpilogue&>(param) = qk;
  return launch_kernel(tc_gemm_pair_kernel<BN, QK>, (unsigned)(2 * pairs), kGemmThreads, PairCfg<BN>::kSmem, s,
                       2, tm_a, tm_w, (const __nv_bfloat16*)bias, out, param, M, Nout, K, d_status);
}

template <int BN, bool QK = false>
int launch_split(const CUtensorMap& tm_a, const CUtensorMap& tm_w, const void* bias, const GemmOut& out, const QkEpilogue& qk,
                 int M, int Nout, int K, int split, int* d_status, cudaStream_t s) {
  static PerDeviceOnce attr_once;
  HERO_TRY(per_device_once(attr_once, [](int) {
    HERO_CUDA_TRY(cudaFuncSetAttribute(tc_gemm_split_kernel<BN, QK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)SplitCfg<BN>::smem(SplitCfg<BN>::kMaxSplit)));
    return HERO_OK;
  }));
  const int tiles = ((M + kBM - 1) / kBM) * ((Nout + BN - 1) / BN);
  QkParam<QK> param;
  if constexpr (QK) static_cast<QkEpilogue&>(param) = qk;
  return launch_kernel(tc_gemm_split_kernel<BN, QK>, (unsigned)(tiles * split), kGemmThreads, SplitCfg<BN>::smem(split), s,
                       (unsigned)split, tm_a, tm_w, (const __nv_bfloat16*)bias, out, param, M, Nout, K, split, d_status);
}

}  // namespace

int launch_tc_gemm(const void* a, const void* w, const void* bias, int M, int Nout, int K, const GemmOut& out,
                   const QkEpilogue* qk, int* d_status, cudaStream_t s) {
  if (M <= 0) return HERO_OK;
  if (K % 8 || Nout % 8 || out.seg_cols % 32) return HERO_ERR_ALIGN;
  if (!aligned16(a) || !aligned16(w) || !aligned16(bias)) return HERO_ERR_ALIGN;
  for (int i = 0; i < 3; ++i)
    if (out.ptr[i] && (!aligned16(out.ptr[i]) || out.ld[i] % 8)) return HERO_ERR_ALIGN;
  const TcGemmPlan plan = plan_tc_gemm(M, Nout, K, qk != nullptr, num_sms());
  CUtensorMap tm_a, tm_w;
  {
    const uint64_t dims[2] = {(uint64_t)K, (uint64_t)M};
    const uint64_t str[1] = {(uint64_t)K * 2};
    const uint32_t box[2] = {(uint32_t)kBK, (uint32_t)kBM};
    HERO_TRY(make_tmap_bf16(&tm_a, a, 2, dims, str, box));
  }
  {
    const uint64_t dims[2] = {(uint64_t)K, (uint64_t)Nout};
    const uint64_t str[1] = {(uint64_t)K * 2};
    const uint32_t box[2] = {(uint32_t)kBK, (uint32_t)(plan.split == 0 ? plan.bn / 2 : plan.bn)};
    HERO_TRY(make_tmap_bf16(&tm_w, w, 2, dims, str, box));
  }
  if (qk) {
    if (out.seg_cols % 64 || Nout != 3 * out.seg_cols || out.act || out.gate || out.seg0_scale != 0.f) return HERO_ERR_ARG;
    if (plan.split)
      return plan.bn == 128 ? launch_split<128, true>(tm_a, tm_w, bias, out, *qk, M, Nout, K, 1, d_status, s)
                            : launch_split<64, true>(tm_a, tm_w, bias, out, *qk, M, Nout, K, 1, d_status, s);
    return plan.bn == 256 ? launch_pair<256, true>(tm_a, tm_w, bias, out, *qk, M, Nout, K, d_status, s)
                          : launch_pair<128, true>(tm_a, tm_w, bias, out, *qk, M, Nout, K, d_status, s);
  }
  const QkEpilogue none = {};
  if (plan.split == 0) {
    switch (plan.bn) {
      case 256: return launch_pair<256>(tm_a, tm_w, bias, out, none, M, Nout, K, d_status, s);
      case 224: return launch_pair<224>(tm_a, tm_w, bias, out, none, M, Nout, K, d_status, s);
      case 192: return launch_pair<192>(tm_a, tm_w, bias, out, none, M, Nout, K, d_status, s);
      default: return launch_pair<128>(tm_a, tm_w, bias, out, none, M, Nout, K, d_status, s);
    }
  }
  return plan.bn == 128 ? launch_split<128>(tm_a, tm_w, bias, out, none, M, Nout, K, plan.split, d_status, s)
                        : launch_split<64>(tm_a, tm_w, bias, out, none, M, Nout, K, plan.split, d_status, s);
}

}  // namespace hero
