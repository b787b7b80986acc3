// Flash-attention for the refresh path (Eq. 3 with the refreshed queries attending to the
// full cached K/V): O = softmax(Q K^T / sqrt(64)) V per (batch, head), bf16 in, fp32 softmax,
// no score matrix ever leaves the SM.
//
// One CTA = 256 query rows (two tiles of 128) of one (batch, head); it streams all N cached
// keys in tiles of 96 through a 6-stage TMA ring shared by both query tiles.  TMEM (512
// columns): per query tile two score buffers of 96 columns (key tile parity) and one 64-column
// output accumulator; P (bf16) is written over the scores it was computed from and is the TMEM
// operand of O += P V.  S of tile j+2 is issued right after P V of tile j (same issuer, executed
// in issue order), so a score tile is normally ready a whole softmax iteration before it is needed.
//
// Two kernels share this layout and these warps:
//
//  * tc_attention_fast_kernel, the one that normally does all the work.  20 warps: TMA producer, one
//    tcgen05.mma issuer warp per query tile (all lanes run the loop, one elected lane issues, so that
//    the operands stay warp-uniform), and SIXTEEN softmax warps: every query row is shared by two
//    threads, each owning 48 of a key tile's 96 score columns.  A warp issues in order and stalls on
//    every ex2 while the special-function unit is busy and on every barrier, fence and TMEM round
//    trip at a tile boundary; with four softmax warps per SM sub-partition instead of two there is
//    always another warp with exponentials ready, which is what keeps that unit (the bound of this
//    kernel at head_dim 64: 16 ex2 per clock per SM against 256 tensor flops per score) busy.
//    The two threads of a row never talk in steady state: the row's scaling maximum is fixed by the
//    first key tile (one exchange through shared memory) and never moves, so a tile is ONE pass -
//    p = 2^((s - m) c), row sum, bf16 pack, store - with no running maximum, no vote and no redo.
//    That is exact as long as no later score exceeds the first tile's maximum by more than 2^100
//    (69 in natural-log units; bf16 and fp32 share their exponent range, so a large p loses no
//    precision, and the final division by the row sum makes the result independent of the maximum
//    used).  The row sum tells whether that held; slices of 32 rows in which it did not go to the safe path.
//    In the step the QKV projection hands over q already multiplied by log2(e) / sqrt(64), so a score is
//    the exponent of its weight: that instantiation (PRESCALED) takes p = 2^s as it stands - no maximum,
//    no first-tile exchange, no multiply-add per pair of scores - and is exact while a row's largest score
//    stays within about +-100; its row sum must then lie in [2^-100, 2^100), else the same.
//  * The safe path (safe_roles) keeps a running maximum that moves whenever a tile exceeds it by 2^8, rescaling the
//    accumulator in TMEM.  The warps are those of the fast kernel; the two threads of a row trade their halves' maxima for
//    every key tile.  A thread block of the fast kernel whose row sums say that the range assumption failed recomputes its
//    queries with it before it ends (a second launch for the failed blocks, as it
//    used to be, cost every attention 2-4 us at small sizes and 14 us at 1728 blocks for finding nothing to do);
//    tc_attention_safe_kernel is the same path as a kernel of its own.  Two threads a row, so that a row's scores stay in
//    registers beside the fast path's (96 a thread): recomputed by eight warps, a thread a row, in two passes over TMEM, all
//    rows of 2 x 1755 x 17776 x 48 out of range took 2696 us (1859 so, 1913 with the second launch), of 2 x 371 x 1562 x 12
//    59 (43, 57); with no range to check, 4 x 2403 x 9894 x 22 takes 787 us, where the fast path takes 579.
//
// The fast kernel comes in three modes (attention_plan says which runs when).  With the scale folded into Q there is no
// maximum, so the partial results of a query group over disjoint runs of keys simply add; that is what the last two use:
//  * kWhole: one thread block per query group (256 queries of one batch item and head), all keys;
//  * kCluster, for grids that leave SMs idle: a cluster of blocks per group, each with a run of the key tiles; they trade
//    16-column pieces of their accumulators through distributed shared memory, each finishing its own;
//  * kCut, for grids of several rounds over long key sequences: persistent blocks, one per SM, work through whole groups a
//    grid apart (so that the blocks in flight stay on few heads and share their K and V in L2), and what is left for the
//    last, partly filled round is cut into runs of key tiles over ALL blocks.  Every warp lays its rows of a part out in a
//    workspace and counts itself in; the one that completes the count adds all parts and writes the rows.
// Parts are added in a fixed order, so that no result depends on timing, and nobody ever waits for another block of kCut.
//
#include <cuda.h>

#include <mutex>
#include <type_traits>

#include "hero_internal.h"
#include "tc_common.cuh"

namespace hero {

int make_tmap_bf16(CUtensorMap* m, const void* base, int rank, const uint64_t* dims, const uint64_t* strides_bytes,
                   const uint32_t* box);

namespace {
using namespace tc;

constexpr int kQT = 128, kQTiles = 2, kKT = 96, kHD = 64, kKvStages = 6;
constexpr int kQBytes = kQT * kHD * 2;       // 16 KB per query tile
constexpr int kKBytes = kKT * kHD * 2;       // 12 KB (a multiple of the 1024-byte swizzle atom)
constexpr int kKvStageBytes = 2 * kKBytes;   // K tile then V tile
constexpr int kFirstSoftmaxWarp = 4;
constexpr int kSoftmaxWarps = 16;            // 2 query tiles x 4 TMEM lane quadrants x 2 column halves
constexpr int kAttThreads = 32 * (kFirstSoftmaxWarp + kSoftmaxWarps);        // 20 warps
constexpr int kHalf = kKT / 2;               // score columns of a key tile that one thread owns
constexpr int kXchgFloats = kQTiles * kQT * 2;   // one slot per (query row, column half)
constexpr size_t kSafeSmem = 1024 + kQTiles * kQBytes + (size_t)kKvStages * kKvStageBytes + 512 + 2 * kXchgFloats * sizeof(float);
constexpr uint32_t kTileCols = 256, kColO = 2 * kKT, kAttTmemCols = 512;   // per tile: S0 | S1 | O
constexpr float kRescaleLog2 = 8.0f;           // the scaling maximum moves only when exceeded by 2^8
static_assert(2 * kKT + kHD <= (int)kTileCols && kQTiles * kTileCols <= kAttTmemCols, "TMEM layout");
static_assert(kKBytes % 1024 == 0 && kKT % 16 == 0, "tile shape");
static_assert(kHalf % 16 == 0 && (kHalf / 16) % 2 == 1, "three 16-column reads per half: half_tile's ping-pong ends on ra");

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float y;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
  return y;
}
__device__ __forceinline__ float2 f2(uint32_t a, uint32_t b) { return make_float2(__uint_as_float(a), __uint_as_float(b)); }

// 16 output features of one row: accumulator times 1 / row sum, bf16, as one 32-byte store where the output is aligned to
// that (every lane has a row of its own, so what counts is the number of requests a row is made of: 256 rows of 128 bytes
// take an SM 1700 clocks in 32-byte stores, 3700 in 16-byte ones).
__device__ __forceinline__ void emit16(const uint32_t (&r)[16], float inv, __nv_bfloat16* dst) {
  uint32_t w[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const __nv_bfloat162 pk = __floats2bfloat162_rn(__uint_as_float(r[2 * q]) * inv, __uint_as_float(r[2 * q + 1]) * inv);
    w[q] = *reinterpret_cast<const uint32_t*>(&pk);
  }
  if ((reinterpret_cast<uintptr_t>(dst) & 31) == 0) {          // (the same for every row of a launch)
    st_global_v8(dst, w);
  } else {
    *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
    *reinterpret_cast<uint4*>(dst + 8) = make_uint4(w[4], w[5], w[6], w[7]);
  }
}

// One thread block's work on the safe path.
struct SafeWork {
  const CUtensorMap *tm_q, *tm_k, *tm_v;
  __nv_bfloat16* O;
  int n_q, N, heads, qg, h, b;
  float c;                       // factor that turns a score into the exponent of its weight
  uint32_t row_mask;             // which 32-row slices (query tile * 4 + quadrant) of the group are written
  uint8_t *s_q, *s_kv;
  uint64_t* bars;                // kSafeBars barriers, set up by safe_init_barriers, never used before
  float* xchg;                   // [2][kXchgFloats] between the two threads of a row
  volatile int* abort_flag;
  uint32_t tmem_base;
};
constexpr int kSafeBars = 1 + 2 * kKvStages + 4 + 4 + 2 * kQTiles + 4 * kQTiles;
// The last query group of a (batch, head) may reach into its second tile by no row at all: that tile's
// issuer and softmax warps then have nothing to do and the K/V stages are released by one issuer alone.
__device__ __forceinline__ int live_tiles(int qg, int n_q) { return (qg * kQTiles + 1) * kQT < n_q ? kQTiles : 1; }
__device__ __forceinline__ void safe_init_barriers(uint64_t* bars, int n_tiles) {
  mbar_init(bars, 1);
  for (int i = 0; i < kKvStages; ++i) { mbar_init(bars + 1 + i, 1); mbar_init(bars + 1 + kKvStages + i, n_tiles); }
  for (int i = 0; i < 4; ++i) { mbar_init(bars + 1 + 2 * kKvStages + i, 1); mbar_init(bars + 5 + 2 * kKvStages + i, 8); }
  for (int i = 0; i < 2 * kQTiles; ++i) mbar_init(bars + 9 + 2 * kKvStages + i, 1);
  for (int i = 0; i < 4 * kQTiles; ++i) mbar_init(bars + 9 + 2 * kKvStages + 2 * kQTiles + i, 2);
}

// Warp 0: TMA producer, warps 1 and 2: MMA issuers, warps 4 .. 19: softmax, as in the fast kernel.
__device__ __forceinline__ void safe_roles(const SafeWork& w) {
  const CUtensorMap &tm_q = *w.tm_q, &tm_k = *w.tm_k, &tm_v = *w.tm_v;
  const int n_q = w.n_q, N = w.N, heads = w.heads, qg = w.qg, h = w.h, b = w.b;
  const float c = w.c;
  const uint32_t row_mask = w.row_mask;
  uint8_t *const s_q = w.s_q, *const s_kv = w.s_kv;
  volatile int* const abort_flag = w.abort_flag;
  const uint32_t tmem_base = w.tmem_base;
  __nv_bfloat16* const O = w.O;
  uint64_t* q_full = w.bars;
  uint64_t* kv_full = q_full + 1;                  // [kKvStages]           TMA -> both issuers
  uint64_t* kv_empty = kv_full + kKvStages;        // [kKvStages], count 2  both issuers -> TMA
  uint64_t* s_full = kv_empty + kKvStages;         // [qt][parity]  issuer -> softmax: S is ready
  uint64_t* p_full = s_full + 4;                   // [qt][parity]  softmax -> issuer: P is in TMEM (8 warps)
  uint64_t* pv_full = p_full + 4;                  // [qt]          issuer -> softmax: P V of tile j done (phase j)
  uint64_t* pv_last = pv_full + kQTiles;           // [qt]          issuer -> softmax: all P V done
  uint64_t* pair_bar = pv_last + kQTiles;          // [qt][quadrant] the two warps that share 32 query rows
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_kv = (N + kKT - 1) / kKT;
  const int n_tiles = live_tiles(qg, n_q);

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      mbar_expect_tx(q_full, n_tiles * kQBytes);
      for (int t = 0; t < n_tiles; ++t)
        tma_load_2d(s_q + t * kQBytes, &tm_q, q_full, h * kHD, b * n_q + (qg * kQTiles + t) * kQT);
      int stage = 0; uint32_t phase = 0;
      for (int j = 0; j < n_kv; ++j) {
        if (!mbar_wait(&kv_empty[stage], phase ^ 1, abort_flag)) break;
        uint8_t* sk = s_kv + (size_t)stage * kKvStageBytes;
        mbar_expect_tx(&kv_full[stage], kKvStageBytes);
        tma_load_3d(sk, &tm_k, &kv_full[stage], h * kHD, j * kKT, b);
        tma_load_3d(sk + kKBytes, &tm_v, &kv_full[stage], h * kHD, j * kKT, b);
        if (++stage == kKvStages) { stage = 0; phase ^= 1; }
      }
      for (int i = 0; i < kKvStages; ++i) {      // all armed stages consumed before the CTA retires
        if (!mbar_wait(&kv_empty[stage], phase ^ 1, abort_flag)) break;
        if (++stage == kKvStages) { stage = 0; phase ^= 1; }
      }
    }
  } else if (warp == 1 || warp == 2) {
    // ------------------------------------------------------------ MMA issuer of query tile t
    if (lane == 0 && warp - 1 < n_tiles) {
      const int t = warp - 1;
      constexpr uint32_t idesc_s = idesc_bf16(kQT, kKT, 0);    // S = Q K^T : both operands K-contiguous
      constexpr uint32_t idesc_pv = idesc_bf16(kQT, kHD, 1);   // O += P V  : V is N(head_dim)-contiguous
      const uint64_t dq = smem_desc_sw128(smem_u32(s_q + t * kQBytes), 1024);
      const uint32_t t_tile = tmem_base + (uint32_t)t * kTileCols;
      auto issue_s = [&](int j) {
        const int st = j % kKvStages;
        const uint64_t dk = smem_desc_sw128(smem_u32(s_kv + (size_t)st * kKvStageBytes), 1024);
        const uint32_t d = t_tile + (uint32_t)(j & 1) * kKT;
#pragma unroll
        for (int k = 0; k < kHD / 16; ++k) mma_ss(d, dq + 2 * k, dk + 2 * k, idesc_s, k != 0);
        mma_commit(&s_full[t * 2 + (j & 1)]);
      };
      bool ok = mbar_wait(q_full, 0, abort_flag);
      for (int j = 0; j < 2 && j < n_kv && ok; ++j) {           // two score tiles ahead of the softmax
        if ((ok = mbar_wait(&kv_full[j], 0, abort_flag))) { tc_fence_after(); issue_s(j); }
      }
      for (int j = 0; j < n_kv && ok; ++j) {
        const int st = j % kKvStages;
        // V tile: rows = keys (128 bytes each), 8-key groups 1024 bytes apart; 16 keys per MMA = 2048 bytes
        const uint64_t dv = smem_desc_sw128(smem_u32(s_kv + (size_t)st * kKvStageBytes + kKBytes), 1024);
        if (!(ok = mbar_wait(&p_full[t * 2 + (j & 1)], (j >> 1) & 1, abort_flag))) break;
        tc_fence_after();
        const uint32_t buf = t_tile + (uint32_t)(j & 1) * kKT;
#pragma unroll
        for (int k = 0; k < kKT / 16; ++k)         // (each half of the softmax writes P inside its own score columns)
          mma_ts(t_tile + kColO, buf + (k / 3) * kHalf + (k % 3) * 8, dv + 128 * k, idesc_pv, (j | k) != 0);
        mma_commit(&pv_full[t]);
        if (j == n_kv - 1) mma_commit(&pv_last[t]);
        mma_commit(&kv_empty[st]);               // second arrival comes from the other tile's issuer
        if (j + 2 < n_kv) {
          // S of tile j+2 overwrites the buffer whose P the product above reads: safe because the
          // tensor core executes this thread's MMAs in issue order
          if (!(ok = mbar_wait(&kv_full[(j + 2) % kKvStages], ((j + 2) / kKvStages) & 1, abort_flag))) break;
          tc_fence_after();
          issue_s(j + 2);
        }
      }
    }
  } else if (warp >= kFirstSoftmaxWarp && (((warp - kFirstSoftmaxWarp) >> 2) & 1) < n_tiles) {
    // ------------------------------------------------------------ softmax
    const int sid = warp - kFirstSoftmaxWarp;
    const int t = (sid >> 2) & 1, hh = sid >> 3;       // query tile, and which 48 of a tile's 96 score columns
    const int quad = warp & 3;                         // TMEM lane quadrant this warp may touch
    const int row = quad * 32 + lane;
    const uint32_t lane_base = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)t * kTileCols;
    uint64_t* my_pair = &pair_bar[t * 4 + quad];
    uint32_t pair_phase = 0;
    // One value of this thread and its partner's.  (Two exchange buffers in turn: a warp may be one exchange ahead of its
    // partner, not two.)
    auto slot = [&]() { return w.xchg + pair_phase * kXchgFloats + (t * kQT + row) * 2; };
    auto offer = [&](float mine) {
      slot()[hh] = mine;
      __syncwarp();
      if (lane == 0) mbar_arrive(my_pair);
    };
    auto take = [&](float2& both) -> bool {
      if (!mbar_wait_warp(my_pair, pair_phase, abort_flag)) return false;
      both = make_float2(slot()[0], slot()[1]);
      pair_phase ^= 1;
      return true;
    };
    float m_used = -INFINITY, l_run = 0.f;             // the maximum that the row's P and accumulator are scaled by
    float2 both;
    bool ok = true;
    for (int j = 0; j < n_kv; ++j) {
      ok = mbar_wait_warp(&s_full[t * 2 + (j & 1)], (j >> 1) & 1, abort_flag);
      if (!ok) break;
      tc_fence_after();
      const uint32_t t_s = lane_base + (uint32_t)(j & 1) * kKT + (uint32_t)hh * kHalf;
      const int valid = N - j * kKT - hh * kHalf;      // columns of this half that are keys
      uint32_t s[kHalf];
#pragma unroll
      for (int ch = 0; ch < kHalf / 16; ++ch) tmem_ld16(t_s + ch * 16, *reinterpret_cast<uint32_t(*)[16]>(&s[ch * 16]));
      tmem_ld_wait();
      if (valid < kHalf) {                             // warp-uniform
#pragma unroll
        for (int i = 0; i < kHalf; ++i)
          if (i >= valid) s[i] = 0xFF800000u;          // -inf: weight 0 under any finite maximum
      }
      float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
      for (int i = 0; i < kHalf; i += 4) {
        mx[0] = max3(mx[0], __uint_as_float(s[i]), __uint_as_float(s[i + 1]));
        mx[1] = max3(mx[1], __uint_as_float(s[i + 2]), __uint_as_float(s[i + 3]));
      }
      offer(fmaxf(mx[0], mx[1]));
      // P under the maximum that the row has: where this tile's does not move it, that is all, and the partner's half of
      // the maximum has arrived meanwhile.
      const float2 c2 = make_float2(c, c);
      auto weights = [&]() -> float {
        const float2 nm2 = make_float2(-m_used * c, -m_used * c);
        float2 acc[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
        for (int ch = 0; ch < kHalf / 16; ++ch) {
          uint32_t pk[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float2 x = __ffma2_rn(f2(s[ch * 16 + 2 * i], s[ch * 16 + 2 * i + 1]), c2, nm2);
            const float2 p = make_float2(ex2(x.x), ex2(x.y));
            acc[i & 1] = __fadd2_rn(acc[i & 1], p);
            const __nv_bfloat162 bb = __floats2bfloat162_rn(p.x, p.y);
            pk[i] = *reinterpret_cast<const uint32_t*>(&bb);
          }
          tmem_st8(t_s + ch * 8, pk);
        }
        const float2 a01 = __fadd2_rn(acc[0], acc[1]);
        return a01.x + a01.y;
      };
      float sum = j > 0 ? weights() : 0.f;
      if (!(ok = take(both))) break;
      const float m_tile = fmaxf(both.x, both.y);      // (the same in both threads of the row, and so is what follows)
      const bool grow = (m_tile - m_used) * c > kRescaleLog2;               // true at the first tile
      const float alpha = grow ? ex2((m_used - m_tile) * c) : 1.0f;         // 0 at the first tile
      if (grow) m_used = m_tile;
      const bool moved = __any_sync(0xFFFFFFFFu, grow);
      if (j == 0 || moved) sum = weights();
      l_run = fmaf(l_run, alpha, sum);
      if (j > 0 && moved) {
        // Rare: the maximum moved, so the accumulator is scaled down before this tile's
        // product is added to it - once P V of tile j-1 has completed.  pv_full is only looked at here, yet the
        // parity wait is unambiguous: S of tile j was issued after P V of tile j-2
        // (so that one is complete) and P V of tile j cannot start before this warp's arrival below, hence
        // the barrier has completed either j-1 or j phases and "phase j-1 complete" is exactly the question.
        ok = mbar_wait_warp(&pv_full[t], (j - 1) & 1, abort_flag);
        if (!ok) break;
        tc_fence_after();
        const float2 a2 = make_float2(alpha, alpha);     // alpha is 1 for rows that did not move
#pragma unroll
        for (int ch = 0; ch < 2; ++ch) {                 // each half 32 of the 64 features
          uint32_t r[16];
          tmem_ld16(lane_base + kColO + hh * 32 + ch * 16, r);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 16; i += 2) {
            const float2 v = __fmul2_rn(f2(r[i], r[i + 1]), a2);
            r[i] = __float_as_uint(v.x); r[i + 1] = __float_as_uint(v.y);
          }
          tmem_st16(lane_base + kColO + hh * 32 + ch * 16, r);
        }
      }
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&p_full[t * 2 + (j & 1)]);
    }
    if (ok) {
      offer(l_run);
      ok = take(both);
    }
    // (Not pv_full: the other warps may still be two tiles behind this one, and its parity cannot tell that.)
    if (ok) ok = mbar_wait_warp(&pv_last[t], 0, abort_flag);
    if (ok) {
      tc_fence_after();
      const int qi = (qg * kQTiles + t) * kQT + row;
      const float inv = 1.0f / (both.x + both.y);
      __nv_bfloat16* dst = O + ((long long)b * n_q + qi) * ((long long)heads * kHD) + h * kHD + hh * 32;
#pragma unroll
      for (int ch = 0; ch < 2; ++ch) {
        uint32_t r[16];
        tmem_ld16(lane_base + kColO + hh * 32 + ch * 16, r);     // warp-collective: every lane loads
        tmem_ld_wait();
        if (qi < n_q && (row_mask >> (t * 4 + quad) & 1)) emit16(r, inv, dst + ch * 16);
      }
    }
  }
}

// status[0] counts the thread blocks that gave up on a bounded wait.
__global__ void __launch_bounds__(kAttThreads, 1)
tc_attention_safe_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                         const __grid_constant__ CUtensorMap tm_v, __nv_bfloat16* __restrict__ O, int n_q, int N,
                         int heads, const float c, int* __restrict__ status) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  SafeWork w = {&tm_q, &tm_k, &tm_v, O, n_q, N, heads};
  w.s_q = smem;
  w.s_kv = smem + kQTiles * kQBytes;
  w.bars = reinterpret_cast<uint64_t*>(w.s_kv + (size_t)kKvStages * kKvStageBytes);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(w.bars + kSafeBars);
  w.abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  w.xchg = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(w.bars) + 512);
  static_assert(kSafeBars * 8 + 8 <= 512, "barrier block");
  w.c = c;
  w.row_mask = ~0u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int q_groups = (n_q + kQT * kQTiles - 1) / (kQT * kQTiles);
  w.qg = blockIdx.x % q_groups;
  w.h = (blockIdx.x / q_groups) % heads;
  w.b = blockIdx.x / (q_groups * heads);
  if (threadIdx.x == 0) {
    safe_init_barriers(w.bars, live_tiles(w.qg, n_q));
    *w.abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == 0 && lane == 0) { tma_prefetch_desc(&tm_q); tma_prefetch_desc(&tm_k); tma_prefetch_desc(&tm_v); }
  if (warp == 1) { tmem_alloc(tmem_slot, kAttTmemCols); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  w.tmem_base = *tmem_slot;
  stream_order();
  safe_roles(w);
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *w.abort_flag) atomicAdd(status, 1);
  if (warp == 1) { __syncwarp(); tc_fence_after(); tmem_dealloc(w.tmem_base, kAttTmemCols); }
}

// =============================================================================================
// The fast kernel
// =============================================================================================
constexpr int kMaxBad = 64;                      // out-of-range row slices of whole groups that a block keeps a list of
constexpr size_t kFastBarBytes = 640;
constexpr size_t kFastSmem = 1024 + 2 * kQTiles * kQBytes + (size_t)kKvStages * kKvStageBytes + kFastBarBytes +
                             2 * kXchgFloats * sizeof(float) + (kMaxBad + 4) * sizeof(int);
constexpr float kRowSumLimit = 1.2676506e30f;    // 2^100: a row sum at or beyond it voids the fixed-maximum assumption
constexpr float kRowSumFloor = 7.8886091e-31f;   // 2^-100: below it a row without a maximum has lost its small terms

// 2^x for two scores on the FMA pipe instead of the special-function unit (Cody-Waite reduction + a cubic).
// The unit evaluates 16 ex2 per clock per SM and is what bounds this kernel; every pair moved here frees two of
// its slots for ten FMA/ALU-pipe instructions, which the four softmax warps per sub-partition have to spare.
//   xs = sat(x / 250 + 1/2)            x clamped to [-125, 125] by the saturating FMA (x = s c - m c is formed here)
//   t  = xs * 250 + (M - 125)          M = 1.5 * 2^23: the sum rounds to M + n, n = round(x), held in t's low bits
//   f  = xs * 250 + ((M - 125) - t)    x - n, in [-1/2, 1/2]
//   2^f ~ C0 + f (C1 + f (C2 + f C3))  minimax cubic for the relative error on [-1/2, 1/2]: 7.5e-5, a fiftieth of the
//                                      bf16 rounding P goes through (coefficients from a Lawson-weighted least-squares fit)
//   result = bits(2^f) + (bits(t) << 23)   adds n to the exponent field: 127 - 125 .. 127 + 125 stays a normal number
// A score that the clamp cuts off at +125 still yields 2^125, far beyond the row-sum limit, so the row is caught.
#ifndef HERO_ATT_POLY_PAIRS
#define HERO_ATT_POLY_PAIRS 1          // of every 8 pairs of scores (1 measured best: 2.22 ms against 2.40 with none, 2.33 with 2)
#endif
#ifndef HERO_ATT_POLY_PAIRS_PRESCALED
#define HERO_ATT_POLY_PAIRS_PRESCALED 2   // with the scale folded into q a pair costs the pipes one instruction less: 2 is best
#endif
constexpr int kPolyPairs = HERO_ATT_POLY_PAIRS, kPolyPairsPrescaled = HERO_ATT_POLY_PAIRS_PRESCALED;
constexpr float kPolySpan = 250.0f, kPolyMagic = 12582912.0f - 125.0f;
__device__ __forceinline__ float fma_sat(float a, float b, float c) {
  float y;
  asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
  return y;
}
__device__ __forceinline__ float2 exp2_poly_pair(float s0, float s1, float cs, float bs) {
  const float2 xs = make_float2(fma_sat(s0, cs, bs), fma_sat(s1, cs, bs));
  const float2 span = make_float2(kPolySpan, kPolySpan), mg = make_float2(kPolyMagic, kPolyMagic);
  const float2 t = __ffma2_rn(xs, span, mg);
  const float2 f = __ffma2_rn(xs, span, __ffma2_rn(t, make_float2(-1.0f, -1.0f), mg));
  float2 p = __ffma2_rn(f, make_float2(0.0551716648f, 0.0551716648f), make_float2(0.2426111251f, 0.2426111251f));
  p = __ffma2_rn(p, f, make_float2(0.6932609677f, 0.6932609677f));
  p = __ffma2_rn(p, f, make_float2(0.9999280572f, 0.9999280572f));
  return make_float2(__int_as_float(__float_as_int(p.x) + (__float_as_int(t.x) << 23)),
                     __int_as_float(__float_as_int(p.y) + (__float_as_int(t.y) << 23)));
}

// One key tile of one thread's 48 columns, steady state: the scores are read 16 columns at a time (one read
// ahead), turned into p = 2^(s c - m c), summed, packed to bf16 and written back over the columns just read -
// half h keeps its P in the first 24 columns of its own 48, so neither half ever writes what the other reads.
// MASKED (the ragged last tile): columns at or beyond `valid` are keys that do not exist.
// PRESCALED: the scores are exponents already (x = s, see the kernel below), one instruction less per pair.
template <bool MASKED, bool PRESCALED>
__device__ __forceinline__ float half_tile(uint32_t t_s, int valid, const float2 c2, const float2 nm2, float cs, float bs) {
  float2 acc[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  uint32_t ra[16], rb[16];
  tmem_ld16(t_s, ra);
#pragma unroll
  for (int ch = 0; ch < kHalf / 16; ++ch) {
    uint32_t(&cur)[16] = (ch & 1) ? rb : ra;
    uint32_t(&nxt)[16] = (ch & 1) ? ra : rb;
    tmem_ld_wait();
    if (ch + 1 < kHalf / 16) tmem_ld16(t_s + (ch + 1) * 16, nxt);
    uint32_t pk[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float2 p;
      constexpr int kPoly = PRESCALED ? kPolyPairsPrescaled : kPolyPairs;
      if ((i * kPoly) % 8 < kPoly) {                    // spread evenly over the chunk (resolved at compile time)
        p = exp2_poly_pair(__uint_as_float(cur[2 * i]), __uint_as_float(cur[2 * i + 1]), cs, bs);
      } else {
        const float2 x = PRESCALED ? f2(cur[2 * i], cur[2 * i + 1]) : __ffma2_rn(f2(cur[2 * i], cur[2 * i + 1]), c2, nm2);
        p = make_float2(ex2(x.x), ex2(x.y));
      }
      if (MASKED) {
        if (ch * 16 + 2 * i >= valid) p.x = 0.f;
        if (ch * 16 + 2 * i + 1 >= valid) p.y = 0.f;
      }
      acc[i & 3] = __fadd2_rn(acc[i & 3], p);
      const __nv_bfloat162 b = __floats2bfloat162_rn(p.x, p.y);
      pk[i] = *reinterpret_cast<const uint32_t*>(&b);
    }
    tmem_st8(t_s + ch * 8, pk);
  }
  const float2 a01 = __fadd2_rn(acc[0], acc[1]), a23 = __fadd2_rn(acc[2], acc[3]);
  return (a01.x + a01.y) + (a23.x + a23.y);
}

// How one launch's query groups are dealt out.  Block c takes the groups c, c + blocks, ... (`rounds` of them at most), then
// one share of the key tiles of the remaining `tail` groups, laid end to end and numbered from 0.  These fall into spans of
// equal length (one group each, or all of them together), every span into `per_span` shares whose lengths differ by one
// tile at most: share_base, the first share_rest of them one more.
struct AttentionPlan {
  int groups, blocks, rounds, tiles;             // tiles: key tiles of a group
  int tail, span, per_span, share_base, share_rest;
  __device__ __forceinline__ int share_start(int c) const {
    const int s = c / per_span, i = c - s * per_span;
    return min(s * span + i * share_base + min(i, share_rest), tail * tiles);
  }
  __device__ __forceinline__ int share_of(int unit) const {      // the block whose share holds this tile
    const int s = unit / span, v = unit - s * span, border = share_rest * (share_base + 1);
    return s * per_span + (v < border ? v / (share_base + 1) : share_rest + (v - border) / share_base);
  }
};
// A run of key tiles of one group; a block's runs in the order it works on them.
struct Run {
  int group, first, n;                           // key tiles [first, first + n) of the group
};
enum AttentionMode { kWhole, kCluster, kCut };
template <AttentionMode MODE>
struct RunIter {
  const AttentionPlan& plan;
  int block, k = 0, u = 0, end = 0;
  __device__ __forceinline__ RunIter(const AttentionPlan& p, int c) : plan(p), block(c) {}
  __device__ __forceinline__ int number() const { return k - 1; }       // of the current run (all of a share's: the same)
  __device__ __forceinline__ bool next(Run& r) {
    if (MODE != kCut) {                          // one run only
      if (k++) return false;
      r.group = MODE == kWhole ? block : block / plan.per_span;
      r.first = MODE == kWhole ? 0 : plan.share_start(block) - r.group * plan.tiles;
      r.n = MODE == kWhole ? plan.tiles : plan.share_start(block + 1) - r.group * plan.tiles - r.first;
      return true;
    }
    if (k < plan.rounds) {
      r.group = block + k * plan.blocks; r.first = 0; r.n = plan.tiles;
      ++k;
      return r.group < plan.groups;
    }
    if (plan.tail == 0) return false;
    if (k == plan.rounds) { u = plan.share_start(block); end = plan.share_start(block + 1); ++k; }
    if (u >= end) return false;
    const int g = u / plan.tiles;
    r.group = plan.groups - plan.tail + g;
    r.first = u - g * plan.tiles;
    r.n = min(end - u, plan.tiles - r.first);
    u += r.n;
    return true;
  }
};
// Workspace of a launch that cuts groups: per block two slots (its first and its last run), per slot and softmax warp
// 32 rows x 32 accumulator columns (eight float4 planes) and the 32 row sums; one counter per block and warp.
constexpr int kPartFloats = 8 * 32 * 4 + 32;
constexpr size_t kSlotFloats = (size_t)kSoftmaxWarps * kPartFloats;

// Counts one part in and returns how many of this launch came before it.  A counter carries the number of the launch that
// last counted in it (upper half): whatever a launch left behind that could not finish (a block that gave up on a wait
// never counts its parts) is not this launch's count.
__device__ __forceinline__ int count_part(unsigned long long* counter, unsigned launch) {
  const unsigned long long none = (unsigned long long)launch << 32;
  unsigned long long seen = __ldcg(counter);
  for (;;) {                                       // (goes round only where another part has been counted meanwhile)
    const unsigned long long before = seen >> 32 == launch ? seen : none;
    const unsigned long long found = atomicCAS(counter, seen, before + 1);
    if (found == seen) return (int)(unsigned)before;
    seen = found;
  }
}

// The fast kernel's shared memory.  Two query groups (the next one is fetched while this one is worked on) and the ring; in
// kCluster, one query group, a shorter ring, and behind it the place for the other blocks' pieces.
template <AttentionMode MODE>
struct FastSmem {
  static constexpr int kStages = MODE == kCluster ? 4 : kKvStages;
  static constexpr int kQBufs = MODE == kCluster ? 1 : 2;
  static constexpr int kBars = 2 + 2 + 2 * kKvStages + 4 + 4 + 2 + 8;
  uint8_t *q, *kv;
  uint64_t *bars, *safe_bars;                      // (the latter for the safe path, should this block need it)
  uint32_t* tmem_slot;
  volatile int* abort_flag;
  float* xchg;                                     // [2][kXchgFloats]
  int *n_bad, *bad_cut, *bad;                      // see in_range
  __device__ __forceinline__ explicit FastSmem(uint8_t* base) {
    q = base;
    kv = base + kQBufs * kQTiles * kQBytes;
    bars = reinterpret_cast<uint64_t*>(base + 2 * kQTiles * kQBytes + (size_t)kKvStages * kKvStageBytes);
    safe_bars = bars + kBars;
    tmem_slot = reinterpret_cast<uint32_t*>(safe_bars + kSafeBars);
    abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    static_assert((kBars + kSafeBars) * 8 + 8 <= (int)kFastBarBytes, "barrier block");
    xchg = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(bars) + kFastBarBytes);
    n_bad = reinterpret_cast<int*>(xchg + 2 * kXchgFloats);
    bad_cut = n_bad + 1;                           // [2] a bit per slice (query tile * 4 + quadrant) of the share's runs
    bad = n_bad + 3;                               // [kMaxBad] whole runs: number of the run * 8 + slice
  }
};

// The recorded slices once more, on the safe path.  One group at a time: the recorded slices, or, where the list was too
// short, the whole of every whole group.  Of a group that several blocks share exactly the recorded slices: the others are
// another block's to write.  (A call of its own: what it needs in registers stays out of the fast path's allocation.)
template <bool PRESCALED, AttentionMode MODE>
static __device__ __noinline__ void recompute(const CUtensorMap& tm_q, const CUtensorMap& tm_k, const CUtensorMap& tm_v,
                                              __nv_bfloat16* O, int n_q, int N, int heads, const AttentionPlan& plan,
                                              uint8_t* smem) {
  const FastSmem<MODE> sm(smem);
  const int q_groups = (n_q + kQT * kQTiles - 1) / (kQT * kQTiles);
  const int n_marked = *sm.n_bad;
  RunIter<MODE> it(plan, blockIdx.x);
  Run run;
  bool used = false;
  int part = 0;
  while (it.next(run)) {
    uint32_t mask = 0;
    if (MODE == kCut && run.n < plan.tiles) {
      mask = (uint32_t)sm.bad_cut[part++];
    } else if (n_marked <= kMaxBad) {
      for (int k = 0; k < n_marked; ++k)
        if (sm.bad[k] >> 3 == it.number()) mask |= 1u << (sm.bad[k] & 7);
    } else {
      mask = ~0u;
    }
    if (mask == 0) continue;                       // block-uniform
    const int qg = run.group % q_groups, bh = run.group / q_groups;
    if (threadIdx.x == 0) {
      if (used)
        for (int k = 0; k < kSafeBars; ++k) mbar_inval(&sm.safe_bars[k]);
      safe_init_barriers(sm.safe_bars, live_tiles(qg, n_q));
      mbar_fence_init();
    }
    used = true;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // (kCluster has used the ring through plain stores)
    __syncthreads();
    tc_fence_after();
    safe_roles({&tm_q, &tm_k, &tm_v, O, n_q, N, heads, qg, bh % heads, bh / heads, PRESCALED ? 1.0f : kScoreScaleLog2,
                mask, sm.q, sm.kv, sm.safe_bars, sm.xchg, sm.abort_flag, *sm.tmem_slot});
    tc_fence_before();
    __syncthreads();
    if (*sm.abort_flag) break;
  }
}

// cta_words (may be null): one word per query group, set to 2 where a block gave up on a bounded wait.
template <bool PRESCALED, AttentionMode MODE>
__global__ void __launch_bounds__(kAttThreads, 1)
tc_attention_fast_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                         const __grid_constant__ CUtensorMap tm_v, __nv_bfloat16* __restrict__ O, int n_q, int N,
                         int heads, const __grid_constant__ AttentionPlan plan, const __grid_constant__ AttentionParts parts,
                         int* __restrict__ status, int* __restrict__ cta_words) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const FastSmem<MODE> sm(smem);
  constexpr int kStages = FastSmem<MODE>::kStages;
  uint8_t *const s_q = sm.q, *const s_kv = sm.kv;
  uint64_t* const bars = sm.bars;
  uint64_t* q_full = bars;                         // [2]           TMA -> both issuers
  uint64_t* q_empty = q_full + 2;                  // [2], count 2  both issuers -> TMA
  uint64_t* kv_full = q_empty + 2;                 // [kKvStages]           TMA -> both issuers
  uint64_t* kv_empty = kv_full + kKvStages;        // [kKvStages], count 2  both issuers -> TMA
  uint64_t* s_full = kv_empty + kKvStages;         // [qt][parity]  issuer -> softmax: S is ready
  uint64_t* p_full = s_full + 4;                   // [qt][parity]  softmax -> issuer: P is in TMEM (8 warps)
  uint64_t* pv_full = p_full + 4;                  // [qt]          issuer -> softmax: the last P V of a run is done
  uint64_t* pair_bar = pv_full + 2;                // [qt][quadrant] the two warps that share 32 query rows
  uint32_t* const tmem_slot = sm.tmem_slot;
  volatile int* const abort_flag = sm.abort_flag;
  float* const xchg = sm.xchg;
  int *const n_bad = sm.n_bad, *const bad_cut = sm.bad_cut, *const bad = sm.bad;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int q_groups = (n_q + kQT * kQTiles - 1) / (kQT * kQTiles);
  const int block = blockIdx.x;
  const int sid = warp - kFirstSoftmaxWarp;
  const int t_own = (sid >> 2) & 1;                    // a softmax warp's query tile
  const int hh = sid >> 3;                             // ... which 48 of a tile's 96 score columns
  const int quad = warp & 3;                           // ... the TMEM lane quadrant it may touch
  const int row = quad * 32 + lane;                    // ... query row within the tile
  static_assert(PRESCALED || MODE == kWhole, "parts of a group add up only where there is no maximum");

  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) { mbar_init(&q_full[i], 1); mbar_init(&q_empty[i], 2); }
    for (int i = 0; i < kStages; ++i) { mbar_init(&kv_full[i], 1); mbar_init(&kv_empty[i], 2); }
    for (int i = 0; i < 4; ++i) { mbar_init(&s_full[i], 1); mbar_init(&p_full[i], 8); }
    for (int i = 0; i < kQTiles; ++i) mbar_init(&pv_full[i], 1);
    for (int i = 0; i < 8; ++i) mbar_init(&pair_bar[i], 2);
    *abort_flag = 0;
    *n_bad = bad_cut[0] = bad_cut[1] = 0;
    mbar_fence_init();
  }
  if (warp == 0 && lane == 0) { tma_prefetch_desc(&tm_q); tma_prefetch_desc(&tm_k); tma_prefetch_desc(&tm_v); }
  if (warp == 1) { tmem_alloc(tmem_slot, kAttTmemCols); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  if (MODE == kCluster) cluster_arrive();              // waited for before anything is sent to another block
  // The row sum tells whether the fixed scaling was good enough (Inf and NaN are caught too; without a maximum the sum must
  // not be vanishingly small either).  If not, the warp's rows are left to the safe path below; of the warps that come to
  // the same verdict on them, the first half's in the first block records them.  `run`: which of the block's runs; `part`:
  // for a part of a group, which of the (at most two) parts in the block's share, else -1.
  auto in_range = [&](float l_row, int qi, int run, int part) -> bool {
    const bool bad_row = qi < n_q && !(l_row < kRowSumLimit && (!PRESCALED || l_row > kRowSumFloor));
    if (!__any_sync(0xFFFFFFFFu, bad_row)) return true;
    if (lane == 0 && hh == 0 && (MODE != kCluster || block % plan.per_span == 0)) {
      const int slice = t_own * 4 + quad;
      if (part >= 0) {
        atomicOr(&bad_cut[part], 1 << slice);
      } else {
        const int at = atomicAdd(n_bad, 1);
        if (at < kMaxBad) bad[at] = run * 8 + slice;
      }
    }
    return false;
  };
  // First output feature of a row's half (a block of one run knows it from the start).
  auto row_of = [&](int group) { return (group % q_groups * kQTiles + t_own) * kQT + row; };
  auto output_of = [&](int group, int qi) {
    const int bh = group / q_groups, h = bh % heads, b = bh / heads;
    return O + ((long long)b * n_q + qi) * ((long long)heads * kHD) + h * kHD;
  };
  const int only_group = MODE == kCluster ? block / plan.per_span : block;
  int qi = row_of(only_group);
  __nv_bfloat16* dst = output_of(only_group, qi);
  bool finished = false;                               // kCluster: this warp's rows are complete in TMEM, their sum is
  float l_cluster = 0.f;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      RunIter<MODE> it(plan, block);
      Run run;
      int stage = 0, qb = 0; uint32_t phase = 0, q_phase = 0;
      bool ok = true, first = true;
      while (ok && it.next(run)) {
        const int qg = run.group % q_groups, bh = run.group / q_groups, h = bh % heads, b = bh / heads;
        const int n_tiles = live_tiles(qg, n_q);
        if (first) stream_order();                     // (where to begin is known by then)
        first = false;
        if (!(ok = mbar_wait(&q_empty[qb], q_phase ^ 1, abort_flag))) break;
        mbar_expect_tx(&q_full[qb], n_tiles * kQBytes);
        for (int t = 0; t < n_tiles; ++t)
          tma_load_2d(s_q + (qb * kQTiles + t) * kQBytes, &tm_q, &q_full[qb], h * kHD, b * n_q + (qg * kQTiles + t) * kQT);
        for (int j = run.first; j < run.first + run.n; ++j) {
          if (!(ok = mbar_wait(&kv_empty[stage], phase ^ 1, abort_flag))) break;
          uint8_t* sk = s_kv + (size_t)stage * kKvStageBytes;
          mbar_expect_tx(&kv_full[stage], kKvStageBytes);
          tma_load_3d(sk, &tm_k, &kv_full[stage], h * kHD, j * kKT, b);
          tma_load_3d(sk + kKBytes, &tm_v, &kv_full[stage], h * kHD, j * kKT, b);
          if (++stage == kStages) { stage = 0; phase ^= 1; }
        }
        qb ^= 1;
        if (qb == 0) q_phase ^= 1;
      }
      for (int i = 0; i < kStages; ++i) {      // all armed stages consumed before the CTA retires
        if (!mbar_wait(&kv_empty[stage], phase ^ 1, abort_flag)) break;
        if (++stage == kStages) { stage = 0; phase ^= 1; }
      }
    } else {
      stream_order();
    }
  } else if (warp == 1 || warp == 2) {
    // ------------------------------------------------------------ MMA issuer warp of query tile t
    // Scores run two key tiles ahead of P V, across the border between two runs as well (the next run's queries are
    // there by then).  The K/V ring counts every tile of the block; the score buffers count this query tile's.
    stream_order();
    const bool leader = elect_one();
    const int t = warp - 1;
    constexpr uint32_t idesc_s = idesc_bf16(kQT, kKT, 0);    // S = Q K^T : both operands K-contiguous
    constexpr uint32_t idesc_pv = idesc_bf16(kQT, kHD, 1);   // O += P V  : V is N(head_dim)-contiguous
    const uint32_t t_tile = tmem_base + (uint32_t)t * kTileCols;
    RunIter<MODE> ahead(plan, block), it(plan, block);
    Run run;
    int a_left = 0, a_qb = 1, a_stage = 0, s_cnt = 0;
    uint32_t a_phase = 0, aq_phase = 1;
    bool a_live = false;
    // The next score tile, if there is one.  (A run whose second query tile has no row: that tile's issuer follows the
    // ring without issuing anything.)
    auto issue_s = [&]() -> bool {
      if (a_left == 0) {
        Run next;
        if (!ahead.next(next)) return true;
        a_left = next.n;
        a_live = t < live_tiles(next.group % q_groups, n_q);
        a_qb ^= 1;
        if (a_qb == 0) aq_phase ^= 1;
        if (!mbar_wait_warp(&q_full[a_qb], aq_phase, abort_flag)) return false;
      }
      if (!mbar_wait_warp(&kv_full[a_stage], a_phase, abort_flag)) return false;
      tc_fence_after();
      --a_left;
      if (a_live) {
        const uint64_t dq = smem_desc_sw128(smem_u32(s_q + (a_qb * kQTiles + t) * kQBytes), 1024);
        const uint64_t dk = smem_desc_sw128(smem_u32(s_kv + (size_t)a_stage * kKvStageBytes), 1024);
        const uint32_t d = t_tile + (uint32_t)(s_cnt & 1) * kKT;
        if (leader) {
#pragma unroll
          for (int k = 0; k < kHD / 16; ++k) mma_ss(d, dq + 2 * k, dk + 2 * k, idesc_s, k != 0);
          mma_commit(&s_full[t * 2 + (s_cnt & 1)]);
          if (a_left == 0) mma_commit(&q_empty[a_qb]);       // these queries are done with
        }
        ++s_cnt;
      } else if (leader && a_left == 0) {
        mbar_arrive(&q_empty[a_qb]);
      }
      if (++a_stage == kStages) { a_stage = 0; a_phase ^= 1; }
      return true;
    };
    bool ok = issue_s() && issue_s();              // two score tiles ahead of the softmax
    int stage = 0, cnt = 0;
    while (ok && it.next(run)) {
      const bool live = t < live_tiles(run.group % q_groups, n_q);
      for (int j = 0; j < run.n; ++j) {
        if (live) {
          // V tile: rows = keys (128 bytes each), 8-key groups 1024 bytes apart; 16 keys per MMA = 2048 bytes
          const uint64_t dv = smem_desc_sw128(smem_u32(s_kv + (size_t)stage * kKvStageBytes + kKBytes), 1024);
          if (!(ok = mbar_wait_warp(&p_full[t * 2 + (cnt & 1)], (cnt >> 1) & 1, abort_flag))) break;
          tc_fence_after();
          const uint32_t buf = t_tile + (uint32_t)(cnt & 1) * kKT;
          if (leader) {
            // P of keys [16k, 16k+16) sits in 8 columns: the first 48 keys in columns [0, 24) of the buffer,
            // the last 48 in columns [48, 72) (each half of the softmax writes inside its own score columns).
            // (The first product of a run overwrites the accumulator: its P came after the run before was read out.)
#pragma unroll
            for (int k = 0; k < kKT / 16; ++k)
              mma_ts(t_tile + kColO, buf + (k / 3) * kHalf + (k % 3) * 8, dv + 128 * k, idesc_pv, (j | k) != 0);
            if (j == run.n - 1) mma_commit(&pv_full[t]);
            mma_commit(&kv_empty[stage]);          // second arrival comes from the other tile's issuer
          }
          ++cnt;
        } else if (leader) {
          mbar_arrive(&kv_empty[stage]);
        }
        if (++stage == kStages) stage = 0;
        // the scores two tiles on overwrite the buffer whose P the product above reads: safe because the
        // tensor core executes this thread's MMAs in issue order
        if (!(ok = issue_s())) break;
      }
    }
  } else if (warp >= kFirstSoftmaxWarp) {
    // ------------------------------------------------------------ softmax
    stream_order();
    const int t = t_own;
    const uint32_t lane_base = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)t * kTileCols;
    uint64_t* my_pair = &pair_bar[t * 4 + quad];
    const float c = PRESCALED ? 1.0f : kScoreScaleLog2;
    const float2 c2 = make_float2(c, c);
    float2 nm2 = make_float2(0.f, 0.f);
    const float cs = c / kPolySpan;
    float bs = 0.5f;
    uint32_t pair_phase = 0, pv_phase = 0;
    int cnt = 0;                                       // key tiles of this query tile so far
    bool ok = true;
    RunIter<MODE> it(plan, block);
    Run run;
    while (ok && it.next(run)) {
      const int qg = run.group % q_groups;
      if (t >= live_tiles(qg, n_q)) continue;
      float l_half = 0.f;
      const int n_left = N - run.first * kKT - hh * kHalf;
      for (int j = 0; j < run.n; ++j, ++cnt) {
        ok = mbar_wait_warp(&s_full[t * 2 + (cnt & 1)], (cnt >> 1) & 1, abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint32_t t_s = lane_base + (uint32_t)(cnt & 1) * kKT + (uint32_t)hh * kHalf;
        int valid = n_left - j * kKT;                  // columns of this half that are keys
        valid = valid < 0 ? 0 : (valid > kHalf ? kHalf : valid);
        if (!PRESCALED && j == 0) {
          // First tile: the maximum over its (existing) keys becomes the row's scaling maximum for good.
          // Both halves read their columns, trade their maxima through shared memory, and then form P
          // from the scores they still hold in registers.
          uint32_t s[kHalf];
#pragma unroll
          for (int ch = 0; ch < kHalf / 16; ++ch) tmem_ld16(t_s + ch * 16, *reinterpret_cast<uint32_t(*)[16]>(&s[ch * 16]));
          tmem_ld_wait();
          float m = -INFINITY;
#pragma unroll
          for (int i = 0; i < kHalf; ++i)
            if (i < valid) m = fmaxf(m, __uint_as_float(s[i]));
          xchg[(t * kQT + row) * 2 + hh] = m;
          __syncwarp();
          if (lane == 0) mbar_arrive(my_pair);
          if (!(ok = mbar_wait_warp(my_pair, pair_phase, abort_flag))) break;
          pair_phase ^= 1;
          m = fmaxf(xchg[(t * kQT + row) * 2], xchg[(t * kQT + row) * 2 + 1]);   // finite: column 0 always exists
          nm2 = make_float2(-m * c, -m * c);
          bs = fmaf(-m, cs, 0.5f);
          float2 acc = make_float2(0.f, 0.f);
#pragma unroll
          for (int ch = 0; ch < kHalf / 16; ++ch) {
            uint32_t pk[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const int col = ch * 16 + 2 * i;
              const float2 x = __ffma2_rn(f2(s[col], s[col + 1]), c2, nm2);
              float2 p = make_float2(ex2(x.x), ex2(x.y));
              if (col >= valid) p.x = 0.f;
              if (col + 1 >= valid) p.y = 0.f;
              acc = __fadd2_rn(acc, p);
              const __nv_bfloat162 bb = __floats2bfloat162_rn(p.x, p.y);
              pk[i] = *reinterpret_cast<const uint32_t*>(&bb);
            }
            tmem_st8(t_s + ch * 8, pk);
          }
          l_half = acc.x + acc.y;
        } else if (valid == kHalf) {
          l_half += half_tile<false, PRESCALED>(t_s, valid, c2, nm2, cs, bs);
        } else {
          l_half += half_tile<true, PRESCALED>(t_s, valid, c2, nm2, cs, bs);
        }
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&p_full[t * 2 + (cnt & 1)]);
      }
      if (!ok) break;
      // The row sum is the sum of the halves'.  (Two exchange buffers in turn: a warp may be a run ahead of its partner
      // but not two.  Without a maximum to trade, PRESCALED has both; otherwise the exchange of the maxima lies between.)
      float* const xl = xchg + (PRESCALED ? (int)(pair_phase & 1) : 1) * kXchgFloats;
      xl[(t * kQT + row) * 2 + hh] = l_half;
      __syncwarp();
      if (lane == 0) mbar_arrive(my_pair);
      if (!(ok = mbar_wait_warp(my_pair, pair_phase, abort_flag))) break;
      pair_phase ^= 1;
      float l_row = xl[(t * kQT + row) * 2] + xl[(t * kQT + row) * 2 + 1];
      if (!(ok = mbar_wait_warp(&pv_full[t], pv_phase, abort_flag))) break;
      pv_phase ^= 1;
      tc_fence_after();

      if (MODE == kCluster) {
        finished = true;
        l_cluster = l_row;
        break;
      }

      // Each half finishes 32 of the row's 64 output features.
      const uint32_t t_out = lane_base + kColO + hh * 32;
      if (MODE == kCut) {
        qi = row_of(run.group);
        dst = output_of(run.group, qi);
      }
      if (MODE == kWhole || run.n == plan.tiles) {
        if (in_range(l_row, qi, it.number(), -1)) {
          const float inv = 1.0f / l_row;
#pragma unroll
          for (int ch = 0; ch < 2; ++ch) {
            uint32_t r[16];
            tmem_ld16(t_out + ch * 16, r);             // warp-collective: every lane loads
            tmem_ld_wait();
            if (qi < n_q) emit16(r, inv, dst + hh * 32 + ch * 16);
          }
        }
        continue;
      }
      // A part of the keys only.  The first of a group's parts may be the second run of its block, the others are the
      // first runs of theirs.
      const int u0 = (run.group - plan.groups + plan.tail) * plan.tiles;
      const int c_first = plan.share_of(u0), c_last = plan.share_of(u0 + plan.tiles - 1);
      const int first_slot = 2 * c_first + (plan.share_start(c_first) >= u0 ? 0 : 1);
      const int my_slot = block == c_first ? first_slot : 2 * block;
      {
        float* const part = parts.rows + (size_t)my_slot * kSlotFloats + sid * kPartFloats;
#pragma unroll 1
        for (int ch = 0; ch < 2; ++ch) {
          uint32_t r[16];
          tmem_ld16(t_out + ch * 16, r);
          tmem_ld_wait();
#pragma unroll
          for (int q = 0; q < 4; ++q)
            __stcg(reinterpret_cast<float4*>(part) + (ch * 4 + q) * 32 + lane,
                   make_float4(__uint_as_float(r[4 * q]), __uint_as_float(r[4 * q + 1]), __uint_as_float(r[4 * q + 2]),
                               __uint_as_float(r[4 * q + 3])));
        }
        __stcg(part + 8 * 32 * 4 + lane, l_row);
      }
      __threadfence();
      __syncwarp();
      int before = 0;
      if (lane == 0) before = count_part(parts.count + c_first * kSoftmaxWarps + sid, parts.launch);
      before = __shfl_sync(0xFFFFFFFFu, before, 0);
      if (before < c_last - c_first) continue;         // the others are not all there yet
      __threadfence();
      if (lane == 0) parts.count[c_first * kSoftmaxWarps + sid] = 0;         // (launches are numbered from 1)
      l_row = 0.f;
      for (int k = c_first; k <= c_last; ++k)
        l_row += __ldcg(parts.rows + (size_t)(k == c_first ? first_slot : 2 * k) * kSlotFloats + sid * kPartFloats + 8 * 32 * 4 + lane);
      if (!in_range(l_row, qi, it.number(), my_slot & 1)) continue;
#pragma unroll 1
      for (int ch = 0; ch < 2; ++ch) {
        float4 sum[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) sum[q] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
        for (int k = c_first; k <= c_last; ++k) {
          const float4* part = reinterpret_cast<const float4*>(
              parts.rows + (size_t)(k == c_first ? first_slot : 2 * k) * kSlotFloats + sid * kPartFloats);
          float4 v[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) v[q] = __ldcg(part + (ch * 4 + q) * 32 + lane);
#pragma unroll
          for (int q = 0; q < 4; ++q) { sum[q].x += v[q].x; sum[q].y += v[q].y; sum[q].z += v[q].z; sum[q].w += v[q].w; }
        }
        uint32_t r[16];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          r[4 * q] = __float_as_uint(sum[q].x); r[4 * q + 1] = __float_as_uint(sum[q].y);
          r[4 * q + 2] = __float_as_uint(sum[q].z); r[4 * q + 3] = __float_as_uint(sum[q].w);
        }
        if (qi < n_q) emit16(r, 1.0f / l_row, dst + hh * 32 + ch * 16);
      }
    }
  }

  if (warp == 3) stream_order();
  if (MODE == kCluster) {
    // ---------------------------------------------------------------- the cluster's parts
    // Piece p (16 columns) of the accumulators is finished by rank p % split, which receives the others' in turn:
    // [piece / split][sender][four columns][row of 256] words of 16 bytes, behind them the row sums.
    const int rank = block % plan.per_span;
    constexpr int kRows = kQTiles * kQT;
    float4* const pieces = reinterpret_cast<float4*>(s_kv + (size_t)kStages * kKvStageBytes);
    float* const sums = reinterpret_cast<float*>(pieces + 4 * 4 * kRows);        // (behind four pieces, the most there are)
    static_assert(kQTiles * kQBytes + 4 * kKvStageBytes + (4 * 4 * 16 + 3 * 4) * kRows <=
                  2 * kQTiles * kQBytes + kKvStages * kKvStageBytes, "ring and pieces fit");
    const int my_row = t_own * kQT + row;
    const uint32_t t_out = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)t_own * kTileCols + kColO;
    auto merge = [&](auto split_c) {
      constexpr int S = decltype(split_c)::value;
      __syncwarp();
      cluster_wait();                                  // the other blocks have started (long since)
      if (finished) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {                  // each half sends two pieces, or keeps them
          const int p = hh * 2 + i, to = p % S;
          if (to == rank) continue;                    // warp-uniform
          uint32_t r[16];
          tmem_ld16(t_out + p * 16, r);
          tmem_ld_wait();
          const int slot = (p / S) * (S - 1) + (rank < to ? rank : rank - 1);
          const uint32_t at = cluster_map(smem_u32(pieces + slot * 4 * kRows + my_row), (uint32_t)to);
#pragma unroll
          for (int q = 0; q < 4; ++q)
            st_cluster_v4(at + q * kRows * 16, __uint_as_float(r[4 * q]), __uint_as_float(r[4 * q + 1]),
                          __uint_as_float(r[4 * q + 2]), __uint_as_float(r[4 * q + 3]));
        }
        if (hh == 0) {
#pragma unroll
          for (int to = 0; to < S; ++to)
            if (to != rank)
              st_cluster_f32(cluster_map(smem_u32(sums + (rank < to ? rank : rank - 1) * kRows + my_row), (uint32_t)to), l_cluster);
        }
      }
      __syncwarp();
      cluster_sync();
      if (!finished) return;
      float l_row = 0.f;                               // (added in rank order, as everything here)
#pragma unroll
      for (int k = 0; k < S; ++k) l_row += k == rank ? l_cluster : sums[(k < rank ? k : k - 1) * kRows + my_row];
      if (!in_range(l_row, qi, 0, -1)) return;         // (all ranks come to the same verdict; the first records it)
      const float inv = 1.0f / l_row;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int p = S == 4 ? rank : hh * 2 + i;      // of four ranks each has one piece: its first half finishes it
        if (p % S != rank || (S == 4 && (hh != 0 || i != 0))) continue;          // warp-uniform
        uint32_t r[16];
        tmem_ld16(t_out + p * 16, r);
        tmem_ld_wait();
        const float4* at = pieces + (p / S) * (S - 1) * 4 * kRows + my_row;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int k = 0; k < S; ++k) {
            const float4 o = k == rank ? make_float4(__uint_as_float(r[4 * q]), __uint_as_float(r[4 * q + 1]),
                                                     __uint_as_float(r[4 * q + 2]), __uint_as_float(r[4 * q + 3]))
                                       : at[((k < rank ? k : k - 1) * 4 + q) * kRows];
            v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
          }
          r[4 * q] = __float_as_uint(v.x); r[4 * q + 1] = __float_as_uint(v.y);
          r[4 * q + 2] = __float_as_uint(v.z); r[4 * q + 3] = __float_as_uint(v.w);
        }
        if (qi < n_q) emit16(r, inv, dst + p * 16);
      }
    };
    if (plan.per_span == 2) merge(std::integral_constant<int, 2>{});
    else if (plan.per_span == 3) merge(std::integral_constant<int, 3>{});
    else merge(std::integral_constant<int, 4>{});
  }

  // ---------------------------------------------------------------- rows out of range: once more, on the safe path
  tc_fence_before();
  __syncthreads();
  // (What is needed from here on is worked out anew, so that it does not sit in a register until now.)
  uint32_t smem_again = smem_u32(smem_raw);
  asm volatile("" : "+r"(smem_again));
  const FastSmem<MODE> end(static_cast<uint8_t*>(__cvta_shared_to_generic((smem_again + 1023) & ~1023u)));
  if ((*end.n_bad | end.bad_cut[0] | end.bad_cut[1]) != 0 && !*end.abort_flag)             // block-uniform
    recompute<PRESCALED, MODE>(tm_q, tm_k, tm_v, O, n_q, N, heads, plan, end.q);

  // ---------------------------------------------------------------- teardown
  if (threadIdx.x == 0 && *end.abort_flag) {
    atomicAdd(status, 1);
    if (cta_words != nullptr) {
      RunIter<MODE> it(plan, blockIdx.x);
      Run run;
      while (it.next(run)) cta_words[run.group] = 2;
    }
  }
  if (threadIdx.x >> 5 == 1) { __syncwarp(); tc_fence_after(); tmem_dealloc(*end.tmem_slot, kAttTmemCols); }
}

}  // namespace

// Tensor maps of one attention problem: Q as [B * n_q, D] rows, K and V as [B][N][D].
static int make_attention_maps(const void* q, const void* k, const void* v, int B, int n_q, int N, int heads,
                               CUtensorMap* tm_q, CUtensorMap* tm_k, CUtensorMap* tm_v) {
  const uint64_t D = (uint64_t)heads * kHD;
  {
    const uint64_t dims[2] = {D, (uint64_t)B * n_q};
    const uint64_t str[1] = {D * 2};
    const uint32_t box[2] = {(uint32_t)kHD, (uint32_t)kQT};
    HERO_TRY(make_tmap_bf16(tm_q, q, 2, dims, str, box));
  }
  {
    const uint64_t dims[3] = {D, (uint64_t)N, (uint64_t)B};
    const uint64_t str[2] = {D * 2, (uint64_t)N * D * 2};
    const uint32_t box[3] = {(uint32_t)kHD, (uint32_t)kKT, 1};
    HERO_TRY(make_tmap_bf16(tm_k, k, 3, dims, str, box));
    HERO_TRY(make_tmap_bf16(tm_v, v, 3, dims, str, box));
  }
  return HERO_OK;
}

constexpr int kMaxSplit = 4;
static int g_resident_clusters[kMaxDevices][kMaxSplit + 1];      // clusters of this many blocks that a device holds at once

static int attention_kernel_attributes() {
  static PerDeviceOnce attr_once;            // the opt-in is a property of the kernel ON a device
  return per_device_once(attr_once, [](int dev) {
    HERO_CUDA_TRY(cudaFuncSetAttribute(tc_attention_safe_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kSafeSmem));
    for (auto kernel : {tc_attention_fast_kernel<false, kWhole>, tc_attention_fast_kernel<true, kWhole>,
                        tc_attention_fast_kernel<true, kCluster>, tc_attention_fast_kernel<true, kCut>})
      HERO_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFastSmem));
    for (int split = 2; split <= kMaxSplit; ++split) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)(split * 64));
      cfg.blockDim = dim3(kAttThreads);
      cfg.dynamicSmemBytes = kFastSmem;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = (unsigned)split; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      HERO_CUDA_TRY(cudaOccupancyMaxActiveClusters(&g_resident_clusters[dev][split],
                                                   tc_attention_fast_kernel<true, kCluster>, &cfg));
    }
    return HERO_OK;
  });
}

long long tc_attention_grid(int B, int n_q, int heads) {
  const long long q_groups = ((long long)n_q + kQT * kQTiles - 1) / (kQT * kQTiles);
  return q_groups * heads * B;
}

// Which mode, and how the groups are dealt out.  Measured (us; queries x keys x heads x batch):
//   * a cluster wherever all clusters are on the chip at once (what does not fit waits for a whole cluster's worth of free
//     SMs): 371 x 1562 x 12, 24 groups, whole 18.9, over four 12.8; 620 x 1319 x 8 x 2, 48 groups, whole 15.8, over two 15.4,
//     over three (which do not all fit) 24.1.  Under six key tiles there is nothing to win.
//   * cutting the last round pays from about 64 key tiles on (a part costs some 5 us of fences, counting and adding up):
//     1755 x 17776 x 48 x 2, 672 groups, 860 -> 851, 4388 x 17776 x 48 x 2, 1728 groups, 2087 -> 2069, the whole 3072-wide
//     cached step 59.6 -> 58.7 ms; but 2970 x 3196 x 48 x 2 (34 tiles) 295 -> 299 and 2627 x 2627 x 18 x 2 84 -> 90.
constexpr int kMinCutTiles = 64;
struct PlannedAttention { AttentionMode mode; AttentionPlan plan; };
static PlannedAttention attention_plan(long long groups, int N, bool may_cluster, bool may_cut) {
  const long long tiles = (N + kKT - 1) / kKT, sms = num_sms(), tail = groups % sms;
  AttentionPlan plan = {(int)groups, (int)groups, 1, (int)tiles, 0, 1, 1, 1, 0};
  auto spans = [&](long long n_spans, long long span, long long shares) {
    plan.span = (int)span; plan.per_span = (int)shares;
    plan.share_base = (int)(span / shares); plan.share_rest = (int)(span % shares);
    plan.tail = (int)(n_spans * span / tiles);
  };
  int dev = 0;
  if (may_cluster && tiles >= 6 && cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < kMaxDevices)
    for (int split = kMaxSplit; split >= 2; --split)
      if (groups <= g_resident_clusters[dev][split]) {
        spans(groups, tiles, split);
        plan.blocks = (int)(groups * split);
        return {kCluster, plan};
      }
  if (may_cut && groups > sms && tail > 0 && tiles >= kMinCutTiles && tail * tiles <= 0x3FFFFFFF) {
    plan.blocks = (int)sms;
    plan.rounds = (int)(groups / sms);
    spans(1, tail * tiles, sms);
    return {kCut, plan};
  }
  return {kWhole, plan};
}

bool tc_attention_may_cut(int B, int n_rows, int heads) {
  return tc_attention_grid(B, n_rows, heads) > num_sms() && (n_rows + kKT - 1) / kKT >= kMinCutTiles;
}
size_t tc_attention_part_bytes() { return (size_t)2 * num_sms() * kSlotFloats * sizeof(float); }
size_t tc_attention_part_counters() { return (size_t)num_sms() * kSoftmaxWarps; }

// What a launch leaves in the counters when every block gives up with one part of each group counted in.
static __global__ void strand_counters_kernel(AttentionParts parts, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) parts.count[i] = ((unsigned long long)parts.launch << 32) + 1;
}
int launch_strand_attention_counters(const AttentionParts& parts, cudaStream_t s) {
  const int n = (int)tc_attention_part_counters();
  strand_counters_kernel<<<(n + 255) / 256, 256, 0, s>>>(parts, n);
  HERO_CUDA_TRY(cudaGetLastError());
  return HERO_OK;
}

// d_status[0] counts thread blocks that gave up on a wait; cta_words may be null.  q_prescaled: the caller has multiplied Q
// by log2(e) / sqrt(head_dim) already, so a score IS the exponent of its weight; the kernel then takes 2^s as it stands,
// with no maximum at all (exact while a row's largest score stays within about +-100, the row sum telling when it did not).
// parts: the caller's for one launch at a time (no rows: groups stay whole).
int launch_tc_attention(const void* q, const void* k, const void* v, void* o, int B, int n_q, int N, int heads,
                        bool q_prescaled, const AttentionParts& parts, int* d_status, int* cta_words, cudaStream_t s) {
  if (B <= 0 || n_q <= 0) return HERO_OK;
  if (N <= 0 || heads <= 0) return HERO_ERR_ARG;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(o)) return HERO_ERR_ALIGN;
  CUtensorMap tm_q, tm_k, tm_v;
  HERO_TRY(make_attention_maps(q, k, v, B, n_q, N, heads, &tm_q, &tm_k, &tm_v));
  HERO_TRY(attention_kernel_attributes());
  const long long groups = tc_attention_grid(B, n_q, heads);
  if (groups > 0x7FFFFFFFll) return HERO_ERR_ARG;
  const PlannedAttention p = attention_plan(groups, N, q_prescaled, q_prescaled && parts.rows != nullptr);
  return launch_kernel(!q_prescaled ? tc_attention_fast_kernel<false, kWhole>
                       : p.mode == kWhole ? tc_attention_fast_kernel<true, kWhole>
                       : p.mode == kCluster ? tc_attention_fast_kernel<true, kCluster> : tc_attention_fast_kernel<true, kCut>,
                       (unsigned)p.plan.blocks, kAttThreads, kFastSmem, s,
                       p.mode == kCluster ? (unsigned)p.plan.per_span : 1u, tm_q, tm_k, tm_v, (__nv_bfloat16*)o, n_q, N,
                       heads, p.plan, parts, d_status, cta_words);
}

// The safe path alone, as a kernel of its own.
int launch_tc_attention_safe(const void* q, const void* k, const void* v, void* o, int B, int n_q, int N, int heads,
                             bool q_prescaled, int* d_status, cudaStream_t s) {
  if (B <= 0 || n_q <= 0) return HERO_OK;
  if (N <= 0 || heads <= 0) return HERO_ERR_ARG;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(o)) return HERO_ERR_ALIGN;
  CUtensorMap tm_q, tm_k, tm_v;
  HERO_TRY(make_attention_maps(q, k, v, B, n_q, N, heads, &tm_q, &tm_k, &tm_v));
  HERO_TRY(attention_kernel_attributes());
  const long long groups = tc_attention_grid(B, n_q, heads);
  if (groups > 0x7FFFFFFFll) return HERO_ERR_ARG;
  return launch_kernel(tc_attention_safe_kernel, (unsigned)groups, kAttThreads, kSafeSmem, s, 1, tm_q, tm_k, tm_v,
                       (__nv_bfloat16*)o, n_q, N, heads, q_prescaled ? 1.0f : kScoreScaleLog2, d_status);
}

}  // namespace hero

// =============================================================================
// hero_attention_bf16_static: the same attention, for callers that must not allocate
// =============================================================================
// hero_attention_bf16 takes its status words from a cudaMalloc made on first use.  Some
// callers cannot afford that: a host thread inside a latency-critical serving loop (cudaMalloc
// and cudaFree synchronise the whole device), a process whose framework has already reserved all
// device memory for its own pool (the allocation would fail), or code that runs where the CUDA
// allocator must not be entered at all.  For them the scratch lives in the library image itself:
// a file-scope __device__ array that every GPU loading the library carries until the process
// exits (kStaticScratchInts * 4 bytes = 64.25 KiB per GPU).
//
// Layout: word 0 counts the CTAs of the latest call that gave up on a bounded wait, word 1 + i
// is CTA i's word (0 = done, 2 = gave up).  The
// array is shared by every call and keeps the previous call's contents, so each call clears the
// words it is going to use on its stream before the kernels run; two calls that overlap on the
// GPU (different streams, no dependency) race on it.
namespace hero {
namespace {

constexpr int kStaticMaxCtas = 16384;                 // largest grid the static scratch can serve
constexpr int kStaticScratchInts = 64 + kStaticMaxCtas;
static __device__ __align__(256) int g_att_static_scratch[kStaticScratchInts];

struct StaticSetup { bool done = false; int* scratch = nullptr; };
StaticSetup g_static_setup[kMaxDevices];
std::mutex g_static_mutex;

// Once per device, with that device current: resolve the DEVICE address of the array (in host
// code the array's name is only a host-side handle, never a pointer a kernel may be given) and
// raise the kernels' dynamic shared-memory limit.
int static_setup(int** scratch) {
  int dev = -1;
  HERO_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return HERO_ERR_ARG;
  HERO_TRY(attention_kernel_attributes());
  std::lock_guard<std::mutex> lock(g_static_mutex);
  StaticSetup& st = g_static_setup[dev];
  if (!st.done) {
    int* p = nullptr;
    HERO_CUDA_TRY(cudaGetSymbolAddress((void**)&p, g_att_static_scratch));
    st.scratch = p;
    st.done = true;
  }
  *scratch = st.scratch;
  return HERO_OK;
}

}  // namespace
}  // namespace hero

extern "C" int hero_attention_bf16_static(const void* d_q, const void* d_k, const void* d_v, void* d_o, int B,
                                          int n_q, int N, int heads, void* stream, int* h_gave_up) {
  using namespace hero;
  if (h_gave_up) *h_gave_up = 0;
  if (B < 0 || n_q < 0 || N <= 0 || heads <= 0) return HERO_ERR_ARG;
  if (B == 0 || n_q == 0) return HERO_OK;
  if (!d_q || !d_k || !d_v || !d_o) return HERO_ERR_ARG;
  if (!aligned16(d_q) || !aligned16(d_k) || !aligned16(d_v) || !aligned16(d_o)) return HERO_ERR_ALIGN;
  const long long grid = tc_attention_grid(B, n_q, heads);
  if (grid > kStaticMaxCtas) {
    set_cuda_error(cudaErrorInvalidConfiguration,
                   "hero_attention_bf16_static: ceil(n_q/256)*heads*B exceeds the 16384 CTAs its static scratch "
                   "serves; split the call or use hero_attention_bf16");
    return HERO_ERR_CAP;
  }
  cudaStream_t s = (cudaStream_t)stream;
  int* scratch = nullptr;
  HERO_TRY(static_setup(&scratch));
  // the array still holds the previous call's records: clear the words this grid will use
  HERO_CUDA_TRY(cudaMemsetAsync(scratch, 0, (size_t)(1 + grid) * sizeof(int), s));
  HERO_TRY(launch_tc_attention(d_q, d_k, d_v, d_o, B, n_q, N, heads, false, AttentionParts{}, scratch, scratch + 1, s));
  if (h_gave_up) {
    HERO_CUDA_TRY(cudaMemcpyAsync(h_gave_up, scratch, sizeof(int), cudaMemcpyDeviceToHost, s));
    HERO_CUDA_TRY(cudaStreamSynchronize(s));
    if (*h_gave_up != 0) return HERO_ERR_TIMEOUT;
  }
  return HERO_OK;
}

// The verdict of the latest hero_attention_bf16_static call on the current device, for callers that passed
// h_gave_up == NULL to stay asynchronous: copies the counter (and, on request, the per-thread-block records)
// out of the static array behind everything queued on `stream`, and waits for that copy.  Allocates nothing.
extern "C" int hero_attention_bf16_static_status(void* stream, int* h_gave_up, int* h_records, int n_records) {
  using namespace hero;
  if (!h_gave_up || n_records < 0 || n_records > kStaticMaxCtas || (n_records > 0 && !h_records)) return HERO_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  int* scratch = nullptr;
  HERO_TRY(static_setup(&scratch));
  HERO_CUDA_TRY(cudaMemcpyAsync(h_gave_up, scratch, sizeof(int), cudaMemcpyDeviceToHost, s));
  if (n_records > 0)
    HERO_CUDA_TRY(cudaMemcpyAsync(h_records, scratch + 1, (size_t)n_records * sizeof(int), cudaMemcpyDeviceToHost, s));
  HERO_CUDA_TRY(cudaStreamSynchronize(s));
  return *h_gave_up != 0 ? HERO_ERR_TIMEOUT : HERO_OK;
}
