// Internal declarations shared by the translation units of libhero.so.
// Nothing here is part of the public ABI (see include/hero.h).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "hero.h"

namespace hero {

// ---------------------------------------------------------------------------
// Error plumbing
// ---------------------------------------------------------------------------
void set_cuda_error(cudaError_t e, const char* what);
#define HERO_CUDA_TRY(expr)                                  \
  do {                                                       \
    cudaError_t e__ = (expr);                                \
    if (e__ != cudaSuccess) {                                \
      ::hero::set_cuda_error(e__, #expr);                    \
      (void)cudaGetLastError();  /* (it is reported here, not by the caller's next CUDA call) */ \
      return HERO_ERR_CUDA;                                  \
    }                                                        \
  } while (0)
#define HERO_TRY(expr)                  \
  do {                                  \
    int r__ = (expr);                   \
    if (r__ != HERO_OK) return r__;     \
  } while (0)

static inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// ---------------------------------------------------------------------------
// Set-up that has to happen once PER DEVICE (a kernel's shared-memory opt-in, a status word in that
// device's memory, its SM count): a process may drive several GPUs, so nothing of this kind may be
// cached per process.  `fn` runs under the table's lock, with the calling thread's device current, the
// first time that device comes by; a failure is not remembered and is retried on the next call.
// ---------------------------------------------------------------------------
constexpr int kMaxDevices = 64;
struct PerDeviceOnce {
  std::mutex mu;
  bool done[kMaxDevices] = {};
};
template <class F>
int per_device_once(PerDeviceOnce& once, F&& fn) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return HERO_ERR_CUDA;
  std::lock_guard<std::mutex> lock(once.mu);
  if (!once.done[dev]) {
    const int rc = fn(dev);
    if (rc != HERO_OK) return rc;
    once.done[dev] = true;
  }
  return HERO_OK;
}

// ---------------------------------------------------------------------------
// Launches.  Kernels are launched with programmatic stream serialisation: their blocks may be placed while the kernel
// before them on the stream still runs, so that launch latency, block start and set-up (barriers, TMEM, tensor-map
// prefetch) are over when that kernel ends.  In return every block of every kernel calls stream_order() before it writes
// anything and before it reads what the kernel in front writes:
//   * the wait returns when all earlier work on the stream is complete and visible (the kernel before has itself waited
//     for its own predecessor, so completion carries over), and
//   * only then may the next kernel's blocks be placed.  A block that uses tensor memory has to have its columns by
//     then: a block of the next kernel on the same SM could otherwise take them and hold them until this kernel ends.
//     (stream_order_wait is the first half alone; the second then happens when the block ends.)
// So a block that runs finds everything complete up to the kernel before the one in front, and may read that before its wait:
// the weights of a GEMM (GemmOut::weights_settled), a step's lists and vectors and the rows of x in the LayerNorm kernels
// (LnSettled, launch_residual_ln), the list of launch_attend_rows.  What a launcher takes for granted stands at its declaration.
// Work of another stream is not among it: behind a wait for an event, a kernel that reads early is launched as an ordinary one.
// Measured, all kernels against none (which is the launch order the kernels had before): mini42 schedule (307 rows, 42
// blocks) 5.36 -> 3.54 ms, width 768 cached step 0.391 -> 0.294, width 1024 cached step 1.156 -> 1.021, fp32 model of width
// 128 0.141 -> 0.108; the 3072-wide 42-block cached step 59.74 -> 59.39.  Kernels that stream large tensors through more
// blocks than fit the chip are the exception (launch_streaming): placed early, the residual and extrapolation passes of
// that step made it 60.5 ms.
// ---------------------------------------------------------------------------
#ifdef __CUDACC__
__device__ __forceinline__ void stream_order_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void stream_order() {
  stream_order_wait();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
#endif
template <class... Params, class... Args>
int launch_kernel_as(bool early, void (*kernel)(Params...), dim3 grid, unsigned threads, size_t smem, cudaStream_t s,
                     unsigned cluster, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = early ? 1 : 0;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = cluster; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  HERO_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, static_cast<Args&&>(args)...));
  return HERO_OK;
}
template <class... Params, class... Args>
int launch_kernel(void (*kernel)(Params...), dim3 grid, unsigned threads, size_t smem, cudaStream_t s, unsigned cluster,
                  Args&&... args) {
  return launch_kernel_as(true, kernel, grid, threads, smem, s, cluster, static_cast<Args&&>(args)...);
}
// A kernel that streams large tensors through many small blocks (256 threads, eight resident per SM): placed early only
// where all its blocks are resident at once.
int num_sms();
template <class... Params, class... Args>
int launch_streaming(void (*kernel)(Params...), long long blocks, unsigned threads, cudaStream_t s, Args&&... args) {
  return launch_kernel_as(blocks <= 8ll * num_sms(), kernel, (unsigned)blocks, threads, 0, s, 1,
                          static_cast<Args&&>(args)...);
}
static inline size_t dtype_size(int dtype) { return dtype == HERO_DTYPE_BF16 ? 2 : 4; }

// ---------------------------------------------------------------------------
// Where a GEMM's output goes (Eq. 3's merge happens in the epilogue).
// The N dimension is cut into up to three segments of seg_cols columns (q | k | v for the
// QKV projection, one segment otherwise).  Row m of the compact operand belongs to batch
// b = m / n_sel and list position i = m % n_sel; a scattered segment writes it to row
// b * n_rows + (idx ? idx[i] : i) of its destination, a compact segment to row m.
// ---------------------------------------------------------------------------
struct GemmOut {
  void* ptr[3];
  long long ld[3];
  int scatter[3];
  int seg_cols;
  const int* idx;
  int n_sel;
  int n_rows;
  const float* gate;   // optional multiplier [B, gate_ld], indexed by column within the segment
  int gate_ld;
  int act;             // 0 = identity, 1 = GELU-tanh
  int weights_settled; // W, bias and idx were complete before the kernel in front was placed: no need to wait for that
  float seg0_scale;    // when not 0: factor on the columns of segment 0 (applied after the bias, before rounding)
};

// Geometry of the selection problem (Sec. 4.3).
struct SelectGeom {
  int frames, grid_h, grid_w, n_text;
  int patch_h, patch_w;
  int ratio_num, ratio_den, quota_mode, track_mode;
  uint32_t seed_lo;
};
constexpr int kMaxSelectBatch = 64;
struct SelectBatch {
  int n;                                  // number of blocks selected in this launch
  int block[kMaxSelectBatch];             // block id (enters the hash)
  int call[kMaxSelectBatch];              // per-block call counter value
  const uint16_t* ages_in[kMaxSelectBatch];
  uint16_t* ages_out[kMaxSelectBatch];
  int* idx[kMaxSelectBatch];
  int* pos[kMaxSelectBatch];              // place of every video token in its list, -1 where it is not in it
};

// ---------------------------------------------------------------------------
// Kernel launchers (each returns HERO_OK or HERO_ERR_CUDA; all asynchronous)
// ---------------------------------------------------------------------------
int launch_select(const SelectGeom& g, const SelectBatch& batch, cudaStream_t s);

int launch_extrapolate(const void* g_prev, const void* g_last, void* out, long long n, int k, int d,
                       int dtype, cudaStream_t s);
// x += e(attn history) ; x += e(ffn history)
int launch_extrapolate_residual(void* x, const void* ga_prev, const void* ga_last, const void* gf_prev,
                                const void* gf_last, long long n, int k, int d, int dtype, cudaStream_t s);
// Several extrapolated blocks in one pass: x += sum over the group's (block, branch) entries of Eq. 5,
// added in the order of the entries, for elements [first, first + n) of every tensor.
constexpr int kMaxDeepGroup = 32;           // blocks per launch (two entries each)
struct DeepGroup {
  int n_plain;                              // 0 or 2: the first entries' `last` is added as it is (a refreshed block's branches)
  int n_entries;
  const void* prev[2 * kMaxDeepGroup];
  const void* last[2 * kMaxDeepGroup];
};
int launch_extrapolate_group(void* x, const DeepGroup& grp, long long first, long long n, int k, int d, int dtype,
                             cudaStream_t s);
// x = (x + ga) + gf
int launch_residual2(void* x, const void* ga, const void* gf, long long n, int dtype, cudaStream_t s);
// deep-stack collapse: x = (x + ga) + gf, acc += ga + gf (fp32);  x += s_last + (s_last - s_prev) * k/d
int launch_residual2_acc(void* x, const void* ga, const void* gf, float* acc, long long n, int dtype, cudaStream_t s);
int launch_extrapolate_stack(void* x, const float* s_prev, const float* s_last, long long n, int k, int d, int dtype,
                             cudaStream_t s);
// Per-head LayerNorm and rotary embedding of bf16 q and k rows (head_dim 64), by the QKV projection's epilogue, before the
// rows are rounded and stored.
struct QkEpilogue {
  const void *qn_w, *qn_b, *kn_w, *kn_b;   // [64] bf16, or all null
  const float2* rope;                      // (cos, sin) per (axis position, pair) or null
  int n_text, frames, grid_h, grid_w;
  float eps, q_scale;
};
// The same for fp32 rows, as a pass of its own over fresh q (compact) and k (in the cache) rows.
struct QkPrepArgs {
  void* q;                 // [B, n_sel, D]
  void* k;                 // [B, N, D], rows idx[i] (or i when idx is null)
  const int* idx;
  const void *qn_w, *qn_b, *kn_w, *kn_b;   // [head_dim], or all null
  const float2* rope;      // (cos, sin) per (axis position, pair) or null
  int B, N, n_sel, D, n_heads, head_dim;
  int n_text, frames, grid_h, grid_w;
  int p_t, p_h, p_w;       // rotary pairs per axis
  float eps;
};
int launch_qk_prep(const QkPrepArgs& a, cudaStream_t s);
// Of K and V [B, N, D] the first n_text rows and the listed ones, compact: [B, n_text + n_sel, D] (what a literal Eq. 3 attends
// to).  The list was complete before the kernel in front on the stream was placed.
int launch_attend_rows(const void* k, const void* v, const int* idx, void* k_out, void* v_out, int B, int N, int n_text,
                       int n_sel, int D, int dtype, cudaStream_t s);
int launch_gather_rows(const void* src, const int* idx, void* dst, int B, int N, int n_sel, int D,
                       int dtype, cudaStream_t s);
int launch_scatter_rows(const void* src, const int* idx, void* dst, int B, int N, int n_sel, int D,
                        int dtype, cudaStream_t s);
// mod[b, j] = b_mod[j] + sum_e silu(temb[b,e]) * w_mod[j,e]   (fp32 output)
// The adaLN vectors of several blocks in one launch (they depend on the timestep embedding only).
constexpr int kMaxModBatch = 64;
struct ModBatch {
  int n;
  const void* w_mod[kMaxModBatch];
  const void* b_mod[kMaxModBatch];
  float* mod[kMaxModBatch];
};
// (beside: the kernel in front on the stream is this step's launch_select)
int launch_modulation_batch(const void* temb, const ModBatch& batch, int B, int n_out, int E, bool beside, int dtype,
                            cudaStream_t s);
int launch_modulation(const void* temb, const void* w_mod, const void* b_mod, float* mod, int B,
                      int n_out, int E, int dtype, cudaStream_t s);
// a[m,:] = LN(x[row(m),:] (+ add[row(m),:])) * (1 + scale[b,:]) + shift[b,:]
// settled: what was complete before the kernel in front on the stream was placed and need not be waited for: nothing, the
// vectors and the list, or the rows of x as well.
enum LnSettled { kLnNothingSettled, kLnModSettled, kLnRowsSettled };
int launch_gather_ln_modulate(const void* x, const void* add, const int* idx, const float* shift,
                              const float* scale, int mod_ld, void* a, int B, int N, int n_sel, int D,
                              float eps, int dtype, int settled, cudaStream_t s);

// x = (x + ga) + gf for all rows and the LayerNorm + modulate of the rows that the next
// block refreshes (pos: as SelectBatch::pos; null: all rows) into a [B, n_sel, D].  Rows as wide as residual_ln_serves.
// Placed early, it reads all but gf before it waits for the kernel in front, which then has to be the only one on the stream
// that may still be running, and the writer of gf alone.  early: that holds, and nothing else (an event of another stream)
// stands between the two launches.
bool residual_ln_serves(int D, int dtype);
int launch_residual_ln(void* x, const void* ga, const void* gf, const int* pos, int n_text, const float* shift,
                       const float* scale, int mod_ld, void* a, int B, int N, int n_sel, int D, float eps, int dtype,
                       bool early, cudaStream_t s);

// fp32 CUDA-core path (config 1 runs in fp32, where tensor cores would break parity)
int launch_simt_gemm(const float* a, const float* w, const float* bias, int M, int Nout, int K, const GemmOut& out,
                     cudaStream_t s);
// Which tile (64 or 32 square) over how many CTAs; tile 0: a problem of more rows than any tile serves.
struct SimtGemmPlan { int tile, split; };
SimtGemmPlan plan_simt_gemm(int M, int Nout, int K, int sms);
int launch_simt_attention(const float* q, const float* k, const float* v, float* o, int B, int n_q, int N, int heads,
                          int head_dim, cudaStream_t s);
constexpr int kSimtAttQ = 32, kSimtAttK = 64;                // queries of a group, keys of a tile
int plan_simt_attention(long long groups, int tiles, int head_dim, int sms);     // CTAs that share a group's keys

// bf16 tensor-core path (tcgen05 + TMEM + TMA)
int tc_init_driver_api();   // resolves cuTensorMapEncodeTiled once
int launch_tc_gemm(const void* a, const void* w, const void* bias, int M, int Nout, int K,
                   const GemmOut& out, const QkEpilogue* qk, int* d_status, cudaStream_t s);
// Columns of a tile and the CTAs that share its K (0: the kernel on CTA pairs).
struct TcGemmPlan { int bn, split; };
TcGemmPlan plan_tc_gemm(int M, int Nout, int K, bool qk, int sms);
// The tensor-core attention serves head_dim 64: a score s enters the softmax as 2^(s * kScoreScaleLog2).
constexpr float kScoreScaleLog2 = 0.125f * 1.4426950408889634f;   // 1/sqrt(64) * log2(e)
// Workspace of an attention launch that may cut query groups.
struct AttentionParts {
  float* rows;                          // tc_attention_part_bytes()
  unsigned long long* count;            // tc_attention_part_counters() of them, zero before the first launch
  unsigned launch;                      // another number, not 0, for every launch on this workspace
};
// q_prescaled: Q holds q * kScoreScaleLog2 (the softmax scale folded into the projection)
int launch_tc_attention(const void* q, const void* k, const void* v, void* o, int B, int n_q, int N,
                        int heads, bool q_prescaled, const AttentionParts& parts, int* d_status, int* cta_words,
                        cudaStream_t s);
bool tc_attention_may_cut(int B, int n_rows, int heads);     // with at most n_rows queries and keys
size_t tc_attention_part_bytes();
size_t tc_attention_part_counters();
// (for the self-test of the give-up path)
int launch_strand_attention_counters(const AttentionParts& parts, cudaStream_t s);
int launch_tc_attention_safe(const void* q, const void* k, const void* v, void* o, int B, int n_q, int N,
                             int heads, bool q_prescaled, int* d_status, cudaStream_t s);
long long tc_attention_grid(int B, int n_q, int heads);   // CTAs of one attention launch

// one thread block, no TMA, no TMEM: a bounded wait on a barrier nobody arms; raises *d_status and returns
int launch_wait_timeout_selftest(int* d_status, int budget_us, cudaStream_t s);

}  // namespace hero
