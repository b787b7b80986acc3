// Treatment of the fresh q and k rows between the QKV projection and attention, as in the base
// video DiT the method is applied to (Sec. 3 leaves the block's internals to the base model):
// an optional LayerNorm over every head's features with a learned gain and bias, then an optional
// 3-D rotary position embedding of the video rows.  q is the compact [B, n_sel, D] projection
// output; k is rewritten in place in the block's K cache at the rows of the index list, so the
// cache always holds keys in their final form (a row never changes position, so cached keys stay
// valid across steps).  HBM-bound: every element is read once and written once.  This is the fp32 form
// (any even head_dim <= 256): one warp owns one (row, head) slice, a lane the rotary pairs (2p, 2p+1)
// for p = lane, lane + 32, ...; in bf16 runs the projection's epilogue does it (emit_head in tc_gemm.cu).
#include "hero_internal.h"

namespace hero {
namespace {

constexpr int kMaxPairsPerLane = 4;  // head_dim <= 256

__device__ __forceinline__ float2 load_pair(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ void store_pair(float* p, float2 v) { *reinterpret_cast<float2*>(p) = v; }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__global__ void __launch_bounds__(256) qk_prep_kernel(QkPrepArgs a) {
  stream_order();
  const int lane = threadIdx.x & 31;
  const long long n_warps = ((long long)gridDim.x * blockDim.x) >> 5;
  const long long n_items = (long long)a.B * a.n_sel * a.n_heads * 2;
  const int pairs = a.head_dim >> 1;
  const float inv_hd = 1.0f / (float)a.head_dim;
  for (long long item = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; item < n_items; item += n_warps) {
    const int which = (int)(item & 1);                // 0: q, 1: k
    long long rest = item >> 1;
    const int head = (int)(rest % a.n_heads); rest /= a.n_heads;
    const int i = (int)(rest % a.n_sel);
    const int b = (int)(rest / a.n_sel);
    const int row = a.idx ? a.idx[i] : i;
    float* p = which ? static_cast<float*>(a.k) + ((long long)b * a.N + row) * a.D + head * a.head_dim
                 : static_cast<float*>(a.q) + ((long long)b * a.n_sel + i) * a.D + head * a.head_dim;
    float2 v[kMaxPairsPerLane];
#pragma unroll
    for (int j = 0; j < kMaxPairsPerLane; ++j) {
      const int pr = lane + 32 * j;
      v[j] = pr < pairs ? load_pair(p + 2 * pr) : make_float2(0.f, 0.f);
    }
    if (a.qn_w) {
      const float* gw = static_cast<const float*>(which ? a.kn_w : a.qn_w);
      const float* gb = static_cast<const float*>(which ? a.kn_b : a.qn_b);
      float s = 0.f;
#pragma unroll
      for (int j = 0; j < kMaxPairsPerLane; ++j) s += v[j].x + v[j].y;   // absent pairs hold zeros
      const float mu = warp_sum(s) * inv_hd;
      float q2 = 0.f;
#pragma unroll
      for (int j = 0; j < kMaxPairsPerLane; ++j)
        if (lane + 32 * j < pairs) q2 += (v[j].x - mu) * (v[j].x - mu) + (v[j].y - mu) * (v[j].y - mu);
      const float rstd = rsqrtf(warp_sum(q2) * inv_hd + a.eps);
#pragma unroll
      for (int j = 0; j < kMaxPairsPerLane; ++j) {
        const int pr = lane + 32 * j;
        if (pr < pairs) {
          const float2 w = load_pair(gw + 2 * pr), bb = load_pair(gb + 2 * pr);
          v[j].x = (v[j].x - mu) * rstd * w.x + bb.x;
          v[j].y = (v[j].y - mu) * rstd * w.y + bb.y;
        }
      }
    }
    if (a.rope && row >= a.n_text) {
      const int t = row - a.n_text;
      const int pos_t = t / (a.grid_h * a.grid_w), pos_h = (t / a.grid_w) % a.grid_h, pos_w = t % a.grid_w;
#pragma unroll
      for (int j = 0; j < kMaxPairsPerLane; ++j) {
        const int pr = lane + 32 * j;
        if (pr < pairs) {
          int at;                                     // entry of the (cos, sin) table
          if (pr < a.p_t) at = pos_t * a.p_t + pr;
          else if (pr < a.p_t + a.p_h) at = a.frames * a.p_t + pos_h * a.p_h + (pr - a.p_t);
          else at = a.frames * a.p_t + a.grid_h * a.p_h + pos_w * a.p_w + (pr - a.p_t - a.p_h);
          const float2 cs = a.rope[at];
          const float x = v[j].x, y = v[j].y;
          v[j].x = x * cs.x - y * cs.y;
          v[j].y = x * cs.y + y * cs.x;
        }
      }
    }
#pragma unroll
    for (int j = 0; j < kMaxPairsPerLane; ++j) {
      const int pr = lane + 32 * j;
      if (pr < pairs) store_pair(p + 2 * pr, v[j]);
    }
  }
}

}  // namespace

int launch_qk_prep(const QkPrepArgs& a, cudaStream_t s) {
  if (a.head_dim % 2 != 0 || a.head_dim > 64 * kMaxPairsPerLane) return HERO_ERR_ARG;
  const long long n_items = (long long)a.B * a.n_sel * a.n_heads * 2;
  if (n_items <= 0) return HERO_OK;
  const long long want = (n_items + 7) / 8, most = num_sms() * 8ll;      // 8 warps per block
  return launch_streaming(qk_prep_kernel, want < most ? want : most, 256, s, a);
}

}  // namespace hero
