// HBM-bound kernels of the cached step: linear extrapolation (Eq. 5), residual adds
// (Algorithm 1), row gather / scatter (Eq. 3's merge), the adaLN modulation vectors and the
// fused gather + LayerNorm + modulate prologue of Eq. 2.  All of them move each byte once
// with 128-bit accesses; grids are sized in multiples of the SM count.
#include "hero_internal.h"

namespace hero {

// SM count of the calling thread's current device (looked up once per device).
int num_sms() {
  static PerDeviceOnce once;
  static int count[kMaxDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 148;
  per_device_once(once, [](int d) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, d) != cudaSuccess || n <= 0) n = 148;
    count[d] = n;
    return HERO_OK;
  });
  return count[dev] > 0 ? count[dev] : 148;
}

namespace {

// ------------------------------------------------------------------ 128-bit packets
template <typename T>
struct Vec;  // 16 bytes of T
template <>
struct Vec<float> {
  static constexpr int N = 4;
  float4 raw;
  __device__ __forceinline__ void unpack(float (&f)[4]) const {
    f[0] = raw.x; f[1] = raw.y; f[2] = raw.z; f[3] = raw.w;
  }
  __device__ __forceinline__ void pack(const float (&f)[4]) { raw = make_float4(f[0], f[1], f[2], f[3]); }
};
template <>
struct Vec<__nv_bfloat16> {
  static constexpr int N = 8;
  uint4 raw;
  __device__ __forceinline__ void unpack(float (&f)[8]) const {
    const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      f[2 * i] = __uint_as_float(w[i] << 16);
      f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
    }
  }
  __device__ __forceinline__ void pack(const float (&f)[8]) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const __nv_bfloat162 p = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
      w[i] = *reinterpret_cast<const uint32_t*>(&p);
    }
    raw = make_uint4(w[0], w[1], w[2], w[3]);
  }
};

template <typename T>
__device__ __forceinline__ float to_f(T v);
template <>
__device__ __forceinline__ float to_f<float>(float v) { return v; }
template <>
__device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T>
__device__ __forceinline__ T from_f(float v);
template <>
__device__ __forceinline__ float from_f<float>(float v) { return v; }
template <>
__device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// streaming loads/stores: these tensors are touched once per step, keep them out of L1
template <typename V>
__device__ __forceinline__ V ld_stream(const V* p) {
  V v;
  v.raw = __ldcs(&p->raw);
  return v;
}
template <typename V>
__device__ __forceinline__ void st_stream(V* p, const V& v) { __stcs(&p->raw, v.raw); }

constexpr int kStreamThreads = 256;
constexpr int kStreamUnroll = 2;

static inline int stream_grid(long long n_vec) {
  const long long per_block = (long long)kStreamThreads * kStreamUnroll;
  long long blocks = (n_vec + per_block - 1) / per_block;
  const long long cap = (long long)num_sms() * 16;   // grid-stride beyond 16 CTAs per SM
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  return (int)blocks;
}

// ------------------------------------------------------------------ Eq. 5
// e = g_last + (g_last - g_prev) * (k/d), evaluated as one fp32 FMA per element.
template <typename T>
__global__ void __launch_bounds__(kStreamThreads) extrapolate_kernel(const T* __restrict__ g_prev,
                                                                     const T* __restrict__ g_last,
                                                                     T* __restrict__ out, long long n, float c) {
  stream_order();
  using V = Vec<T>;
  const long long n_vec = n / V::N;
  const V* p = reinterpret_cast<const V*>(g_prev);
  const V* l = reinterpret_cast<const V*>(g_last);
  V* o = reinterpret_cast<V*>(out);
  const long long stride = (long long)gridDim.x * kStreamThreads * kStreamUnroll;
  for (long long i0 = (long long)blockIdx.x * kStreamThreads * kStreamUnroll + threadIdx.x; i0 < n_vec; i0 += stride) {
    V vp[kStreamUnroll], vl[kStreamUnroll];
#pragma unroll
    for (int u = 0; u < kStreamUnroll; ++u) {
      const long long i = i0 + (long long)u * kStreamThreads;
      if (i < n_vec) { vp[u] = ld_stream(p + i); vl[u] = ld_stream(l + i); }
    }
#pragma unroll
    for (int u = 0; u < kStreamUnroll; ++u) {
      const long long i = i0 + (long long)u * kStreamThreads;
      if (i < n_vec) {
        float fp[V::N], fl[V::N];
        vp[u].unpack(fp); vl[u].unpack(fl);
#pragma unroll
        for (int j = 0; j < V::N; ++j) fl[j] = fmaf(fl[j] - fp[j], c, fl[j]);
        V r; r.pack(fl);
        st_stream(o + i, r);
      }
    }
  }
  // ragged tail (fewer than one packet)
  const long long tail0 = n_vec * V::N;
  if (blockIdx.x == 0 && threadIdx.x < n - tail0) {
    const long long i = tail0 + threadIdx.x;
    const float a = to_f(g_last[i]), b = to_f(g_prev[i]);
    out[i] = from_f<T>(fmaf(a - b, c, a));
  }
}

// x += e(attn) ; x += e(ffn)  (both branches of a deep block in one pass: 5 reads, 1 write)
template <typename T>
__global__ void __launch_bounds__(kStreamThreads)
extrapolate_residual_kernel(T* __restrict__ x, const T* __restrict__ ga_prev, const T* __restrict__ ga_last,
                            const T* __restrict__ gf_prev, const T* __restrict__ gf_last, long long n, float c) {
  stream_order();
  using V = Vec<T>;
  const long long n_vec = n / V::N;
  V* xv = reinterpret_cast<V*>(x);
  const V* ap = reinterpret_cast<const V*>(ga_prev);
  const V* al = reinterpret_cast<const V*>(ga_last);
  const V* fp_ = reinterpret_cast<const V*>(gf_prev);
  const V* fl_ = reinterpret_cast<const V*>(gf_last);
  const long long stride = (long long)gridDim.x * kStreamThreads;
  for (long long i = (long long)blockIdx.x * kStreamThreads + threadIdx.x; i < n_vec; i += stride) {
    const V vx = ld_stream(xv + i), v1 = ld_stream(ap + i), v2 = ld_stream(al + i), v3 = ld_stream(fp_ + i),
            v4 = ld_stream(fl_ + i);
    float fx[V::N], f1[V::N], f2[V::N], f3[V::N], f4[V::N];
    vx.unpack(fx); v1.unpack(f1); v2.unpack(f2); v3.unpack(f3); v4.unpack(f4);
#pragma unroll
    for (int j = 0; j < V::N; ++j) {
      const float ea = fmaf(f2[j] - f1[j], c, f2[j]);
      const float ef = fmaf(f4[j] - f3[j], c, f4[j]);
      fx[j] = (fx[j] + ea) + ef;
    }
    V r; r.pack(fx);
    st_stream(xv + i, r);
  }
  const long long tail0 = n_vec * V::N;
  if (blockIdx.x == 0 && threadIdx.x < n - tail0) {
    const long long i = tail0 + threadIdx.x;
    const float a1 = to_f(ga_prev[i]), a2 = to_f(ga_last[i]), b1 = to_f(gf_prev[i]), b2 = to_f(gf_last[i]);
    x[i] = from_f<T>((to_f(x[i]) + fmaf(a2 - a1, c, a2)) + fmaf(b2 - b1, c, b2));
  }
}

// Eq. 5 for a run of consecutive extrapolated blocks in ONE pass over x: a deep block touches nothing but
// the residual stream, so x can stay in registers while the blocks' four history tensors stream by.  Per
// element and block that is 8 bytes read instead of 12 moved (x is read and written once per launch, not
// once per block), and the sum is rounded to the storage type once.  The adds keep the order of the blocks.  The branches
// of the last refreshed block in front can come along (n_plain): its residual pass over x is then saved altogether.
// E entries of the group are in flight per thread: four keep a large pass at the memory's rate (25 GB: 6.6 TB/s); where the
// elements give every SM less than two blocks the pass is a chain of loads, and sixteen make it shorter (56 entries of
// 157k elements: 36 -> 14 us).
template <typename T, int E>
__global__ void __launch_bounds__(kStreamThreads) extrapolate_group_kernel(T* __restrict__ x, const DeepGroup grp,
                                                                           long long first, long long n, float c) {
  stream_order();
  using V = Vec<T>;
  const long long n_vec = n / V::N;
  V* xv = reinterpret_cast<V*>(x + first);
  const long long stride = (long long)gridDim.x * kStreamThreads;
  for (long long i = (long long)blockIdx.x * kStreamThreads + threadIdx.x; i < n_vec; i += stride) {
    float fx[V::N];
    const V vx = ld_stream(xv + i);
    if (grp.n_plain) {                     // (both branches of one block)
      float fa[V::N], ff[V::N];
      const V va = ld_stream(reinterpret_cast<const V*>(static_cast<const T*>(grp.last[0]) + first) + i);
      const V vf = ld_stream(reinterpret_cast<const V*>(static_cast<const T*>(grp.last[1]) + first) + i);
      vx.unpack(fx); va.unpack(fa); vf.unpack(ff);
#pragma unroll
      for (int j = 0; j < V::N; ++j) fx[j] = (fx[j] + fa[j]) + ff[j];
    } else {
      vx.unpack(fx);
    }
    for (int e0 = grp.n_plain; e0 < grp.n_entries; e0 += E) {
      V vp[E], vl[E];
#pragma unroll
      for (int u = 0; u < E; ++u)
        if (e0 + u < grp.n_entries) {
          vp[u] = ld_stream(reinterpret_cast<const V*>(static_cast<const T*>(grp.prev[e0 + u]) + first) + i);
          vl[u] = ld_stream(reinterpret_cast<const V*>(static_cast<const T*>(grp.last[e0 + u]) + first) + i);
        }
#pragma unroll
      for (int u = 0; u < E; ++u)
        if (e0 + u < grp.n_entries) {
          float fp_[V::N], fl_[V::N];
          vp[u].unpack(fp_); vl[u].unpack(fl_);
#pragma unroll
          for (int j = 0; j < V::N; ++j) fx[j] += fmaf(fl_[j] - fp_[j], c, fl_[j]);
        }
    }
    V r; r.pack(fx);
    st_stream(xv + i, r);
  }
  const long long tail0 = n_vec * V::N;
  if (blockIdx.x == 0 && threadIdx.x < n - tail0) {
    const long long i = first + tail0 + threadIdx.x;
    float v = to_f(x[i]);
    for (int e = 0; e < grp.n_plain; ++e) v += to_f(static_cast<const T*>(grp.last[e])[i]);
    for (int e = grp.n_plain; e < grp.n_entries; ++e) {
      const float a = to_f(static_cast<const T*>(grp.prev[e])[i]), b = to_f(static_cast<const T*>(grp.last[e])[i]);
      v += fmaf(b - a, c, b);
    }
    x[i] = from_f<T>(v);
  }
}

// x = (x + ga) + gf  (both residual adds of a refresh block in one pass)
template <typename T>
__global__ void __launch_bounds__(kStreamThreads) residual2_kernel(T* __restrict__ x, const T* __restrict__ ga,
                                                                   const T* __restrict__ gf, long long n) {
  stream_order();
  using V = Vec<T>;
  const long long n_vec = n / V::N;
  V* xv = reinterpret_cast<V*>(x);
  const V* a = reinterpret_cast<const V*>(ga);
  const V* f = reinterpret_cast<const V*>(gf);
  const long long stride = (long long)gridDim.x * kStreamThreads * kStreamUnroll;
  for (long long i0 = (long long)blockIdx.x * kStreamThreads * kStreamUnroll + threadIdx.x; i0 < n_vec; i0 += stride) {
    V vx[kStreamUnroll], va[kStreamUnroll], vf[kStreamUnroll];
#pragma unroll
    for (int u = 0; u < kStreamUnroll; ++u) {
      const long long i = i0 + (long long)u * kStreamThreads;
      if (i < n_vec) { vx[u] = ld_stream(xv + i); va[u] = ld_stream(a + i); vf[u] = ld_stream(f + i); }
    }
#pragma unroll
    for (int u = 0; u < kStreamUnroll; ++u) {
      const long long i = i0 + (long long)u * kStreamThreads;
      if (i < n_vec) {
        float fx[V::N], fa[V::N], ff[V::N];
        vx[u].unpack(fx); va[u].unpack(fa); vf[u].unpack(ff);
#pragma unroll
        for (int j = 0; j < V::N; ++j) fx[j] = (fx[j] + fa[j]) + ff[j];
        V r; r.pack(fx);
        st_stream(xv + i, r);
      }
    }
  }
  const long long tail0 = n_vec * V::N;
  if (blockIdx.x == 0 && threadIdx.x < n - tail0) {
    const long long i = tail0 + threadIdx.x;
    x[i] = from_f<T>((to_f(x[i]) + to_f(ga[i])) + to_f(gf[i]));
  }
}

// ------------------------------------------------------------------ deep-stack collapse
// fp32 side-band packets matching one 16-byte packet of T
template <typename T>
struct AccVec;
template <>
struct AccVec<float> {
  __device__ static void load(const float* p, long long i, float (&f)[4]) {
    const float4 v = __ldcs(reinterpret_cast<const float4*>(p) + i);
    f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w;
  }
  __device__ static void store(float* p, long long i, const float (&f)[4]) {
    __stcs(reinterpret_cast<float4*>(p) + i, make_float4(f[0], f[1], f[2], f[3]));
  }
};
template <>
struct AccVec<__nv_bfloat16> {
  __device__ static void load(const float* p, long long i, float (&f)[8]) {
    const float4 a = __ldcs(reinterpret_cast<const float4*>(p) + 2 * i), b = __ldcs(reinterpret_cast<const float4*>(p) + 2 * i + 1);
    f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w; f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
  }
  __device__ static void store(float* p, long long i, const float (&f)[8]) {
    __stcs(reinterpret_cast<float4*>(p) + 2 * i, make_float4(f[0], f[1], f[2], f[3]));
    __stcs(reinterpret_cast<float4*>(p) + 2 * i + 1, make_float4(f[4], f[5], f[6], f[7]));
  }
};

// Full step, deep block, collapse mode: x = (x + ga) + gf and acc += ga + gf (fp32 running sum of the
// deep stack's branch outputs, the quantity Eq. 5 is applied to on cached steps).
template <typename T>
__global__ void __launch_bounds__(kStreamThreads) residual2_acc_kernel(T* __restrict__ x, const T* __restrict__ ga,
                                                                       const T* __restrict__ gf,
                                                                       float* __restrict__ acc, long long n) {
  stream_order();
  using V = Vec<T>;
  const long long n_vec = n / V::N;
  V* xv = reinterpret_cast<V*>(x);
  const V* a = reinterpret_cast<const V*>(ga);
  const V* f = reinterpret_cast<const V*>(gf);
  const long long stride = (long long)gridDim.x * kStreamThreads;
  for (long long i = (long long)blockIdx.x * kStreamThreads + threadIdx.x; i < n_vec; i += stride) {
    const V vx = ld_stream(xv + i), va = ld_stream(a + i), vf = ld_stream(f + i);
    float fx[V::N], fa[V::N], ff[V::N], fs[V::N];
    vx.unpack(fx); va.unpack(fa); vf.unpack(ff);
    AccVec<T>::load(acc, i, fs);
#pragma unroll
    for (int j = 0; j < V::N; ++j) { fx[j] = (fx[j] + fa[j]) + ff[j]; fs[j] += fa[j] + ff[j]; }
    V r; r.pack(fx);
    st_stream(xv + i, r);
    AccVec<T>::store(acc, i, fs);
  }
  const long long tail0 = n_vec * V::N;
  if (blockIdx.x == 0 && threadIdx.x < n - tail0) {
    const long long i = tail0 + threadIdx.x;
    const float va = to_f(ga[i]), vf = to_f(gf[i]);
    x[i] = from_f<T>((to_f(x[i]) + va) + vf);
    acc[i] += va + vf;
  }
}

// Cached step, whole deep stack in one pass: x += s_last + (s_last - s_prev) * c  (Eq. 5 on the sums).
template <typename T>
__global__ void __launch_bounds__(kStreamThreads) extrapolate_stack_kernel(T* __restrict__ x,
                                                                           const float* __restrict__ s_prev,
                                                                           const float* __restrict__ s_last,
                                                                           long long n, float c) {
  stream_order();
  using V = Vec<T>;
  const long long n_vec = n / V::N;
  V* xv = reinterpret_cast<V*>(x);
  const long long stride = (long long)gridDim.x * kStreamThreads;
  for (long long i = (long long)blockIdx.x * kStreamThreads + threadIdx.x; i < n_vec; i += stride) {
    const V vx = ld_stream(xv + i);
    float fx[V::N], fp[V::N], fl[V::N];
    vx.unpack(fx);
    AccVec<T>::load(s_prev, i, fp);
    AccVec<T>::load(s_last, i, fl);
#pragma unroll
    for (int j = 0; j < V::N; ++j) fx[j] += fmaf(fl[j] - fp[j], c, fl[j]);
    V r; r.pack(fx);
    st_stream(xv + i, r);
  }
  const long long tail0 = n_vec * V::N;
  if (blockIdx.x == 0 && threadIdx.x < n - tail0) {
    const long long i = tail0 + threadIdx.x;
    x[i] = from_f<T>(to_f(x[i]) + fmaf(s_last[i] - s_prev[i], c, s_last[i]));
  }
}

// ------------------------------------------------------------------ gather / scatter of rows
// One warp moves one row in 16-byte packets, four packets per lane in flight at a time (2 KB per
// warp, 16 KB per CTA); GATHER reads row idx[i] and writes row i, SCATTER the reverse.  Rows not
// listed are never touched.
constexpr int kMoveUnroll = 4;
template <bool GATHER>
__global__ void __launch_bounds__(256) move_rows_kernel(const uint4* __restrict__ src, const int* __restrict__ idx,
                                                        uint4* __restrict__ dst, int B, int N, int n_sel,
                                                        int row_vec) {
  stream_order();
  const long long warp_global = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long n_warps = ((long long)gridDim.x * blockDim.x) >> 5;
  const int lane = threadIdx.x & 31;
  const long long total = (long long)B * n_sel;
  for (long long m = warp_global; m < total; m += n_warps) {
    const int b = (int)(m / n_sel), i = (int)(m - (long long)b * n_sel);
    const long long far = ((long long)b * N + __ldg(idx + i)) * row_vec, near = m * row_vec;
    const uint4* s = src + (GATHER ? far : near);
    uint4* d = dst + (GATHER ? near : far);
    for (int c0 = lane; c0 < row_vec; c0 += 32 * kMoveUnroll) {
      uint4 v[kMoveUnroll];
#pragma unroll
      for (int u = 0; u < kMoveUnroll; ++u)
        if (c0 + 32 * u < row_vec) v[u] = __ldcs(s + c0 + 32 * u);
#pragma unroll
      for (int u = 0; u < kMoveUnroll; ++u)
        if (c0 + 32 * u < row_vec) __stcs(d + c0 + 32 * u, v[u]);
    }
  }
}

// The rows of K and V that a literal Eq. 3 attends to, compact: the text rows, then the listed ones.  As move_rows_kernel, both
// tensors in one launch; where a row lies is found before the wait for the projection in front.  Against a launch that wrote the
// list out and a gather for each tensor: cached step of 4 blocks of 371 x 768 212 -> 200 us, of 8 blocks of 1394 x 1024 831 ->
// 814, of 6 blocks of 5940 x 3072 9.56 -> 9.54 ms.
__global__ void __launch_bounds__(256) attend_rows_kernel(const uint4* __restrict__ k, const uint4* __restrict__ v,
                                                          const int* __restrict__ idx, uint4* __restrict__ k_out,
                                                          uint4* __restrict__ v_out, int B, int N, int n_text, int n_att,
                                                          int row_vec) {
  const long long n_warps = ((long long)gridDim.x * blockDim.x) >> 5, rows = (long long)B * n_att;
  const int lane = threadIdx.x & 31;
  long long m = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5, far = 0;
  auto find = [&]() {
    const long long in_tensor = m < rows ? m : m - rows;
    const int b = (int)(in_tensor / n_att), i = (int)(in_tensor - (long long)b * n_att);
    far = ((long long)b * N + (i < n_text ? i : __ldg(idx + i - n_text))) * row_vec;
  };
  if (m < 2 * rows) find();
  stream_order();
  while (m < 2 * rows) {
    const uint4* s = (m < rows ? k : v) + far;
    uint4* d = m < rows ? k_out + m * row_vec : v_out + (m - rows) * row_vec;
    for (int c0 = lane; c0 < row_vec; c0 += 32 * kMoveUnroll) {
      uint4 r[kMoveUnroll];
#pragma unroll
      for (int u = 0; u < kMoveUnroll; ++u)
        if (c0 + 32 * u < row_vec) r[u] = __ldcs(s + c0 + 32 * u);
#pragma unroll
      for (int u = 0; u < kMoveUnroll; ++u)
        if (c0 + 32 * u < row_vec) d[c0 + 32 * u] = r[u];
    }
    m += n_warps;
    if (m < 2 * rows) find();
  }
}

// ------------------------------------------------------------------ adaLN modulation vectors
// mod[b, j] = b_mod[j] + sum_e silu(temb[b, e]) * w_mod[j, e].  A warp owns kModRows consecutive output columns
// j at a time: their weight rows are read once with 16-byte loads, all kModRows loads of a step in flight
// together (a row of 512 weights is two loads per lane: one row at a time leaves the warp waiting on DRAM
// latency for most of its life), and reused for every batch item.
constexpr int kModMaxB = 8, kModRows = 4;

// silu(temb) into shared memory, laid out [B][V::N][E / V::N]: element e of a row sits at
// (e % V::N) * (E / V::N) + e / V::N, so that the lanes of a warp, which hold consecutive 16-byte packets of a
// weight row, read consecutive words
template <typename T>
__device__ __forceinline__ void modulation_stage_activations(const T* __restrict__ temb, float* s_act, int B, int E) {
  for (int i = threadIdx.x; i < B * E; i += blockDim.x) {
    const float t = to_f(temb[i]);
    const int b = i / E, e = i - b * E;
    s_act[b * E + (e % Vec<T>::N) * (E / Vec<T>::N) + e / Vec<T>::N] = t / (1.0f + expf(-t));
  }
  __syncthreads();
}

template <typename T, int MAXB>
__device__ __forceinline__ void modulation_rows(const float* s_act, const T* __restrict__ w_mod,
                                                const T* __restrict__ b_mod, float* __restrict__ mod, int B,
                                                int n_out, int E) {
  using V = Vec<T>;
  const int lane = threadIdx.x & 31;
  const int warps = gridDim.x * (blockDim.x >> 5), warp = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int packets = E / V::N;
  for (int j0 = warp * kModRows; j0 < n_out; j0 += warps * kModRows) {
    float acc[kModRows][MAXB];
#pragma unroll
    for (int r = 0; r < kModRows; ++r)
#pragma unroll
      for (int b = 0; b < MAXB; ++b) acc[r][b] = 0.f;
#pragma unroll(MAXB <= 2 ? 2 : 1)
    for (int c = lane; c < packets; c += 32) {
      V wv[kModRows];
#pragma unroll
      for (int r = 0; r < kModRows; ++r) {
        const int j = j0 + r < n_out ? j0 + r : n_out - 1;           // a row past the end repeats the last one
        wv[r].raw = __ldg(&reinterpret_cast<const V*>(w_mod + (long long)j * E)[c].raw);
      }
      float wf[kModRows][V::N];
#pragma unroll
      for (int r = 0; r < kModRows; ++r) wv[r].unpack(wf[r]);
#pragma unroll
      for (int b = 0; b < MAXB; ++b) {
        if (b < B) {
#pragma unroll
          for (int q = 0; q < V::N; ++q) {
            const float a = s_act[b * E + q * packets + c];
#pragma unroll
            for (int r = 0; r < kModRows; ++r) acc[r][b] = fmaf(a, wf[r][q], acc[r][b]);
          }
        }
      }
    }
    // Sums over the warp, all of them together: as long as a lane holds more than one value, the two halves of a pair of
    // lanes share them out (a quarter of the shuffles of one butterfly per value).
    constexpr int kSums = kModRows * MAXB;
    float v[kSums];
#pragma unroll
    for (int r = 0; r < kModRows; ++r)
#pragma unroll
      for (int b = 0; b < MAXB; ++b) v[r * MAXB + b] = acc[r][b];
    int which = 0;                                     // which value ends up in this lane
    int n = kSums;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      if (n > 1) {
        n >>= 1;
        const bool upper = lane & o;
#pragma unroll
        for (int i = 0; i < kSums / 2; ++i) {
          if (i < n) {
            const float give = upper ? v[i] : v[i + n], keep = upper ? v[i + n] : v[i];
            v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, o);
          }
        }
        which += upper ? n : 0;
      } else {
        v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], o);
      }
    }
    static_assert(kSums <= 32, "a lane per value");
    const int r = which / MAXB, b = which - r * MAXB;
    if ((lane & (32 / kSums - 1)) == 0 && b < B && j0 + r < n_out)
      mod[(long long)b * n_out + j0 + r] = v[0] + to_f(b_mod[j0 + r]);
  }
}

template <typename T, int MAXB>
__global__ void __launch_bounds__(256, 2) modulation_kernel(const T* __restrict__ temb, const T* __restrict__ w_mod,
                                                         const T* __restrict__ b_mod, float* __restrict__ mod,
                                                         int B, int n_out, int E) {
  stream_order();
  extern __shared__ float s_act[];
  modulation_stage_activations<T>(temb, s_act, B, E);
  modulation_rows<T, MAXB>(s_act, w_mod, b_mod, mod, B, n_out, E);
}

// The same for several blocks at once: blockIdx.y picks the block's weights and output.  `beside`: the kernel in front is
// the token selection of the same step, which has nothing to do with this one (and which has itself waited for everything
// that came before): the two run side by side, and the wait that makes this kernel's end stand for both comes last.
template <typename T, int MAXB>
__global__ void __launch_bounds__(256, 2) modulation_batch_kernel(const T* __restrict__ temb, const ModBatch batch, int B,
                                                               int n_out, int E, bool beside) {
  if (!beside) stream_order();
  extern __shared__ float s_act[];
  modulation_stage_activations<T>(temb, s_act, B, E);
  modulation_rows<T, MAXB>(s_act, static_cast<const T*>(batch.w_mod[blockIdx.y]), static_cast<const T*>(batch.b_mod[blockIdx.y]),
                     batch.mod[blockIdx.y], B, n_out, E);
  if (beside) stream_order();
}

// ------------------------------------------------------------------ gather + LayerNorm + modulate (Eq. 2 prologue)
// One CTA per refreshed row: the row (plus, for the FFN branch, the not-yet-added attention
// output of the same row) is read once into shared memory as fp32, mean and biased variance
// are reduced in two passes over that copy, and the modulated row is written compactly.
constexpr int kLnThreads = 256;
__device__ __forceinline__ float block_sum(float v, float* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  float t = (lane < kLnThreads / 32) ? red[lane] : 0.f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
  return t;
}

template <typename T>
__global__ void __launch_bounds__(kLnThreads)
gather_ln_modulate_kernel(const T* __restrict__ x, const T* __restrict__ add, const int* __restrict__ idx,
                          const float* __restrict__ shift, const float* __restrict__ scale, int mod_ld,
                          T* __restrict__ a, int N, int n_sel, int D, float eps) {
  stream_order();
  extern __shared__ float s_row[];   // [D]
  __shared__ float red[kLnThreads / 32];
  using V = Vec<T>;
  const int m = blockIdx.x;
  const int b = m / n_sel, i = m - b * n_sel;
  const long long row = (long long)b * N + (idx ? idx[i] : i);
  const V* xr = reinterpret_cast<const V*>(x + row * D);
  const V* ar = add ? reinterpret_cast<const V*>(add + row * D) : nullptr;
  const int n_vec = D / V::N;
  float sum = 0.f;
  for (int c = threadIdx.x; c < n_vec; c += kLnThreads) {
    float f[V::N];
    V v; v.raw = __ldg(&xr[c].raw);
    v.unpack(f);
    if (ar) {
      float g[V::N];
      V w; w.raw = __ldg(&ar[c].raw);
      w.unpack(g);
#pragma unroll
      for (int q = 0; q < V::N; ++q) f[q] += g[q];
    }
#pragma unroll
    for (int q = 0; q < V::N; ++q) { s_row[c * V::N + q] = f[q]; sum += f[q]; }
  }
  const float mean = block_sum(sum, red) / (float)D;
  float sq = 0.f;
  for (int c = threadIdx.x; c < D; c += kLnThreads) { const float d = s_row[c] - mean; sq = fmaf(d, d, sq); }
  const float var = block_sum(sq, red) / (float)D;
  const float rstd = 1.0f / sqrtf(var + eps);
  const float* sh = shift + (long long)b * mod_ld;
  const float* sc = scale + (long long)b * mod_ld;
  V* out = reinterpret_cast<V*>(a + (long long)m * D);
  for (int c = threadIdx.x; c < n_vec; c += kLnThreads) {
    float f[V::N];
#pragma unroll
    for (int q = 0; q < V::N; ++q) {
      const int col = c * V::N + q;
      f[q] = fmaf((s_row[col] - mean) * rstd, 1.0f + sc[col], sh[col]);
    }
    V r; r.pack(f);
    out[c] = r;
  }
}

// Rows of up to 32 * VPL packets of 16 bytes: one WARP per refreshed row, the row held in registers (VPL packets per
// lane, the last of them predicated), statistics by warp shuffles alone - no block barrier per row, 8 independent rows
// in flight per CTA.  Each CTA serves ONE batch item.
// The CTAs are persistent and first put their item's (1 + scale) and shift vectors into shared memory in fp32 (24 KB at
// D = 3072, once per CTA), so a row costs its own 6 KB in and 6 KB out of HBM plus shared-memory reads - not 24 KB of
// L1/L2 traffic for the vectors again (reading them straight into registers was slower even with one row per warp: 4.6
// against 4.1 us for 1394 rows of 1024).  Layout: planes of float4, [quarter q of a packet's (1 + scale), of its
// shift][packet], so that the lanes of a warp read consecutive words.
// Measured (bf16), against one CTA per row through shared memory: 5254 rows of 1152 26.0 -> 8.0 us, 371 of 768
// 3.8 -> 3.4, 614 of 256 3.2 -> 2.8; 3510 rows of 3072 12.8 us (3.4 TB/s, mostly ramp), 35552 rows 94 us (4.6 TB/s).
//
// An instantiation serves every row width up to its own that the next smaller one does not: the chunks beyond that
// one's are predicated.
__host__ __device__ constexpr int ln_full_chunks(int vpl) {
  return vpl <= 6 ? vpl - 1 : (vpl == 8 ? 6 : (vpl == 10 ? 8 : (vpl == 12 ? 10 : 12)));
}
__host__ __device__ constexpr int ln_ctas_per_sm(int vpl, bool one) {      // what the registers of a row allow
  return vpl <= 2 && !one ? 6 : (vpl <= 4 ? 4 : (vpl <= 6 ? 3 : (vpl <= 12 ? 2 : 1)));
}
// One batch item's (1 + scale) and shift into shared memory: [2 * Q][packets] float4.
template <typename T>
__device__ __forceinline__ void ln_stage_modulation(float4* s_mod, const float* __restrict__ scale, const float* __restrict__ shift,
                                                    int packets) {
  constexpr int Q = Vec<T>::N / 4;                  // float4s of modulation per packet and vector
  const float4* sc = reinterpret_cast<const float4*>(scale);
  const float4* sh = reinterpret_cast<const float4*>(shift);
  for (int i = threadIdx.x; i < Q * packets; i += 256) {         // float4 i covers columns [4i, 4i + 4)
    const float4 s4 = __ldg(sc + i), h4 = __ldg(sh + i);
    s_mod[(i % Q) * packets + i / Q] = make_float4(1.0f + s4.x, 1.0f + s4.y, 1.0f + s4.z, 1.0f + s4.w);
    s_mod[(Q + i % Q) * packets + i / Q] = h4;
  }
  __syncthreads();
}
// Statistics of a row held by a warp (absent packets are zeros), normalised, modulated and written to `out`.
template <typename T, int VPL, int FULL>
__device__ __forceinline__ void ln_finish_row(const float (&f)[VPL][Vec<T>::N], const float4* s_mod, int packets, int D, float eps,
                                              int lane, T* out_row) {
  using V = Vec<T>;
  constexpr int Q = V::N / 4;
  float sum = 0.f;
#pragma unroll
  for (int c = 0; c < VPL; ++c)
#pragma unroll
    for (int q = 0; q < V::N; ++q) sum += f[c][q];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
  const float mean = sum / (float)D;
  float sq = 0.f;
#pragma unroll
  for (int c = 0; c < VPL; ++c)
    if (c < FULL || c * 32 + lane < packets) {
#pragma unroll
      for (int q = 0; q < V::N; ++q) { const float d = f[c][q] - mean; sq = fmaf(d, d, sq); }
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xFFFFFFFFu, sq, o);
  const float rstd = 1.0f / sqrtf(sq / (float)D + eps);
  V* out = reinterpret_cast<V*>(out_row);
#pragma unroll
  for (int c = 0; c < VPL; ++c) {
    const int v = c * 32 + lane;         // packet index: columns [V::N * v, V::N * (v + 1))
    if (c < FULL || v < packets) {
      float r[V::N];
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const float4 s4 = s_mod[q * packets + v], h4 = s_mod[(Q + q) * packets + v];
        r[4 * q] = fmaf((f[c][4 * q] - mean) * rstd, s4.x, h4.x);
        r[4 * q + 1] = fmaf((f[c][4 * q + 1] - mean) * rstd, s4.y, h4.y);
        r[4 * q + 2] = fmaf((f[c][4 * q + 2] - mean) * rstd, s4.z, h4.z);
        r[4 * q + 3] = fmaf((f[c][4 * q + 3] - mean) * rstd, s4.w, h4.w);
      }
      V o; o.pack(r);
      __stcs(&out[v].raw, o.raw);
    }
  }
}

// `settled` (launch_gather_ln_modulate) says what was complete before the kernel in front was placed: those loads go out
// before the wait for that kernel, so that of the chain vectors, list, row, row to add only the last link is left behind it.
// A row is fetched so early where every warp has one at most: ahead of a loop it would not stay in registers, and with both in
// one kernel the loop spills (17776 x 2560 32.4 -> 33.7 us, 150 x 2816 5.3 -> 5.7).  With the same in the pass from block to block
// and 32-byte stores in the attention, all behind the wait before: schedule of 42 blocks of 614 x 256 2734 -> 2573 us, cached step
// of 4 blocks of 371 x 768 221 -> 210.
//
// Several rows a warp.  (EXACT: the row has exactly 32 * VPL packets, nothing is predicated; the wide rows have no registers to
// spare for it.)
template <typename T, int VPL, bool EXACT>
__global__ void __launch_bounds__(256, ln_ctas_per_sm(VPL, false))
gather_ln_modulate_rows_kernel(const T* __restrict__ x, const T* __restrict__ add, const int* __restrict__ idx,
                               const float* __restrict__ shift, const float* __restrict__ scale, int mod_ld,
                               T* __restrict__ a, int N, int n_sel, int B, int D, float eps, int settled) {
  using V = Vec<T>;
  constexpr int kFull = EXACT ? VPL : ln_full_chunks(VPL);    // chunks of 32 packets that every row it serves has
  const int packets = EXACT ? VPL * 32 : D / V::N;
  if (EXACT) D = VPL * 32 * V::N;
  extern __shared__ float4 s_mod[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b = blockIdx.x % B, slot = blockIdx.x / B, slots = gridDim.x / B;
  if (settled < kLnModSettled) stream_order();
  ln_stage_modulation<T>(s_mod, scale + (long long)b * mod_ld, shift + (long long)b * mod_ld, packets);
  if (settled >= kLnModSettled) stream_order();
  for (int i = slot * 8 + warp; i < n_sel; i += slots * 8) {
    const long long row = (long long)b * N + (idx ? __ldg(idx + i) : i);
    const V* xr = reinterpret_cast<const V*>(x + row * D);
    V raw[VPL];
#pragma unroll
    for (int c = 0; c < VPL; ++c)
      if (c < kFull || c * 32 + lane < packets) raw[c].raw = __ldcs(&xr[c * 32 + lane].raw);
    float f[VPL][V::N];
#pragma unroll
    for (int c = 0; c < VPL; ++c) {
      if (c < kFull || c * 32 + lane < packets) {
        raw[c].unpack(f[c]);
      } else {
#pragma unroll
        for (int q = 0; q < V::N; ++q) f[c][q] = 0.f;
      }
    }
    if (add) {
      const V* ar = reinterpret_cast<const V*>(add + row * D);
#pragma unroll
      for (int c = 0; c < VPL; ++c)
        if (c < kFull || c * 32 + lane < packets) raw[c].raw = __ldcs(&ar[c * 32 + lane].raw);
#pragma unroll
      for (int c = 0; c < VPL; ++c) {
        if (c < kFull || c * 32 + lane < packets) {
          float g[V::N];
          raw[c].unpack(g);
#pragma unroll
          for (int q = 0; q < V::N; ++q) f[c][q] += g[q];
        }
      }
    }
    ln_finish_row<T, VPL, kFull>(f, s_mod, packets, D, eps, lane, a + ((long long)b * n_sel + i) * D);
  }
}

// One row a warp at most.  What need not be waited for is on its way before the wait; with nothing settled x is, before the
// vectors are staged (600 x 256 2.21 -> 1.99 us, 4400 x 512 4.34 -> 3.25 against the loop).
template <typename T, int VPL>
__global__ void __launch_bounds__(256, ln_ctas_per_sm(VPL, true))
gather_ln_modulate_row_kernel(const T* __restrict__ x, const T* __restrict__ add, const int* __restrict__ idx,
                              const float* __restrict__ shift, const float* __restrict__ scale, int mod_ld,
                              T* __restrict__ a, int N, int n_sel, int B, int D, float eps, int settled) {
  using V = Vec<T>;
  constexpr int kFull = ln_full_chunks(VPL);
  const int packets = D / V::N;
  extern __shared__ float4 s_mod[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b = blockIdx.x % B, i = blockIdx.x / B * 8 + warp;
  const bool there = i < n_sel;                               // warp-uniform
  long long row = 0;
  V raw[VPL];
  auto load = [&](const T* from) {
    const V* r = reinterpret_cast<const V*>(from + row * D);
#pragma unroll
    for (int c = 0; c < VPL; ++c)
      if (c < kFull || c * 32 + lane < packets) raw[c].raw = __ldcs(&r[c * 32 + lane].raw);
  };
  if (settled < kLnModSettled) stream_order();
  if (there) {
    row = (long long)b * N + (idx ? __ldg(idx + i) : i);
    if (settled != kLnModSettled) load(x);
  }
  ln_stage_modulation<T>(s_mod, scale + (long long)b * mod_ld, shift + (long long)b * mod_ld, packets);
  if (settled >= kLnModSettled) stream_order();
  if (!there) return;
  if (settled == kLnModSettled) load(x);
  float f[VPL][V::N];
#pragma unroll
  for (int c = 0; c < VPL; ++c) {
    if (c < kFull || c * 32 + lane < packets) {
      raw[c].unpack(f[c]);
    } else {
#pragma unroll
      for (int q = 0; q < V::N; ++q) f[c][q] = 0.f;
    }
  }
  if (add) {
    load(add);
#pragma unroll
    for (int c = 0; c < VPL; ++c) {
      if (c < kFull || c * 32 + lane < packets) {
        float g[V::N];
        raw[c].unpack(g);
#pragma unroll
        for (int q = 0; q < V::N; ++q) f[c][q] += g[q];
      }
    }
  }
  ln_finish_row<T, VPL, kFull>(f, s_mod, packets, D, eps, lane, a + ((long long)b * n_sel + i) * D);
}

// The end of one refreshed block and the start of the next in one pass: x = (x + ga) + gf for every row, and the rows that
// the next block refreshes, as stored, normalised and modulated into their places in its compact input.  pos gives a video
// row's place (-1: not refreshed; null: every row of x, in order).  Against the two passes one after the other it saves a
// launch and the second reading of x: in a whole step of 42 blocks of 614 rows x 256 1.3 us a block (2.92 -> 2.80 ms), of
// 8 blocks of 5820 x 1024 0.8, of 4 blocks of 1562 x 768 1.1.  A collapsed deep stack's blocks, which add a fp32 sum to the
// streams of a row, keep the two passes (16 blocks of 5254 x 1152: 4.46 ms apart, 4.47 in one).
constexpr int rln_ctas_per_sm(int vpl) { return vpl <= 3 ? 3 : 2; }      // what the registers of three rows allow
template <typename T, int VPL, bool ONE>
__global__ void __launch_bounds__(256, rln_ctas_per_sm(VPL))
residual_ln_kernel(T* __restrict__ x, const T* __restrict__ ga, const T* __restrict__ gf,
                   const int* __restrict__ pos, int n_text, const float* __restrict__ shift, const float* __restrict__ scale,
                   int mod_ld, T* __restrict__ a, int N, int n_sel, int B, int D, float eps) {
  using V = Vec<T>;
  constexpr int kFull = ln_full_chunks(VPL);
  const int packets = D / V::N;
  extern __shared__ float4 s_mod[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b = blockIdx.x % B, slot = blockIdx.x / B, slots = gridDim.x / B;
  // The kernel in front writes gf (the FFN's down-projection).  All else has been complete since before that kernel was
  // placed (x was last written a block ago, ga three launches ago, the lists and the vectors at the start of the step) and is
  // fetched before the wait, the rows of x and ga where a warp has one row at most (ONE).
  int place = 0;
  V* xr = nullptr;
  V vx[VPL], va[VPL], vf[VPL];
  auto load_early = [&](int i) {
    place = pos == nullptr ? i : (i < n_text ? -1 : __ldg(pos + i - n_text));
    xr = reinterpret_cast<V*>(x + ((long long)b * N + i) * D);
    const V* ar = reinterpret_cast<const V*>(ga + ((long long)b * N + i) * D);
#pragma unroll
    for (int c = 0; c < VPL; ++c)
      if (c < kFull || c * 32 + lane < packets) { vx[c] = ld_stream(xr + c * 32 + lane); va[c] = ld_stream(ar + c * 32 + lane); }
  };
  auto load_late = [&](int i) {
    const V* fr = reinterpret_cast<const V*>(gf + ((long long)b * N + i) * D);
#pragma unroll
    for (int c = 0; c < VPL; ++c)
      if (c < kFull || c * 32 + lane < packets) vf[c] = ld_stream(fr + c * 32 + lane);
  };
  const int first = slot * 8 + warp;
  if (ONE && first < N) load_early(first);
  ln_stage_modulation<T>(s_mod, scale + (long long)b * mod_ld, shift + (long long)b * mod_ld, packets);
  stream_order();
  for (int i = first; i < N; i += slots * 8) {
    if (!ONE) load_early(i);
    load_late(i);
    float f[VPL][V::N];
#pragma unroll
    for (int c = 0; c < VPL; ++c) {
      if (c < kFull || c * 32 + lane < packets) {
        float fa[V::N], ff[V::N];
        vx[c].unpack(f[c]); va[c].unpack(fa); vf[c].unpack(ff);
#pragma unroll
        for (int q = 0; q < V::N; ++q) f[c][q] = (f[c][q] + fa[q]) + ff[q];
        V r; r.pack(f[c]);
        st_stream(xr + c * 32 + lane, r);
        r.unpack(f[c]);                    // (the next block sees x as it is stored)
      } else {
#pragma unroll
        for (int q = 0; q < V::N; ++q) f[c][q] = 0.f;
      }
    }
    if (place >= 0) ln_finish_row<T, VPL, kFull>(f, s_mod, packets, D, eps, lane, a + ((long long)b * n_sel + place) * D);
    if (ONE) break;
  }
}

template <typename T, int VPL>
int residual_ln_launch(void* x, const void* ga, const void* gf, const int* pos, int n_text, const float* shift,
                       const float* scale, int mod_ld, void* a, int N, int n_sel, int B, int D, float eps, bool early,
                       cudaStream_t s) {
  const int resident = (num_sms() * rln_ctas_per_sm(VPL) + B - 1) / B, need = (N + 7) / 8;
  return launch_kernel_as(early, need <= resident ? residual_ln_kernel<T, VPL, true> : residual_ln_kernel<T, VPL, false>,
                          (unsigned)((need < resident ? need : resident) * B), 256,
                          (size_t)2 * D * sizeof(float), s, 1, (T*)x, (const T*)ga, (const T*)gf, pos, n_text, shift, scale,
                          mod_ld, (T*)a, N, n_sel, B, D, eps);
}
constexpr int kResidualLnPackets = 6;        // a lane's packets of three tensors stay in registers up to here
template <typename T>
int residual_ln_dispatch(void* x, const void* ga, const void* gf, const int* pos, int n_text, const float* shift,
                         const float* scale, int mod_ld, void* a, int N, int n_sel, int B, int D, float eps, bool early,
                         cudaStream_t s) {
  const int vpl = (D / Vec<T>::N + 31) / 32;
#define HERO_RLN(V) \
  if (vpl <= V) \
    return residual_ln_launch<T, V>(x, ga, gf, pos, n_text, shift, scale, mod_ld, a, N, n_sel, B, D, eps, early, s)
  HERO_RLN(1); HERO_RLN(2); HERO_RLN(3); HERO_RLN(4); HERO_RLN(5); HERO_RLN(6);
#undef HERO_RLN
  return HERO_ERR_ARG;
}

template <typename T, int VPL>
int gather_ln_warp(const void* x, const void* add, const int* idx, const float* shift, const float* scale, int mod_ld,
                   void* a, int N, int n_sel, int B, int D, float eps, int settled, cudaStream_t s) {
  // the same number of CTAs for every batch item, at most as many as stay resident
  const int need = (n_sel + 7) / 8;
  const bool one = VPL < 8 && need <= num_sms() * ln_ctas_per_sm(VPL, true) / B;
  const int resident = (num_sms() * ln_ctas_per_sm(VPL, one) + B - 1) / B;
  const unsigned grid = (unsigned)((need < resident ? need : resident) * B);
  const size_t smem = (size_t)2 * D * sizeof(float);
  auto kernel = gather_ln_modulate_rows_kernel<T, VPL, false>;
  if constexpr (VPL >= 8) {
    if (D == VPL * 32 * Vec<T>::N) kernel = gather_ln_modulate_rows_kernel<T, VPL, true>;
  } else {
    if (one) kernel = gather_ln_modulate_row_kernel<T, VPL>;
  }
  return launch_kernel(kernel, grid, 256, smem, s, 1, (const T*)x, (const T*)add, idx, shift, scale, mod_ld, (T*)a, N, n_sel,
                       B, D, eps, settled);
}

// Rows of at most 16 packets a lane; wider ones go through shared memory (gather_ln_modulate_kernel).
constexpr int kLnMaxPackets = 16;
template <typename T>
int gather_ln_dispatch(const void* x, const void* add, const int* idx, const float* shift, const float* scale, int mod_ld,
                       void* a, int N, int n_sel, int B, int D, float eps, int settled, cudaStream_t s) {
  const int vpl = (D / Vec<T>::N + 31) / 32;
#define HERO_LN(V) \
  if (vpl <= V) return gather_ln_warp<T, V>(x, add, idx, shift, scale, mod_ld, a, N, n_sel, B, D, eps, settled, s)
  HERO_LN(1); HERO_LN(2); HERO_LN(3); HERO_LN(4); HERO_LN(5); HERO_LN(6); HERO_LN(8); HERO_LN(10); HERO_LN(12); HERO_LN(16);
#undef HERO_LN
  return HERO_ERR_ARG;
}

template <typename T>
int extrapolate_t(const void* p, const void* l, void* o, long long n, float c, cudaStream_t s) {
  HERO_TRY(launch_streaming(extrapolate_kernel<T>, stream_grid(n / Vec<T>::N), kStreamThreads, s, (const T*)p,
                         (const T*)l, (T*)o, n, c));
  return HERO_OK;
}

}  // namespace

int launch_extrapolate(const void* g_prev, const void* g_last, void* out, long long n, int k, int d, int dtype,
                       cudaStream_t s) {
  const float c = (float)k / (float)d;
  return dtype == HERO_DTYPE_BF16 ? extrapolate_t<__nv_bfloat16>(g_prev, g_last, out, n, c, s)
                                  : extrapolate_t<float>(g_prev, g_last, out, n, c, s);
}

int launch_extrapolate_residual(void* x, const void* ga_prev, const void* ga_last, const void* gf_prev,
                                const void* gf_last, long long n, int k, int d, int dtype, cudaStream_t s) {
  const float c = (float)k / (float)d;
  if (dtype == HERO_DTYPE_BF16) {
    using T = __nv_bfloat16;
    const long long n_vec = n / Vec<T>::N;
    long long blocks = (n_vec + kStreamThreads - 1) / kStreamThreads;
    blocks = blocks < 1 ? 1 : (blocks > (long long)num_sms() * 32 ? (long long)num_sms() * 32 : blocks);
    HERO_TRY(launch_streaming(extrapolate_residual_kernel<T>, blocks, kStreamThreads, s, (T*)x,
                           (const T*)ga_prev, (const T*)ga_last, (const T*)gf_prev, (const T*)gf_last, n, c));
  } else {
    using T = float;
    const long long n_vec = n / Vec<T>::N;
    long long blocks = (n_vec + kStreamThreads - 1) / kStreamThreads;
    blocks = blocks < 1 ? 1 : (blocks > (long long)num_sms() * 32 ? (long long)num_sms() * 32 : blocks);
    HERO_TRY(launch_streaming(extrapolate_residual_kernel<T>, blocks, kStreamThreads, s, (T*)x,
                           (const T*)ga_prev, (const T*)ga_last, (const T*)gf_prev, (const T*)gf_last, n, c));
  }
  return HERO_OK;
}

int launch_extrapolate_group(void* x, const DeepGroup& grp, long long first, long long n, int k, int d, int dtype,
                             cudaStream_t s) {
  if (grp.n_entries <= 0 || n <= 0) return HERO_OK;
  const float c = (float)k / (float)d;
  const int per = dtype == HERO_DTYPE_BF16 ? 8 : 4;
  if (first % per != 0) return HERO_ERR_ALIGN;            // keeps every 16-byte access aligned
  long long blocks = (n / per + kStreamThreads - 1) / kStreamThreads;
  blocks = blocks < 1 ? 1 : (blocks > (long long)num_sms() * 16 ? (long long)num_sms() * 16 : blocks);
  const bool few = blocks < 2ll * num_sms();
  if (dtype == HERO_DTYPE_BF16) {
    using T = __nv_bfloat16;
    HERO_TRY(launch_streaming(few ? extrapolate_group_kernel<T, 16> : extrapolate_group_kernel<T, 4>, blocks, kStreamThreads,
                              s, (T*)x, grp, first, n, c));
  } else {
    HERO_TRY(launch_streaming(few ? extrapolate_group_kernel<float, 16> : extrapolate_group_kernel<float, 4>, blocks,
                              kStreamThreads, s, (float*)x, grp, first, n, c));
  }
  return HERO_OK;
}

int launch_residual2(void* x, const void* ga, const void* gf, long long n, int dtype, cudaStream_t s) {
  if (dtype == HERO_DTYPE_BF16) {
    using T = __nv_bfloat16;
    HERO_TRY(launch_streaming(residual2_kernel<T>, stream_grid(n / Vec<T>::N), kStreamThreads, s, (T*)x,
                           (const T*)ga, (const T*)gf, n));
  } else {
    HERO_TRY(launch_streaming(residual2_kernel<float>, stream_grid(n / 4), kStreamThreads, s, (float*)x,
                           (const float*)ga, (const float*)gf, n));
  }
  return HERO_OK;
}

static int wide_grid(long long n_vec) {
  long long blocks = (n_vec + kStreamThreads - 1) / kStreamThreads;
  const long long cap = (long long)num_sms() * 32;
  return (int)(blocks < 1 ? 1 : (blocks > cap ? cap : blocks));
}

int launch_residual2_acc(void* x, const void* ga, const void* gf, float* acc, long long n, int dtype, cudaStream_t s) {
  if (dtype == HERO_DTYPE_BF16) {
    using T = __nv_bfloat16;
    HERO_TRY(launch_streaming(residual2_acc_kernel<T>, wide_grid(n / Vec<T>::N), kStreamThreads, s, (T*)x,
                           (const T*)ga, (const T*)gf, acc, n));
  } else {
    HERO_TRY(launch_streaming(residual2_acc_kernel<float>, wide_grid(n / 4), kStreamThreads, s, (float*)x,
                           (const float*)ga, (const float*)gf, acc, n));
  }
  return HERO_OK;
}

int launch_extrapolate_stack(void* x, const float* s_prev, const float* s_last, long long n, int k, int d, int dtype,
                             cudaStream_t s) {
  const float c = (float)k / (float)d;
  if (dtype == HERO_DTYPE_BF16) {
    using T = __nv_bfloat16;
    HERO_TRY(launch_streaming(extrapolate_stack_kernel<T>, wide_grid(n / Vec<T>::N), kStreamThreads, s, (T*)x,
                           s_prev, s_last, n, c));
  } else {
    HERO_TRY(launch_streaming(extrapolate_stack_kernel<float>, wide_grid(n / 4), kStreamThreads, s, (float*)x,
                           s_prev, s_last, n, c));
  }
  return HERO_OK;
}

int launch_attend_rows(const void* k, const void* v, const int* idx, void* k_out, void* v_out, int B, int N, int n_text,
                       int n_sel, int D, int dtype, cudaStream_t s) {
  const long long row_bytes = (long long)D * dtype_size(dtype), rows = 2ll * B * (n_text + n_sel);
  if (row_bytes % 16 != 0) return HERO_ERR_ALIGN;
  if (rows == 0) return HERO_OK;
  const long long blocks = (rows + 7) / 8, cap = (long long)num_sms() * 16;          // a warp per row
  return launch_streaming(attend_rows_kernel, blocks < cap ? blocks : cap, 256, s, (const uint4*)k, (const uint4*)v, idx,
                          (uint4*)k_out, (uint4*)v_out, B, N, n_text, n_text + n_sel, (int)(row_bytes / 16));
}
static int move_rows(bool gather, const void* src, const int* idx, void* dst, int B, int N, int n_sel, int D,
                     int dtype, cudaStream_t s) {
  const long long row_bytes = (long long)D * dtype_size(dtype);
  if (row_bytes % 16 != 0) return HERO_ERR_ALIGN;
  const long long rows = (long long)B * n_sel;
  if (rows == 0) return HERO_OK;
  long long blocks = (rows + 7) / 8;   // 8 warps per CTA, one row per warp
  const long long cap = (long long)num_sms() * 16;
  if (blocks > cap) blocks = cap;
  if (gather)
    HERO_TRY(launch_streaming(move_rows_kernel<true>, blocks, 256, s, (const uint4*)src, idx,
                           (uint4*)dst, B, N, n_sel, (int)(row_bytes / 16)));
  else
    HERO_TRY(launch_streaming(move_rows_kernel<false>, blocks, 256, s, (const uint4*)src, idx,
                           (uint4*)dst, B, N, n_sel, (int)(row_bytes / 16)));
  return HERO_OK;
}

int launch_gather_rows(const void* src, const int* idx, void* dst, int B, int N, int n_sel, int D, int dtype,
                       cudaStream_t s) {
  return move_rows(true, src, idx, dst, B, N, n_sel, D, dtype, s);
}
int launch_scatter_rows(const void* src, const int* idx, void* dst, int B, int N, int n_sel, int D, int dtype,
                        cudaStream_t s) {
  return move_rows(false, src, idx, dst, B, N, n_sel, D, dtype, s);
}

// The kernels are instantiated for 1, 2, 4 and 8 batch items so that a warp's accumulators are as many as it needs.
template <typename T, int MAXB>
static int modulation_batch_launch(const void* temb, const ModBatch& batch, int B, int n_out, int E, bool beside, dim3 grid,
                                    size_t smem, cudaStream_t s) {
  return launch_kernel(modulation_batch_kernel<T, MAXB>, grid, 256, smem, s, 1, (const T*)temb, batch, B, n_out, E, beside);
}
template <typename T, int MAXB>
static int modulation_launch(const void* temb, const void* w_mod, const void* b_mod, float* mod, int B, int n_out,
                              int E, int blocks, size_t smem, cudaStream_t s) {
  return launch_kernel(modulation_kernel<T, MAXB>, (unsigned)blocks, 256, smem, s, 1, (const T*)temb, (const T*)w_mod,
                       (const T*)b_mod, mod, B, n_out, E);
}
#define HERO_MOD_DISPATCH(FN, T, ...)                      \
  do {                                                     \
    if (B <= 1) return FN<T, 1>(__VA_ARGS__);              \
    if (B <= 2) return FN<T, 2>(__VA_ARGS__);              \
    if (B <= 4) return FN<T, 4>(__VA_ARGS__);              \
    return FN<T, kModMaxB>(__VA_ARGS__);                   \
  } while (0)

int launch_modulation_batch(const void* temb, const ModBatch& batch, int B, int n_out, int E, bool beside, int dtype,
                            cudaStream_t s) {
  if (B > kModMaxB || batch.n < 0 || batch.n > kMaxModBatch) return HERO_ERR_ARG;
  if (batch.n == 0) return HERO_OK;
  const size_t smem = (size_t)B * E * sizeof(float);
  int bx = (n_out + 8 * kModRows - 1) / (8 * kModRows);     // eight warps per CTA, kModRows columns per warp and turn
  const int cap = num_sms() * 2 / batch.n;     // two CTAs per SM over the whole grid (what the registers allow): one wave
  if (bx > cap) bx = cap < 1 ? 1 : cap;
  const dim3 grid(bx, batch.n);
  if (dtype == HERO_DTYPE_BF16) {
    if (E % 8) return HERO_ERR_ALIGN;
    HERO_MOD_DISPATCH(modulation_batch_launch, __nv_bfloat16, temb, batch, B, n_out, E, beside, grid, smem, s);
  } else {
    if (E % 4) return HERO_ERR_ALIGN;
    HERO_MOD_DISPATCH(modulation_batch_launch, float, temb, batch, B, n_out, E, beside, grid, smem, s);
  }
}

int launch_modulation(const void* temb, const void* w_mod, const void* b_mod, float* mod, int B, int n_out, int E,
                      int dtype, cudaStream_t s) {
  if (B > kModMaxB) return HERO_ERR_ARG;
  const size_t smem = (size_t)B * E * sizeof(float);
  int blocks = (n_out + 8 * kModRows - 1) / (8 * kModRows);
  const int cap = num_sms() * 2;
  if (blocks > cap) blocks = cap;
  if (dtype == HERO_DTYPE_BF16) {
    if (E % 8) return HERO_ERR_ALIGN;
    HERO_MOD_DISPATCH(modulation_launch, __nv_bfloat16, temb, w_mod, b_mod, mod, B, n_out, E, blocks, smem, s);
  } else {
    if (E % 4) return HERO_ERR_ALIGN;
    HERO_MOD_DISPATCH(modulation_launch, float, temb, w_mod, b_mod, mod, B, n_out, E, blocks, smem, s);
  }
}
#undef HERO_MOD_DISPATCH

bool residual_ln_serves(int D, int dtype) { return D / (dtype == HERO_DTYPE_BF16 ? 8 : 4) <= 32 * kResidualLnPackets; }

int launch_residual_ln(void* x, const void* ga, const void* gf, const int* pos, int n_text, const float* shift,
                       const float* scale, int mod_ld, void* a, int B, int N, int n_sel, int D, float eps, int dtype,
                       bool early, cudaStream_t s) {
  return dtype == HERO_DTYPE_BF16
             ? residual_ln_dispatch<__nv_bfloat16>(x, ga, gf, pos, n_text, shift, scale, mod_ld, a, N, n_sel, B, D, eps, early, s)
             : residual_ln_dispatch<float>(x, ga, gf, pos, n_text, shift, scale, mod_ld, a, N, n_sel, B, D, eps, early, s);
}

int launch_gather_ln_modulate(const void* x, const void* add, const int* idx, const float* shift,
                              const float* scale, int mod_ld, void* a, int B, int N, int n_sel, int D, float eps,
                              int dtype, int settled, cudaStream_t s) {
  const long long rows = (long long)B * n_sel;
  if (rows == 0) return HERO_OK;
  const bool bf16 = dtype == HERO_DTYPE_BF16;
  const int per = bf16 ? 8 : 4;
  if (D % per) return HERO_ERR_ALIGN;
  // the warp kernel reads the adaLN vectors as float4: every item's slice starts 16-byte aligned when mod_ld % 4 == 0
  const bool vec_ok = mod_ld % 4 == 0 && ((reinterpret_cast<uintptr_t>(shift) | reinterpret_cast<uintptr_t>(scale)) & 15) == 0;
  if (vec_ok && D / per <= 32 * kLnMaxPackets)
    return bf16 ? gather_ln_dispatch<__nv_bfloat16>(x, add, idx, shift, scale, mod_ld, a, N, n_sel, B, D, eps, settled, s)
                : gather_ln_dispatch<float>(x, add, idx, shift, scale, mod_ld, a, N, n_sel, B, D, eps, settled, s);
  // The widest row, 12288 features, fills the 48 KB a kernel may have without an opt-in; the reduction's words come on top.
  static PerDeviceOnce once;
  HERO_TRY(per_device_once(once, [](int) {
    HERO_CUDA_TRY(cudaFuncSetAttribute(gather_ln_modulate_kernel<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, 48 * 1024));
    HERO_CUDA_TRY(cudaFuncSetAttribute(gather_ln_modulate_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, 48 * 1024));
    return HERO_OK;
  }));
  const size_t smem = (size_t)D * sizeof(float);
  if (bf16)
    HERO_TRY(launch_kernel(gather_ln_modulate_kernel<__nv_bfloat16>, (unsigned)rows, kLnThreads, smem, s, 1,
                           (const __nv_bfloat16*)x, (const __nv_bfloat16*)add, idx, shift, scale, mod_ld,
                           (__nv_bfloat16*)a, N, n_sel, D, eps));
  else
    HERO_TRY(launch_kernel(gather_ln_modulate_kernel<float>, (unsigned)rows, kLnThreads, smem, s, 1, (const float*)x,
                           (const float*)add, idx, shift, scale, mod_ld, (float*)a, N, n_sel, D, eps));
  return HERO_OK;
}

}  // namespace hero
