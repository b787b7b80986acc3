// Token selection S(z) = union_i Sample(P^i, R) (Eq. 4) with frequency-aware tracking
// (Sec. 4.3): integer-only, data-independent, bit-exact against the CPU oracle.
//
// One WARP per band (the grid rows of one row of patches in one frame: ph x W consecutive tokens) and block to select,
// all shallow blocks of a step in one launch.  A patch never leaves its band, and the quotas of the patches before a
// band sum to a closed form, so a warp knows where its part of the list starts without asking anybody; inside the band
// each lane rebuilds the keys of its token's patch mates from the old ages, ranks the token, and the warp compacts the
// winners in ascending row order with ballots.  Bands of more than 32 tokens get a thread block instead, whose warps take
// 32 tokens each at a time and count their winners for one another (launch_select says when).  Ages are double-buffered
// (read old, write new) because a patch spans several grid rows.  Bound by latency (integer work, a few hundred bytes per
// warp) and, where a patch has hundreds of tokens, by the hashes.
#include "hero_internal.h"

namespace hero {
namespace {

constexpr int kSelWarps = 8;

__device__ __forceinline__ uint32_t mix32(uint32_t x) {
  // xor-shift / odd-multiply avalanche rounds (the published MurmurHash3 finaliser)
  x ^= x >> 16;
  x *= 0x85EBCA6Bu;
  x ^= x >> 13;
  x *= 0xC2B2AE35u;
  x ^= x >> 16;
  return x;
}

// Sampling key of a token: larger wins.  Mode 0: (age+1) * (hash+1), a uniform draw on (0, age+1] up to
// scale, so the chance of being picked grows with the time a token has gone unsampled.  Mode 1: age first,
// hash second - strict oldest-first, the draw only orders tokens of equal age.
__device__ __forceinline__ unsigned long long make_key(int track_mode, uint32_t age, uint32_t hash) {
  return track_mode == 0 ? (unsigned long long)(age + 1u) * ((unsigned long long)hash + 1ull)
                         : ((unsigned long long)age << 32) | (unsigned long long)hash;
}

// Tokens that the patches of one band take in quota_mode 1 (each patch rounds for itself), `rows` grid rows high.
__device__ __forceinline__ int band_total_rounded(const SelectGeom& g, int rows) {
  const long long ra = g.ratio_num, rb = g.ratio_den;
  auto quota = [&](int n) { return min(n, (int)((2ll * n * ra + rb) / (2 * rb))); };
  const int whole = g.grid_w / g.patch_w, rest = g.grid_w - whole * g.patch_w;
  return whole * quota(rows * g.patch_w) + (rest ? quota(rows * rest) : 0);
}

// LONG: a thread block per band, else a warp.
template <bool LONG>
__global__ void __launch_bounds__(LONG ? 1024 : kSelWarps * 32) select_kernel(const SelectGeom g, const SelectBatch batch) {
  stream_order();
  __shared__ int s_count[2][32];                           // (of this turn and of the one before)
  const int e = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int H = g.grid_h, W = g.grid_w, ph = g.patch_h, pw = g.patch_w;
  const int bands_per_frame = (H + ph - 1) / ph;
  const int band = LONG ? blockIdx.x : blockIdx.x * kSelWarps + warp;
  if (band >= g.frames * bands_per_frame) return;          // (of whole warps, and never of a warp of a LONG block)
  const uint16_t* __restrict__ ages_in = batch.ages_in[e];
  uint16_t* __restrict__ ages_out = batch.ages_out[e];
  int* __restrict__ idx = batch.idx[e];
  int* __restrict__ pos = batch.pos[e];
  const int call = batch.call[e];
  const uint32_t h_block = mix32(mix32(g.seed_lo ^ (uint32_t)batch.block[e]) + (uint32_t)call);
  const long long off = (long long)call * ph * pw, ra = g.ratio_num, rb = g.ratio_den;

  const int t = band / bands_per_frame, py = band - t * bands_per_frame;
  const int y0 = py * ph, hh = min(ph, H - y0);
  const long long band_first = (long long)t * H * W + (long long)y0 * W;     // tokens before this band
  // list entries before this band
  int start;
  if (g.quota_mode == 0) {
    start = (int)(((band_first + off) * ra) / rb - (off * ra) / rb);
  } else {
    const int full = band_total_rounded(g, ph);
    const int tail = H % ph ? band_total_rounded(g, H % ph) : 0;
    start = t * ((H / ph) * full + tail) + py * full;
  }
  const int n_band = hh * W;
  const int step = LONG ? (int)blockDim.x : 32;
  int turn = 0;
  for (int base = 0; base < n_band; base += step, turn ^= 1) {
    const int i = base + (LONG ? (int)threadIdx.x : lane);
    bool pick = false;
    uint32_t age_v = 0;
    const int v = (int)band_first + i;
    if (i < n_band) {
      const int x = i % W;
      const int x0 = x / pw * pw, ww = min(pw, W - x0);
      const int n_here = hh * ww;
      int quota;
      if (g.quota_mode == 0) {
        // patches that precede this one (patch-id order: frame, patch row, patch column)
        const long long before = band_first + (long long)hh * x0 + off;
        quota = (int)(((before + n_here) * ra) / rb - (before * ra) / rb);
      } else {
        quota = min(n_here, (int)((2ll * n_here * ra + rb) / (2 * rb)));
      }
      age_v = ages_in[v];
      const unsigned long long key_v = make_key(g.track_mode, age_v, mix32(h_block + (uint32_t)v));
      int beaten_by = 0;
      for (int dy = 0; dy < hh; ++dy) {
        for (int dx = 0; dx < ww; ++dx) {
          const int u = (int)band_first + dy * W + x0 + dx;
          if (u == v) continue;
          const unsigned long long key_u = make_key(g.track_mode, (uint32_t)ages_in[u], mix32(h_block + (uint32_t)u));
          beaten_by += (key_u > key_v || (key_u == key_v && u < v)) ? 1 : 0;
        }
      }
      pick = beaten_by < quota;
    }
    const unsigned ballot = __ballot_sync(0xFFFFFFFFu, pick);
    int before = 0, total = __popc(ballot);                // winners of the warps in front, and of all of them
    if (LONG) {
      if (lane == 0) s_count[turn][warp] = total;
      __syncthreads();
      const int c = lane < step / 32 ? s_count[turn][lane] : 0;
      before = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? c : 0);
      total = __reduce_add_sync(0xFFFFFFFFu, c);
    }
    if (i < n_band) {
      const int place = start + before + __popc(ballot & ((1u << lane) - 1u));
      if (pick) idx[place] = g.n_text + v;
      if (pos) pos[v] = pick ? place : -1;
      ages_out[v] = pick ? (uint16_t)0 : (uint16_t)min(age_v + 1u, 65535u);
    }
    start += total;
  }
}

}  // namespace

int launch_select(const SelectGeom& g, const SelectBatch& batch, cudaStream_t s) {
  if (batch.n <= 0) return HERO_OK;
  const int bands = g.frames * ((g.grid_h + g.patch_h - 1) / g.patch_h);
  const long long longest = (long long)(g.patch_h < g.grid_h ? g.patch_h : g.grid_h) * g.grid_w;
  // A warp per band is the better split only where every band is one turn of it, or where there are more tokens than the
  // chip holds threads and enough bands (16 warps an SM) to fill it.  Measured in us, a block / a warp a band, and in
  // brackets one block a list, in turns of 1024 tokens (lists x frames x grid, patch): 1 x 1 x 64 x 64, 8 x 8 8.9 / 103 (51),
  // 64 x 64 2509 / 36621 (2460); 1 x 1 x 2 x 127, 2 x 2 6.9 / 14.6 (7.7); 1 x 1 x 2 x 8775, 2 x 2 39 / 602 (49);
  // 14 x 13 x 30 x 45, 2 x 2 12.7 / 12.5 (58), 3 x 3 14.7 / 16.7 (72); 14 x 13 x 60 x 90, 2 x 2 29.2 / 22.9 (215);
  // 14 x 3 x 9 x 11, 2 x 2 (22 tokens a band) 8.4 / 8.1 (8.5).
  const long long tokens = (long long)g.frames * g.grid_h * g.grid_w * batch.n, sms = num_sms();
  if (longest > 32 && (tokens <= sms * 2048 || (long long)bands * batch.n < sms * 16))
    return launch_kernel(select_kernel<true>, dim3((unsigned)bands, (unsigned)batch.n),
                         longest < 1024 ? (unsigned)((longest + 31) / 32 * 32) : 1024u, 0, s, 1, g, batch);
  return launch_kernel(select_kernel<false>, dim3((unsigned)((bands + kSelWarps - 1) / kSelWarps), (unsigned)batch.n),
                       kSelWarps * 32, 0, s, 1, g, batch);
}

}  // namespace hero
