// Token-granular prefill compression of fixed heads, and of tidal heads' permanent base ("Prefill Compression";
// retention per head from Eq. 1).
//
// Runs once per (sequence, layer) at placement, after the chunk-granular placement has staged the prefix: the staging
// buffer holds every head's audio K,V in the chunk-padded row layout and the text store holds the text rows.
//   1. wnw_token_logits_kernel, wnw_token_mass_kernel: p[tau] = sum over the text queries and the head's q-heads of the
//                               softmax weight of audio position tau (softmax over the whole prefix), fp32, sums in a
//                               fixed order so that they are reproducible;
//   2. wnw_token_select_kernel: per segment of n_s tokens the floor(retention * length) positions with the largest p
//                               (equal p: the earlier position), or the same total from the whole head (the ablation's
//                               global top-k); kept positions in ascending order; block table of the compact store;
//   3. wnw_token_gather_kernel: K,V rows of the kept positions from staging into the head's compact fixed store.
// The decode kernel then reads a fixed head as blocks of nc rows whose table entries carry their row count (-(2 + rows))
// instead of a chunk id.
#include <algorithm>

#include "wnw_internal.cuh"

namespace wnw {

namespace {

constexpr int TOK_THREADS = 512;
constexpr int TOK_TILE = 128;

// Compressed head x of a layer: the fixed heads first, then (token-granular tidal bases) the tidal heads.  Returns the
// KV-head, and in `head` its index among the sequence's compact stores.
__device__ __forceinline__ int comp_head(const CacheView &cv, int layer, int x, int &head) {
  const Geometry &G = cv.geo;
  const LayerInfo &li = cv.layers[layer];
  const int role = x < li.n_fixed ? ROLE_FIXED : ROLE_TIDAL, idx = x < li.n_fixed ? x : x - li.n_fixed;
  head = role == ROLE_FIXED ? li.fixed_off + idx : G.F_fix + li.tid_prefix + idx;
  for (int h = 0; h < G.Hkv; ++h)
    if (cv.roles[layer * G.Hkv + h] == role && cv.role_idx[layer * G.Hkv + h] == idx) return h;
  return -1;
}

}  // namespace

// Scores in two kernels over tiles of TOK_TILE positions, so that the tiles of all heads fill the machine (one CTA per head, as
// it was, left 141 of 148 SMs idle: 523 us a layer at 3064 positions, 7 heads, 4 queries of 4 heads; now 21 + 10 us).
//
// (1) grid (tiles, compressed heads), a thread per position: its logits for up to TOK_QR query rows (a row = one q-head of one
// text query).  The position's K row passes through registers once, 16 bytes at a time, the query rows sit in shared memory
// (broadcast reads).  Bound by the fp32 multiply-adds of the warps in flight, 128 x TOK_QR per position.  A tile also leaves
// each row's (max, sum of 2^(logit - max)).
__global__ void __launch_bounds__(TOK_TILE) wnw_token_logits_kernel(const __grid_constant__ CacheView cv, int b, int layer,
                                                                   const bf16 *stage, const bf16 *q_rows, int n_q, int T_t, int T_a,
                                                                   float *work, float2 *tile_ml) {
  const Geometry &G = cv.geo;
  extern __shared__ float tok_smem[];   // [n_q * g][d] query rows, then [n_q * g][warps] (max, sum)
  const int n = T_t + T_a, d = G.d, g = G.g, n_row = n_q * g, i = blockIdx.x * TOK_TILE + threadIdx.x;
  int head;
  const int f = blockIdx.y, h = comp_head(cv, layer, f, head);
  if (h < 0) return;
  float2 *red = reinterpret_cast<float2 *>(tok_smem + n_row * d);
  for (int x = threadIdx.x; x < n_row * d; x += TOK_TILE) {
    const int r = x / d;
    tok_smem[x] = __bfloat162float(q_rows[((long long)(r / g) * G.Hq + h * g + r % g) * d + (x - r * d)]);
  }
  __syncthreads();
  float acc[TOK_QR];
#pragma unroll
  for (int r = 0; r < TOK_QR; ++r) acc[r] = 0.f;
  if (i < n) {
    const bf16 *row;
    if (i < T_t) row = cv.text + text_off(G, b, layer, h, 0) + (long long)i * d;
    else { const int tau = i - T_t; row = stage + anchor_off(G, 0, 0, h, 0) + ((long long)(tau / G.nc) * G.ncp + tau % G.nc) * d; }
    const uint4 *r4 = reinterpret_cast<const uint4 *>(row);
#pragma unroll 2
    for (int v = 0; v < d / 8; ++v) {
      const uint4 u = r4[v];
      const __nv_bfloat162 *h2 = reinterpret_cast<const __nv_bfloat162 *>(&u);
      float kf[8];
#pragma unroll
      for (int e = 0; e < 4; ++e) { const float2 x = __bfloat1622float2(h2[e]); kf[2 * e] = x.x; kf[2 * e + 1] = x.y; }
#pragma unroll
      for (int r = 0; r < TOK_QR; ++r)
        if (r < n_row) {
          const float4 qa = *reinterpret_cast<const float4 *>(tok_smem + r * d + v * 8), qb = *reinterpret_cast<const float4 *>(tok_smem + r * d + v * 8 + 4);
          acc[r] = fmaf(qa.x, kf[0], acc[r]); acc[r] = fmaf(qa.y, kf[1], acc[r]); acc[r] = fmaf(qa.z, kf[2], acc[r]); acc[r] = fmaf(qa.w, kf[3], acc[r]);
          acc[r] = fmaf(qb.x, kf[4], acc[r]); acc[r] = fmaf(qb.y, kf[5], acc[r]); acc[r] = fmaf(qb.z, kf[6], acc[r]); acc[r] = fmaf(qb.w, kf[7], acc[r]);
        }
    }
  }
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int r = 0; r < TOK_QR; ++r)
    if (r < n_row) {
      const float l2 = i < n ? acc[r] * G.scale_log2 : -INFINITY;
      if (i < n) work[((long long)f * TOK_QR + r) * n + i] = l2;
      float m = l2;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      float z = m > -INFINITY ? exp2f(l2 - m) : 0.f;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
      if (lane == 0) red[r * (TOK_TILE / 32) + w] = make_float2(m, z);
    }
  __syncthreads();
  for (int r = threadIdx.x; r < n_row; r += TOK_TILE) {
    float M = -INFINITY, Z = 0.f;
    for (int x = 0; x < TOK_TILE / 32; ++x) M = fmaxf(M, red[r * (TOK_TILE / 32) + x].x);
    for (int x = 0; x < TOK_TILE / 32; ++x) Z += red[r * (TOK_TILE / 32) + x].y * exp2f(red[r * (TOK_TILE / 32) + x].x - M);
    tile_ml[((long long)f * TOK_QR + r) * gridDim.x + blockIdx.x] = make_float2(M, Z);
  }
}

// (2) grid (tiles of the audio, compressed heads): the rows' final (max, denominator) from the tiles' (a warp per row, fixed
// tree), then p[tau] += 2^(logit - max) / denominator, row by row in order.
__global__ void __launch_bounds__(TOK_TILE) wnw_token_mass_kernel(const __grid_constant__ CacheView cv, int n_q, int T_t, int T_a,
                                                                 int n_tiles, const float *work, const float2 *tile_ml, float *p_tok,
                                                                 long long p_stride, int first) {
  const int n = T_t + T_a, n_row = n_q * cv.geo.g, f = blockIdx.y, lane = threadIdx.x & 31;
  __shared__ float2 mz[TOK_QR];
  for (int r = threadIdx.x >> 5; r < n_row; r += TOK_TILE / 32) {
    const float2 *ml = tile_ml + ((long long)f * TOK_QR + r) * n_tiles;
    float M = -INFINITY, Z = 0.f;
    for (int x = lane; x < n_tiles; x += 32) M = fmaxf(M, ml[x].x);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
    for (int x = lane; x < n_tiles; x += 32) Z += ml[x].y * exp2f(ml[x].x - M);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) Z += __shfl_xor_sync(0xffffffffu, Z, o);
    if (lane == 0) mz[r] = make_float2(M, Z);
  }
  __syncthreads();
  const int tau = blockIdx.x * TOK_TILE + threadIdx.x;
  if (tau >= T_a) return;
  float p = first ? 0.f : p_tok[(long long)f * p_stride + tau];
  for (int r = 0; r < n_row; ++r) p += __fdiv_rn(exp2f(work[((long long)f * TOK_QR + r) * n + T_t + tau] - mz[r].x), mz[r].y);
  p_tok[(long long)f * p_stride + tau] = p;
}

// grid: fixed heads of the layer; block: TOK_THREADS.  flags: [n_fixed][p_stride] int32 scratch.
__global__ void __launch_bounds__(TOK_THREADS) wnw_token_select_kernel(const __grid_constant__ CacheView cv, int b, int layer,
                                                                      const float *p_tok, long long p_stride, int T_a, int seg,
                                                                      const __grid_constant__ TokenRetention ret_h, int variant, int32_t *flags,
                                                                      int32_t *fixed_tok, int tok_cap, int32_t *tok_n) {
  const Geometry &G = cv.geo;
  __shared__ int counts[TOK_THREADS + 1];
  int head;
  const int f = blockIdx.x, h = comp_head(cv, layer, f, head);
  if (h < 0) return;
  const long long fh = (long long)b * G.F_tot + head;
  const float *key = p_tok + (long long)f * p_stride;
  int32_t *fl = flags + (long long)f * p_stride, *out = fixed_tok + fh * tok_cap;
  const double ret = (double)ret_h.r[h];
  int total = 0;
  if (variant != 0)
    for (int lo = 0; lo < T_a; lo += seg) total += (int)floor(ret * (double)min(seg, T_a - lo));
  for (int tau = threadIdx.x; tau < T_a; tau += TOK_THREADS) {
    const float me = key[tau];
    int lo = 0, hi = T_a, m = total;
    if (variant == 0) {
      lo = tau / seg * seg; hi = min(lo + seg, T_a);
      m = (int)floor(ret * (double)(hi - lo));
    }
    int rank = 0;
    for (int t = lo; t < hi && rank < m; ++t) rank += (key[t] > me) || (key[t] == me && t < tau);
    fl[tau] = rank < m;
  }
  __syncthreads();
  // kept positions in ascending order: every thread owns a contiguous range of positions
  const int per = (T_a + TOK_THREADS - 1) / TOK_THREADS, t0 = min(T_a, (int)threadIdx.x * per), t1 = min(T_a, t0 + per);
  int cnt = 0;
  for (int t = t0; t < t1; ++t) cnt += fl[t];
  counts[threadIdx.x] = cnt;
  __syncthreads();
  if (threadIdx.x == 0) {
    int run = 0;
    for (int i = 0; i < TOK_THREADS; ++i) { const int c = counts[i]; counts[i] = run; run += c; }
    counts[TOK_THREADS] = run;
  }
  __syncthreads();
  int at = counts[threadIdx.x];
  for (int t = t0; t < t1; ++t)
    if (fl[t]) out[at++] = t;
  const int n = counts[TOK_THREADS], n_blk = (n + G.nc - 1) / G.nc;
  for (int s = threadIdx.x; s < G.FB; s += TOK_THREADS)   // block s of the compact store holds min(nc, n - s*nc) rows
    cv.fixed_chunks[fh * G.FB + s] = s < n_blk ? -(2 + min(G.nc, n - s * G.nc)) : -1;
  if (threadIdx.x == 0) { cv.fixed_n[fh] = n_blk; tok_n[fh] = n; }
  const LayerInfo &li = cv.layers[layer];
  if (f >= li.n_fixed && threadIdx.x == 0) {   // (the global variant keeps a different number per segment: the table below says)
    const int tail_len = T_a - (T_a - 1) / G.nc * G.nc;
    cv.tok_m[((long long)b * G.L + layer) * G.Hkv + h] =
        variant != 0 ? make_int2(-1, -1) : make_int2((int)floor(ret * (double)G.nc), (int)floor(ret * (double)tail_len));
  }
  if (f >= li.n_fixed) {   // a tidal head's base: how many positions of every segment it holds (what a fetched segment must skip)
    int32_t *sk = cv.seg_kept + ((long long)b * cv.tid_total + li.tid_prefix + (f - li.n_fixed)) * G.C_max;
    for (int c = threadIdx.x; c * G.nc < T_a; c += TOK_THREADS) {
      int k = 0;
      for (int t = c * G.nc; t < min(T_a, (c + 1) * G.nc); ++t) k += fl[t];
      sk[c] = k;
    }
  }
}

// grid (FB, fixed heads of the layer); block 128.  Fills block blockIdx.x of the head's compact store.
__global__ void __launch_bounds__(128) wnw_token_gather_kernel(const __grid_constant__ CacheView cv, int b, int layer,
                                                               const bf16 *stage, const int32_t *fixed_tok, int tok_cap,
                                                               const int32_t *tok_n) {
  const Geometry &G = cv.geo;
  int head;
  const int blk = blockIdx.x, f = blockIdx.y, h = comp_head(cv, layer, f, head);
  if (h < 0) return;
  const long long fh = (long long)b * G.F_tot + head;
  const int n = tok_n[fh];
  if (blk * G.nc >= n) return;
  const int pieces = G.d / 8;
  const int32_t *pos = fixed_tok + fh * tok_cap;
  for (int kv = 0; kv < 2; ++kv) {
    const uint4 *src = reinterpret_cast<const uint4 *>(stage + anchor_off(G, 0, 0, h, kv));
    uint4 *dst = reinterpret_cast<uint4 *>(cv.fixed + compact_off(G, b, head, kv) + (long long)blk * G.ncp * G.d);
    for (int v = threadIdx.x; v < G.ncp * pieces; v += blockDim.x) {
      const int r = v / pieces, x = v - r * pieces, i = blk * G.nc + r;
      uint4 val = make_uint4(0, 0, 0, 0);   // rows past the block's last token are zero
      if (r < G.nc && i < n) {
        const int tau = pos[i];
        val = src[((long long)(tau / G.nc) * G.ncp + tau % G.nc) * pieces + x];
      }
      dst[v] = val;
    }
  }
}

// grid (segments, tidal heads of the layer); block 128.  Token-granular tidal base: rewrites segment blockIdx.x of the
// head in the layer's outgoing mirror image with the positions that are NOT in the base first (ascending), the kept ones after them, so that
// the first (length - kept) rows of a fetched segment are exactly its complement.
__global__ void __launch_bounds__(128) wnw_token_mirror_kernel(const __grid_constant__ CacheView cv, int b, int layer,
                                                               const bf16 *stage, const int32_t *flags, long long p_stride,
                                                               int T_a, bf16 *mirror_out) {
  const Geometry &G = cv.geo;
  extern __shared__ int mirror_dst[];   // [nc] destination row of every position of the segment
  const LayerInfo li = cv.layers[layer];
  const int c = blockIdx.x, t = blockIdx.y, x = li.n_fixed + t;
  int head;
  const int h = comp_head(cv, layer, x, head);
  if (h < 0) return;
  const int lo = c * G.nc, len = min(G.nc, T_a - lo);
  const int32_t *fl = flags + (long long)x * p_stride + lo;
  int n_out = 0;
  for (int r = 0; r < len; ++r) n_out += fl[r] == 0;
  for (int r = threadIdx.x; r < len; r += blockDim.x) {
    int before_same = 0;
    for (int q = 0; q < r; ++q) before_same += fl[q] == fl[r];
    mirror_dst[r] = fl[r] ? n_out + before_same : before_same;
  }
  __syncthreads();
  const int pieces = G.d / 8;
  for (int kv = 0; kv < 2; ++kv) {
    const uint4 *src = reinterpret_cast<const uint4 *>(stage + anchor_off(G, 0, 0, h, kv) + (long long)c * G.ncp * G.d);
    uint4 *dst = reinterpret_cast<uint4 *>(mirror_out + mirror_block_off(G, li, c, t, kv));
    for (int v = threadIdx.x; v < len * pieces; v += blockDim.x) {
      const int r = v / pieces, piece = v - r * pieces;
      dst[(long long)mirror_dst[r] * pieces + piece] = src[v];
    }
  }
}

// n_comp: compressed heads of the layer (its fixed heads, then its tidal heads when they keep a token base)
cudaError_t launch_token_compress(const CacheView &cv, int b, int layer, int n_comp, int n_tidal_base, const bf16 *stage,
                                  const bf16 *q_text, int n_q, int T_t, int T_a, int seg, const TokenRetention &ret,
                                  int variant, float *work, float2 *tile_ml, float *p_tok, int32_t *flags, long long p_stride,
                                  int32_t *fixed_tok, int tok_cap, int32_t *tok_n, bf16 *mirror_out, cudaStream_t st) {
  if (n_comp <= 0 || T_a <= 0) return cudaSuccess;
  const Geometry &G = cv.geo;
  const int n_tiles = (T_t + T_a + TOK_TILE - 1) / TOK_TILE, per = TOK_QR / G.g;   // whole queries per pass
  for (int q0 = 0; q0 < n_q; q0 += per) {
    const int nq = std::min(per, n_q - q0);
    const size_t smem = (size_t)nq * G.g * (G.d + 2 * (TOK_TILE / 32)) * sizeof(float);
    wnw_token_logits_kernel<<<dim3(n_tiles, n_comp), TOK_TILE, smem, st>>>(cv, b, layer, stage, q_text + (size_t)q0 * G.Hq * G.d, nq, T_t,
                                                                          T_a, work, tile_ml);
    wnw_token_mass_kernel<<<dim3((T_a + TOK_TILE - 1) / TOK_TILE, n_comp), TOK_TILE, 0, st>>>(cv, nq, T_t, T_a, n_tiles, work, tile_ml, p_tok,
                                                                                            p_stride, q0 == 0);
  }
  wnw_token_select_kernel<<<n_comp, TOK_THREADS, 0, st>>>(cv, b, layer, p_tok, p_stride, T_a, seg, ret, variant, flags,
                                                         fixed_tok, tok_cap, tok_n);
  wnw_token_gather_kernel<<<dim3(cv.geo.FB, n_comp), 128, 0, st>>>(cv, b, layer, stage, fixed_tok, tok_cap, tok_n);
  if (n_tidal_base > 0) {
    const int C_b = (T_a + cv.geo.nc - 1) / cv.geo.nc;
    wnw_token_mirror_kernel<<<dim3(C_b, n_tidal_base), 128, (size_t)cv.geo.nc * sizeof(int), st>>>(cv, b, layer, stage, flags,
                                                                                                  p_stride, T_a, mirror_out);
  }
  return cudaGetLastError();
}

}  // namespace wnw
