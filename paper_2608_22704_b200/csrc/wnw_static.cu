// wnw_attend_static: one-query full attention over a caller-owned K/V buffer, with every byte of scratch taken
// from a fixed array inside the library image.  It reuses the attention kernels of wnw_attn.cu and wnw_attn_short.cu;
// what differs from the cache-based entry points is only where the split partials, the completion counters and
// the per-head split table live.
//
// Who this is for: callers that cannot allocate device memory at the point of the call.  A serving loop that has
// handed the whole device to its own pool allocator, or a latency-critical decode thread for which the implicit
// device-wide synchronisation of cudaMalloc/cudaFree is not acceptable, can still run an attention step through
// this entry point: it calls no cudaMalloc, no cudaFree and no allocating library routine, and its host side keeps
// no list at all.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <mutex>

#include "../../include/wnw.h"
#include "../../include/wnw_debug.h"
#include "wnw_internal.cuh"

using namespace wnw;

namespace {

constexpr int ST_MAX_KV_HEADS = 64;
constexpr int ST_MAX_Q_HEADS = 128;
constexpr int ST_MAX_ROWS = 96 * MAX_G;              // partial rows: (pieces of a head) x (query heads)
constexpr long long ST_MAX_TOKENS = 1ll << 20;
constexpr int ST_MAX_DEVICES = 64;

// layout of the scratch array (byte offsets, all multiples of 256)
constexpr size_t OFF_STATUS = 0;                                                   // int32: sticky STATUS_* bits of the kernels' bounded waits,
                                                                                   //   reset when it is read
constexpr size_t OFF_COUNTERS = 256;                                               // int32 [ST_MAX_KV_HEADS], zero between calls: the CTA
                                                                                   //   that finishes a head resets the head's
constexpr size_t OFF_HEAD_MZ = 1024;                                               // float2 [ST_MAX_Q_HEADS]
constexpr size_t OFF_PART_ML = 2048;                                               // float2 [ST_MAX_ROWS]
constexpr size_t OFF_PART_O = OFF_PART_ML + (size_t)ST_MAX_ROWS * 8;               // float  [ST_MAX_ROWS][128]
constexpr size_t SCRATCH_BYTES = OFF_PART_O + (size_t)ST_MAX_ROWS * 128 * 4;       // about 0.8 MB
static_assert(OFF_PART_O % 256 == 0, "scratch sections are 256-byte aligned");

// Every GPU that loads the library holds this array until the process exits.
static __device__ __align__(256) unsigned char g_static_scratch[SCRATCH_BYTES];

// What the calls need to know of a device, found once: a call among others takes no lock and asks the driver nothing.
struct StaticDevice {
  std::atomic<unsigned char *> scratch;   // device address of the array (in host code its name is only a stand-in); set last
  int n_sm;
  std::atomic<int> room[2][2][3];         // [group of more than 8][head_dim 128][k]: 1 + the clusters of 4 << k CTAs that fit at once, 0: not asked yet
};
StaticDevice g_devices[ST_MAX_DEVICES];

wnw_status_t current_device(int device, StaticDevice **out) {
  if (device < 0 || device >= ST_MAX_DEVICES) return WNW_ERR_INVALID_ARG;
  StaticDevice &dv = g_devices[device];
  if (!dv.scratch.load(std::memory_order_acquire)) {
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    void *p = nullptr;
    if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || !p) { cudaGetLastError(); return WNW_ERR_CUDA; }
    if (configure_attn_kernels() != cudaSuccess) { cudaGetLastError(); return WNW_ERR_CUDA; }  // shared-memory opt-in, no allocation
    int n_sm = 0;
    if (cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) { cudaGetLastError(); return WNW_ERR_CUDA; }
    if (!dv.scratch.load(std::memory_order_relaxed)) {
      dv.n_sm = n_sm;
      dv.scratch.store((unsigned char *)p, std::memory_order_release);
    }
  }
  *out = &dv;
  return WNW_OK;
}

// How the heads of a call are cut.  cluster: CTAs of a cluster that a head's pieces share; 0: the pieces meet in global memory.
struct StaticCut { int pieces, cluster; };

wnw_status_t check_shape(int n_tokens, int n_q_heads, int n_kv_heads, int head_dim) {
  if (n_q_heads < 1 || n_kv_heads < 1 || n_q_heads % n_kv_heads || n_tokens < 1) return WNW_ERR_INVALID_ARG;
  if (head_dim != 64 && head_dim != 128) return WNW_ERR_UNSUPPORTED;
  // beyond the fixed scratch: refuse rather than overrun
  if (n_kv_heads > ST_MAX_KV_HEADS || n_q_heads > ST_MAX_Q_HEADS || n_q_heads / n_kv_heads > MAX_G || n_tokens > ST_MAX_TOKENS) return WNW_ERR_CAPACITY;
  return WNW_OK;
}

wnw_status_t cut_heads(StaticDevice &dv, int n_tokens, int n_q_heads, int n_kv_heads, int head_dim, StaticCut *cut) {
  const int n_gran = (n_tokens + GR - 1) / GR, nw = attn_warps(false), g = n_q_heads / n_kv_heads;
  // Where a head would be split and its pieces of 16 granules fit a cluster, all heads' clusters on the GPU at once: they meet inside
  // the cluster instead of in global memory.  us a call among others, through global memory / in clusters: 4 KV heads of 64 (8 query
  // heads), 129 tokens 5.6 / 4.2, 777 5.6 / 4.3, 4096 8.9 / 4.4; 2 of 128 (16 query heads) 777 6.8 / 5.1, 4096 10.3 / 5.0.  Not one
  // piece a head (16 tokens 3.4 / 4.1), nor a second wave of clusters (8 KV heads of 128, 4096 tokens 8.6 / 9.7; 64 of 64 7.7 / 8.5).
  const int n_short = (n_gran + SHORT_GRANULES - 1) / SHORT_GRANULES, k = n_short <= 4 ? 0 : n_short <= 8 ? 1 : 2;
  if (n_gran > nw && n_short <= 16) {
    std::atomic<int> &room = dv.room[g > 8][head_dim == 128][k];
    int n = room.load(std::memory_order_acquire) - 1;
    if (n < 0) {   // (some 0.5 ms; threads that ask at the same time get the same answer)
      if (short_uniform_room(g, head_dim, 4 << k, &n) != cudaSuccess) { cudaGetLastError(); return WNW_ERR_CUDA; }
      room.store(n + 1, std::memory_order_release);
    }
    if (n_kv_heads <= n) { *cut = StaticCut{n_short, 4 << k}; return WNW_OK; }
  }
  // Every head in the same number of pieces: at least a granule for every warp of a CTA, one wave of CTAs (one fits an SM),
  // and no more partial rows than the scratch holds (binds only for one KV head with more than eight query heads).  All heads
  // are alike, so a CTA computes its piece from its index and no list is built or passed.  Before, at most 96 CTAs ran, what
  // a list in the kernel parameters held, behind a kernel that cleared counters: 50001 tokens x 8 heads 47.5 -> 40.9 us,
  // 777 tokens x 4 heads of 64: 13.1 -> 8.5 us.
  *cut = StaticCut{std::max(1, std::min({(n_gran + nw - 1) / nw, dv.n_sm / n_kv_heads, ST_MAX_ROWS / n_q_heads})), 0};
  return WNW_OK;
}

struct OnDevice {   // the device is current while this lives
  int prev = -1, dev;
  bool ok;
  explicit OnDevice(int device) : dev(device) {
    ok = cudaGetDevice(&prev) == cudaSuccess && (prev == device || cudaSetDevice(device) == cudaSuccess);
    if (!ok) cudaGetLastError();
  }
  ~OnDevice() { if (ok && prev != dev) cudaSetDevice(prev); }
};

}  // namespace

extern "C" wnw_status_t wnw_attend_static_status(int32_t device, void *cuda_stream, int32_t *timed_out) {
  if (!timed_out) return WNW_ERR_INVALID_ARG;
  OnDevice on(device);
  if (!on.ok) return WNW_ERR_CUDA;
  StaticDevice *dv = nullptr;
  const wnw_status_t rc = current_device(device, &dv);
  if (rc != WNW_OK) return rc;
  unsigned char *scr = dv->scratch.load(std::memory_order_relaxed);
  cudaStream_t st = (cudaStream_t)cuda_stream;
  int32_t word = 0;
  if (cudaMemcpyAsync(&word, scr + OFF_STATUS, sizeof(word), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaMemsetAsync(scr + OFF_STATUS, 0, sizeof(word), st) != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) {
    cudaGetLastError();
    return WNW_ERR_CUDA;
  }
  *timed_out = (word & STATUS_TIMEOUT) ? 1 : 0;
  return WNW_OK;
}

extern "C" wnw_status_t wnw_attend_static(const void *kv_dev, int32_t n_tokens, int32_t padded_tokens, const void *q_dev,
                                          void *out_dev, int32_t n_q_heads, int32_t n_kv_heads, int32_t head_dim,
                                          float softmax_scale, int32_t device, void *cuda_stream) {
  if (!kv_dev || !q_dev || !out_dev) return WNW_ERR_INVALID_ARG;
  if (n_tokens < 1 || padded_tokens < n_tokens || padded_tokens % GR) return WNW_ERR_INVALID_ARG;
  if (!(softmax_scale >= 0.f) || std::isinf(softmax_scale)) return WNW_ERR_INVALID_ARG;
  wnw_status_t rc = check_shape(padded_tokens, n_q_heads, n_kv_heads, head_dim);
  if (rc != WNW_OK) return rc;
  OnDevice on(device);
  if (!on.ok) return WNW_ERR_CUDA;
  StaticDevice *dv = nullptr;
  StaticCut cut;
  if ((rc = current_device(device, &dv)) != WNW_OK || (rc = cut_heads(*dv, n_tokens, n_q_heads, n_kv_heads, head_dim, &cut)) != WNW_OK) return rc;
  unsigned char *scr = dv->scratch.load(std::memory_order_relaxed);
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const int n_gran = (n_tokens + GR - 1) / GR;

  CacheView cv;
  memset(&cv, 0, sizeof(cv));
  Geometry &G = cv.geo;
  G.L = 1; G.Hq = n_q_heads; G.Hkv = n_kv_heads; G.d = head_dim; G.g = n_q_heads / n_kv_heads;
  G.nc = GR; G.ncp = GR; G.gpc = 1; G.topk = 0;
  G.T_cap_pad = GR; G.n_tg = 0;                        // no text region: every key comes from kv_dev
  G.C_max = padded_tokens / GR; G.S_max = 0; G.T_a_pad = padded_tokens;
  G.max_batch = 1;
  const double scale = softmax_scale > 0.f ? (double)softmax_scale : 1.0 / std::sqrt((double)head_dim);
  G.scale_log2 = (float)(scale * 1.4426950408889634);
  cv.status = reinterpret_cast<int32_t *>(scr + OFF_STATUS);   // where a bounded wait that ran out leaves its mark

  // descriptor of the caller's buffer (a host-side encode, no allocation); every role points at it
  TmaMaps maps;
  if (!encode_store_map(&maps.anchor, kv_dev, (unsigned long long)n_kv_heads * 2 * padded_tokens, head_dim, padded_tokens, 2)) return WNW_ERR_CUDA;
  maps.text = maps.pool = maps.fixed = maps.anchor;
  AttnArgs a{};
  a.maps = &maps;
  a.mode = ATTN_FULL; a.layer = 0; a.n_active = 1; a.has_new = 0; a.score_on = 0;
  a.uni = WorkItem{0, 0, 0, n_gran, 0, ROLE_ANCHOR, 0, n_tokens, n_gran, 0, 0, 0, cut.pieces};
  a.pdl = 1;   // the launch overlaps the tail of the preceding kernel; nothing is read before that has completed
  a.q = (const bf16 *)q_dev;
  a.anchor_base = (const bf16 *)kv_dev; a.anchor_seq_stride = 0; a.anchor_head0 = 0;
  a.part_o = reinterpret_cast<float *>(scr + OFF_PART_O);
  a.part_ml = reinterpret_cast<float2 *>(scr + OFF_PART_ML);
  a.gran_em = nullptr; a.n_aq = 1; a.n_ag_max = 1;
  a.head_done = reinterpret_cast<int32_t *>(scr + OFF_COUNTERS);
  a.head_mz = reinterpret_cast<float2 *>(scr + OFF_HEAD_MZ);
  a.out = (bf16 *)out_dev;
  a.cluster = cut.cluster;
  const cudaError_t e = cut.cluster ? launch_attn_short_uniform(cv, a, n_kv_heads, st) : launch_attn_uniform(cv, a, n_kv_heads, 1, st);
  if (e != cudaSuccess) { cudaGetLastError(); return WNW_ERR_CUDA; }
  return WNW_OK;
}

extern "C" wnw_status_t wnw_debug_attend_static_cluster(int32_t device, int32_t n_tokens, int32_t n_q_heads, int32_t n_kv_heads,
                                                        int32_t head_dim, int32_t *cluster) {
  if (!cluster) return WNW_ERR_INVALID_ARG;
  wnw_status_t rc = check_shape(n_tokens, n_q_heads, n_kv_heads, head_dim);
  if (rc != WNW_OK) return rc;
  OnDevice on(device);
  if (!on.ok) return WNW_ERR_CUDA;
  StaticDevice *dv = nullptr;
  StaticCut cut;
  if ((rc = current_device(device, &dv)) != WNW_OK || (rc = cut_heads(*dv, n_tokens, n_q_heads, n_kv_heads, head_dim, &cut)) != WNW_OK) return rc;
  *cluster = cut.cluster;
  return WNW_OK;
}
