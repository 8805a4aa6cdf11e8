// Chained or serial layers whose heads are cut into pieces of at most two granules a warp, the pieces of a head in one
// thread-block cluster or, of long heads, in several (PARTS): the layer's span is what counts (sm_100a).
//
// What bounds such a layer is a chain of latencies, not bytes (config 1 moves 4 MB a layer, 0.6 us of HBM): inputs visible, query
// into registers, K q^T, softmax, P V, merge over the warps, merge over the head's pieces, output.  The kernel of longer pieces (wnw_attn.cu) gives
// every warp the whole head_dim of its own tokens and merges eight warps' accumulators through shared memory.  Here the tokens are
// split over the warps for the first product alone and head_dim for the second, and what does not depend on the query is done
// ahead of it:
//   - before the inputs are waited for: the piece's bytes land, masked V rows are cleared, the fragments of K (the warp's own two
//     granules) and, one CTA to an SM, of V (the warp's 16 elements of head_dim, all tokens) sit in registers;
//   - behind them: 16 products from registers, the piece's maximum over one barrier, weights to shared memory (4 KB for all warps
//     instead of 32 KB of accumulators), a second barrier, 16 products of V with everybody's weights.  Nothing is merged over the
//     warps: a warp holds its share of head_dim complete and sends it to the pieces that finish it;
//   - (maximum, denominator) of the piece leave ahead of P V, so that the weights of the pieces are ready when the accumulators
//     arrive; the softmax-mass partials of anchor heads are added up while these travel.
// From the inputs to the output a piece takes 4 200 cycles: query 600 to 1 050 (near and far half of L2), K q^T 330 (mma.sync at its
// rate: 16 a warp, two warps a scheduler), softmax 650, P V 760, exchange 820, last sums 400.  30 chained layers of 3000
// tokens with the program's copies: 149 -> 136 us a step; the paper's form 207 -> 156; 16 query heads a KV head 235 -> 174.  Registers: wide
// forms 148 to 197, dense ones 107 to 120 (bounds 208 and 120; of those only the ones of 16 query heads a KV head of 64 spill, 12 bytes).
// tcgen05 does not pay here: with 8 to 16 query heads its M = 128, N = 16, K = 16 steps take 50 to 59 cycles each (485 to 567 for
// 128 tokens), where mma.sync needs 256 for 256 tokens with its operands in registers.
#include <mutex>
#include <set>
#include <tuple>

#include "wnw_attn_dev.cuh"
#include "wnw_internal.cuh"

namespace wnw {

namespace {

// DENSE: two CTAs to an SM, so that the layers behind this one start beside it: V fragments follow the K fragments into their
// registers, and at head_dim 128 V rows land in the place of the K rows (TWICE).  Else one CTA to an SM, both ahead of the query.
template <int D, bool G16, bool DENSE>
struct ShortShape {
  static constexpr bool TWICE = DENSE && D == 128;
  static constexpr bool V_AHEAD = !DENSE && !(G16 && D == 128);   // (the registers do not reach)
  static constexpr int NW = NW_LAT, HALVES = D / 64, HALFB = GR * 128, TILEB = HALVES * HALFB, STAGEB = TWICE ? TILEB : 2 * TILEB, KK = D / 16;
  static constexpr int V_AT = TWICE ? 0 : TILEB;   // V rows inside a stage
  static constexpr int NTN = G16 ? 2 : 1, HEADS = 8 * NTN, PPR = D / 8, QROW = D * 2 + 16;
  static constexpr int TILES = D / 16;             // 16-wide tiles of head_dim, one to a warp; with warps to spare (head_dim 64) ...
  static constexpr bool SPLIT_NT = TILES < NW && G16;   // ... the n-tiles are dealt over them too
  static constexpr int NTV = SPLIT_NT ? 1 : NTN;   // n-tiles of a warp's share of the second product
  // shared memory behind the stages (bytes): weights of the piece's tokens, units that arrive, (max, denominator) of the pieces
  static constexpr int STAGES_B = NW * 2 * STAGEB, P_B = NTN * NW * 32 * 16;
};

}  // namespace

// tokens x heads accumulators in units of four values as a lane holds them: heads 2p and 2p + 1 at d = 16 t + r and 16 t + r + 8.
// Unit u = p * D / 2 + 8 t + r; piece u % np finishes it, in place u / np of its receive buffer.
// UNI: the allocation-free call: all heads alike, one cluster each; a CTA's item follows from its index and nothing is chained.
template <int D, bool G16, bool TB, bool DENSE, bool PARTS, bool UNI>
__device__ __forceinline__ void short_body(const CacheView &cv, const AttnArgs &a, const TmaMaps &maps) {
  typedef ShortShape<D, G16, DENSE> X;
  constexpr int NW = X::NW, HALVES = X::HALVES, HALFB = X::HALFB, TILEB = X::TILEB, STAGEB = X::STAGEB, KK = X::KK, NTN = X::NTN, PPR = X::PPR,
                QROW = X::QROW, TILES = X::TILES, NTV = X::NTV;
  extern __shared__ unsigned char smem_raw[];
  unsigned char *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);   // the 128-byte swizzle wants 1024-byte stages
  const Geometry &G = cv.geo;
  const LayerInfo &li = a.li;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, bid = (int)blockIdx.x, g = G.g;
  if (UNI) asm volatile("griddepcontrol.wait;\n" ::: "memory");   // the caller's buffer may be what the preceding work wrote
  WorkItem it;
  if constexpr (UNI) {
    const int np = a.uni.hd_count, n = a.uni.g1, h = bid / a.cluster, x = bid - h * a.cluster;
    it = a.uni;
    it.h = it.ridx = h; it.hd_first = h * a.cluster; it.hd_count = x < np ? np : 0;
    it.g0 = (int)((long long)n * x / np); it.g1 = (int)((long long)n * (x + 1) / np);
  } else it = a.items[bid];           // the first load of the chain item -> granule -> bytes: on its way before anything else
  if (warp == NW - 1 && lane < 4)     // the copies' descriptors, beside it
    asm volatile("prefetch.tensormap [%0];\n" ::"l"(lane == 0 ? &maps.text : lane == 1 ? &maps.anchor : lane == 2 ? &maps.pool : &maps.fixed) : "memory");
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");   // (what later work may rely on: see attn_body)
  __shared__ __align__(8) unsigned long long bars[NW][2];        // one mbarrier per stage
  __shared__ __align__(8) unsigned long long cl_bars[2];         // bytes of the other pieces: (max, denominator); accumulators
  __shared__ float2 cl_m[NW][X::HEADS / 2], cl_l[NW][X::HEADS / 2];   // maximum, denominator of every warp and pair of heads
  __shared__ __align__(16) unsigned char new_k[D * 2];           // the K row of the token being generated
  __shared__ __align__(16) unsigned char cl_q[X::HEADS * QROW];  // the query, rows padded: ldmatrix reads eight of them without conflicts
  const uint32_t base = smem_u32(smem), my_base = base + (uint32_t)warp * 2 * STAGEB, p_base = base + X::STAGES_B;
  if (lane == 0) {
    mbar_init(smem_u32(&bars[warp][0]), 1);
    mbar_init(smem_u32(&bars[warp][1]), 1);
    if (warp == 0) { mbar_init(smem_u32(&cl_bars[0]), 1); mbar_init(smem_u32(&cl_bars[1]), 1); }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    fence_proxy_async();
  }
  __syncwarp();
  // the pieces' barriers exist before anything is sent to them: waited for ahead of the first send, long after
  asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
  // (the recall epochs a tidal item will ask for, read beside the item: the later acquire is then the only round trip left)
  const bool may_wait = a.wait_epoch != nullptr;
  int expect = 0;
  if (may_wait) expect = __ldcg(a.expect_epoch);
  auto finish = [&]() { if (bid == 0) asm volatile("griddepcontrol.wait;\n" ::: "memory"); };   // a completed kernel implies its predecessors
  if (it.hd_count == 0) {   // a place in the cluster without work
    asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    finish();
    return;
  }
  const int T_t = UNI ? 0 : cv.text_len[it.b] + a.has_new, ridx = it.ridx;
  if (!UNI && it.h == 0 && it.g0 == 0 && threadIdx.x == 0) cv.step_snap[(long long)it.b * G.L + a.layer] = cv.steps[it.b];
  const int parity = it.role == ROLE_TIDAL ? (int)(cv.steps[it.b] & 1) : 0;   // which copy of the slot table this step reads

  // ---- the warp's two granules: lane n holds granule n's descriptor and queues its copy ----
  const int j = it.g0 + warp + lane * NW;
  const bool mine = lane < 2 && j < it.g1;
  GranDesc gd;
  gd.row = 0; gd.meta = 0; gd.cid = -1; gd.off = 0; gd.score_idx = -1;
  if (mine) gd = decode_granule<TB, D>(cv, a, li, it, j, parity);
  const bool is_text = j < G.n_tg, base_blk = TB && gd.score_idx == -2;   // (base_blk: a tidal head's permanent token base, compact store)
  int m_full = 0, m_tail = 0;
  const int32_t *seg_kept = nullptr;
  if (TB && it.role == ROLE_TIDAL) {
    const int2 m = cv.tok_m[((long long)it.b * G.L + a.layer) * G.Hkv + it.h];
    m_full = m.x; m_tail = m.y;
    seg_kept = cv.seg_kept + ((long long)it.b * cv.tid_total + li.tid_prefix + it.ridx) * G.C_max;
  }
  auto rows_of = [&]() { return visible_rows<TB>(G, it, T_t, gd.meta, gd.cid, gd.off, j, m_full, m_tail, seg_kept); };
  auto map_of = [&]() -> const CUtensorMap * {
    return is_text ? &maps.text : base_blk ? &maps.fixed : it.role == ROLE_ANCHOR ? &maps.anchor : it.role == ROLE_TIDAL ? &maps.pool : &maps.fixed;
  };
  bool loaded = false, timed_out = false;
  auto copy = [&]() {
    const uint32_t bar = smem_u32(&bars[warp][lane]);
    mbar_expect_tx(bar, X::TWICE ? TILEB : STAGEB);
    if (X::TWICE) tma_load_rows(my_base + lane * STAGEB, map_of(), gd.row, 0, bar);
    else tma_load_granule(my_base + lane * STAGEB, map_of(), gd.row, bar);
    loaded = true;
  };
  auto queue = [&](bool now) {
    if (!mine || !now) return;
    if (gd.meta != -1 && gd.meta != -3) { if (gd.meta != 0) copy(); }    // the row is known: nothing loaded is waited for
    else if (gd.meta == -1 ? rows_of() > 0 : gd.cid >= 0) copy();        // the text length, the table entry
  };
  // Replayed steps: the slots may still be refilled by the recall behind the previous step; bounded wait for the layer's epoch word
  // before the first of them is fetched, other granules first.
  const bool slot = mine && !is_text && !base_blk;
  if (may_wait && it.role == ROLE_TIDAL && __any_sync(0xffffffffu, slot)) {
    queue(!slot);
    if (lane == 0) {
      const long long t0 = clock64();
      for (;;) {
        int seen;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];\n" : "=r"(seen) : "l"(a.wait_epoch) : "memory");
        if (seen >= expect) break;
        if (clock64() - t0 > 2000000000ll) { timed_out = true; break; }
      }
    }
    timed_out = __shfl_sync(0xffffffffu, (int)timed_out, 0) != 0;
    asm volatile("fence.proxy.async.global;\n" ::: "memory");   // the slots are read by TMA (async proxy)
    __syncwarp();
    queue(slot);
  } else {
    queue(true);
  }
  auto load_q = [&]() {
    if (threadIdx.x < g * PPR) {
      const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(a.q + ((long long)it.i * G.Hq + (long long)it.h * g) * D) + threadIdx.x);
      *reinterpret_cast<uint4 *>(cl_q + (threadIdx.x / PPR) * QROW + (threadIdx.x % PPR) * 16) = v;
    }
  };
  if (UNI) load_q();   // (nothing to wait for: beside the bytes)
  const int mtx = lane >> 3, r0 = lane >> 2, cq = (lane & 3) * 2;
  const int tile = warp % TILES, nt0 = X::SPLIT_NT ? warp / TILES : 0;   // this warp's share of the second product
  const bool pv = X::SPLIT_NT || warp < TILES;
  // ---- what the exchange needs, while the bytes are in flight ----
  const int new_j = a.has_new ? (T_t - 1) / GR : -1;               // the text granule that takes the row of the token being generated
  const bool new_here = new_j >= it.g0 && new_j < it.g1;           // (the same on every warp)
  const int new_x = new_here ? new_j - it.g0 : 0, new_w = new_x & (NW - 1), new_n = new_x / NW;
  const int np = it.hd_count, piece = bid - it.hd_first, GP = (g + 1) / 2, U = GP * (D / 2), slots = (U - piece + np - 1) / np;
  const uint32_t recv = p_base + X::P_B, ml_recv = recv + (uint32_t)(U + 16) * 16, ml_bar = smem_u32(&cl_bars[0]), o_bar = smem_u32(&cl_bars[1]);
  const uint32_t rank0 = (uint32_t)(it.hd_first % a.cluster);
  auto peer = [&](uint32_t addr, int to) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(addr), "r"(rank0 + to));
    return r;
  };
  auto send = [&](uint32_t dst, uint32_t bar, float x, float y, float z, float w) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];\n" ::"r"(dst), "f"(x), "f"(y), "f"(z),
                 "f"(w), "r"(bar) : "memory");
  };
  uint32_t o_dst[NTV], o_dbar[NTV], ml_dst = 0, ml_dbar = 0;
#pragma unroll
  for (int y = 0; y < NTV; ++y) {
    const int p = (nt0 + y) * 4 + (lane & 3), u = p * (D / 2) + tile * 8 + r0, slot_u = u / np, dest = u - slot_u * np;
    o_dst[y] = peer(recv + (uint32_t)(slot_u * np + piece) * 16, p < GP ? dest : 0);
    o_dbar[y] = peer(o_bar, p < GP ? dest : 0);
  }
  const int ml_to = warp * 8 + r0;   // the piece this lane tells (max, denominator)
  if (ml_to < np) { ml_dst = peer(ml_recv + (uint32_t)piece * 16, ml_to); ml_dbar = peer(ml_bar, ml_to); }   // + p * 256 for head pair p
  if (threadIdx.x == 0) {
    mbar_expect_tx(ml_bar, (uint32_t)(np * GP * 16));
    mbar_expect_tx(o_bar, (uint32_t)(np * slots * 16));
  }
  for (int x = threadIdx.x; x < (X::HEADS - g) * PPR; x += NW * 32)   // query heads beyond the group
    *reinterpret_cast<uint4 *>(cl_q + (g + x / PPR) * QROW + (x % PPR) * 16) = make_uint4(0, 0, 0, 0);
  asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");

  // ---- fragments that need no query ----
  // a lane's ldmatrix row address inside a 16 x 128-byte box with the 128-byte swizzle; a k-step is one XOR (see attn_body)
  const uint32_t lane_k = (uint32_t)((((mtx >> 1) << 3) + (lane & 7)) * 128 + (((mtx & 1) ^ (lane & 7)) << 4));
  const uint32_t lane_v = (uint32_t)((((mtx & 1) << 3) + (lane & 7)) * 128 + (((mtx >> 1) ^ (lane & 7)) << 4));
  const int vis_mine = mine ? rows_of() : 0;
  const unsigned in_flight = __ballot_sync(0xffffffffu, loaded);
  int vis[2], sidx[2];
  uint32_t kf[2][KK][4];
#pragma unroll
  for (int n = 0; n < 2; ++n) {
    vis[n] = __shfl_sync(0xffffffffu, vis_mine, n);
    sidx[n] = __shfl_sync(0xffffffffu, gd.score_idx, n);
    if ((in_flight >> n & 1u) && !mbar_wait(smem_u32(&bars[warp][n]), 0)) timed_out = true;
    // (masked K rows, and shared memory without a copy, only spoil logits that are replaced anyway)
#pragma unroll
    for (int kk = 0; kk < KK; ++kk) ldsm_x4(kf[n][kk], ((my_base + n * STAGEB + lane_k) ^ (uint32_t)(((2 * kk) & 7) << 4)) + (kk >> 2) * HALFB);
  }
  __syncwarp();
  if (X::TWICE) {
    if (loaded) {
      const uint32_t bar = smem_u32(&bars[warp][lane]);
      fence_proxy_async();   // the rows were read through the generic proxy
      mbar_expect_tx(bar, TILEB);
      tma_load_rows(my_base + lane * STAGEB, map_of(), gd.row, 1, bar);
    }
#pragma unroll
    for (int n = 0; n < 2; ++n)
      if ((in_flight >> n & 1u) && !mbar_wait(smem_u32(&bars[warp][n]), 1)) timed_out = true;
  }
  // rows past the visible ones get weight 0, but 0 x NaN is NaN and shared memory without a copy may hold anything: cleared
#pragma unroll
  for (int n = 0; n < 2; ++n)
    for (int r = vis[n] + (lane >> 3); r < GR; r += 4)
#pragma unroll
      for (int hf = 0; hf < HALVES; ++hf)
        asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};\n" ::"r"(my_base + n * STAGEB + X::V_AT + hf * HALFB + r * 128 + ((lane & 7) << 4)), "r"(0u) : "memory");
  const uint32_t v_base = base + X::V_AT + (tile >> 2) * HALFB + (lane_v ^ (uint32_t)(((2 * tile) & 7) << 4));
  uint32_t vf[NW][2][4];
  auto load_v = [&](int from, int to) {
#pragma unroll
    for (int w = 0; w < NW; ++w)
      if (w >= from && w < to)
#pragma unroll
        for (int n = 0; n < 2; ++n) ldsm_x4_t(vf[w][n], v_base + (uint32_t)(w * 2 + n) * STAGEB);
  };
  if (X::V_AHEAD) {
    __syncthreads();   // every warp's bytes are there, masked rows cleared
    if (pv) load_v(0, NW);
  }

  // ---- the inputs: lines asked into L2 (where the preceding work's stores land) ahead of the wait, loads past L1 behind it ----
  if (a.wait_inputs) {
    const char *qline = reinterpret_cast<const char *>(a.q + ((long long)it.i * G.Hq + (long long)it.h * g) * D);
    if (threadIdx.x * 128 < g * D * 2) asm volatile("prefetch.global.L2 [%0];\n" ::"l"(qline + threadIdx.x * 128));
    if (a.has_new && threadIdx.x < 2) {
      const bf16 *nb = (threadIdx.x ? a.v_new : a.k_new) + ((long long)it.i * G.Hkv + it.h) * D;
      asm volatile("prefetch.global.L2 [%0];\n" ::"l"(nb));
      if (D * 2 > 128) asm volatile("prefetch.global.L2 [%0];\n" ::"l"(reinterpret_cast<const char *>(nb) + 128));
    }
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
  }
  const int new_kv = lane / PPR, new_pc = lane - new_kv * PPR, nr = (T_t - 1) & (GR - 1);
  const bool new_mine = new_here && warp == new_w && lane < 2 * PPR;
  uint4 new_val = make_uint4(0, 0, 0, 0);
  if (new_mine) new_val = __ldcg(reinterpret_cast<const uint4 *>((new_kv ? a.v_new : a.k_new) + ((long long)it.i * G.Hkv + it.h) * D + new_pc * 8));
  if (!UNI) load_q();
  if (new_mine) {   // the row of the token being generated: V into its granule, K beside the query, both to the text region
    // (at once: a store still under way when the kernel ends holds up the next layer)
    *reinterpret_cast<uint4 *>(cv.text + text_off(G, it.b, a.layer, it.h, new_kv) + (long long)(T_t - 1) * D + new_pc * 8) = new_val;
    const uint32_t dst = new_kv ? my_base + new_n * STAGEB + X::V_AT + (new_pc >> 3) * HALFB + nr * 128 + (((new_pc & 7) ^ (nr & 7)) << 4)
                                : smem_u32(new_k) + new_pc * 16;
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(dst), "r"(new_val.x), "r"(new_val.y), "r"(new_val.z), "r"(new_val.w) : "memory");
  }
  __syncthreads();
  uint32_t qa[KK][2 * NTN];
#pragma unroll
  for (int kk = 0; kk < KK; kk += 2)
#pragma unroll
    for (int nt = 0; nt < NTN; ++nt) {
      uint32_t r[4];
      ldsm_x4(r, smem_u32(cl_q) + (uint32_t)((nt * 8 + (lane & 7)) * QROW + (kk * 2 + (lane >> 3)) * 16));
      qa[kk][2 * nt] = r[0]; qa[kk][2 * nt + 1] = r[1]; qa[kk + 1][2 * nt] = r[2]; qa[kk + 1][2 * nt + 1] = r[3];
    }

  if (new_here && warp == new_w && r0 == (nr & 7)) {   // K fragments were taken ahead of the new row: its lanes take it now
#pragma unroll
    for (int kk = 0; kk < KK; ++kk) {
      const uint32_t lo = *reinterpret_cast<const uint32_t *>(new_k + kk * 32 + cq * 2), hi = *reinterpret_cast<const uint32_t *>(new_k + kk * 32 + 16 + cq * 2);
#pragma unroll
      for (int n = 0; n < 2; ++n) {
        if (n == new_n && nr < 8) { kf[n][kk][0] = lo; kf[n][kk][1] = hi; }
        if (n == new_n && nr >= 8) { kf[n][kk][2] = lo; kf[n][kk][3] = hi; }
      }
    }
  }
  // ---- S^T = K q^T of the warp's own tokens; V fragments that were not taken ahead take the registers that the K fragments leave ----
  float sT[2][NTN][4], sO[2][NTN][4];   // even and odd k-steps: shorter dependent mma chains
#pragma unroll
  for (int n = 0; n < 2; ++n) {
#pragma unroll
    for (int kk = 0; kk < KK; ++kk)
#pragma unroll
      for (int nt = 0; nt < NTN; ++nt) {
        float(&acc)[4] = (kk & 1) ? sO[n][nt] : sT[n][nt];
        if (kk < 2) mma16816_z(acc, kf[n][kk][0], kf[n][kk][2], kf[n][kk][1], kf[n][kk][3], qa[kk][2 * nt], qa[kk][2 * nt + 1]);
        else mma16816(acc, kf[n][kk][0], kf[n][kk][2], kf[n][kk][1], kf[n][kk][3], qa[kk][2 * nt], qa[kk][2 * nt + 1]);
      }
    if (!X::V_AHEAD && pv) load_v(n * (NW / 2), (n + 1) * (NW / 2));
  }
  // ---- softmax of the warp's own tokens (log2 units, fp32), relative to the piece's maximum ----
  float v[NTN][2][4];
#pragma unroll
  for (int nt = 0; nt < NTN; ++nt) {
    float mA = -INFINITY, mB = -INFINITY;
#pragma unroll
    for (int n = 0; n < 2; ++n) {
      const bool lo = r0 < vis[n], hi = r0 + 8 < vis[n];
#pragma unroll
      for (int e = 0; e < 4; ++e) v[nt][n][e] = (e < 2 ? lo : hi) ? (sT[n][nt][e] + sO[n][nt][e]) * G.scale_log2 : -INFINITY;
      mA = fmaxf(mA, fmaxf(v[nt][n][0], v[nt][n][2])); mB = fmaxf(mB, fmaxf(v[nt][n][1], v[nt][n][3]));
    }
#pragma unroll
    for (int sh = 4; sh <= 16; sh <<= 1) {
      mA = fmaxf(mA, __shfl_xor_sync(0xffffffffu, mA, sh));
      mB = fmaxf(mB, __shfl_xor_sync(0xffffffffu, mB, sh));
    }
    if (r0 == 0) cl_m[warp][nt * 4 + (lane & 3)] = make_float2(mA, mB);
  }
  __syncthreads();
  if (X::V_AHEAD && new_here && pv) {   // (V fragments were taken ahead of the new row)
#pragma unroll
    for (int w = 0; w < NW; ++w)
#pragma unroll
      for (int n = 0; n < 2; ++n)
        if (w == new_w && n == new_n) ldsm_x4_t(vf[w][n], v_base + (uint32_t)(w * 2 + n) * STAGEB);
  }
  float M[NTN][2], eA[NTN][2], eB[NTN][2];   // the piece's maximum, this lane's share of the granules' softmax mass
#pragma unroll
  for (int nt = 0; nt < NTN; ++nt) {
    float mA = -INFINITY, mB = -INFINITY;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      const float2 m = cl_m[w][nt * 4 + (lane & 3)];
      mA = fmaxf(mA, m.x); mB = fmaxf(mB, m.y);
    }
    M[nt][0] = mA; M[nt][1] = mB;
    const float refA = mA > -INFINITY ? mA : 0.f, refB = mB > -INFINITY ? mB : 0.f;   // a piece without a visible token: all weights 0
#pragma unroll
    for (int n = 0; n < 2; ++n) {
      float(&x)[4] = v[nt][n];
      x[0] = ex2(x[0] - refA); x[2] = ex2(x[2] - refA);
      x[1] = ex2(x[1] - refB); x[3] = ex2(x[3] - refB);
      eA[nt][n] = x[0] + x[2]; eB[nt][n] = x[1] + x[3];
      // [token][8 heads]: ldmatrix hands it out transposed, as the second product's B operand
      const uint32_t dst = p_base + (uint32_t)((nt * NW + warp) * 2 + n) * 256 + (uint32_t)(r0 * 16 + cq * 2);
      asm volatile("st.shared.b32 [%0], %1;\n" ::"r"(dst), "r"(pack_bf16(x[0], x[1])) : "memory");
      asm volatile("st.shared.b32 [%0], %1;\n" ::"r"(dst + 128), "r"(pack_bf16(x[2], x[3])) : "memory");
    }
    float lA = eA[nt][0] + eA[nt][1], lB = eB[nt][0] + eB[nt][1];
#pragma unroll
    for (int sh = 4; sh <= 16; sh <<= 1) {
      lA += __shfl_xor_sync(0xffffffffu, lA, sh);
      lB += __shfl_xor_sync(0xffffffffu, lB, sh);
    }
    if (r0 == 0) cl_l[warp][nt * 4 + (lane & 3)] = make_float2(lA, lB);
  }
  __syncthreads();
  // ---- the piece's (max, denominator) to all pieces, by the first two warps ----
  if (ml_to < np) {
#pragma unroll
    for (int nt = 0; nt < NTN; ++nt) {
      float LA = 0.f, LB = 0.f;
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        const float2 l = cl_l[w][nt * 4 + (lane & 3)];
        LA += l.x; LB += l.y;
      }
      const int p = nt * 4 + (lane & 3);
      if (p < GP) send(ml_dst + (uint32_t)p * 256, ml_dbar, M[nt][0], LA, M[nt][1], LB);
    }
  }
  // ---- O^T = V^T P^T: this warp's 16 elements of head_dim over all tokens of the piece ----
  if (pv) {
#pragma unroll
    for (int y = 0; y < NTV; ++y) {
      float acc[4][4];   // independent chains
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        uint32_t pb[4];   // both granules' weights: tokens 0-7 | 8-15 of each x this lane's head
        ldsm_x4_t(pb, p_base + (uint32_t)(((nt0 + y) * NW + w) * 2) * 256 + (uint32_t)lane * 16);
#pragma unroll
        for (int n = 0; n < 2; ++n) {
          float(&c)[4] = acc[(w & 1) * 2 + n];
          if (w < 2) mma16816_z(c, vf[w][n][0], vf[w][n][2], vf[w][n][1], vf[w][n][3], pb[2 * n], pb[2 * n + 1]);
          else mma16816(c, vf[w][n][0], vf[w][n][2], vf[w][n][1], vf[w][n][3], pb[2 * n], pb[2 * n + 1]);
        }
      }
      float o[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) o[e] = (acc[0][e] + acc[1][e]) + (acc[2][e] + acc[3][e]);
      if ((nt0 + y) * 4 + (lane & 3) < GP) send(o_dst[y], o_dbar[y], o[0], o[1], o[2], o[3]);
    }
  }
  // ---- while the pieces' shares travel: softmax-mass partials per granule (fp32, before any bf16 rounding) of anchor-like heads ----
  if (sidx[0] >= 0 || sidx[1] >= 0) {
#pragma unroll
    for (int nt = 0; nt < NTN; ++nt)
#pragma unroll
      for (int n = 0; n < 2; ++n) {
#pragma unroll
        for (int sh = 4; sh <= 16; sh <<= 1) {
          eA[nt][n] += __shfl_xor_sync(0xffffffffu, eA[nt][n], sh);
          eB[nt][n] += __shfl_xor_sync(0xffffffffu, eB[nt][n], sh);
        }
        const int hq = nt * 8 + cq;
        if (r0 == 0 && sidx[n] >= 0 && vis[n] > 0) {
          float2 *ge = a.gran_em + ((long long)it.i * a.n_aq + (long long)ridx * g + hq) * a.n_ag_max + sidx[n];
          if (hq < g) ge[0] = make_float2(eA[nt][n], M[nt][0]);
          if (hq + 1 < g) ge[a.n_ag_max] = make_float2(eB[nt][n], M[nt][1]);
        }
      }
  }
  timed_out = __any_sync(0xffffffffu, timed_out);
  if (timed_out && lane == 0 && cv.status) atomicOr(cv.status, STATUS_TIMEOUT);

  const ItemPart pt = PARTS ? a.parts[bid] : ItemPart{0, 1, 0, 0};
  // ---- finish this piece's share: four lanes per unit, each adds up every fourth source ----
  // a peer may be late by its own bounded waits; these waits are long enough for all of them, so that nobody sends to a CTA that has left
  bool late = !mbar_wait_cluster(ml_bar, 0);
  bf16 *ob = a.out + ((long long)it.i * G.Hq + (long long)it.h * g) * D;
  const int src = threadIdx.x & 3;
  constexpr int XS = 4;
  for (int s0 = 0; s0 < slots; s0 += NW * 8) {
    const int slot = s0 + (threadIdx.x >> 2), u = slot * np + piece, p = u / (D / 2), td = u % (D / 2);
    const bool on = slot < slots;
    float4 f[XS];   // (max, denominator), then the weights of the sources
    float MA = -INFINITY, MB = -INFINITY, LA = 0.f, LB = 0.f;
#pragma unroll
    for (int x = 0; x < XS; ++x) {
      const int s = src + 4 * x;
      f[x] = make_float4(-INFINITY, 0.f, -INFINITY, 0.f);
      if (on && s < np)
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n" : "=f"(f[x].x), "=f"(f[x].y), "=f"(f[x].z), "=f"(f[x].w)
                     : "r"(ml_recv + (uint32_t)(p * 16 + s) * 16) : "memory");
      MA = fmaxf(MA, f[x].x); MB = fmaxf(MB, f[x].z);
    }
#pragma unroll
    for (int sh = 2; sh > 0; sh >>= 1) { MA = fmaxf(MA, __shfl_xor_sync(0xffffffffu, MA, sh)); MB = fmaxf(MB, __shfl_xor_sync(0xffffffffu, MB, sh)); }
    const float MA0 = MA > -INFINITY ? MA : 0.f, MB0 = MB > -INFINITY ? MB : 0.f;
#pragma unroll
    for (int x = 0; x < XS; ++x) {
      const float wA = ex2(f[x].x - MA0), wB = ex2(f[x].z - MB0);
      LA += f[x].y * wA; LB += f[x].w * wB;
      f[x].x = wA; f[x].z = wB;
    }
#pragma unroll
    for (int sh = 2; sh > 0; sh >>= 1) { LA += __shfl_xor_sync(0xffffffffu, LA, sh); LB += __shfl_xor_sync(0xffffffffu, LB, sh); }
    const float L = (src & 1) ? LB : LA, inv = L > 0.f ? 1.f / L : 0.f;
    if (s0 == 0) late = !mbar_wait_cluster(o_bar, 0) || late;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int x = 0; x < XS; ++x) {
      const int s = src + 4 * x;
      if (on && s < np) {
        float4 o;
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n" : "=f"(o.x), "=f"(o.y), "=f"(o.z), "=f"(o.w)
                     : "r"(recv + (uint32_t)(slot * np + s) * 16) : "memory");
        acc.x += o.x * f[x].x; acc.y += o.y * f[x].z; acc.z += o.z * f[x].x; acc.w += o.w * f[x].z;
      }
    }
    // lane e of the four ends up with value e of the unit and stores it
    const bool up = src & 2, odd = src & 1;
    float k0 = up ? acc.z : acc.x, k1 = up ? acc.w : acc.y;
    k0 += __shfl_xor_sync(0xffffffffu, up ? acc.x : acc.z, 2);
    k1 += __shfl_xor_sync(0xffffffffu, up ? acc.y : acc.w, 2);
    const float val = (odd ? k1 : k0) + __shfl_xor_sync(0xffffffffu, odd ? k0 : k1, 1);
    const int hq = 2 * p + (src & 1), dd = (td >> 3) * 16 + (td & 7) + (src >> 1) * 8;
    if (PARTS && pt.n > 1) {
      if (on && hq < g) {
        const long long row = (long long)(pt.base + pt.part) * g + hq;
        a.part_o[row * D + dd] = val;
        if (td == 0 && src < 2) a.part_ml[row] = make_float2(src ? MB : MA, L);
      }
    } else if (on && hq < g) {
      ob[hq * D + dd] = __float2bfloat16_rn(val * inv);
      if (td == 0 && src < 2) a.head_mz[(long long)it.i * G.Hq + it.h * g + hq] = make_float2(src ? MB : MA, L);
    }
  }
  if (late && threadIdx.x == 0 && cv.status) atomicOr(cv.status, STATUS_TIMEOUT);
  // ---- a head of several clusters: the piece that comes last adds up what the clusters left in global memory ----
  // (No cluster waits for another: two steps on two streams may hold a part of the machine each.)  Every thread's stores are ordered
  // before the barrier, thread 0's fence makes them visible device-wide before the head's counter moves.
  if (PARTS && pt.n > 1) {
    __shared__ int s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
      int *ctr = a.head_done + it.i * G.Hkv + it.h;
      __threadfence();
      s_last = atomicAdd(ctr, 1) == pt.pieces - 1;
      if (s_last) *ctr = 0;
    }
    __syncthreads();
    if (s_last) {
      constexpr int MB = 8;   // parts a batch of loads takes
      for (int x = threadIdx.x; x < g * (D / 4); x += NW * 32) {
        const int row = x / (D / 4), col = x % (D / 4);
        float m = -INFINITY, z = 0.f;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int c0 = 0; c0 < pt.n; c0 += MB) {
          float2 ml[MB];
          float4 o[MB];
          float mb = m;
#pragma unroll
          for (int c = 0; c < MB; ++c) {
            ml[c] = make_float2(-INFINITY, 0.f); o[c] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (c0 + c < pt.n) {
              const long long r = (long long)(pt.base + c0 + c) * g + row;
              ml[c] = __ldcg(a.part_ml + r);
              o[c] = __ldcg(reinterpret_cast<const float4 *>(a.part_o + r * D) + col);
            }
          }
#pragma unroll
          for (int c = 0; c < MB; ++c) mb = fmaxf(mb, ml[c].x);
          if (mb == -INFINITY) continue;   // nothing visible so far
          const float f0 = ex2(m - mb);    // (m = -inf on the first batch: 0)
          acc.x *= f0; acc.y *= f0; acc.z *= f0; acc.w *= f0; z *= f0;
#pragma unroll
          for (int c = 0; c < MB; ++c) {
            const float f = ex2(ml[c].x - mb);
            acc.x += o[c].x * f; acc.y += o[c].y * f; acc.z += o[c].z * f; acc.w += o[c].w * f;
            z += ml[c].y * f;
          }
          m = mb;
        }
        const float inv = z > 0.f ? 1.f / z : 0.f;
        *reinterpret_cast<uint2 *>(ob + row * D + col * 4) = make_uint2(pack_bf16(acc.x * inv, acc.y * inv), pack_bf16(acc.z * inv, acc.w * inv));
        if (col == 0) a.head_mz[(long long)it.i * G.Hq + it.h * g + row] = make_float2(m, z);
      }
    }
  }
  // after a timeout copies may still be in flight towards this CTA's shared memory: bounded wait before it is released
  if (timed_out && lane < 2 && loaded) mbar_wait(smem_u32(&bars[warp][lane]), X::TWICE ? 1 : 0);
  finish();
}

template <int D, bool G16, bool TB, bool DENSE, bool PARTS>
__global__ void __maxnreg__(DENSE ? 120 : 208) wnw_attn_short_kernel(const __grid_constant__ CacheView cv, const __grid_constant__ AttnArgs a,
                                                                     const __grid_constant__ TmaMaps maps) {
  short_body<D, G16, TB, DENSE, PARTS, false>(cv, a, maps);
}
template <int D, bool G16>
__global__ void __maxnreg__(208) wnw_attn_short_uniform_kernel(const __grid_constant__ CacheView cv, const __grid_constant__ AttnArgs a,
                                                               const __grid_constant__ TmaMaps maps) {
  short_body<D, G16, false, false, false, true>(cv, a, maps);
}

// ---- host: one list of the forms there are ----
namespace {

template <int D, bool G16, bool TB, bool DENSE, bool PARTS, bool UNI = false>
struct ShortForm {
  typedef ShortShape<D, G16, DENSE> X;
  static auto kernel() {
    if constexpr (UNI) return wnw_attn_short_uniform_kernel<D, G16>;
    else return wnw_attn_short_kernel<D, G16, TB, DENSE, PARTS>;
  }
  static size_t smem(int g) { return (size_t)X::STAGES_B + X::P_B + (size_t)((g + 1) / 2 * (D / 2) + 16) * 16 + 8 * 16 * 16 + 1024; }
  static void config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute (&attr)[2], int g, int n_ctas, int cluster, bool pdl, cudaStream_t st) {
    cfg.gridDim = dim3((unsigned)n_ctas, 1, 1);
    cfg.blockDim = dim3(NW_LAT * 32, 1, 1);
    cfg.dynamicSmemBytes = smem(g);
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cluster; attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = pdl ? 2 : 1;
  }
  static cudaError_t launch(const CacheView &cv, const AttnArgs &a, cudaStream_t st) {
    const TmaMaps *maps = X::TWICE ? a.maps_rows : a.maps;
    if (!maps || !a.cluster || a.n_items % a.cluster) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[2];
    config(cfg, attr, cv.geo.g, a.n_items, a.cluster, a.pdl, st);
    return cudaLaunchKernelEx(&cfg, kernel(), cv, a, *maps);
  }
  static cudaError_t configure() {
    const cudaError_t e = cudaFuncSetAttribute(kernel(), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem(G16 ? 16 : 8));
    return e != cudaSuccess ? e : cudaFuncSetAttribute(kernel(), cudaFuncAttributeNonPortableClusterSizeAllowed, 1);   // up to 16 CTAs
  }
  // The answer depends on what the kernel is allowed, so it is configured here and not left to whoever launches it.
  static cudaError_t cluster_room(int g, int cluster, int *n) {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[2];
    config(cfg, attr, g, cluster, cluster, false, nullptr);
    const cudaError_t e = configure();
    return e != cudaSuccess ? e : max_active_clusters((const void *)kernel(), cfg, n);
  }
  static bool leaves_recall_room(int g, int rt) { return recall_room((const void *)kernel(), NW_LAT * 32, smem(g), rt); }
};
// f: called with the form's ShortForm
template <bool TB, bool DENSE, bool PARTS, class F>
auto with_form_t(int g, int d, F f) {
  if (d == 128) return g > 8 ? f(ShortForm<128, true, TB, false, PARTS>{}) : f(ShortForm<128, false, TB, DENSE, PARTS>{});   // (two n-tiles at 128: one form)
  return g > 8 ? f(ShortForm<64, true, TB, DENSE, PARTS>{}) : f(ShortForm<64, false, TB, DENSE, PARTS>{});
}
template <class F>
auto with_form(int g, int d, bool tb, bool dense, bool parts, F f) {
  if (parts) {
    if (tb) return dense ? with_form_t<true, true, true>(g, d, f) : with_form_t<true, false, true>(g, d, f);
    return dense ? with_form_t<false, true, true>(g, d, f) : with_form_t<false, false, true>(g, d, f);
  }
  if (tb) return dense ? with_form_t<true, true, false>(g, d, f) : with_form_t<true, false, false>(g, d, f);
  return dense ? with_form_t<false, true, false>(g, d, f) : with_form_t<false, false, false>(g, d, f);
}

template <class F>
auto with_uniform_form(int g, int d, F f) {
  if (d == 128) return g > 8 ? f(ShortForm<128, true, false, false, false, true>{}) : f(ShortForm<128, false, false, false, false, true>{});
  return g > 8 ? f(ShortForm<64, true, false, false, false, true>{}) : f(ShortForm<64, false, false, false, false, true>{});
}

}  // namespace

// a.uni as for launch_attn_uniform, pieces of at most SHORT_GRANULES granules, a cluster of a.cluster CTAs a head
cudaError_t launch_attn_short_uniform(const CacheView &cv, AttnArgs a, int n_heads, cudaStream_t st) {
  const int np = a.uni.hd_count;
  if (np < 1 || np > a.cluster || a.cluster > 16 || a.uni.g1 > np * SHORT_GRANULES || n_heads < 1 || (cv.geo.d != 64 && cv.geo.d != 128)) return cudaErrorInvalidValue;
  a.n_items = n_heads * a.cluster;
  return with_uniform_form(cv.geo.g, cv.geo.d, [&](auto x) { return x.launch(cv, a, st); });
}
cudaError_t launch_attn_short(const CacheView &cv, const AttnArgs &a, cudaStream_t st) {
  if (cv.geo.kv8 || (cv.geo.d != 64 && cv.geo.d != 128)) return cudaErrorInvalidValue;
  return with_form(cv.geo.g, cv.geo.d, cv.geo.token_base != 0, a.short_pieces == SHORT_DENSE, a.parts != nullptr, [&](auto x) { return x.launch(cv, a, st); });
}
// Opt-in shared memory and cluster sizes, once per device: of the forms a cache of that shape uses (a kernel's first attribute call
// loads it: some 0.3 ms each).
cudaError_t configure_short_kernels(int device, int g, int d, bool token_base) {
  static std::mutex mu;
  static std::set<std::tuple<int, bool, int, bool>> done;
  std::lock_guard<std::mutex> lock(mu);
  const auto key = std::make_tuple(device, g > 8, d, token_base);
  if (done.count(key)) return cudaSuccess;
  cudaError_t e = cudaSuccess;
  for (int k = 0; k < 4 && e == cudaSuccess; ++k) e = with_form(g, d, token_base, k & 1, k & 2, [](auto x) { return x.configure(); });
  if (e == cudaSuccess) done.insert(key);
  return e;
}
// One answer for all groups that share a uniform form: 208 registers a thread hold an SM to one CTA.
cudaError_t short_uniform_room(int g, int d, int cluster, int *n) {
  return with_uniform_form(g, d, [&](auto x) { return x.cluster_room(g > 8 ? 16 : 8, cluster, n); });
}
cudaError_t short_cluster_room(int g, int d, bool token_base, bool dense, int cluster, int *n) {
  return with_form(g, d, token_base, dense, false, [&](auto x) { return x.cluster_room(g, cluster, n); });
}
bool short_leaves_recall_room(int g, int d, bool token_base, bool dense, int recall_threads) {
  return with_form(g, d, token_base, dense, false, [&](auto x) { return x.leaves_recall_room(g, recall_threads); }) &&
         with_form(g, d, token_base, dense, true, [&](auto x) { return x.leaves_recall_room(g, recall_threads); });
}

}  // namespace wnw
