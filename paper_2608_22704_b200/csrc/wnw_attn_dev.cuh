// Device pieces the attention kernels share: mbarriers, TMA copies of granules, ldmatrix / mma.sync wrappers, and the map from a
// head's virtual key space to the stores.
#pragma once
#include <cuda_fp16.h>

#include "wnw_internal.cuh"

namespace wnw {

constexpr int NW_LAT = 8;  // warps of a one-shot CTA (one work item each): 1 CTA per SM

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
// ---- mbarrier + TMA (every CTA fetches its own tiles) ----
__device__ __forceinline__ void mbar_init(uint32_t bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ uint32_t mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok;
}
// Bounded wait: gives up after about a second of SM clocks and reports it instead of hanging.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity))
    if (clock64() - t0 > 2000000000ll) return false;
  return true;
}
// The same for bytes that other CTAs of the cluster send, eight times as long (their own waits may have run out before).
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity) {
  for (const long long t0 = clock64();;) {
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    if (ok) return true;
    if (clock64() - t0 > 16000000000ll) return false;
  }
}
// One granule of a store: 16 rows from `row` on, K and V, both 64-element halves (see encode_store_map)
__device__ __forceinline__ void tma_load_granule(uint32_t dst, const CUtensorMap *map, int row, uint32_t bar) {
  asm volatile("cp.async.bulk.tensor.4d.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %3, %3}], [%2];\n"
               ::"r"(dst), "l"(map), "r"(bar), "r"(0), "r"(row) : "memory");
}
// K (kv 0) or V (kv 1) rows of a granule alone (maps with boxes of one of them)
__device__ __forceinline__ void tma_load_rows(uint32_t dst, const CUtensorMap *map, int row, int kv, uint32_t bar) {
  asm volatile("cp.async.bulk.tensor.4d.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %3, %5}], [%2];\n"
               ::"r"(dst), "l"(map), "r"(bar), "r"(0), "r"(row), "r"(kv) : "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }
__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void mma16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t *>(&v);
}

// 2^x in one instruction; results below the normal range come out as 0
__device__ __forceinline__ float ex2(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(r) : "f"(x));
  return r;
}

// The first product of a chain: the accumulator starts at zero
__device__ __forceinline__ void mma16816_z(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};\n"
               : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}
// (x, y) *= (a, b) in one instruction
__device__ __forceinline__ void mul2(float &x, float &y, float a, float b) {
  asm("{\n .reg .b64 p, q;\n mov.b64 p, {%0, %1};\n mov.b64 q, {%2, %3};\n mul.rn.f32x2 p, p, q;\n mov.b64 {%0, %1}, p;\n}\n" : "+f"(x), "+f"(y) : "f"(a), "f"(b));
}

// Two e4m3 bytes (low 16 bits of x) as two fp16 numbers: one instruction, exact (every e4m3 value is an fp16 value).
__device__ __forceinline__ uint32_t e4m3x2_to_f16x2(uint32_t x) {
  uint32_t h;
  asm("cvt.rn.f16x2.e4m3x2 %0, %1;\n" : "=r"(h) : "h"((unsigned short)x));
  return h;
}
__device__ __forceinline__ uint32_t pack_f16(float lo, float hi) {
  __half2 v = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<uint32_t *>(&v);
}
// bf16 pair -> fp16 pair: exact for magnitudes inside fp16's normal range
__device__ __forceinline__ uint32_t bf16x2_to_f16x2(uint32_t x) { return pack_f16(__uint_as_float(x << 16), __uint_as_float(x & 0xffff0000u)); }
__device__ __forceinline__ void mma16816_f16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                             uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

struct GranDesc {
  int row;         // first K row of the granule in its store (the store's tensor map knows how far its V row is)
  int meta;        // >= 0: visible tokens, known statically; -1: text granule, needs the text length; -2: needs `cid`;
                   // -3: needs `cid` and is not fetched at all when the slot is empty
  int cid;         // chunk id held by the slot / compact position (filled by a load that is not waited on here)
  int off;         // token offset of the granule inside its chunk
  int score_idx;   // audio granule index for score partials, -1 = none
  int ex;          // e4m3 tidal tier: K scale exponent | V scale exponent << 8 | 1 << 16 for a slot granule (filled with the metadata)
  bool loaded;     // a copy has been (or will be) queued
  uint32_t word;   // the granule's ring entry, once its metadata is resolved
  const CUtensorMap *map;
  int vis;         // visible rows, resolved with the first metadata of the descriptor's block of 32 granules
};

// Maps granule j of a head's virtual key space [text capacity | audio] to memory WITHOUT waiting on any global load:
// the row of every granule is static; what may be unknown yet is how many of its 16 rows are visible.
template <bool TB, int D>
__device__ __forceinline__ GranDesc decode_granule(const CacheView &cv, const AttnArgs &a, const LayerInfo &li,
                                                   const WorkItem &it, int j, int table_parity) {
  const Geometry &G = cv.geo;
  GranDesc r;
  r.cid = -1; r.off = 0; r.score_idx = -1; r.ex = 0; r.vis = 0; r.loaded = false; r.word = 0; r.map = nullptr;
  if (j < G.n_tg) {
    const int tok0 = j * GR;
    r.row = (int)(text_off(G, it.b, a.layer, it.h, 0) / D) + tok0;
    r.meta = tok0 + GR <= it.T_hint ? GR : -1;
    return r;
  }
  const int ag = j - G.n_tg, ci = ag / G.gpc, off = (ag - ci * G.gpc) * GR;
  r.off = off;
  if (it.role == ROLE_ANCHOR) {
    r.row = (int)(anchor_off(G, a.anchor_seq_stride, it.b, a.anchor_head0 + it.ridx, 0) / D) + ci * G.ncp + off;
    int len = it.T_a - ci * G.nc;
    if (len > G.nc) len = G.nc;
    len -= off;
    r.meta = len <= 0 ? 0 : (len < GR ? len : GR);
    if (a.score_on) r.score_idx = ag;
  } else if (TB && it.role == ROLE_TIDAL && ci < it.S) {
    // token-granular permanent base: the first it.S units of the head are blocks of its compact store
    const int head = G.F_fix + li.tid_prefix + it.ridx;
    r.row = (int)(compact_off(G, it.b, head, 0) / D) + ci * G.ncp + off;
    r.cid = cv.fixed_chunks[((long long)it.b * G.F_tot + head) * G.FB + ci];
    r.meta = -2;
    r.score_idx = -2;               // marks the compact store (its tensor map is not the pool's)
  } else if (it.role == ROLE_TIDAL) {
    const int slot = TB ? ci - it.S : ci;
    r.row = (int)(pool_off(G, li, it.b, slot, it.ridx, 0) / D) + off;
    r.cid = cv.slot_chunk[slot_table_off(G, table_parity, (long long)it.b * G.L + a.layer) + slot];
    // beyond the permanent slots a slot may be empty: its rows are fetched only if it is not
    r.meta = (TB || ci >= it.S) ? -3 : -2;
  } else {
    const long long fh = (long long)it.b * G.F_tot + li.fixed_off + it.ridx;
    r.row = (int)(fixed_off(G, li, it.b, it.ridx, 0) / D) + ci * G.ncp + off;
    r.cid = cv.fixed_chunks[fh * G.FB + ci];
    r.meta = -2;
  }
  return r;
}

// Visible rows of a granule of item `it` once its metadata has arrived (meta, cid, off: see GranDesc; j: its index in the head's
// virtual key space; T_t: text rows).  m_full, m_tail, seg_kept: what of a fetched segment lives in the head's token base already.
template <bool TB>
__device__ __forceinline__ int visible_rows(const Geometry &G, const WorkItem &it, int T_t, int meta, int cid, int off, int j, int m_full, int m_tail,
                                            const int32_t *seg_kept) {
  if (meta >= 0) return meta;
  int len;
  if (meta == -1) len = T_t - j * GR;
  else {
    if (cid == -1) return 0;
    if (cid < -1) len = -cid - 2;   // a block of a token-compacted fixed head: the entry carries its row count
    else {
      len = it.T_a - cid * G.nc;
      if (len > G.nc) len = G.nc;
      // token base: a fetched segment holds its complement first; the last segment has its own count
      if (TB) len -= m_full < 0 ? seg_kept[cid] : (it.T_a - cid * G.nc > G.nc) ? m_full : m_tail;
    }
    len -= off;
  }
  return len <= 0 ? 0 : (len < GR ? len : GR);
}

}  // namespace wnw
