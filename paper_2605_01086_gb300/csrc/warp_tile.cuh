// Shared machinery of the warp-tile kernels: tile constants and the per-window
// dequantization of the Table 1 shape N = 32, E = 16, per-domain tables in
// shared memory, the SymLen word decoder, the TMA store of 32-window output
// tiles, and two ways for a warp to decode its contiguous range of tiles:
//   * stream_tiles (decode_warp.cu, decode_shape.cuh): the range as one stream of
//     passes; a step of the transform runs whenever its symbols are there;
//   * decode_tile with its contexts and their asynchronous prefetch
//     (decode_tc.cu, decode_tcs.cu, backward_warp.cu): one tile after the other,
//     each starting at the word where the one before it ended.
// Either way the first tile of the range is located from the index's chunk
// offsets (symbol_word), and no record per tile is read.
#pragma once

#include <cuda.h>

#include "device_util.cuh"
#include "symlen_chunks.cuh"

namespace fptc {
namespace wt {

constexpr int kN = 32;
constexpr int kE = 16;
constexpr int kT = 128;                    // windows per tile
constexpr int kTS = kT * kE;               // symbols per tile
constexpr int kGuard = 64;                 // entries before and after the tile (a word holds <= 64 codewords)
constexpr int kStage = kTS + kGuard;       // level bytes per warp after the first-pass words (see kStageOff)
constexpr int kZStride = 257;              // floats per zone row (zero levels of the zones in different banks)
constexpr int kZRows = 2;                  // zone rows in shared memory: zone 2 reconstructs 0 without a row
constexpr uint32_t kDeqBytes = (kZRows * kZStride * 4 + 15) / 16 * 16;  // a domain's dequantization rows
constexpr int kWPL = 2;                    // consecutive words per lane per decode pass
constexpr int kPassWords = 32 * kWPL;
constexpr int kStepWin = 32;               // windows per transform step (one per lane)
constexpr int kOutTile = kStepWin * kN * 4;  // bytes of a step's output (TMA box 32 x 32 floats)
// Per warp: the first-pass words, then the level bytes.  The guard before tile
// position 0 is the last kGuard bytes of the first-pass words: those words are
// in registers before the decode writes there, and the next tile's words are
// requested only after it (decode_tile ends with a warp barrier).
constexpr int kMiscBytes = kPassWords * 8 + kStage;
constexpr int kStageOff = kPassWords * 8;  // tile position 0 from the start of the warp's area
static_assert(kGuard <= kPassWords * 8, "the guard before the tile lies inside the first-pass words");
static_assert(kStageOff % 16 == 0 && kMiscBytes % 16 == 0, "level rows are read as 16-byte vectors");
// zone mask of Table 1 (B1 = 2, B2 = 16): bins 0, 1 in zone 0, the rest in zone 1
constexpr uint32_t kZmaskTable1 = 0x55555550u;

// 32-byte streaming store (one full sector per thread)
__device__ __forceinline__ void st_cs_v8(float *p, const float (&v)[8]) {
  asm volatile("st.global.cs.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]), "f"(v[1]),
               "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}

// TMA tensor store of a staged 32 x 32-float tile to rows [row, row + 32) of
// the output, and the waits on it (bulk async-group of the issuing thread).
__device__ __forceinline__ void tma_store_rows(const CUtensorMap *map, const void *smem_tile, int32_t row) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(0), "r"(row), "r"(static_cast<uint32_t>(__cvta_generic_to_shared(smem_tile)))
               : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// ---- bounded mbarrier waits ---------------------------------------------------
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint32_t addr, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(addr), "r"(count) : "memory");
}
// One test of the phase of parity `parity`; the thread may be suspended up to
// hint_ns until that phase completes (it does not spin meanwhile).
__device__ __forceinline__ bool mbar_try_wait_for(uint32_t addr, uint32_t parity, uint32_t hint_ns) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(addr), "r"(parity), "r"(hint_ns)
      : "memory");
  return ok != 0;
}
constexpr uint64_t kWaitNs = 1000000000ull;  // a wait gives up after 1 s of global time
// Waits for the phase of parity `parity` of the mbarrier at addr, sleeping in
// try_wait between tests; false if it has not completed after kWaitNs.
__device__ __forceinline__ bool mbar_wait(uint32_t addr, uint32_t parity) {
  if (mbar_try_wait_for(addr, parity, 20000u)) return true;
  const uint64_t t0 = global_ns();
  do {
    if (mbar_try_wait_for(addr, parity, 1000000u)) return true;
  } while (global_ns() - t0 < kWaitNs);
  return false;
}

__device__ __forceinline__ void tma_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void tma_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_async_shared() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

struct DomW {
  uint32_t lut_off;   // bytes from the start of shared memory: 16-bit entries len | level << 8
  uint32_t deq_off;   // bytes: zone rows [kZRows][kZStride] floats (zones 0 and 1)
  uint32_t shift;     // 32 - lmax
  uint32_t zmask;     // zone of bin k at bits 2k..2k+1
  uint32_t complete;  // every prefix decodes (no zero entry)
  uint32_t pad[3];
};

// Codewords of one SymLen word, MSB first.  w's bits sit in hi:lo with a marker
// bit right under them (mk); each codeword shifts the 96 bits left by its
// length (the entry's low 5 bits: the funnel shifts use the amount mod 32).
// The marker leaves the buffer iff the codewords used more than 64 bits.
// CHECKED (incomplete code): an entry of length 0 marks a prefix with no
// codeword.  SHIFT: 32 - lmax when the caller knows it at compile time (the
// table index is then one shift-and-add), else 0 and `shift` holds it.
// Returns error flags.
template <bool CHECKED, uint32_t SHIFT = 0>
__device__ __forceinline__ uint32_t decode_word(uint64_t w, uint32_t n, uint8_t *__restrict__ dst,
                                                const uint16_t *__restrict__ lut, uint32_t shift) {
  uint32_t hi = (uint32_t)(w >> 32), lo = (uint32_t)w, mk = 0x80000000u;
  uint32_t low = 31u;
  auto step = [&]() -> uint32_t {
    const uint32_t e = lut[hi >> (SHIFT ? SHIFT : shift)];
    hi = __funnelshift_l(lo, hi, e);
    lo = __funnelshift_l(mk, lo, e);
    mk = __funnelshift_l(0u, mk, e);
    if (CHECKED) low = min(low, e & 31u);
    return e;
  };
  // levels go out two per 16-bit store where both are this word's
  uint32_t j = 0;
  if (n && (reinterpret_cast<uintptr_t>(dst) & 1u)) {
    dst[0] = (uint8_t)(step() >> 8);
    j = 1;
  }
  for (; j + 4 <= n; j += 4) {  // four codewords an iteration (less loop overhead per codeword)
    const uint32_t e0 = step();
    const uint32_t e1 = step();
    const uint32_t e2 = step();
    const uint32_t e3 = step();
    *reinterpret_cast<uint16_t *>(dst + j) = (uint16_t)__byte_perm(e0, e1, 0x0051);
    *reinterpret_cast<uint16_t *>(dst + j + 2) = (uint16_t)__byte_perm(e2, e3, 0x0051);
  }
  if (j + 2 <= n) {
    const uint32_t e0 = step();
    const uint32_t e1 = step();
    *reinterpret_cast<uint16_t *>(dst + j) = (uint16_t)__byte_perm(e0, e1, 0x0051);
    j += 2;
  }
  if (j < n) dst[j] = (uint8_t)(step() >> 8);
  return ((hi | lo | mk) == 0u ? kFlagBitOverrun : 0u) | ((CHECKED && low == 0u) ? kFlagInvalidCode : 0u);
}

// Where a tile's words are (first word, words that may belong to it, codewords
// of the first word that belong to the previous tile) and its segment.
struct Ctx {
  uint64_t fw;
  uint32_t nw;
  uint32_t skip;
  uint32_t seg;
  uint32_t ok;  // 0: segment flagged by the index, or no tile
};

// Context of a tile of segment s starting at word fw after `skip` symbols.  A
// tile holds at most kTS symbols and every word of a valid stream at least
// one, so it spans at most kTS + 1 words (fewer at the segment's end).
__device__ __forceinline__ Ctx make_ctx(const DecodeParams &p, uint32_t s, uint64_t fw, uint32_t skip) {
  Ctx c{fw, 0, skip, s, 0};
  if (p.seg_bad[s] != 0) return c;
  const SegDev &sg = p.segs[s];
  const uint64_t end = sg.word_offset + sg.n_words;
  c.nw = fw < end ? (uint32_t)min(end - fw, (uint64_t)kTS + 1u) : 0u;
  c.ok = 1;
  return c;
}

// Context of tile g of segment s (tiles of tile_syms symbols) located from the
// index (warp-collective).
__device__ __forceinline__ Ctx first_ctx(const DecodeParams &p, uint32_t s, uint64_t g, uint32_t lane,
                                         uint64_t tile_syms = kTS) {
  const SegDev &sg = p.segs[s];
  if (p.seg_bad[s] != 0) return Ctx{0, 0, 0, s, 0};
  const uint64_t tin = g - sg.tile_base;
  if (tin == 0) return make_ctx(p, s, sg.word_offset, 0u);
  const TileRec r = symbol_word(p.symlen, p.chunk_off, sg, tin * tile_syms, lane);
  if (r.pad != 0) return Ctx{0, 0, 0, s, 0};
  return make_ctx(p, s, r.first_word, r.skip);
}

// Where a decoded tile ended: the word (from the tile's first word) holding
// the next tile's first symbol and the symbols of it that were this tile's.
struct TileEnd {
  uint32_t bad;  // error flags (OR over the warp)
  uint32_t word;
  uint32_t skip;
};

// Context of tile g + 1 after tile g (segment s, context cur) ended at e.
__device__ __forceinline__ Ctx next_ctx(const DecodeParams &p, uint64_t g, uint32_t s, const Ctx &cur,
                                        const TileEnd &e) {
  if (g + 1 < p.segs[s].tile_base + p.segs[s].n_tiles) {
    if (!cur.ok) return Ctx{0, 0, 0, s, 0};
    return make_ctx(p, s, cur.fw + e.word, e.skip);
  }
  uint32_t s1 = s + 1;
  while (g + 1 >= p.segs[s1].tile_base + p.segs[s1].n_tiles) ++s1;  // segments without tiles
  return make_ctx(p, s1, p.segs[s1].word_offset, 0u);
}

// Words i0 + kWPL lane + u (u < kWPL) of a tile (zero beyond its word count).
__device__ __forceinline__ void load_pass(const DecodeParams &p, const Ctx &c, uint32_t i0, uint32_t lane,
                                          uint64_t (&w)[kWPL], uint32_t (&n)[kWPL]) {
#pragma unroll
  for (int u = 0; u < kWPL; ++u) {
    const uint32_t i = i0 + kWPL * lane + u;
    const bool in = c.ok && i < c.nw;
    w[u] = in ? __ldg(p.words + c.fw + i) : 0ull;
    n[u] = in ? (uint32_t)__ldg(p.symlen + c.fw + i) : 0u;
  }
}

__device__ __forceinline__ uint32_t smem_addr(const void *ptr) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(ptr));
}

// Asynchronous global -> shared copies (no register staging; completion by
// cp.async.wait_all in the copying thread).
__device__ __forceinline__ void cp_async8(void *dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(dst)), "l"(__cvta_generic_to_global(src))
               : "memory");
}
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(__cvta_generic_to_global(src))
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// First pass of a tile: words kWPL lane + u into wbuf (copies), their symbol
// counts packed one per byte into a register (zero beyond the tile's words).
__device__ __forceinline__ uint32_t fetch_pass0(const DecodeParams &p, const Ctx &c, uint32_t lane, uint64_t *wbuf) {
  uint32_t packed = 0;
#pragma unroll
  for (int u = 0; u < kWPL; ++u) {
    const uint32_t i = kWPL * lane + u;
    if (c.ok && i < c.nw) {
      cp_async8(wbuf + i, p.words + c.fw + i);
      packed |= (uint32_t)__ldg(p.symlen + c.fw + i) << (8 * u);
    }
  }
  cp_async_commit();
  return packed;
}

// A domain's decode table into shared memory with its entries' bytes swapped
// (len | level << 8), eight entries a load (the tables start on 16-byte boundaries).
template <int THREADS>
__device__ __forceinline__ void load_warp_lut(const uint16_t *g_lut, uint32_t lmax, unsigned char *dst) {
  const uint32_t entries = 1u << lmax;
  if (entries >= 8) {
    for (uint32_t i = threadIdx.x; i < entries / 8; i += THREADS) {
      const uint4 v = __ldg(reinterpret_cast<const uint4 *>(g_lut) + i);
      reinterpret_cast<uint4 *>(dst)[i] = make_uint4(__byte_perm(v.x, 0u, 0x2301), __byte_perm(v.y, 0u, 0x2301),
                                                     __byte_perm(v.z, 0u, 0x2301), __byte_perm(v.w, 0u, 0x2301));
    }
  } else {
    for (uint32_t i = threadIdx.x; i < entries; i += THREADS) {
      const uint32_t v = __ldg(g_lut + i);
      reinterpret_cast<uint16_t *>(dst)[i] = (uint16_t)((v >> 8) | ((v & 0xffu) << 8));
    }
  }
}

// Every domain's tables into shared memory from byte 0 (the layout of
// warp_smem_layout; offsets computed here, not indexed from a parameter
// block): the DomW array, then per domain the decode table (entries rewritten
// len | level << 8) and the dequantization rows.  Returns the end offset.
// Contains no barrier.
template <int THREADS>
__device__ __forceinline__ uint32_t load_domain_tables(const DecodeParams &p, uint32_t n_domains, unsigned char *smem) {
  DomW *const dw = reinterpret_cast<DomW *>(smem);
  uint32_t off = (uint32_t)align16(sizeof(DomW) * (n_domains ? n_domains : 1));
  for (uint32_t d = 0; d < n_domains; ++d) {
    const DomainDev &dm = p.domains[d];
    const uint32_t lut_off = off;
    const uint32_t deq_off = lut_off + (uint32_t)align16((size_t)2 << dm.lmax);
    off = deq_off + kDeqBytes;
    if (threadIdx.x == 0) {
      DomW x;
      x.lut_off = lut_off;
      x.deq_off = deq_off;
      x.shift = 32u - dm.lmax;
      uint32_t zm = 0;
      for (uint32_t k = 0; k < kE; ++k) zm |= (k < dm.B1 ? 0u : (k < dm.B2 ? 1u : 2u)) << (2 * k);
      x.zmask = zm;
      x.complete = dm.complete;
      x.pad[0] = x.pad[1] = x.pad[2] = 0;
      dw[d] = x;
    }
    load_warp_lut<THREADS>(p.luts + dm.lut_offset, dm.lmax, smem + lut_off);
    float a0 = p.scale ? p.scale[d * 3 + 0] : dm.scale[0];
    float a1 = p.scale ? p.scale[d * 3 + 1] : dm.scale[1];
    a0 = a0 > 1e-30f ? a0 : 0.0f;
    a1 = a1 > 1e-30f ? a1 : 0.0f;
    float *deq = reinterpret_cast<float *>(smem + deq_off);
    for (uint32_t i = threadIdx.x; i < (uint32_t)(kZRows * kZStride); i += THREADS) {
      const uint32_t z = i / kZStride, L = i - z * kZStride;
      deq[i] = L < 256u ? (z == 0 ? a0 : a1) * dm.unit[z][L] : 0.0f;
    }
  }
  return off;
}

// SymLen decode of one tile of `te` symbols (Sec. 4.2.1) into the level bytes
// at stage[0..): passes of two consecutive words per lane, a warp scan of their
// symbol counts, the codewords of each word at their tile positions (those of
// the previous tile go to the guard before the tile, those after the tile's
// last symbol to the guard after it).  The pass whose scan reaches te is the
// last: its words that start at or after te are left to the next tile, and the
// word holding symbol te is where the next tile starts.  w/n hold the first
// pass's words; each later pass is loaded while the one before it decodes.
// D: the domain's table view (lut_off, shift, complete).
template <class D>
__device__ __forceinline__ TileEnd decode_tile(const DecodeParams &p, const Ctx &cur, uint32_t te, const D &dd,
                                               const unsigned char *smem, uint8_t *stage, uint32_t lane,
                                               uint64_t (&w)[kWPL], uint32_t (&n)[kWPL]) {
  const uint16_t *lut = reinterpret_cast<const uint16_t *>(smem + dd.lut_off);
  int32_t base = -(int32_t)cur.skip;
  uint32_t bad = 0;
  TileEnd r{0u, 0u, 0u};
  for (uint32_t c0 = 0; c0 < cur.nw; c0 += kPassWords) {
    uint32_t tot = 0;
#pragma unroll
    for (int u = 0; u < kWPL; ++u) tot += n[u];
    uint32_t x = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= (uint32_t)o) x += y;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, x, 31);
    const int32_t p0 = base + (int32_t)(x - tot);  // tile position of this lane's first symbol
    const bool last = base + (int32_t)total >= (int32_t)te;
    uint64_t xw[kWPL];
    uint32_t xn[kWPL];
    if (!last && c0 + kPassWords < cur.nw) {
      load_pass(p, cur, c0 + kPassWords, lane, xw, xn);
    } else {
#pragma unroll
      for (int u = 0; u < kWPL; ++u) {
        xw[u] = 0;
        xn[u] = 0;
      }
    }
    if (last) {
      uint32_t hit = 0u, hw = 0u, hs = 0u;
      int32_t q = p0;
#pragma unroll
      for (int u = 0; u < kWPL; ++u) {
        const int32_t qe = q + (int32_t)n[u];
        if (!hit && q <= (int32_t)te && (int32_t)te < qe) {
          hit = 1u;
          hw = c0 + kWPL * lane + u;
          hs = (uint32_t)((int32_t)te - q);
        }
        if (q >= (int32_t)te) n[u] = 0u;
        q = qe;
      }
      const uint32_t m = __ballot_sync(0xffffffffu, hit);
      if (m) {
        const uint32_t src = (uint32_t)(__ffs(m) - 1);
        r.word = __shfl_sync(0xffffffffu, hw, src);
        r.skip = __shfl_sync(0xffffffffu, hs, src);
      } else {  // the tile ends with this pass's last word
        r.word = c0 + kPassWords;
        r.skip = 0u;
      }
    }
    uint8_t *dst = stage + p0;
    if (dd.complete && dd.shift == 20u) {  // L_max = 12, the trained tables' limit
#pragma unroll
      for (int u = 0; u < kWPL; ++u) {
        bad |= decode_word<false, 20u>(w[u], n[u], dst, lut, 20u);
        dst += n[u];
      }
    } else if (dd.complete) {
#pragma unroll
      for (int u = 0; u < kWPL; ++u) {
        bad |= decode_word<false>(w[u], n[u], dst, lut, dd.shift);
        dst += n[u];
      }
    } else {
#pragma unroll
      for (int u = 0; u < kWPL; ++u) {
        bad |= decode_word<true>(w[u], n[u], dst, lut, dd.shift);
        dst += n[u];
      }
    }
    if (last) break;
    base += (int32_t)total;
#pragma unroll
    for (int u = 0; u < kWPL; ++u) {
      w[u] = xw[u];
      n[u] = xn[u];
    }
  }
  r.bad = __reduce_or_sync(0xffffffffu, bad);
  __syncwarp();  // the guard before the tile is the first-pass words' area, refilled after this
  return r;
}

// The 16 coefficients A_z * unit_z(level) of a window from its 16 level bytes
// (Eq. 2 / Eq. 3 inverted by table: one shared-memory read per bin).
__device__ __forceinline__ void window_coefs(const uint4 &sv, const float *deq, uint32_t zmask, float (&c)[16]) {
  const uint32_t sw[4] = {sv.x, sv.y, sv.z, sv.w};
  if (zmask == kZmaskTable1) {
#pragma unroll
    for (int k = 0; k < 16; ++k) c[k] = deq[(k < 2 ? 0 : kZStride) + ((sw[k >> 2] >> (8 * (k & 3))) & 0xffu)];
  } else {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const uint32_t z = (zmask >> (2 * k)) & 3u;
      c[k] = z < 2u ? deq[z * kZStride + ((sw[k >> 2] >> (8 * (k & 3))) & 0xffu)] : 0.0f;  // zone 2: 0
    }
  }
}

// The window's levels to the caller's level buffer (16 bytes).
__device__ __forceinline__ void put_levels(uint8_t *dl, const uint4 &sv) {
  if ((reinterpret_cast<uintptr_t>(dl) & 15u) == 0) {
    *reinterpret_cast<uint4 *>(dl) = sv;
  } else {
    const uint32_t sw[4] = {sv.x, sv.y, sv.z, sv.w};
#pragma unroll
    for (int j = 0; j < 16; ++j) dl[j] = (uint8_t)(sw[j >> 2] >> (8 * (j & 3)));
  }
}

// A row of 32 samples from the staging tile (16-byte chunk c at c ^ (row & 7),
// sx = row & 7) to dst: m samples, 32-byte or 16-byte streaming stores where
// the alignment allows.
__device__ __forceinline__ void store_row(const unsigned char *row, uint32_t sx, float *dst, uint32_t m, bool vec32,
                                          bool vec16) {
  if (m == 32 && (vec32 || vec16)) {
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const float4 u = *reinterpret_cast<const float4 *>(row + (((2 * b) ^ sx) << 4));
      const float4 v = *reinterpret_cast<const float4 *>(row + (((2 * b + 1) ^ sx) << 4));
      if (vec32) {
        const float x[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
        st_cs_v8(dst + 8 * b, x);
      } else {
        __stcs(reinterpret_cast<float4 *>(dst + 8 * b), u);
        __stcs(reinterpret_cast<float4 *>(dst + 8 * b) + 1, v);
      }
    }
  } else {
    for (uint32_t n = 0; n < m; ++n)
      dst[n] = *reinterpret_cast<const float *>(row + ((((n >> 2) ^ sx) << 4) | ((n & 3u) << 2)));
  }
}

// ---- streaming decode -----------------------------------------------------------
// A warp's range of tiles, segment by segment, decoded as one stream of passes:
// a pass gives every lane two consecutive words, a scan of their symbol counts
// their places behind the symbols already in the warp's stage; whenever a step's
// symbols are there the caller's transform takes them, and what is left moves to
// the front.  Nothing is decoded twice or left idle where a tile ends, so the
// tile (the unit in which ranges are split) can be as small as a step.  The words
// of a pass are loaded while the pass before it decodes and its steps run.

constexpr int kStreamGuard = kGuard;  // bytes before (symbols of a unit's first word that are not its) and after the stage

// What a unit's passes and steps read of its segment.  In shared memory: beside
// 200 KB of tables and stages L1 keeps little, and a pass that read the segment
// record again waited for L2.
struct UnitSeg {
  int64_t word_end;
  uint64_t n_samples, out_offset, level_offset;
  uint32_t out_aligned;
  uint32_t caller_index;
  uint32_t pad[6];
};
static_assert(sizeof(UnitSeg) == 64, "a warp's streaming area keeps its 16-byte alignment");
__host__ __device__ constexpr int stream_bytes(int cap) { return (int)sizeof(UnitSeg) + 2 * kStreamGuard + cap; }
// A warp's streaming area: the unit's segment, guard, stage, guard.
constexpr int kStreamStage = (int)sizeof(UnitSeg) + kStreamGuard;

// Words of a pass: two consecutive words per lane, their counts n0 | n1 << 8.
struct PassWords {
  ulonglong2 w;
  uint32_t n;
};

// Words base + 2 lane, + 1 of [lo, hi) (zero outside).  base: a 16-byte boundary.
__device__ __forceinline__ PassWords load_pass_words(const DecodeParams &p, int64_t base, int64_t lo, int64_t hi,
                                                     uint32_t lane) {
  PassWords r{{0ull, 0ull}, 0u};
  const int64_t i = base + 2 * (int64_t)lane;
  if (base >= lo && base + kPassWords <= hi && (reinterpret_cast<uintptr_t>(p.symlen + base) & 1u) == 0) {
    r.w = __ldg(reinterpret_cast<const ulonglong2 *>(p.words + i));
    r.n = __ldg(reinterpret_cast<const uint16_t *>(p.symlen + i));
  } else {
    if (i >= lo && i < hi) {
      r.w.x = __ldg(p.words + i);
      r.n = __ldg(p.symlen + i);
    }
    if (i + 1 >= lo && i + 1 < hi) {
      r.w.y = __ldg(p.words + i + 1);
      r.n |= (uint32_t)__ldg(p.symlen + i + 1) << 8;
    }
  }
  return r;
}

// One pass's words of a lane into the level bytes at dst (their order).
template <class D>
__device__ __forceinline__ uint32_t decode_pair(const PassWords &c, uint32_t n0, uint32_t n1, uint32_t gap,
                                                uint8_t *dst, const uint16_t *lut, const D &dd) {
  uint32_t bad;
  if (dd.complete && dd.shift == 20u) {  // L_max = 12, the trained tables' limit
    bad = decode_word<false, 20u>(c.w.x, n0, dst, lut, 20u);
    bad |= decode_word<false, 20u>(c.w.y, n1, dst + gap, lut, 20u);
  } else if (dd.complete) {
    bad = decode_word<false>(c.w.x, n0, dst, lut, dd.shift);
    bad |= decode_word<false>(c.w.y, n1, dst + gap, lut, dd.shift);
  } else {
    bad = decode_word<true>(c.w.x, n0, dst, lut, dd.shift);
    bad |= decode_word<true>(c.w.y, n1, dst + gap, lut, dd.shift);
  }
  return bad;
}

// The tiles [t0, t1) (of T windows each, T = tile_windows(dd)) of a launch.
// stage: kStreamStage bytes into the warp's stream_bytes(CAP);
// step(sg, dd, levels, win, n): n windows of the unit's segment from window win, levels
// at `levels` (16-byte aligned where every step is a multiple of 16 symbols);
// step_windows(dd): windows of a whole step, whose symbols and a word's 64 are at
// most CAP.
// Barriers: step is entered with the levels visible to the warp; they are
// rewritten only after a warp barrier of stream_tiles itself, so a step needs
// none of its own behind its reads.
template <int CAP, class Dom, class Geo, class Step>
__device__ __forceinline__ void stream_tiles(const DecodeParams &p, uint64_t t0, uint64_t t1, const Dom *doms,
                                             const unsigned char *smem, uint8_t *stage, uint32_t lane, const Geo &geo,
                                             const Step &step) {
  const uint32_t odd = (uint32_t)(reinterpret_cast<uintptr_t>(p.words) >> 3) & 1u;  // word 0 is off a 16-byte boundary
  auto floor2 = [&](int64_t w) -> int64_t { return w - (int64_t)(((uint32_t)w + odd) & 1u); };
  uint32_t s = warp_find_segment(p.segs, p.seg_begin, p.seg_end, t0, lane);
  int64_t base;         // the pass's first word
  int32_t fill = 0;     // symbols in the stage (negative: those of the unit's first word before it)
  auto bad_segment = [&](uint32_t i) -> bool { return p.seg_bad[p.form_order ? p.segs[i].queue_index : i] != 0; };
  bool ok = !bad_segment(s);
  PassWords nx;
  {
    const SegDev &sg = p.segs[s];
    int64_t lo = (int64_t)sg.word_offset;
    if (ok && t0 != sg.tile_base) {
      const TileRec r = symbol_word(p.symlen, p.chunk_off, sg, (t0 - sg.tile_base) * geo.tile_symbols(doms[sg.domain]), lane);
      ok = r.pad == 0;
      lo = (int64_t)r.first_word;
      fill = -(int32_t)r.skip;
    }
    base = floor2(lo);
    nx = load_pass_words(p, base, lo, ok ? (int64_t)(sg.word_offset + sg.n_words) : lo, lane);
  }
  uint64_t t = t0;
  while (true) {
    // ---- a unit: the range's tiles of segment s, from tile t
    const SegDev &seg = p.segs[s];
    const Dom &dd = doms[seg.domain];
    UnitSeg &sg = *reinterpret_cast<UnitSeg *>(stage - kStreamStage);
    if (lane == 0) {
      sg.word_end = (int64_t)(seg.word_offset + seg.n_words);
      sg.n_samples = seg.n_samples;
      sg.out_offset = seg.out_offset;
      sg.level_offset = seg.level_offset;
      sg.out_aligned = seg.out_aligned;
      sg.caller_index = seg.caller_index;
    }
    __syncwarp();
    const uint32_t E = geo.bins(dd), sw = geo.step_windows(dd);
    uint64_t win = (t - seg.tile_base) * geo.tile_windows(dd);
    // windows of the unit left (a warp's share of what device memory holds fits 32 bits)
    uint32_t left;
    {
      const uint64_t seg_end = seg.tile_base + seg.n_tiles;
      left = (uint32_t)((t1 < seg_end ? (t1 - seg.tile_base) * geo.tile_windows(dd) : seg.n_windows) - win);
      t = t1 < seg_end ? t1 : seg_end;  // the next unit's first tile
    }
    uint32_t bad = 0;
    uint32_t s1 = s;   // the next unit's segment, its words and whether it is decoded
    int64_t lo1 = 0;
    bool ok1 = false;
    bool more = ok;
    auto next_segment = [&](int64_t &hi1) {
      do ++s1; while (t >= p.segs[s1].tile_base + p.segs[s1].n_tiles);  // segments without tiles
      lo1 = (int64_t)p.segs[s1].word_offset;
      hi1 = lo1 + (int64_t)p.segs[s1].n_words;
      ok1 = !bad_segment(s1);
      if (!ok1) hi1 = lo1;
    };
    if (!ok && t < t1) {  // a segment the index rejected: only the next unit's first words
      int64_t hi1;
      next_segment(hi1);
      nx = load_pass_words(p, floor2(lo1), lo1, hi1, lane);
    }
    while (more) {
      const PassWords cw = nx;
      uint32_t n0 = cw.n & 0xffu, n1 = cw.n >> 8;
      const uint32_t gap = n0, tot = n0 + n1;
      uint32_t x = tot;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= (uint32_t)o) x += y;
      }
      const int32_t after = fill + (int32_t)__shfl_sync(0xffffffffu, x, 31);
      const int32_t p0 = fill + (int32_t)(x - tot);  // place of the lane's first symbol
      // symbols from the stage's front to the unit's end (clipped: a pass adds 4096 at most)
      const int32_t rem = (int32_t)((left < 65536u ? left : 65536u) * E);
      const int64_t hi = sg.word_end;
      base += kPassWords;
      const int32_t upto = after < rem ? after : rem;  // symbols this pass completes, less where the stage is too small
      const bool last = (after >= rem || base >= hi) && upto <= CAP;
      int64_t hi1 = 0;
      if (last) {
        // words that start at or after the unit's end are not decoded
        if (p0 >= rem) n0 = 0u;
        if (p0 + (int32_t)gap >= rem) n1 = 0u;
        if (t < t1) next_segment(hi1);
        fill = upto;  // (an inconsistent stream can run out of words before its end)
      } else if (after > CAP) {
        // the words that fit; the next pass starts behind them
        const bool a0 = p0 + (int32_t)gap <= CAP, a1 = p0 + (int32_t)tot <= CAP;
        const uint32_t m0 = __ballot_sync(0xffffffffu, a0), m1 = __ballot_sync(0xffffffffu, a1);
        const uint32_t words = (uint32_t)(__popc(m0) + __popc(m1));
        fill = (int32_t)__shfl_sync(0xffffffffu, (uint32_t)(p0 + (int32_t)(words & 1u ? gap : tot)), (words - 1) >> 1);
        if (!a0) n0 = 0u;
        if (!a1) n1 = 0u;
        const int64_t lo = base - kPassWords + words;
        base = floor2(lo);
        nx = load_pass_words(p, base, lo, hi, lane);
      } else {
        fill = after;
        nx = load_pass_words(p, base, base, hi, lane);
      }
      bad |= decode_pair(cw, n0, n1, gap, stage + p0, reinterpret_cast<const uint16_t *>(smem + dd.lut_off), dd);
      if (last && t < t1) nx = load_pass_words(p, floor2(lo1), lo1, hi1, lane);
      __syncwarp();
      // ---- the steps that are complete
      int32_t off = 0;
      const int32_t need = (int32_t)(sw * E);
      while (fill - off >= need || (last && off < fill)) {
        const uint32_t n = left < sw ? left : sw;
        step(sg, dd, stage + off, win, n);
        win += n;
        left -= n;
        off += need;
      }
      more = !last;
      if (more && off) {  // the symbols left, to the front
        __syncwarp();  // over levels the step has just read: not every step ends with a barrier (lane stores)
        const int32_t r = fill - off;  // fewer than a step's, so the two places do not overlap
        if ((off & 15) == 0) {
          for (int32_t at = 16 * (int32_t)lane; at < r; at += 512)
            *reinterpret_cast<uint4 *>(stage + at) = *reinterpret_cast<const uint4 *>(stage + off + at);
        } else {  // a step that is not a multiple of 16 symbols
          for (int32_t at = (int32_t)lane; at < r; at += 32) stage[at] = stage[off + at];
        }
        fill = r;
      }
      __syncwarp();
    }
    bad = __reduce_or_sync(0xffffffffu, bad);
    if (bad && lane == 0) flag_bad(p.status, bad, sg.caller_index);
    if (t >= t1) break;
    __syncwarp();  // the unit's segment has been read
    s = s1;
    ok = ok1;
    base = floor2(lo1);
    fill = 0;
  }
}

// The warp's tile range of a launch, for tiles handed out `per` at a time to
// `units` units (warps, or warpgroups of `per` warps).
__device__ __forceinline__ void unit_tiles(const DecodeParams &p, uint64_t unit, uint64_t units, uint64_t &t0,
                                           uint64_t &t1) {
  const uint64_t n_all = p.tile_end - p.tile_begin;
  t0 = p.tile_begin + n_all * unit / units;
  t1 = p.tile_begin + n_all * (unit + 1) / units;
}

}  // namespace wt
}  // namespace fptc
