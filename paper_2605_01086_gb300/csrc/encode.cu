// The FPTC encoder on the GPU (include/fptc_encoder.h): Eq. 1, the three-zone
// quantizer of Sec. 3.2 and the SymLen packing of Alg. 1 for many streams.
//
//   k_enc_levels_w32  (every domain N = 32, E = 16) one thread per window: the
//                 window's 16 bins of Eq. 1 by the even/odd butterfly in FP32
//                 (dct32.cuh) with a bound on its error, and the zone
//                 quantizer bracketed by that bound.
//   k_enc_levels_any  (other shapes) a warp per tile of windows, folded once
//                 by the mirror symmetry of the basis: four windows by four
//                 bins per lane in FP32 with a bound on the sums' error.
//   k_enc_levels_bins  (other shapes, streams of a window or a few bins, where
//                 there are many or no others) one thread per bin.
//                 In all, every zone map is monotone in the coefficient, so
//                 when the levels at c - err and c + err agree the FP64
//                 coefficient (which lies between) has that level too;
//                 otherwise the bin goes to a list that k_enc_fallback
//                 computes again in FP64 (products and sums rounded
//                 separately, in sample order, then scaled by 2/N, as the host
//                 encoder does), one bin per lane, and quantizes from that.
//   k_enc_short  one lane per short stream, where there are very many: its
//                 words, one after the other.  The other streams:
//   k_enc_starts  one warp per packing block of kPackBlock symbols: where
//                 words start in it (Alg. 1), as a bitmap of its symbols.
//   k_enc_scan    one warp per stream: the words before each block; the
//                 stream's word count, room and code checks.
//   k_enc_pack    one warp per 2048 symbols, one lane per word: the words'
//                 codewords put together and written, with their counts.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <limits>
#include <memory>
#include <vector>

#include "dct32.cuh"
#include "device_util.cuh"
#include "fptc_codec.h"
#include "fptc_encoder.h"
#include "fptc_internal.h"
#include "host_util.h"

namespace fptc {
namespace {

constexpr uint32_t kPackBlock = 8192;            // symbols per packing block
constexpr uint32_t kMaskWords = kPackBlock / 32;  // words of its bitmap of word starts

struct EncDomain {
  uint32_t N, E, B1, B2;
  uint32_t cos_off;   // first entry of the E x N cosine tables (FP64 and FP32 copies)
  // FP32 forms for the fast evaluation of the quantizer
  float A0f, A1f, muf, d1f, inv_A0f, inv_span1f, inv_log1pmuf;
  float slack0, slack1;  // per zone: an input width that covers the FP32 evaluation error
  uint32_t on0, on1;     // A0 > 1e-30; A1 > 1e-30 and A1 > d1 (as the FP64 quantizer tests them): the zone is in use
  // zone 1 in units of the unscaled sum (c N / 2), for the window kernel's
  // branch-free first tier: d1, A1, slack1 scaled by N / 2 (exactly, N = 32),
  // and 126 / (A1 - d1), 127 / (A1 - d1) scaled by 2 / N
  float u1_d1, u1_A1, u1_slack, u1_kp, u1_kn;
  // zone 1's linear map may be evaluated in FP32 (A1 - d1 >= 2^-12 A1): the
  // FP32 roundings of A1 and d1 (2^-24 A1 each) then move the map's top by at
  // most 126 2^-23 / 2^-12 = 0.06 of a level; otherwise FP64 decides every
  // zone-1 bin outside the deadzone
  uint32_t z1_f32;
  uint32_t dot_off;      // first of its cosines in rows of any_pairs4(N) (k_enc_levels_any)
  float two_over_n;
  uint32_t bnd_off;      // first of the domain's 2 x 255 boundaries of the host encoder's zone maps
};

struct EncSeg {
  uint64_t in_offset;   // first sample in d_x
  uint64_t n_samples;
  uint64_t word_offset;
  uint64_t room;
  uint64_t level_offset;
  uint64_t n_windows;
  uint64_t block_base;  // first global packing block (not of a stream k_enc_short packs)
  uint32_t domain;
  uint32_t pad;
};

struct EncStatus {
  unsigned int flags;
  unsigned int pad;
  unsigned long long first_bad;
};

struct PackRec;
struct EncUnit;
struct EncBins;

struct EncParams {
  const float *x;
  uint64_t *words;
  uint8_t *symlen;
  uint64_t *n_words;
  uint8_t *levels;
  const EncSeg *segs;
  const EncDomain *doms;
  const double *cosv;
  const float *cosf;
  PackRec *recs;         // per packing block: its words and states
  uint32_t *masks;       // per packing block: kMaskWords words, where words start in it
  uint64_t *first_word;  // per packing block: the stream's words that start before it
  const uint32_t *block_seg;  // per packing block: its segment
  const uint32_t *code_tab;   // per domain, 256 entries: codeword << (32 - length) | length, 0: no codeword
  const uint32_t *short_seg;  // k_enc_short: its streams
  uint64_t n_short;
  const uint32_t *scan_seg;   // k_enc_scan: the others, or null: every stream
  uint64_t n_scan;
  const EncUnit *units;       // k_enc_levels_any: the windows of each warp
  const float *dots;          // and its cosines
  const EncBins *bins;        // k_enc_levels_bins: its streams
  const uint32_t *bin_first;  // and of every 32 of their bins the first one's entry
  uint32_t n_bin_segs, n_bins;
  const uint32_t *lv_seg;     // k_enc_levels_w32: the segment of each warp's first window
  const long long *bound_keys;  // per domain: zone 0's, then zone 1's 255 level boundaries (order keys)
  uint32_t n_doms;
  uint32_t *seg_bad;
  unsigned long long *fb_list;   // bins whose level the FP64 coefficient decides
  unsigned int *fb_count;
  uint32_t fb_cap;
  EncStatus *status;
  uint64_t n_segs;
  uint64_t n_levels;
  uint64_t n_blocks;
};

__device__ __forceinline__ void enc_flag(EncStatus *st, unsigned int f, uint64_t seg) {
  atomicOr(&st->flags, f);
  atomicMin(&st->first_bad, (unsigned long long)seg);
}

// The host encoder's FP64 map of a zone (Eq. 2 or Eq. 3) is given as its 255
// ascending boundaries (the smallest double with level L or more, L = 1 ..
// 255, computed on the host from the host encoder's own map), stored as
// order keys: signed 64-bit integers that order like the doubles (the
// magnitude bits of a negative double flipped; a level no double reaches has
// the largest key), so that comparisons run on the integer pipe.  The level
// of a non-NaN c is the number of keys <= key(c).
__device__ __forceinline__ long long order_key(double c) {
  const long long b = __double_as_longlong(c);
  return b < 0 ? b ^ 0x7fffffffffffffffll : b;
}

__device__ __forceinline__ uint32_t level_by_keys(const long long *kb, long long kc) {
  uint32_t n = 0;
#pragma unroll
  for (uint32_t step = 128; step; step >>= 1)
    if (n + step <= 255u && __ldg(kb + n + step - 1) <= kc) n += step;
  return n;
}

__device__ __forceinline__ const long long *zone_keys(const EncParams &p, const EncDomain &d, uint32_t k) {
  return p.bound_keys + d.bnd_off + (k < d.B1 ? 0u : 255u);
}

// The host encoder's level of bin k for its FP64 coefficient c.
__device__ __forceinline__ uint32_t bin_level(const EncParams &p, uint32_t k, double c, const EncDomain &d) {
  if (k >= d.B2 || isnan(c)) return 128u;
  return level_by_keys(zone_keys(p, d, k), order_key(c));
}

// The level of bin k when the FP64 coefficient lies within err of cd: level
// L0 (an estimate) when both ends of [cd - err, cd + err] lie between
// boundaries L0 - 1 and L0 (two loads), else the map's level at both ends (the
// map is monotone); false when those differ or cd is not finite (the FP64
// coefficient decides).
__device__ __forceinline__ bool level_bracket64(const EncParams &p, uint32_t k, double cd, double err,
                                                uint32_t L0, const EncDomain &d, uint32_t &L) {
  if (k >= d.B2) {
    L = 128u;
    return true;
  }
  const double e = err + fabs(cd) * 0x1p-50;  // and the rounding of cd -+ e
  if (!(fabs(cd) + e <= 1.0e300)) return false;
  const long long *kb = zone_keys(p, d, k);
  const long long lo = order_key(cd - e), hi = order_key(cd + e);
  if ((L0 == 0u || __ldg(kb + L0 - 1) <= lo) && (L0 == 255u || hi < __ldg(kb + L0))) {
    L = L0;
    return true;
  }
  const uint32_t l0 = level_by_keys(kb, lo), l1 = level_by_keys(kb, hi);
  L = l0;
  return l0 == l1;
}

// Zone 0's map evaluated in FP32 (reciprocals, log1pf): off from the FP64
// evaluation by less than the zone's slack in the coefficient (both are close
// to the exact monotone map), so used only to bracket it.
__device__ __forceinline__ uint32_t zone0_level32(float c, const EncDomain &d) {
  if (!d.on0 || isnan(c)) return 128u;
  const float a = fminf(fabsf(c), d.A0f);
  const float q = log1pf(d.muf * (a * d.inv_A0f)) * d.inv_log1pmuf;
  const int v = c >= 0.0f ? 128 + (int)floorf(fmaf(127.0f, q, 0.5f)) : 128 - (int)floorf(fmaf(128.0f, q, 0.5f));
  return (uint32_t)(v < 0 ? 0 : (v > 255 ? 255 : v));
}

// A level near the FP32 coefficient c (the FP32 map at c; a start for
// level_bracket64, which checks it).
__device__ __forceinline__ uint32_t level_estimate(uint32_t k, float c, const EncDomain &d) {
  if (k >= d.B2) return 128u;
  if (k < d.B1) return zone0_level32(c, d);
  const float a = fabsf(c);
  if (!d.on1 || isnan(c) || a <= d.d1f) return 128u;
  const float r = fminf((fminf(a, d.A1f) - d.d1f) * d.inv_span1f, 1.0f);
  const int v = c > 0.0f ? 129 + (int)floorf(fmaf(r, 126.0f, 0.5f)) : 127 - (int)floorf(fmaf(r, 127.0f, 0.5f));
  return (uint32_t)(v < 0 ? 0 : (v > 255 ? 255 : v));
}

// Zone 1 decided in FP32 alone from c with |c - c64| <= m - slack1 (the first
// tier of the level kernels): the deadzone test against d1 rounded to FP32
// (|d1f - d1| <= 2^-24 A1, far inside the slack A1 2^-20 that m carries), then
// the linear map at both ends of the bracket.  Returns false when the bin has
// to be decided more closely.
__device__ __forceinline__ bool zone1_decide32(float c, float m, const EncDomain &d, uint32_t &L) {
  if (!d.on1 || isnan(c)) {
    L = 128u;
    return true;
  }
  const float a = fabsf(c);
  if (a + m < d.d1f) {
    L = 128u;
    return true;
  }
  if (a - m <= d.d1f || !d.z1_f32) return false;  // at the deadzone edge, or FP32 cannot map it
  const float k = c > 0.0f ? 126.0f : 127.0f;
  const float r0 = fmaxf((fminf(a - m, d.A1f) - d.d1f) * d.inv_span1f, 0.0f);
  const float r1 = fmaxf((fminf(a + m, d.A1f) - d.d1f) * d.inv_span1f, 0.0f);
  const int v0 = (int)floorf(fmaf(r0, k, 0.5f)), v1 = (int)floorf(fmaf(r1, k, 0.5f));
  if (v0 != v1) return false;
  const int v = c > 0.0f ? 129 + v0 : 127 - v0;
  L = (uint32_t)(v < 0 ? 0 : (v > 255 ? 255 : v));
  return true;
}

// Level of bin g (global level index) of segment s from the FP64 coefficient,
// computed as the host encoder does: products and sums rounded separately, in
// sample order, then scaled by 2/N.
__device__ __forceinline__ uint32_t level_fp64_seg(const EncParams &p, uint64_t g, uint64_t s) {
  const EncSeg sg = p.segs[s];
  const EncDomain d = p.doms[sg.domain];
  const uint64_t local = g - sg.level_offset;
  const uint64_t w = local / d.E;
  const uint32_t k = (uint32_t)(local - w * d.E);
  const uint64_t avail = sg.n_samples - w * d.N;
  const float *src = p.x + sg.in_offset + w * d.N;
  const double *row = p.cosv + d.cos_off + (size_t)k * d.N;
  double a64 = 0.0;
  for (uint32_t n = 0; n < d.N; ++n) a64 = __dadd_rn(a64, __dmul_rn(n < avail ? (double)src[n] : 0.0, row[n]));
  return bin_level(p, k, __dmul_rn(a64, 2.0 / (double)d.N), d);
}

// FP64 list entries: level index (bits 0-39) and segment (bits 40-63).
__device__ __forceinline__ unsigned long long fb_entry(uint64_t g, uint64_t s) {
  return (unsigned long long)(g | (s << 40));
}
// A slot of the FP64 list for this thread, one atomic per warp (the lanes
// that call it at the same time share it); ~0u when the list is full.
__device__ __forceinline__ unsigned int fb_slot(const EncParams &p) {
  const uint32_t am = __activemask();
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t leader = (uint32_t)(__ffs(am) - 1);
  unsigned int base = 0;
  if (lane == leader) base = atomicAdd(p.fb_count, (unsigned int)__popc(am));
  base = __shfl_sync(am, base, leader);
  const unsigned int slot = base + (unsigned int)__popc(am & ((1u << lane) - 1u));
  return slot < p.fb_cap ? slot : ~0u;
}

// First tier of k_enc_levels_w32 for the 16 bins of a window: levels into lv,
// the bins the bound cannot settle into the mask undecided (their level 0).
// T1: the zones of Table 1 (B1 = 2, B2 = 16), fixed per bin at compile time.
template <bool T1>
__device__ __forceinline__ void tier1_bins(const float (&a)[16], const float (&eb)[16], float err64,
                                           const EncDomain &d, uint32_t (&lv)[4], uint32_t &undecided) {
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const float sc = k == 0 ? 4.0f / 32.0f : 2.0f / 32.0f;
    const float c = a[k] * sc;
    const bool z2 = T1 ? false : (uint32_t)k >= d.B2;
    const bool z0 = T1 ? k < 2 : (uint32_t)k < d.B1;
    uint32_t L = 128u;
    if (!z2) {
      const float err = eb[k] * sc + err64;
      const float m = err + (z0 ? d.slack0 : d.slack1) + fabsf(c) * 0x1p-21f;
      bool decided;
      if (z0) {
        const uint32_t l0 = zone0_level32(c - m, d), l1 = zone0_level32(c + m, d);
        decided = l0 == l1;
        L = l0;
      } else {
        decided = zone1_decide32(c, m, d, L);
      }
      if (!decided) {
        undecided |= 1u << k;
        L = 0u;
      }
    }
    lv[k >> 2] |= L << (8 * (k & 3));
  }
}

// The window kernel's first tier for Table 1's zones (B1 = 2, B2 = 16) when
// the window's samples are finite (so are its bins) and zone 1 is in use:
// bins 0 and 1 as in tier1_bins, bins 2 .. 15 branch-free in units of the
// unscaled sum a = c N / 2 (every constant scaled by the power of two N / 2
// = 16, so each comparison and rounding is the one zone1_decide32 makes on c,
// up to the level map's FP32 evaluation, whose error, a few ulp of a level
// index, is far inside the slack 2^-18 A1 that the bracket carries).
__device__ __forceinline__ void tier1_bins_fast(const float (&a)[16], const float (&eb)[16], float err64,
                                                const EncDomain &d, uint32_t (&lv)[4], uint32_t &undecided) {
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const float sc = k == 0 ? 4.0f / 32.0f : 2.0f / 32.0f;
    const float c = a[k] * sc;
    const float m = eb[k] * sc + err64 + d.slack0 + fabsf(c) * 0x1p-21f;
    const uint32_t l0 = zone0_level32(c - m, d), l1 = zone0_level32(c + m, d);
    undecided |= l0 == l1 ? 0u : 1u << k;
    lv[0] |= (l0 == l1 ? l0 : 0u) << (8 * k);
  }
  const float base = err64 * 16.0f + d.u1_slack;  // err64 and slack1 in units of a
#pragma unroll
  for (int k = 2; k < 16; ++k) {
    const float ak = fabsf(a[k]);
    const float m = eb[k] + base + ak * 0x1p-21f;
    const float lo = ak - m, hi = ak + m;
    const bool dz = hi < d.u1_d1;              // settled: inside the deadzone
    const bool edge = lo <= d.u1_d1;           // else the deadzone edge is inside the bracket
    const bool pos = a[k] > 0.0f;
    const float kk = pos ? d.u1_kp : d.u1_kn;
    const int v0 = __float2int_rd(fmaf(fminf(lo, d.u1_A1) - d.u1_d1, kk, 0.5f));
    const int v1 = __float2int_rd(fmaf(fminf(hi, d.u1_A1) - d.u1_d1, kk, 0.5f));
    const bool und = !dz && (edge || v0 != v1);
    const uint32_t L = dz ? 128u : (und ? 0u : (uint32_t)(pos ? 129 + v0 : 127 - v0));
    undecided |= und ? 1u << k : 0u;
    lv[k >> 2] |= L << (8 * (k & 3));
  }
}

// Inclusive warp scan.
__device__ __forceinline__ uint32_t lane_prefix(uint32_t v, uint32_t lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= (uint32_t)o) v += y;
  }
  return v;  // inclusive
}

constexpr uint32_t kLvThreads = 128;  // threads per CTA of k_enc_levels_w32 (4 warps)
constexpr uint32_t kTier2Inline = 8;  // a warp with more undecided bins settles them itself
constexpr uint32_t kLvGroups = 8;     // groups of 32 windows per warp, each loaded while the previous is computed
constexpr uint32_t kRowPitch = 36;    // floats per window row in shared memory (144 bytes: 16-byte reads conflict-free)

__device__ __forceinline__ uint32_t lds_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
// 16 bytes, or src_bytes of them with zeros after (0: all zeros; src is not read)
__device__ __forceinline__ void cp_async_16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(lds_addr(dst)), "l"(__cvta_generic_to_global(src))
               : "memory");
}
__device__ __forceinline__ void cp_async_4z(void *dst, const void *src, uint32_t src_bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(lds_addr(dst)),
               "l"(__cvta_generic_to_global(src)), "r"(src_bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit_group() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait_group() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Where a window's samples are: its segment, the window within it, its first sample.
struct LvWin {
  uint64_t s = 0;           // segment
  uint64_t g0 = 0;          // its first level
  const float *src = nullptr;
  uint64_t avail = 0;       // samples from src on in the stream (>= 1), 0 for no window
};

__device__ __forceinline__ LvWin lv_window(const EncParams &p, uint64_t gw, uint64_t n_windows, uint64_t s_from) {
  LvWin r;
  r.s = s_from;
  if (gw >= n_windows) return r;
  r.g0 = gw * 16u;
  while (r.s + 1 < p.n_segs && p.segs[r.s + 1].level_offset <= r.g0) ++r.s;
  const EncSeg &sg = p.segs[r.s];
  const uint64_t i0 = ((r.g0 - sg.level_offset) >> 4) * 32u;
  r.avail = sg.n_samples - i0;
  r.src = p.x + sg.in_offset + i0;
  return r;
}

// The group's samples into its shared-memory rows (one window each),
// asynchronously.  32 whole windows of one stream are 1024 consecutive
// samples: consecutive lanes copy consecutive 16 bytes (4 where the stream does
// not start on a 16-byte boundary, as in a batch of ragged lengths).  Where
// windows of several streams or a stream's end meet, each lane copies its own
// window, a whole one on a 16-byte boundary in 16-byte pieces (zero past the
// stream's end; no window: zeros).  That is every group of a batch of short
// streams: 50,000 of 600 samples take 80 us, 145 in 4-byte pieces alone.
// Each lane its own row for every group made a ragged batch of 86 M samples
// take 317 us (50 M of the 70 M shared-memory wavefronts bank conflicts, 32
// lines a copy); consecutive lanes take 122 us.
__device__ __forceinline__ void lv_load_async(const EncParams &p, const LvWin &wn, float *rows, uint32_t lane) {
  const uint64_t s0 = __shfl_sync(0xffffffffu, wn.s, 0);
  if (__all_sync(0xffffffffu, wn.avail >= 32 && wn.s == s0)) {
    const uint64_t b0 = __shfl_sync(0xffffffffu, (uint64_t)reinterpret_cast<uintptr_t>(wn.src), 0);
    const float *const src = reinterpret_cast<const float *>((uintptr_t)b0);
    if ((b0 & 15u) == 0) {
#pragma unroll
      for (uint32_t j = 0; j < 8; ++j) {
        const uint32_t c = 32 * j + lane;  // 16-byte piece of the group
        cp_async_16(rows + (c >> 3) * kRowPitch + (c & 7u) * 4, src + 4 * c);
      }
    } else {
#pragma unroll 8
      for (uint32_t j = 0; j < 32; ++j) cp_async_4z(rows + j * kRowPitch + lane, src + 32 * j + lane, 4u);
    }
    return;
  }
  float *const row = rows + lane * kRowPitch;
  if (wn.avail >= 32 && (reinterpret_cast<uintptr_t>(wn.src) & 15u) == 0) {
#pragma unroll
    for (int j = 0; j < 8; ++j) cp_async_16(row + 4 * j, wn.src + 4 * j);
    return;
  }
  const float *base = wn.avail ? wn.src : p.x;  // a valid address where nothing is read
#pragma unroll 8
  for (int j = 0; j < 32; ++j)
    cp_async_4z(row + j, (uint64_t)j < wn.avail ? wn.src + j : base, (uint64_t)j < wn.avail ? 4u : 0u);
}

// One thread per window, for encoders whose every domain has N = 32, E = 16:
// the window's 16 Eq. 1 bins at once by the even/odd butterfly in FP32, with
// a bound on each bin's error from the butterfly's own intermediate sums
// (dct32.cuh dct2_16_bounded; the exact scale 2/N, 4/N for bin 0), plus the
// FP64 encoder's own rounding; the zone quantizer is bracketed by that bound
// as in k_enc_levels_any.  Bins it cannot settle are computed again, spread over
// the warp's lanes, as compensated dot products; what those cannot settle goes
// to the FP64 list.  A warp takes `groups` groups of 32 consecutive windows
// (kLvGroups, fewer where a batch has too few windows to fill the chip with
// that); each group's samples come into shared memory by asynchronous copies while
// the warp computes the group before.
__global__ void __launch_bounds__(kLvThreads, 5) k_enc_levels_w32(EncParams p, uint64_t n_windows, uint32_t groups) {
  dependents_may_start();
  // per warp: two groups' samples (one row per window), and the second tier's
  // work list (window lane, bin), the windows' levels, segments, sample sums
  __shared__ __align__(16) float rows[kLvThreads / 32][2][32 * kRowPitch];
  __shared__ uint16_t work[kLvThreads / 32][512];
  __shared__ uint32_t lvs[kLvThreads / 32][32][4];
  __shared__ uint32_t segs_s[kLvThreads / 32][32];
  __shared__ float s1s[kLvThreads / 32][32];
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  const uint64_t chunk = (uint64_t)blockIdx.x * (kLvThreads / 32) + wid;
  if (chunk * groups * 32u >= n_windows) return;  // the whole warp
  const uint64_t first_group = chunk * groups;
  // the segment of the warp's first window from a table, then a step forward
  // per window (a warp's windows span few segments)
  const uint64_t s_first = p.lv_seg[first_group / kLvGroups];
  LvWin cur = lv_window(p, first_group * 32u + lane, n_windows, s_first);
  lv_load_async(p, cur, rows[wid][0], lane);
  cp_async_commit_group();
#pragma unroll 1
  for (uint32_t t = 0; t < groups; ++t) {
    const uint64_t grp = first_group + t;
    if (grp * 32u >= n_windows) break;  // the whole warp
    // the next group's copies in flight
    LvWin nxt = cur;
    if (t + 1 < groups) {
      nxt = lv_window(p, (grp + 1) * 32u + lane, n_windows, cur.s);
      lv_load_async(p, nxt, rows[wid][(t + 1) & 1], lane);
    }
    cp_async_commit_group();
    cp_async_wait_group<1>();
    __syncwarp();
    const float *const xr = rows[wid][t & 1];
    const bool valid = cur.avail > 0;  // every lane stays for the warp's shuffles
    const uint64_t s = cur.s;
    const uint64_t g0 = cur.g0;
    const EncDomain d = p.doms[p.segs[s].domain];
    float x[32];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float4 v = *reinterpret_cast<const float4 *>(xr + lane * kRowPitch + 4 * j);
      x[4 * j] = v.x;
      x[4 * j + 1] = v.y;
      x[4 * j + 2] = v.z;
      x[4 * j + 3] = v.w;
    }
    float s1 = 0.0f;
#pragma unroll
    for (int j = 0; j < 32; ++j) s1 += fabsf(x[j]);
    float a[16], eb[16];
    dct32::dct2_16_bounded(x, a, eb);
    // |c - c64| <= the butterfly's bound for bin k (scaled like c) + the FP64 encoder's own rounding
    const float err64 = s1 * (2.0f / 32.0f) * 0x1p-40f + 1e-30f;
    uint32_t lv[4] = {0u, 0u, 0u, 0u};
    uint32_t undecided = 0;  // bins the butterfly's bound cannot settle
    if (d.B1 == 2u && d.B2 == 16u && d.z1_f32 && s1 <= 3.0e38f)  // Table 1's zones, finite bins
      tier1_bins_fast(a, eb, err64, d, lv, undecided);
    else if (d.B1 == 2u && d.B2 == 16u)  // the zone of every bin known at compile time
      tier1_bins<true>(a, eb, err64, d, lv, undecided);
    else
      tier1_bins<false>(a, eb, err64, d, lv, undecided);
    if (!valid) undecided = 0u;
    // second tier, spread over the warp's lanes: each undecided bin again as a
    // compensated FP32 dot product (|error| <= 2^-34 (2/N) sum |x|, as in
    // level_compensated); what that cannot settle goes to the FP64 list
    const uint32_t cnt = (uint32_t)__popc(undecided);
    const uint32_t incl = lane_prefix(cnt, lane);
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    if (total && total <= kTier2Inline) {  // a few: k_enc_fallback settles them (compensated, then FP64)
      uint64_t lo8 = ((uint64_t)lv[1] << 32) | lv[0], hi8 = ((uint64_t)lv[3] << 32) | lv[2];
      uint32_t u = undecided;
      while (u) {
        const uint32_t k = (uint32_t)(__ffs(u) - 1);
        u &= u - 1u;
        const unsigned int slot = fb_slot(p);
        if (slot != ~0u) {
          p.fb_list[slot] = fb_entry(g0 + k, s);  // its level (0 here) is written after the window's store
        } else {
          const uint64_t L = level_fp64_seg(p, g0 + k, s);
          if (k < 8)
            lo8 |= L << (8 * k);
          else
            hi8 |= L << (8 * (k - 8));
        }
      }
      lv[0] = (uint32_t)lo8;
      lv[1] = (uint32_t)(lo8 >> 32);
      lv[2] = (uint32_t)hi8;
      lv[3] = (uint32_t)(hi8 >> 32);
    } else if (total) {  // many (re-encoded signals): settled here, spread over the warp's lanes
      if (cnt) {
        segs_s[wid][lane] = (uint32_t)s;
        s1s[wid][lane] = s1;
        uint32_t u = undecided, o = incl - cnt;
        while (u) {
          work[wid][o++] = (uint16_t)((lane << 4) | (uint32_t)(__ffs(u) - 1));
          u &= u - 1u;
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) lvs[wid][lane][q] = lv[q];
      __syncwarp();
      const uint64_t gw_base = grp * 32u;
      for (uint32_t i = lane; i < total; i += 32) {
        const uint32_t e = work[wid][i], own = e >> 4, k = e & 15u;
        const uint64_t so = segs_s[wid][own];
        const EncDomain od = p.doms[p.segs[so].domain];
        const float2 *ct = reinterpret_cast<const float2 *>(p.cosf) + od.cos_off + k;
        const float *xo = xr + own * kRowPitch;
        float hi = 0.0f, lo = 0.0f;
#pragma unroll 8
        for (int n = 0; n < 32; ++n) {
          const float xv = xo[n];
          const float2 cs = ct[(size_t)n * 16u];
          const float pr = __fmul_rn(xv, cs.x);
          const float pe = __fadd_rn(__fmaf_rn(xv, cs.x, -pr), __fmul_rn(xv, cs.y));
          const float tt = __fadd_rn(hi, pr);
          const float bp = __fsub_rn(tt, hi);
          lo = __fadd_rn(lo, __fadd_rn(__fadd_rn(__fsub_rn(hi, __fsub_rn(tt, bp)), __fsub_rn(pr, bp)), pe));
          hi = tt;
        }
        const float err2 = s1s[wid][own] * (2.0f / 32.0f) * 0x1p-34f + 1e-30f;
        const double cd = ((double)hi + (double)lo) * (2.0 / 32.0);
        uint32_t L = 0u;
        const bool decided =
            level_bracket64(p, k, cd, 2.0 * (double)err2, level_estimate(k, (float)cd, od), od, L);
        const uint64_t g = (gw_base + own) * 16u + k;
        if (!decided) {
          const unsigned int slot = fb_slot(p);
          if (slot != ~0u) {
            p.fb_list[slot] = fb_entry(g, so);
            L = 0u;  // k_enc_fallback writes this level after the window's store
          } else {
            L = level_fp64_seg(p, g, so);
          }
        }
        reinterpret_cast<uint8_t *>(lvs[wid][own])[k] = (uint8_t)L;
      }
      __syncwarp();
#pragma unroll
      for (int q = 0; q < 4; ++q) lv[q] = lvs[wid][lane][q];
    }
    if (valid) {
      uint8_t *const dst = p.levels + g0;
      if ((reinterpret_cast<uintptr_t>(dst) & 15u) == 0) {
        *reinterpret_cast<uint4 *>(dst) = make_uint4(lv[0], lv[1], lv[2], lv[3]);
      } else {
#pragma unroll
        for (int k = 0; k < 16; ++k) dst[k] = (uint8_t)(lv[k >> 2] >> (8 * (k & 3)));
      }
    }
    __syncwarp();  // every lane is done with this group's rows and tier-2 lists before they are refilled
    cur = nxt;
  }
  cp_async_wait_group<0>();
}

// ---- SymLen packing (Alg. 1) in parallel ---------------------------------------
// Alg. 1 starts a word at the first codeword that does not fit the open one,
// so where words start in a run of symbols depends only on the bits u of the
// open word that are used when the run is entered (1 .. 64; 64 also when no
// word is open).  A codeword of c bits starts a word when u + c > 64, and u
// becomes c, else u + c.  Held as s = u + kOff with kOff = 2^16 - 65 (or 2^32 -
// 65), u + c > 64 is the carry out of s + c, so the step is
// s = max(s + c, c + kOff) in modular arithmetic: one instruction, and one for
// two packings at once in 16-bit halves.
//
// Where the first word of a run starts is the only thing its entry state
// decides: at the symbol j whose codeword no longer fits, one of the (about
// ten) symbols that begin in the run's first 64 bits.  So a run's effect on the
// state is a small table: the run packed once for every such j, two packings
// per instruction.  A run of kSub symbols per lane keeps the serial chain
// short; the tables of 32 runs are put together step by step, again for every
// first start at once (one per lane), which gives the table of the block of
// kPackBlock symbols.  Packings of the same symbols from different states meet
// sooner or later (on the trained codes the chance that two have not falls by
// e every 900 symbols) and coincide from there on: the table of a block nearly
// always gives one and the same state, which is then where the next block is
// entered whatever came before.
//   k_enc_starts  a warp per block: the tables, then, entered as the block
//                 before it (of the same CTA, or packed along for this) says,
//                 the word starts as a bitmap of the block's symbols.
//   k_enc_scan    a warp per stream: the word starts added up block after
//                 block; a block entered in another state than assumed is
//                 walked again from the true one until the two packings meet.
//   k_enc_pack    a warp per 2048 symbols, one lane per word: the word starts
//                 give every word's symbols, so the words are put together
//                 independently of one another and written once, consecutive
//                 lanes to consecutive words.
// All three are bound by instruction issue on large batches and by the length
// of a run (256 symbols) on small ones.  With a block's packing done by one
// thread twice (its reference, then the words) the chain was 16,384 symbols
// and more: 43 M levels of a mixed batch took 1,112 us for the packing, now
// 113 us (69 + 2 + 42); one stream of 32,768 levels 677 us, now 24 us.  The loops
// of k_enc_starts are rolled up: unrolled, its 50 KB of code came from L2 once per
// SM and cost 10 us more (21 us for one stream, 14 now).  Runs of
// 2048 symbols by one thread without tables left 5 to 14 % of the blocks
// unmet, and the scan that walked them took 380 us.

// What k_enc_starts leaves of a block.
struct PackRec {
  uint32_t starts;  // words that start in the block, entered as assumed
  uint32_t u_in;    // the assumed state (64 at a stream's first block)
  uint32_t u_out;   // the state it is left in then (not of a stream's last block)
  uint32_t bad;     // a level of the block has no codeword
};

// A level's code length from the table of a domain (code << (32 - length) |
// length per level, 0: no codeword); 64 for a level without one, which takes a
// word of its own and shows in the OR of a block's lengths.
__device__ __forceinline__ uint32_t entry_len(uint32_t e) { return e ? e & 31u : 64u; }

// The code tables in shared memory (lengths in k_enc_starts, whole entries in
// k_enc_pack), for encoders of at most kTabDomains domains; others read the
// table in global memory.
constexpr uint32_t kTabDomains = 16;

// 16 levels from i (a multiple of 16, i < n) of the run of n at lv, zero past
// n: one vector load where the run is 16-byte aligned, else aligned 4-byte
// words put together (bytes at the run's ends, where a word would reach
// outside it).  Here and below levels are read by plain loads: the grids
// before may still be writing them when this one starts (launch_after).
__device__ __forceinline__ uint4 load_run16(const uint8_t *lv, uint32_t i, uint32_t n) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(lv + i);
  if ((a & 15u) == 0 && i + 16 <= n) return *reinterpret_cast<const uint4 *>(a);
  if (i != 0 && i + 20 <= n) {
    const uint32_t *w = reinterpret_cast<const uint32_t *>(a & ~uintptr_t(3));
    const uint32_t s = (uint32_t)(a & 3u) * 8u;
    const uint32_t w0 = w[0], w1 = w[1], w2 = w[2], w3 = w[3], w4 = w[4];
    return make_uint4(__funnelshift_r(w0, w1, s), __funnelshift_r(w1, w2, s), __funnelshift_r(w2, w3, s),
                      __funnelshift_r(w3, w4, s));
  }
  uint32_t t[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int r = 0; r < 16; ++r)
    if (i + r < n) t[r >> 2] |= (uint32_t)lv[i + r] << (8 * (r & 3));
  return make_uint4(t[0], t[1], t[2], t[3]);
}

// fn(j, level) for the 16 levels of a vector.
template <class F>
__device__ __forceinline__ void each16(const uint4 &q, F fn) {
  const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
  for (int j = 0; j < 16; ++j) fn(j, (w[j >> 2] >> (8 * (j & 3))) & 0xffu);
}

constexpr uint32_t kSub = kPackBlock / 32;       // symbols of a lane's run
constexpr uint32_t kOff16x2 = 0xFFBFFFBFu;       // 2^16 - 65 in both halves
constexpr uint32_t kOff32 = 0xFFFFFFBFu;         // 2^32 - 65
constexpr uint32_t kStartWarps = 8;              // blocks of a CTA of k_enc_starts; one more warp packs the block before
constexpr uint32_t kExitPitch = 68;              // bytes per run: its exits by first start (64 at most), in separate banks
constexpr uint32_t kSeqPitch = 33;               // bytes per first start: the states its 32 runs are entered in, exit
constexpr uint32_t kStartWarpBytes = 32 * kExitPitch + 64 * kSeqPitch + 32 * 8;

// fn(v, levels 16 v .. 16 v + 15) over the run of n at lv, the next three vectors
// in flight.  One place in the code where levels are loaded: a small batch runs
// this once per SM, from a cold instruction cache.
template <class F>
__device__ __forceinline__ void each_vector(const uint8_t *lv, uint32_t first, uint32_t n, F fn) {
  const int nv = (int)((n + 15) / 16);
  uint4 r0, r1, r2, r3;
  r1 = r2 = r3 = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 1
  for (int v = (int)first - 3; v < nv; ++v) {
    r0 = r1;
    r1 = r2;
    r2 = r3;
    if (v + 3 < nv) r3 = load_run16(lv, 16 * (uint32_t)(v + 3), n);
    if (v >= (int)first) fn((uint32_t)v, r0);
  }
}

// Exits of a run by first start into its row (bytes: the states' low bytes,
// u - 65 mod 256), for the first starts base .. base + 2 R - 1 (base a multiple of
// 16, R <= 8): two packings per instruction, c2 a level's code length in both
// halves.
template <int R, class Len2>
__device__ __forceinline__ void run_exits(const uint8_t *lv, uint32_t base, const Len2 &c2, uint8_t *row) {
  uint32_t s[R];
#pragma unroll
  for (int r = 0; r < R; ++r) s[r] = 0xFFFFFFFFu;  // a full word: the next symbol starts one
  each_vector(lv, base / 16, kSub, [&](uint32_t v, const uint4 &q) {
    if (v == base / 16) {  // first start j begins at symbol base + j
      each16(q, [&](int j, uint32_t level) {
        const uint32_t c = c2(level), k = c + kOff16x2;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if (j >= 2 * r) s[r] = __viaddmax_u16x2(s[r], c, k);
          if (j == 2 * r) s[r] |= 0xFFFF0000u;
        }
      });
    } else {
      each16(q, [&](int, uint32_t level) {
        const uint32_t c = c2(level), k = c + kOff16x2;
#pragma unroll
        for (int r = 0; r < R; ++r) s[r] = __viaddmax_u16x2(s[r], c, k);
      });
    }
  });
  // byte 0 and byte 2 of two states
#pragma unroll
  for (int r = 0; r < R; r += 2)
    *reinterpret_cast<uint32_t *>(row + base + 2 * r) = __byte_perm(s[r], r + 1 < R ? s[r + 1] : 0u, 0x6420);
}

// Index of the first start of a run entered with u bits used, from the
// run's symbol boundaries in its first 63 bits (bit t - 1: one after t bits):
// the symbols that fit the 64 - u bits left.
__device__ __forceinline__ uint32_t first_start(uint64_t bounds, uint32_t u) {
  return (uint32_t)__popcll(bounds & ((1ull << (64u - u)) - 1ull));
}

template <bool TAB>
__global__ void __launch_bounds__((kStartWarps + 1) * 32, 4) k_enc_starts(EncParams p) {
  dependents_may_start();
  extern __shared__ uint32_t starts_smem[];
  // per block: what it is (bit 0: there is one, 1: its stream's first, 2: another follows it, 3: every first start
  // gives one exit), the state it is entered in and which first start that is
  __shared__ uint32_t what_s[kStartWarps + 1], in_s[kStartWarps + 1], cand_s[kStartWarps + 1];
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  uint32_t *const tab_s = starts_smem;  // TAB: [n_domains][256] code lengths, in both halves
  uint8_t *const wbase = reinterpret_cast<uint8_t *>(starts_smem + (TAB ? p.n_doms * 256u : 0u)) + wid * kStartWarpBytes;
  uint64_t *const bounds_s = reinterpret_cast<uint64_t *>(wbase);
  uint8_t *const exits = wbase + 32 * 8;                         // [run][kExitPitch]
  uint8_t *const seq = exits + 32 * kExitPitch;                  // [first start][kSeqPitch]
  if (TAB) {
    for (uint32_t i = threadIdx.x; i < p.n_doms * 256u; i += (kStartWarps + 1) * 32)
      tab_s[i] = entry_len(__ldg(p.code_tab + i)) * 0x10001u;
    __syncthreads();
  }
  dependency_wait();  // the levels
  const uint64_t b = (uint64_t)blockIdx.x * kStartWarps + wid - 1;  // warp 0: the block before the CTA's (may wrap: none)
  bool have = b < p.n_blocks;
  const uint8_t *lv = p.levels;  // this lane's run
  uint32_t dom = 0, nb = 0;
  bool head = true, more = false;  // the stream's first block; it has another after it
  if (have) {
    const EncSeg &sg = p.segs[p.block_seg[b]];
    const uint64_t i0 = (b - sg.block_base) * kPackBlock;
    const uint64_t L = sg.n_windows * p.doms[sg.domain].E;
    nb = (uint32_t)(L - i0 < kPackBlock ? L - i0 : kPackBlock);
    lv = p.levels + sg.level_offset + i0 + lane * kSub;
    dom = sg.domain;
    head = i0 == 0;
    more = i0 + nb < L;
  }
  uint32_t what = (have ? 1u : 0u) | (head ? 2u : 0u) | (more ? 4u : 0u);
  if (wid == 0) have = have && more;  // only its exit is wanted
  const uint32_t *const lt = tab_s + dom * 256u;
  const uint32_t *const gt = p.code_tab + dom * 256u;
  auto c2 = [&](uint32_t level) -> uint32_t { return TAB ? lt[level] : entry_len(__ldg(gt + level)) * 0x10001u; };
  const uint32_t nsub = (nb + kSub - 1) / kSub;
  uint32_t n_cand = 1;  // first starts of the block
  if (have) {
    // ---- the runs' tables.  A run needs one when another follows it (it is whole then)
    const bool mine = (lane + 1 < nsub) || (lane + 1 == nsub && more);
    uint32_t blo = 0, bhi = 0;
    {
      uint32_t sum = 0;
#pragma unroll 1
      for (uint32_t i = 0; i < 64; i += 16) {
        if (!__any_sync(0xffffffffu, mine && sum < 64u)) break;
        if (!mine) continue;
        each16(load_run16(lv, i, kSub), [&](int, uint32_t level) {
          sum += c2(level) & 0xffffu;
          const uint32_t bit = 1u << ((sum - 1u) & 31u);
          blo |= sum <= 32u ? bit : 0u;
          bhi |= sum > 32u && sum <= 63u ? bit : 0u;
        });
      }
    }
    const uint64_t bounds = (uint64_t)bhi << 32 | blo;
    bounds_s[lane] = bounds;
    const uint32_t cands = mine ? (uint32_t)__popcll(bounds) + 1u : 0u;
    const uint32_t most = __reduce_max_sync(0xffffffffu, cands);
    uint8_t *const row = exits + lane * kExitPitch;
#pragma unroll 1
    for (uint32_t base = 0; base < most; base += 16) {
      if (!mine) continue;
      // as many packings as the warp's runs want (the instance is the warp's)
      if (most - base > 12)
        run_exits<8>(lv, base, c2, row);
      else
        run_exits<6>(lv, base, c2, row);
    }
    __syncwarp();
    // ---- the block's: lane = first start, run after run
    n_cand = (uint32_t)__popcll(bounds_s[0]) + 1u;
    const uint32_t steps = more ? nsub : (nsub ? nsub - 1u : 0u);  // runs that are left for another
    uint32_t same = 1u, last = 0u;
    for (uint32_t j0 = 0; j0 < n_cand; j0 += 32) {
      const uint32_t j = j0 + lane;
      uint32_t u = 0;
      if (j < n_cand) {
        uint32_t at = j;
#pragma unroll 1
        for (uint32_t k = 0; k < steps; ++k) {
          u = ((uint32_t)exits[k * kExitPitch + at] + 65u) & 0xffu;
          seq[j * kSeqPitch + k + 1] = (uint8_t)u;
          at = k + 1 < 32u ? first_start(bounds_s[k + 1], u) : 0u;
        }
      }
      const uint32_t u0 = __shfl_sync(0xffffffffu, u, 0);
      same &= __all_sync(0xffffffffu, j >= n_cand || u == u0) ? 1u : 0u;
      if (j0) same &= u0 == last ? 1u : 0u;
      last = u0;
    }
    what |= same << 3;
  }
  if (lane == 0) what_s[wid] = what;
  __syncthreads();
  // ---- the states the CTA's blocks are entered in
  if (threadIdx.x == 0) {
    uint32_t u = 64u;
    for (uint32_t w = 0; w <= kStartWarps; ++w) {
      const uint32_t f = what_s[w];
      if (!(f & 1u)) continue;
      const uint8_t *wb = wbase + w * kStartWarpBytes;  // thread 0 is of warp 0
      if (f & 2u) u = 64u;
      in_s[w] = u;
      // warp 0's block stands for itself when its stream starts there or every first
      // start gives one exit; else 64 is assumed, and k_enc_scan sees whether that is so
      const uint32_t cand = w == 0 ? 0u : first_start(*reinterpret_cast<const uint64_t *>(wb), u);
      cand_s[w] = cand;
      if (f & 4u)
        u = w == 0 && (f & 10u) == 0 ? 64u : (uint32_t)wb[32 * 8 + 32 * kExitPitch + cand * kSeqPitch + 32];
    }
  }
  __syncthreads();
  if (wid == 0 || !have) return;
  // ---- the word starts, each lane those of its run (its bitmap in halfwords over its row of exits)
  uint32_t seen = 0, cnt = 0;
  const uint32_t n = lane * kSub < nb ? (nb - lane * kSub < kSub ? nb - lane * kSub : kSub) : 0u;
  const uint32_t u_in = in_s[wid];
  if (n) {
    uint16_t *const bits = reinterpret_cast<uint16_t *>(exits + lane * kExitPitch);
    uint32_t s = (lane ? (uint32_t)seq[cand_s[wid] * kSeqPitch + lane] : u_in) + kOff32;
    auto start = [&](uint32_t level) -> bool {
      const uint32_t c = c2(level) & 0xffffu, k = c + kOff32;
      seen |= c;
      s = __viaddmax_u32(s, c, k);
      return s == k;
    };
    each_vector(lv, 0, n, [&](uint32_t v, const uint4 &q) {
      uint32_t m = 0;
      if (16 * v + 16 <= n) {
        each16(q, [&](int j, uint32_t level) { m |= start(level) ? 1u << j : 0u; });
      } else {  // the stream's last symbols
#pragma unroll 1
        for (uint32_t j = 0; 16 * v + j < n; ++j) m |= start((uint32_t)lv[16 * v + j]) ? 1u << j : 0u;
      }
      cnt += __popc(m);
      bits[v] = (uint16_t)m;
    });
    for (uint32_t v = (n + 15) / 16; v < kSub / 16; ++v) bits[v] = 0;
    const uint32_t *const w = reinterpret_cast<const uint32_t *>(bits);
    uint4 *const row = reinterpret_cast<uint4 *>(p.masks + b * kMaskWords + lane * (kSub / 32));
    static_assert(kSub == 256, "a run's bitmap is two 16-byte vectors");
    row[0] = make_uint4(w[0], w[1], w[2], w[3]);
    row[1] = make_uint4(w[4], w[5], w[6], w[7]);
  }
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  seen = __reduce_or_sync(0xffffffffu, seen);
  if (lane == 0)
    p.recs[b] = PackRec{cnt, u_in, more ? (uint32_t)seq[cand_s[wid] * kSeqPitch + 32] : 64u, seen >> 6};
}

// Word starts of Alg. 1 among the first `valid` symbols of a chunk of 32 (S:
// inclusive prefix of the chunk's code lengths, per lane), entered with v bits
// left, which moves on.  One ballot per word start.
__device__ __forceinline__ uint32_t chunk_starts(uint32_t S, uint32_t lane, uint32_t valid, uint32_t &v) {
  uint32_t mask = 0, from = 0, pre = 0;
  while (true) {
    const uint32_t over = __ballot_sync(0xffffffffu, lane >= from && lane < valid && S - pre > v);
    if (over == 0) {  // the rest of the chunk fits the open word
      v -= __shfl_sync(0xffffffffu, S, valid - 1) - pre;
      return mask;
    }
    from = (uint32_t)(__ffs(over) - 1);  // a word starts at symbol from
    mask |= 1u << from;
    pre = from ? __shfl_sync(0xffffffffu, S, from - 1) : 0u;
    v = 64u;
  }
}

// Block b again, entered with u bits used, by the whole warp, 32 symbols at a
// time, until a start of its bitmap is met (its starts before that one are
// replaced): the words that start in it and the state it is left in.
__device__ void walk_block(const EncParams &p, const EncSeg &sg, const EncDomain &d, uint64_t b, uint32_t &u,
                           uint32_t &starts, uint32_t u_out, uint32_t lane) {
  const uint64_t L = sg.n_windows * d.E;
  const uint64_t i0 = (b - sg.block_base) * kPackBlock;
  const uint32_t nb = (uint32_t)(L - i0 < kPackBlock ? L - i0 : kPackBlock);
  const uint8_t *lv = p.levels + sg.level_offset + i0;
  const uint32_t *tab = p.code_tab + sg.domain * 256u;
  uint32_t *row = p.masks + b * kMaskWords;
  auto fetch = [&](uint32_t at) -> uint32_t { return at + lane < nb ? (uint32_t)lv[at + lane] : 0u; };
  uint32_t cur = fetch(0), v = 64u - u;
  for (uint32_t at = 0; at < nb; at += 32) {
    const uint32_t nxt = fetch(at + 32);
    const uint32_t valid = nb - at < 32 ? nb - at : 32;
    const uint32_t S = lane_prefix(lane < valid ? entry_len(__ldg(tab + cur)) : 0u, lane);
    const uint32_t r = row[at >> 5];
    __syncwarp();
    const uint32_t t = chunk_starts(S, lane, valid, v);
    const uint32_t both = t & r;
    const uint32_t below = both ? (both & (0u - both)) - 1u : 0xffffffffu;
    starts += __popc(t & below) - __popc(r & below);
    if (lane == 0) row[at >> 5] = (t & below) | (r & ~below);
    if (both) {
      u = u_out;
      return;
    }
    cur = nxt;
  }
  u = 64u - v;
}

// One warp per stream: the words before each block from the blocks' records,
// 32 blocks at a time (a warp scan), the next 32 records in flight; a block
// entered in another state than assumed is walked again from the true one;
// code and room checks; the stream's word count.
__global__ void __launch_bounds__(128) k_enc_scan(EncParams p) {
  dependents_may_start();
  dependency_wait();  // the blocks' records
  if (blockIdx.x == 0 && threadIdx.x == 0) *p.fb_count = 0;  // the level kernels' list, for the next encode
  const uint64_t i = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t lane = threadIdx.x & 31u;
  if (i >= p.n_scan) return;  // the whole warp
  const uint64_t s = p.scan_seg ? p.scan_seg[i] : i;
  const EncSeg sg = p.segs[s];
  const EncDomain &d = p.doms[sg.domain];
  const uint64_t L = sg.n_windows * d.E;
  const uint64_t nblk = (L + kPackBlock - 1) / kPackBlock;
  uint64_t w = 0;  // words that start before the group
  bool bad = false;
  auto fetch = [&](uint64_t jb) -> PackRec {
    return jb + lane < nblk ? p.recs[sg.block_base + jb + lane] : PackRec{0u, 0u, 0u, 0u};
  };
  uint32_t u_prev = 64u;  // the state the block before the group is left in
  PackRec rec = fetch(0);
  for (uint64_t jb = 0; jb < nblk; jb += 32) {
    const PackRec nxt = fetch(jb + 32);
    const uint64_t b0 = sg.block_base + jb;
    const uint32_t n = nblk - jb < 32 ? (uint32_t)(nblk - jb) : 32u;
    bad = __any_sync(0xffffffffu, rec.bad != 0u);
    if (bad) break;
    while (true) {  // the first block entered in another state than assumed, until there is none
      uint32_t u = __shfl_up_sync(0xffffffffu, rec.u_out, 1);
      if (lane == 0) u = u_prev;
      const uint32_t off = __ballot_sync(0xffffffffu, lane < n && u != rec.u_in);
      if (!off) break;
      const uint32_t at = (uint32_t)(__ffs(off) - 1);
      uint32_t ua = __shfl_sync(0xffffffffu, u, at), st = __shfl_sync(0xffffffffu, rec.starts, at);
      const uint32_t uo = __shfl_sync(0xffffffffu, rec.u_out, at);
      if (lane == at) rec.u_in = ua;
      walk_block(p, sg, d, b0 + at, ua, st, uo, lane);
      if (lane == at) {
        rec.starts = st;
        rec.u_out = ua;
      }
    }
    const uint32_t add = lane < n ? rec.starts : 0u;
    const uint32_t incl = lane_prefix(add, lane);
    if (lane < n) p.first_word[b0 + lane] = w + (incl - add);
    w += __shfl_sync(0xffffffffu, incl, 31);
    u_prev = __shfl_sync(0xffffffffu, rec.u_out, n - 1);
    rec = nxt;
  }
  if (lane == 0) {
    if (bad) enc_flag(p.status, FPTC_ENC_FLAG_NO_CODE, s);
    if (!bad && w > sg.room) {
      enc_flag(p.status, FPTC_ENC_FLAG_ROOM, s);
      bad = true;
    }
    p.seg_bad[s] = bad ? 1u : 0u;
    p.n_words[s] = bad ? 0u : w;
  }
}

// Level of bin g of segment s from its compensated FP32 coefficient (exact
// products by FMA, exact sums by two-sum: error O((N u)^2 sum |x|) + u |c|; the
// bound 2^-34 (2/N) sum |x| also covers the cosines' representation and the
// FP64 evaluation's own rounding for N <= 128); false when that bound cannot
// settle it.  AHEAD: sixteen samples and cosines are requested at once, for
// kernels with few bins in flight (and registers for it).
template <bool AHEAD = true>
__device__ __forceinline__ bool level_compensated(const EncParams &p, uint64_t g, uint64_t s, uint32_t &L) {
  const EncSeg sg = p.segs[s];
  const EncDomain d = p.doms[sg.domain];
  const uint64_t local = g - sg.level_offset;
  const uint64_t w = local / d.E;
  const uint32_t k = (uint32_t)(local - w * d.E);
  const uint64_t avail = sg.n_samples - w * d.N;
  const uint32_t nn = avail < d.N ? (uint32_t)avail : d.N;
  const float *src = p.x + sg.in_offset + w * d.N;
  const float2 *ct = reinterpret_cast<const float2 *>(p.cosf) + d.cos_off + k;
  float hi = 0.0f, lo = 0.0f, s1 = 0.0f;
  auto step = [&](float xv, float2 cs) {
    const float pr = __fmul_rn(xv, cs.x);
    const float pe = __fadd_rn(__fmaf_rn(xv, cs.x, -pr), __fmul_rn(xv, cs.y));
    const float t = __fadd_rn(hi, pr);
    const float bp = __fsub_rn(t, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fadd_rn(__fsub_rn(hi, __fsub_rn(t, bp)), __fsub_rn(pr, bp)), pe));
    hi = t;
    s1 += fabsf(xv);
  };
  if (!AHEAD) {
    for (uint32_t n = 0; n < nn; ++n) step(__ldg(src + n), __ldg(ct + (size_t)n * d.E));
  } else if (d.N == 32 && nn == 32 && (reinterpret_cast<uintptr_t>(src) & 15u) == 0) {
    // a whole window: its samples and cosines requested at once, the same
    // operations in the same order as below
    float xv[32];
    float2 cs[32];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float4 v = __ldg(reinterpret_cast<const float4 *>(src) + j);
      xv[4 * j] = v.x;
      xv[4 * j + 1] = v.y;
      xv[4 * j + 2] = v.z;
      xv[4 * j + 3] = v.w;
    }
#pragma unroll
    for (int n = 0; n < 32; ++n) cs[n] = __ldg(ct + (size_t)n * d.E);
#pragma unroll
    for (int n = 0; n < 32; ++n) step(xv[n], cs[n]);
  } else {
    for (uint32_t n0 = 0; n0 < nn; n0 += 16) {  // sixteen of each requested at once
      float xv[16];
      float2 cs[16];
#pragma unroll
      for (uint32_t j = 0; j < 16; ++j) {
        xv[j] = n0 + j < nn ? __ldg(src + n0 + j) : 0.0f;
        cs[j] = n0 + j < nn ? __ldg(ct + (size_t)(n0 + j) * d.E) : make_float2(0.0f, 0.0f);
      }
#pragma unroll
      for (uint32_t j = 0; j < 16; ++j)
        if (n0 + j < nn) step(xv[j], cs[j]);
    }
  }
  const float err2 = s1 * (2.0f / (float)d.N) * 0x1p-34f + 1e-30f;
  const double cd = ((double)hi + (double)lo) * (2.0 / (double)d.N);
  return level_bracket64(p, k, cd, 2.0 * (double)err2, level_estimate(k, (float)cd, d), d, L);
}

// ---- level kernel for every other shape (N in [4, 128], any E) ------------------
// A warp takes tiles of `tile` windows.  A window is folded once, u[n] = x[n] +
// x[N-1-n] and v[n] = x[n] - x[N-1-n] for n < P = ceil(N / 2) (the middle sample
// of an odd N alone in u), because bin k of Eq. 1 is sum_n u[n] cos(k, n) for
// even k and the same of v for odd k.  A lane then has four windows and four
// bins of one parity: 64 multiply-adds for four 16-byte reads of the folded
// windows and four of the cosines, in FP32.  The next tile's samples are
// copied into shared memory meanwhile.
//
// Error of such a sum against the exact one: each of the P fused multiply-adds
// (paired: over even and over odd n, added at the end) rounds a partial sum of
// magnitude at most S = sum |u| (or |v|), and so does that addition, the folding
// rounds each u to 2^-24 |u| and the cosines (at most 1) are off by at most
// 2^-25, so (P + 2.5) 2^-24 S and terms of second order; (P + 4) 2^-24 S is
// used, and 2^-40 (sum |u| + sum |v|) for the host encoder's own rounding in FP64
// (N 2^-52 sum |x|, and sum |x| <= sum |u| + sum |v|).  The zone maps are bracketed
// by that bound as in the window kernel; a bin it does not settle (about one
// in 200) goes to the list of k_enc_fallback, or, where a tile has many, is
// settled here by the compensated sum.
// Bound by instruction issue (about 30 instructions a sample at N = 64, E = 32); at
// 128 registers 64 bytes a thread are spilled, around the branch for samples that
// are not finite and zones that the fast map does not take.
// 16.8 M samples at N = 64, E = 32: 70 us (one thread per bin with the compensated
// sum for every bin took 457 us; the zone maps behind a branch per bin, and plain
// multiply-adds, 75).
constexpr uint32_t kAnyWarps = 4;
constexpr uint32_t kAnyTile0 = 4;  // zone-0 bins of a window mapped by all lanes together

struct EncUnit {
  uint64_t win;  // first window in its stream
  uint32_t seg;
  uint32_t n;    // windows
};

// Rows of n floats in 16-byte pieces, an odd number of them (rows of
// different windows start in different banks).
__host__ __device__ constexpr uint32_t any_pitch(uint32_t n) { return ((n + 3) / 4 | 1u) * 4; }
__host__ __device__ constexpr uint32_t any_pairs4(uint32_t N) { return ((N + 1) / 2 + 3) / 4 * 4; }
// Windows per tile: enough for one item of four windows and four bins per
// lane, within 2048 samples.
__host__ __device__ constexpr uint32_t any_groups(uint32_t E) { return ((E + 1) / 2 + 3) / 4 + (E / 2 + 3) / 4; }
__host__ __device__ constexpr uint32_t any_tile(uint32_t N, uint32_t E) {
  uint32_t t = 16;
  while (t < 64 && any_groups(E) * t / 4 < 32 && 2 * t * N <= 2048) t *= 2;
  return t;
}
// Bytes per warp: samples, folded rows, their sums of magnitudes, zone-0 bins,
// the list of bins to settle, levels.
__host__ __device__ constexpr uint32_t any_bytes(uint32_t N, uint32_t E) {
  const uint32_t t = any_tile(N, E);
  return t * any_pitch(N) * 4 + 2 * t * any_pitch(any_pairs4(N)) * 4 + 4 * t * 4 + t * kAnyTile0 * 4 + 512 * 2 +
         (t * E + 15) / 16 * 16;
}

__global__ void __launch_bounds__(kAnyWarps * 32, 4) k_enc_levels_any(EncParams p, uint64_t n_units, uint32_t warp_bytes) {
  extern __shared__ __align__(16) unsigned char any_smem[];
  dependents_may_start();
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  const uint64_t unit = (uint64_t)blockIdx.x * kAnyWarps + wid;
  if (unit >= n_units) return;  // the whole warp
  const EncUnit un = p.units[unit];
  // by value: read through references they are loaded again after every store
  const EncSeg sg = p.segs[un.seg];
  const EncDomain d = p.doms[sg.domain];
  const uint32_t N = d.N, E = d.E, B1 = d.B1, B2 = d.B2;
  const uint32_t P = (N + 1) / 2, P4 = any_pairs4(N), tile = any_tile(N, E);
  const uint32_t xp = any_pitch(N), up = any_pitch(P4);
  const uint32_t evens = (E + 1) / 2, ge = (evens + 3) / 4, go = (E / 2 + 3) / 4;
  float *const xs = reinterpret_cast<float *>(any_smem + (size_t)wid * warp_bytes);
  float *const us = xs + tile * xp;          // [tile][up], then v
  float *const vs = us + tile * up;
  float *const sums = vs + tile * up;        // [u half 0, u half 1, v half 0, v half 1][tile]
  float *const z0 = sums + 4 * tile;         // [tile][kAnyTile0]
  uint16_t *const work = reinterpret_cast<uint16_t *>(z0 + tile * kAnyTile0);
  uint8_t *const lev = reinterpret_cast<uint8_t *>(work + 512);
  const float *const src0 = p.x + sg.in_offset + un.win * N;
  const uint64_t avail0 = sg.n_samples - un.win * N;  // samples of the stream from the unit's first
  const bool vec = N % 4 == 0 && (reinterpret_cast<uintptr_t>(src0) & 15u) == 0;
  const float *const dots = p.dots + d.dot_off;
  // n < 2^16 divided by N or N / 4 by a multiplication
  const uint32_t magic = (uint32_t)((0x100000000ull + N - 1) / N);
  auto load = [&](uint32_t w0) {  // the tile's samples, zero past the stream's end
    const uint32_t nw = un.n - w0 < tile ? un.n - w0 : tile, total = nw * N;
    const float *src = src0 + (uint64_t)w0 * N;
    const uint64_t left = avail0 - (uint64_t)w0 * N;
    if (vec && left >= total) {
      for (uint32_t i = 4 * lane; i < total; i += 128) {
        const uint32_t w = __umulhi(i, magic);
        cp_async_16(xs + w * xp + (i - w * N), src + i);
      }
    } else {
      for (uint32_t i = lane; i < total; i += 32) {
        const uint32_t w = __umulhi(i, magic);
        cp_async_4z(xs + w * xp + (i - w * N), i < left ? src + i : p.x, i < left ? 4u : 0u);
      }
    }
    cp_async_commit_group();
  };
  load(0);
  for (uint32_t w0 = 0; w0 < un.n; w0 += tile) {
    const uint32_t nw = un.n - w0 < tile ? un.n - w0 : tile;
    cp_async_wait_group<0>();
    __syncwarp();
    // ---- fold: lane (or lanes' turn t) = window and every other piece of four pairs
    for (uint32_t t = lane; t < 2 * tile; t += 32) {
      const uint32_t w = t % tile, h = t / tile;
      const float *x = xs + w * xp;
      float su = 0.0f, sv = 0.0f;
      for (uint32_t c = 4 * h; c < P4; c += 8) {
        float a[4], b[4];
        if (N % 4 == 0) {
          const float4 q = *reinterpret_cast<const float4 *>(x + c);
          const float4 r = *reinterpret_cast<const float4 *>(x + N - 4 - c);
          a[0] = q.x, a[1] = q.y, a[2] = q.z, a[3] = q.w;
          b[0] = r.w, b[1] = r.z, b[2] = r.y, b[3] = r.x;
        } else {
#pragma unroll
          for (uint32_t i = 0; i < 4; ++i) {
            a[i] = c + i < P ? x[c + i] : 0.0f;
            b[i] = c + i < P ? x[N - 1 - c - i] : 0.0f;
          }
        }
        float u[4], v[4];
#pragma unroll
        for (uint32_t i = 0; i < 4; ++i) {
          const bool in = c + i < P, mid = 2 * (c + i) + 1 == N;
          u[i] = in ? (mid ? a[i] : a[i] + b[i]) : 0.0f;
          v[i] = in && !mid ? a[i] - b[i] : 0.0f;
          su += fabsf(u[i]);
          sv += fabsf(v[i]);
        }
        *reinterpret_cast<float4 *>(us + w * up + c) = make_float4(u[0], u[1], u[2], u[3]);
        *reinterpret_cast<float4 *>(vs + w * up + c) = make_float4(v[0], v[1], v[2], v[3]);
      }
      sums[h * tile + w] = su;
      sums[(2 + h) * tile + w] = sv;
    }
    __syncwarp();
    if (w0 + tile < un.n) load(w0 + tile);
    // ---- bins, four windows x four bins a lane and round
    const uint64_t win = un.win + w0;
    const uint32_t wgs = tile / 4, items = wgs * (ge + go);
    for (uint32_t i0 = 0; i0 < items; i0 += 32) {
      const uint32_t item = i0 + lane;
      uint32_t undecided = 0, wg = 0, k0 = 0;
      if (item < items) {
        wg = item % wgs;
        const uint32_t bg = item / wgs;
        const bool odd = bg >= ge;
        k0 = odd ? 8 * (bg - ge) + 1 : 8 * bg;  // bins k0, k0 + 2, + 4, + 6
        const float *rows = (odd ? vs : us) + wg * up;
        const float *cs[4];
#pragma unroll
        for (uint32_t j = 0; j < 4; ++j) cs[j] = dots + (k0 + 2 * j < E ? k0 + 2 * j : k0) * P4;
        float2 pair[4][4];  // sums over even and odd n
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) pair[i][j] = make_float2(0.0f, 0.0f);
        for (uint32_t c = 0; c < P4; c += 4) {
          float4 f[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) f[i] = *reinterpret_cast<const float4 *>(rows + i * wgs * up + c);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float4 g = __ldg(reinterpret_cast<const float4 *>(cs[j] + c));
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              pair[i][j] = __ffma2_rn(make_float2(f[i].x, f[i].y), make_float2(g.x, g.y), pair[i][j]);
              pair[i][j] = __ffma2_rn(make_float2(f[i].z, f[i].w), make_float2(g.z, g.w), pair[i][j]);
            }
          }
        }
        float acc[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = pair[i][j].x + pair[i][j].y;
        // bound on |a - a64|, a the unscaled sum (c = a 2 / N), per window
        float eb[4];
        bool finite = true;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint32_t w = wg + i * wgs;
          const float su = sums[w] + sums[tile + w], sv = sums[2 * tile + w] + sums[3 * tile + w];
          eb[i] = (odd ? sv : su) * ((float)(P + 4) * 0x1p-24f) + (su + sv) * 0x1p-40f + 1e-28f;
          finite = finite && (su + sv <= 1.0e38f || w >= nw);
        }
        if (d.z1_f32 && B1 <= kAnyTile0 && finite) {
          // every bin as one of zone 1, branch-free as in tier1_bins_fast; the others
          // masked (zone 0 is mapped below and written over this)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const uint32_t w = wg + i * wgs;
            const float base = eb[i] + d.u1_slack;
            uint8_t *const out = lev + w * E + k0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const uint32_t k = k0 + 2 * j;
              const float ak = fabsf(acc[i][j]);
              const float m = fmaf(ak, 0x1p-21f, base);
              const float lo = ak - m, hi = ak + m;
              const bool dz = hi < d.u1_d1, edge = lo <= d.u1_d1, pos = acc[i][j] > 0.0f;
              const float kk = pos ? d.u1_kp : d.u1_kn;
              const int v0 = __float2int_rd(fmaf(fminf(lo, d.u1_A1) - d.u1_d1, kk, 0.5f));
              const int v1 = __float2int_rd(fmaf(fminf(hi, d.u1_A1) - d.u1_d1, kk, 0.5f));
              const bool und = !dz && (edge || v0 != v1) && k >= B1 && k < B2 && w < nw;
              undecided |= und ? 1u << (4 * i + j) : 0u;
              if (k < E) out[2 * j] = (uint8_t)(dz || k >= B2 ? 128u : und ? 0u : (uint32_t)(pos ? 129 + v0 : 127 - v0));
              if (j < 2 && k < B1) z0[w * kAnyTile0 + k] = acc[i][j];  // k < 4: j = 0, 1
            }
          }
        } else {
#pragma unroll 1
          for (int i = 0; i < 4; ++i) {
            const uint32_t w = wg + i * wgs;
            if (w >= nw) continue;
            const float su = sums[w] + sums[tile + w], sv = sums[2 * tile + w] + sums[3 * tile + w];
            const bool fin = su + sv <= 1.0e38f;
            const float e = i == 0 ? eb[0] : i == 1 ? eb[1] : i == 2 ? eb[2] : eb[3];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const uint32_t k = k0 + 2 * j;
              if (k >= E) continue;
              const float a = i == 0 ? acc[0][j] : i == 1 ? acc[1][j] : i == 2 ? acc[2][j] : acc[3][j];
              if (k < B1 && k < kAnyTile0) {
                z0[w * kAnyTile0 + k] = a;
                continue;
              }
              uint32_t L = 128u;
              bool und = false;
              if (k < B2) {
                const float c = a * d.two_over_n;
                if (!fin) {
                  und = true;
                } else if (k < B1) {
                  const float m = e * d.two_over_n + d.slack0 + fabsf(c) * 0x1p-21f;
                  L = zone0_level32(c - m, d);
                  und = L != zone0_level32(c + m, d);
                } else {
                  und = !zone1_decide32(c, e * d.two_over_n + d.slack1 + fabsf(c) * 0x1p-21f, d, L);
                }
              }
              undecided |= und ? 1u << (4 * i + j) : 0u;
              lev[w * E + k] = (uint8_t)(und ? 0u : L);
            }
          }
        }
      }
      // ---- the bins that bound did not settle: a few to the list (their level, 0
      // here, is written after the tile's), many from the compensated sum
      const uint32_t cnt = (uint32_t)__popc(undecided);
      const uint32_t incl = lane_prefix(cnt, lane);
      const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
      if (total) {
        uint32_t o = incl - cnt;
        for (uint32_t u = undecided; u; u &= u - 1u) {
          const uint32_t q = (uint32_t)(__ffs(u) - 1);
          work[o++] = (uint16_t)((wg + (q >> 2) * wgs) * 128u + k0 + 2 * (q & 3u));
        }
        __syncwarp();
        for (uint32_t i = lane; i < total; i += 32) {
          const uint32_t w = work[i] >> 7, k = work[i] & 127u;
          const uint64_t g = sg.level_offset + (win + w) * E + k;
          uint32_t L = 0u;
          if (total <= kTier2Inline || !level_compensated(p, g, un.seg, L)) {
            const unsigned int slot = fb_slot(p);
            L = 0u;
            if (slot != ~0u)
              p.fb_list[slot] = fb_entry(g, un.seg);
            else
              L = level_fp64_seg(p, g, un.seg);
          }
          lev[w * E + k] = (uint8_t)L;
        }
      }
      __syncwarp();
    }
    // ---- zone 0, a bin a lane
    const uint32_t nz = B1 < kAnyTile0 ? B1 : kAnyTile0;
    for (uint32_t t = lane; t < nw * nz; t += 32) {
      const uint32_t w = t / nz, k = t - w * nz;
      const float su = sums[w] + sums[tile + w], sv = sums[2 * tile + w] + sums[3 * tile + w];
      const float eb = ((k & 1u) ? sv : su) * ((float)(P + 4) * 0x1p-24f) + (su + sv) * 0x1p-40f + 1e-28f;
      const float c = z0[w * kAnyTile0 + k] * d.two_over_n;
      const float m = eb * d.two_over_n + d.slack0 + fabsf(c) * 0x1p-21f;
      uint32_t L = zone0_level32(c - m, d);
      if (!(su + sv <= 1.0e38f) || L != zone0_level32(c + m, d)) {
        const uint64_t g = sg.level_offset + (win + w) * E + k;
        const unsigned int slot = fb_slot(p);
        L = 0u;
        if (slot != ~0u)
          p.fb_list[slot] = fb_entry(g, un.seg);
        else
          L = level_fp64_seg(p, g, un.seg);
      }
      lev[w * E + k] = (uint8_t)L;
    }
    __syncwarp();
    // ---- the tile's levels, consecutive lanes to consecutive bytes
    uint8_t *const dst = p.levels + sg.level_offset + win * E;
    const uint32_t bytes = nw * E;
    if ((reinterpret_cast<uintptr_t>(dst) & 15u) == 0 && (bytes & 15u) == 0) {
      for (uint32_t i = 16 * lane; i < bytes; i += 512)
        *reinterpret_cast<uint4 *>(dst + i) = *reinterpret_cast<const uint4 *>(lev + i);
    } else {
      for (uint32_t i = lane; i < bytes; i += 32) dst[i] = lev[i];
    }
    __syncwarp();
  }
}

// A stream whose bins take a thread each, and how many such bins come before it.
struct EncBins {
  uint32_t seg;
  uint32_t base;
};
// Streams of one window or of at most a warp's bins: a warp of k_enc_levels_any
// takes 2.3 ns (N = 4) to 18 ns (N = E = 128) for one however few windows it has, as
// compensated sums a thread each they take 0.2 to 5.  200,000 streams of four samples
// at N = 4: 466 us there, 36 here, of 32 475 and 254; of twenty at (24, 12) 501 and
// 102; of forty at (64, 32) 638 and 270, at (128, 128) 3645 and 1013.
__host__ __device__ constexpr bool few_bins(uint64_t n_windows, uint32_t E) { return n_windows == 1 || n_windows * E <= 32; }

__global__ void __launch_bounds__(256) k_enc_levels_bins(EncParams p) {
  dependents_may_start();
  dependency_wait();  // k_enc_fallback, behind this kernel, waits for this one only
  const uint32_t b = blockIdx.x * 256u + threadIdx.x;
  if (b >= p.n_bins) return;
  uint32_t i = p.bin_first[b >> 5];
  while (i + 1 < p.n_bin_segs && p.bins[i + 1].base <= b) ++i;
  const uint64_t s = p.bins[i].seg, g = p.segs[s].level_offset + (b - p.bins[i].base);
  uint32_t L;
  if (!level_compensated<false>(p, g, s, L)) {
    const unsigned int slot = fb_slot(p);
    if (slot != ~0u) {
      p.fb_list[slot] = fb_entry(g, s);
      return;  // k_enc_fallback writes the level
    }
    L = level_fp64_seg(p, g, s);
  }
  p.levels[g] = (uint8_t)L;
}

// The listed bins, one per thread: from their compensated FP32 coefficient
// where its bound settles the level, else from their FP64 coefficient.
__global__ void __launch_bounds__(256) k_enc_fallback(EncParams p) {
  dependents_may_start();
  dependency_wait();  // the list
  const unsigned int n = min(*p.fb_count, p.fb_cap);
  for (unsigned int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const unsigned long long e = p.fb_list[i];
    const uint64_t g = e & ((1ull << 40) - 1ull), s = e >> 40;
    uint32_t L;
    if (!level_compensated(p, g, s, L)) L = level_fp64_seg(p, g, s);
    p.levels[g] = (uint8_t)L;
  }
}

// k_enc_pack: one warp per part of a block.  The part's levels (and the 64 after
// it, which its last word may reach into) come into shared memory; the lanes turn
// two words of the start bitmap each into a list of starts; then one lane per
// word: its codewords shifted into 64 bits one after the other (a table entry
// holds the code left-aligned above its length, so a funnel shift by the entry
// appends it), five operations a codeword beside the loop.  A word belongs to
// the part it starts in.
constexpr uint32_t kPackWarps = 4;
constexpr uint32_t kPackPart = 2048;                       // symbols of a part
constexpr uint32_t kPartWords = kPackPart / 32;            // words of its bitmap (two a lane)
constexpr uint32_t kPackSpan = kPackPart + 64;             // symbols a part's words may hold
constexpr uint32_t kPackStage = (kPackSpan + 16 + 15) / 16 * 16;
constexpr uint32_t kPackList = kPackPart / 4 + 2;          // starts of a part (a word holds at least four codewords) + end

template <bool TAB>
__global__ void __launch_bounds__(kPackWarps * 32) k_enc_pack(EncParams p) {
  extern __shared__ uint32_t code_s[];  // TAB: [n_domains][256] table entries
  __shared__ __align__(16) uint8_t stage_s[kPackWarps][kPackStage];
  __shared__ uint16_t list_s[kPackWarps][kPackList];
  if (TAB) {
    for (uint32_t i = threadIdx.x; i < p.n_doms * 256u; i += kPackWarps * 32) code_s[i] = __ldg(p.code_tab + i);
    __syncthreads();
  }
  dependency_wait();  // the scan
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  const uint64_t item = (uint64_t)blockIdx.x * kPackWarps + wid, b = item / (kPackBlock / kPackPart);
  const uint32_t part = (uint32_t)(item % (kPackBlock / kPackPart));
  if (b >= p.n_blocks) return;  // the whole warp
  const uint32_t s = p.block_seg[b];
  if (p.seg_bad[s]) return;
  const EncSeg &sg = p.segs[s];
  const uint64_t L = sg.n_windows * p.doms[sg.domain].E;
  const uint64_t i0 = (b - sg.block_base) * kPackBlock + part * kPackPart;
  if (i0 >= L) return;
  const uint32_t nb = (uint32_t)(L - i0 < kPackPart ? L - i0 : kPackPart);
  const uint32_t span = (uint32_t)(L - i0 < kPackSpan ? L - i0 : kPackSpan);
  const uint8_t *const lv = p.levels + sg.level_offset;  // the stream's levels
  uint8_t *const stage = stage_s[wid];
  uint16_t *const list = list_s[wid];
  // levels: 16-byte pieces from the aligned address at or before the block's first
  const uintptr_t a0 = reinterpret_cast<uintptr_t>(lv + i0);
  const uint32_t sh = (uint32_t)(a0 & 15u);
  const uintptr_t lo = reinterpret_cast<uintptr_t>(lv), hi = lo + L;
  for (uint32_t c = lane * 16u; c < sh + span; c += 512u) {
    const uintptr_t a = a0 - sh + c;
    uint4 q = make_uint4(0u, 0u, 0u, 0u);
    if (a >= lo && a + 16 <= hi) {
      q = *reinterpret_cast<const uint4 *>(a);
    } else {  // the stream's ends: nothing outside it is read
      uint32_t t[4] = {0u, 0u, 0u, 0u};
#pragma unroll
      for (int r = 0; r < 16; ++r)
        if (a + r >= lo && a + r < hi) t[r >> 2] |= (uint32_t)*reinterpret_cast<const uint8_t *>(a + r) << (8 * (r & 3));
      q = make_uint4(t[0], t[1], t[2], t[3]);
    }
    *reinterpret_cast<uint4 *>(stage + c) = q;
  }
  // starts
  const uint32_t *const row = p.masks + b * kMaskWords + part * kPartWords;
  const uint2 m = *(reinterpret_cast<const uint2 *>(row) + lane);
  uint32_t before = 0;  // words that start in the block's parts before this one
  for (uint32_t q = 1; q <= part; ++q) {
    const uint2 x = *(reinterpret_cast<const uint2 *>(row - q * kPartWords) + lane);
    before += __popc(x.x) + __popc(x.y);
  }
  before = __reduce_add_sync(0xffffffffu, before);
  // a row's words past the stream's symbols are not written by k_enc_starts
  uint32_t m0 = 64u * lane < nb ? m.x : 0u, m1 = 64u * lane + 32u < nb ? m.y : 0u;
  const uint32_t cnt = __popc(m0) + __popc(m1);
  const uint32_t incl = lane_prefix(cnt, lane);
  const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
  uint32_t o = incl - cnt;
  for (; m0; m0 &= m0 - 1u) list[o++] = (uint16_t)(64u * lane + (uint32_t)(__ffs(m0) - 1));
  for (; m1; m1 &= m1 - 1u) list[o++] = (uint16_t)(64u * lane + 32u + (uint32_t)(__ffs(m1) - 1));
  if (lane == 0) {
    // the last word ends at the next part's first start (among its first 64
    // symbols), or with the stream
    uint32_t end = span;
    if (i0 + nb < L) {
      const uint32_t *nx = row + kPartWords;  // the next part's row, in this block or the next
      const uint32_t rest = (uint32_t)(L - i0 - nb < 64 ? L - i0 - nb : 64);
      const uint32_t n0 = nx[0], n1 = rest > 32u ? nx[1] : 0u;
      if (n0)
        end = nb + (uint32_t)(__ffs(n0) - 1);
      else if (n1)
        end = nb + 32u + (uint32_t)(__ffs(n1) - 1);
    }
    list[total] = (uint16_t)end;
  }
  __syncwarp();
  const uint64_t g0 = sg.word_offset + p.first_word[b] + before;
  const uint32_t *const tab = TAB ? code_s + sg.domain * 256u : p.code_tab + sg.domain * 256u;
  for (uint32_t j = lane; j < total; j += 32) {
    const uint32_t from = list[j], n = list[j + 1] - from;
    const uint8_t *src = stage + sh + from;
    uint32_t h = 0, l = 0, used = 0;
    auto add = [&](uint32_t level) {
      const uint32_t e = TAB ? tab[level] : __ldg(tab + level);
      h = __funnelshift_l(l, h, e);
      l = __funnelshift_l(e, l, e);
      used += e;  // the lengths add up in the low 16 bits (codes lie above them)
    };
    uint32_t i = 0;
    for (; i + 4 <= n; i += 4) {
      add(src[i]);
      add(src[i + 1]);
      add(src[i + 2]);
      add(src[i + 3]);
    }
    for (; i < n; ++i) add(src[i]);
    p.words[g0 + j] = ((uint64_t)h << 32 | l) << (64u - (used & 0xffffu));
    p.symlen[g0 + j] = (uint8_t)n;
  }
}

// k_enc_short: one lane per stream, by Alg. 1 as it stands, twice: the words
// counted (and the code and room checks), then put together and written.  Bound
// by a lane's chain, 63 ns a symbol for both, until some 20,000 streams fill the
// chip.  A warp per block (and four in k_enc_pack) takes about 10 ns a block of any
// size: 50,000 streams of 304 symbols took 463 us so (43 us when every block was
// a lane's), and take 41 us here.
constexpr uint32_t kShortThreads = 64;

template <bool TAB>
__global__ void __launch_bounds__(kShortThreads) k_enc_short(EncParams p) {
  dependents_may_start();
  extern __shared__ uint32_t short_s[];  // TAB: [n_domains][256] table entries
  if (TAB) {
    for (uint32_t i = threadIdx.x; i < p.n_doms * 256u; i += kShortThreads) short_s[i] = __ldg(p.code_tab + i);
    __syncthreads();
  }
  dependency_wait();  // the levels
  if (blockIdx.x == 0 && threadIdx.x == 0) *p.fb_count = 0;  // as in k_enc_scan
  const uint64_t i = (uint64_t)blockIdx.x * kShortThreads + threadIdx.x;
  if (i >= p.n_short) return;
  const uint32_t s = p.short_seg[i];
  const EncSeg &sg = p.segs[s];
  const uint32_t L = (uint32_t)(sg.n_windows * p.doms[sg.domain].E);
  const uint8_t *const lv = p.levels + sg.level_offset;
  const uint32_t *const tab = TAB ? short_s + sg.domain * 256u : p.code_tab + sg.domain * 256u;
  auto entry = [&](uint32_t level) -> uint32_t { return TAB ? tab[level] : __ldg(tab + level); };
  // fn(level) for the stream's levels in order
  auto each = [&](auto fn) {
    each_vector(lv, 0, L, [&](uint32_t v, const uint4 &q) {
      if (16 * v + 16 <= L) {
        each16(q, [&](int, uint32_t level) { fn(level); });
      } else {
#pragma unroll 1
        for (uint32_t j = 16 * v; j < L; ++j) fn((uint32_t)lv[j]);
      }
    });
  };
  uint32_t state = 0xFFFFFFFFu, words = 0, seen = 0;  // a full word: the first symbol starts one
  each([&](uint32_t level) {
    const uint32_t c = entry_len(entry(level)), k = c + kOff32;
    seen |= c;
    state = __viaddmax_u32(state, c, k);
    words += state == k ? 1u : 0u;
  });
  bool bad = seen >> 6;
  if (bad) enc_flag(p.status, FPTC_ENC_FLAG_NO_CODE, s);
  if (!bad && words > sg.room) {
    enc_flag(p.status, FPTC_ENC_FLAG_ROOM, s);
    bad = true;
  }
  p.seg_bad[s] = bad ? 1u : 0u;
  p.n_words[s] = bad ? 0u : words;
  if (bad || L == 0) return;
  uint64_t *w = p.words + sg.word_offset;
  uint8_t *n = p.symlen + sg.word_offset;
  uint32_t h = 0, l = 0, used = 0, count = 0;
  auto put = [&]() {
    *w++ = ((uint64_t)h << 32 | l) << (64u - used);
    *n++ = (uint8_t)count;
  };
  each([&](uint32_t level) {
    const uint32_t e = entry(level), c = e & 31u;
    if (used + c > 64u) {
      put();
      h = l = used = count = 0u;
    }
    h = __funnelshift_l(l, h, e);
    l = __funnelshift_l(e, l, e);
    used += c;
    ++count;
  });
  put();
}

struct DevGuard {
  int prev = -1;
  bool ok = true;
  explicit DevGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
    if (prev != dev) ok = cudaSetDevice(dev) == cudaSuccess;
  }
  ~DevGuard() {
    if (prev >= 0) cudaSetDevice(prev);
  }
};

fptc_status enc_cuda_fail(cudaError_t e, const char *what) {
  set_error("%s: %s", what, cudaGetErrorString(e));
  return e == cudaErrorMemoryAllocation ? FPTC_ERR_OUT_OF_MEMORY : FPTC_ERR_CUDA;
}

}  // namespace
}  // namespace fptc

using namespace fptc;

struct fptc_encoder {
  int device = 0;
  uint64_t n_segs = 0, n_windows = 0, n_levels = 0;
  std::vector<uint64_t> level_off;  // caller order
  EncSeg *d_segs = nullptr;
  EncDomain *d_doms = nullptr;
  double *d_cos = nullptr;
  float *d_cosf = nullptr;
  PackRec *d_recs = nullptr;                // [n_blocks]
  uint32_t *d_masks = nullptr;              // [n_blocks][kMaskWords]
  uint64_t *d_first_word = nullptr;         // [n_blocks]
  uint32_t *d_block_seg = nullptr;          // [n_blocks]
  uint32_t *d_short_seg = nullptr;          // [n_short]
  uint32_t *d_scan_seg = nullptr;           // [n_scan], null where n_short is 0
  uint64_t n_short = 0, n_scan = 0;
  uint32_t *d_code_tab = nullptr;           // [n_domains][256]
  uint32_t *d_lv_seg = nullptr;             // [warps of k_enc_levels_w32]
  long long *d_bound_keys = nullptr;        // [n_domains][2][255]
  EncUnit *d_units = nullptr;               // [n_units] (k_enc_levels_any)
  float *d_dots = nullptr;                  // its cosines
  EncBins *d_bins = nullptr;                // [n_bin_segs] (k_enc_levels_bins)
  uint32_t *d_bin_first = nullptr;          // [(n_bins + 31) / 32]
  uint64_t n_units = 0;
  uint32_t n_bin_segs = 0, n_bins = 0;
  uint32_t any_warp_bytes = 0;              // its shared memory per warp
  bool w32 = false;               // every domain N = 32, E = 16: the window-per-thread level kernel
  uint32_t *d_seg_bad = nullptr;
  unsigned long long *d_fb_list = nullptr;
  unsigned int *d_fb_count = nullptr;
  uint32_t fb_cap = 0;
  uint64_t n_blocks = 0;
  int sm_count = 1;
  uint32_t n_doms = 0;
  EncStatus *d_status = nullptr;
  uint8_t *d_lev_scratch = nullptr;
};

namespace {

void enc_free(fptc_encoder *e) {
  cudaFree(e->d_segs);
  cudaFree(e->d_doms);
  cudaFree(e->d_cos);
  cudaFree(e->d_cosf);
  cudaFree(e->d_recs);
  cudaFree(e->d_masks);
  cudaFree(e->d_first_word);
  cudaFree(e->d_block_seg);
  cudaFree(e->d_short_seg);
  cudaFree(e->d_scan_seg);
  cudaFree(e->d_code_tab);
  cudaFree(e->d_lv_seg);
  cudaFree(e->d_units);
  cudaFree(e->d_dots);
  cudaFree(e->d_bins);
  cudaFree(e->d_bin_first);
  cudaFree(e->d_bound_keys);
  cudaFree(e->d_seg_bad);
  cudaFree(e->d_fb_list);
  cudaFree(e->d_fb_count);
  cudaFree(e->d_status);
  cudaFree(e->d_lev_scratch);
}

struct EncDeleter {
  void operator()(fptc_encoder *e) const {
    enc_free(e);
    delete e;
  }
};

template <typename T>
cudaError_t enc_upload(T **dst, const T *src, size_t n) {
  cudaError_t e = cudaMalloc(reinterpret_cast<void **>(dst), std::max<size_t>(n, 1) * sizeof(T));
  if (e == cudaSuccess && n) e = cudaMemcpy(*dst, src, n * sizeof(T), cudaMemcpyHostToDevice);
  return e;
}

EncParams enc_params(const fptc_encoder *e, uint64_t *d_words, uint8_t *d_symlen, uint64_t *d_n_words,
                     uint8_t *levels) {
  EncParams p{};
  p.words = d_words;
  p.symlen = d_symlen;
  p.n_words = d_n_words;
  p.levels = levels;
  p.segs = e->d_segs;
  p.doms = e->d_doms;
  p.cosv = e->d_cos;
  p.cosf = e->d_cosf;
  p.recs = e->d_recs;
  p.masks = e->d_masks;
  p.first_word = e->d_first_word;
  p.n_doms = e->n_doms;
  p.block_seg = e->d_block_seg;
  p.short_seg = e->d_short_seg;
  p.n_short = e->n_short;
  p.scan_seg = e->d_scan_seg;
  p.n_scan = e->n_scan;
  p.code_tab = e->d_code_tab;
  p.lv_seg = e->d_lv_seg;
  p.units = e->d_units;
  p.dots = e->d_dots;
  p.bins = e->d_bins;
  p.bin_first = e->d_bin_first;
  p.n_bin_segs = e->n_bin_segs;
  p.n_bins = e->n_bins;
  p.bound_keys = e->d_bound_keys;
  p.seg_bad = e->d_seg_bad;
  p.fb_list = e->d_fb_list;
  p.fb_count = e->d_fb_count;
  p.fb_cap = e->fb_cap;
  p.n_blocks = e->n_blocks;
  p.status = e->d_status;
  p.n_segs = e->n_segs;
  p.n_levels = e->n_levels;
  return p;
}

// The streams that k_enc_short packs: those of at most X symbols, X such that it
// gains most over a warp for each of their blocks, if it gains anything.  In
// nanoseconds, measured: 10 a block and 0.001 a symbol there; here the longest
// stream's 63 a symbol or, of very many, 0.003 for each (16,384 streams of 2048
// symbols: 180 us there, 132 here; 4000 of them 57 and 131; 1000 of 304 symbols 23
// and 23, 4000 of them 52 and 23).
std::vector<uint32_t> choose_short(const std::vector<EncSeg> &segs, const std::vector<EncDomain> &doms) {
  std::vector<std::pair<uint32_t, uint32_t>> single;  // (symbols, segment)
  for (size_t i = 0; i < segs.size(); ++i) {
    const uint64_t L = segs[i].n_windows * doms[segs[i].domain].E;
    if (L <= kPackBlock) single.push_back({(uint32_t)L, (uint32_t)i});
  }
  std::sort(single.begin(), single.end());
  double best = 0.0, symbols = 0.0;
  size_t take = 0;
  for (size_t i = 0; i < single.size(); ++i) {
    symbols += single[i].first;
    if (i + 1 < single.size() && single[i + 1].first == single[i].first) continue;
    const double gain = 10.0 * (double)(i + 1) + 0.001 * symbols - std::max(6000.0 + 63.0 * single[i].first, 0.003 * symbols);
    if (gain > best) {
      best = gain;
      take = i + 1;
    }
  }
  std::vector<uint32_t> r(take);  // neighbours in a warp are as long as one another
  for (size_t i = 0; i < take; ++i) r[i] = single[i].second;
  return r;
}

bool aligned(const void *p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

}  // namespace

extern "C" {

fptc_status fptc_encoder_create(fptc_encoder **enc, int device, const fptc_domain *domains, uint32_t n_domains,
                                const fptc_segment *segments, uint64_t n_segments) {
  return guarded([&]() -> fptc_status {
    clear_error();
    if (!enc) {
      set_error("NULL encoder pointer");
      return FPTC_ERR_INVALID_ARGUMENT;
    }
    *enc = nullptr;
    if (!domains || n_domains == 0 || (n_segments && !segments)) {
      set_error("need at least one domain and a segment array");
      return FPTC_ERR_INVALID_ARGUMENT;
    }
    std::vector<EncDomain> doms(n_domains);
    std::vector<double> cosv;
    uint32_t dots_size = 0;
    std::vector<uint32_t> code_tab;
    std::vector<double> bounds(2 * 255 * (size_t)n_domains);
    std::vector<long long> bound_keys(bounds.size());
    for (uint32_t d = 0; d < n_domains; ++d) {
      const fptc_domain &dm = domains[d];
      fptc_status st = fptc_validate_domain(&dm);
      if (st != FPTC_OK) return st;
      EncDomain &x = doms[d];
      x.N = dm.N;
      x.E = dm.E;
      x.B1 = dm.B1;
      x.B2 = dm.B2;
      x.A0f = (float)dm.scale[0];
      x.A1f = (float)dm.scale[1];
      x.muf = (float)dm.mu;
      const double d1 = dm.alpha1 * dm.scale[1];  // as the FP64 quantizer computes it
      x.d1f = (float)d1;
      x.inv_A0f = dm.scale[0] > 1e-30 ? (float)(1.0 / dm.scale[0]) : 0.0f;
      x.inv_span1f = dm.scale[1] > 1e-30 && dm.scale[1] * (1.0 - dm.alpha1) > 0.0
                         ? (float)(1.0 / (dm.scale[1] - dm.alpha1 * dm.scale[1])) : 0.0f;
      x.inv_log1pmuf = (float)(1.0 / std::log1p(dm.mu));
      // 2^-18 of the zone scale: well above the FP32 evaluation error of either
      // map expressed in the coefficient (a few ulp of the scale: the maps'
      // arguments carry relative errors of a few 2^-24, over slopes of at most
      // mu / log1p(mu) and 1 / (1 - alpha1) per scale)
      x.slack0 = (float)(std::fabs(dm.scale[0]) * 0x1p-18);
      // zone 1's map is linear: its FP32 evaluation errs by a few 2^-24 A1 in
      // the coefficient (an emulation of both FP32 forms still brackets the
      // FP64 map with 2^-22 A1)
      x.slack1 = (float)(std::fabs(dm.scale[1]) * 0x1p-20);
      x.on0 = dm.scale[0] > 1e-30 ? 1u : 0u;
      // zone 1 is in use when A1 > 1e-30 and its linear part is not empty: with
      // alpha1 = 1 every |c| <= min(|c|, A1) <= d1, all level 128
      x.on1 = dm.scale[1] > 1e-30 && dm.scale[1] - d1 > 0.0 ? 1u : 0u;
      {
        const double h = dm.N / 2.0, span = dm.scale[1] - d1;
        x.u1_d1 = (float)(d1 * h);
        x.u1_A1 = (float)(dm.scale[1] * h);
        x.u1_slack = (float)(std::fabs(dm.scale[1]) * 0x1p-20 * h);
        x.u1_kp = span > 0.0 ? (float)(126.0 / span / h) : 0.0f;
        x.u1_kn = span > 0.0 ? (float)(127.0 / span / h) : 0.0f;
        x.z1_f32 = x.on1 && span >= dm.scale[1] * 0x1p-12 ? 1u : 0u;
      }
      // the host encoder's zone maps as boundaries: the levels of the second
      // and third tiers are those maps' own
      x.bnd_off = 2 * 255 * d;
      host_zone_bounds(dm, 0, bounds.data() + x.bnd_off);
      host_zone_bounds(dm, 1, bounds.data() + x.bnd_off + 255);
      x.cos_off = (uint32_t)cosv.size();
      x.dot_off = dots_size;
      dots_size += any_pairs4(dm.N) * dm.E;
      x.two_over_n = (float)(2.0 / dm.N);
      for (uint32_t k = 0; k < dm.E; ++k)
        for (uint32_t n = 0; n < dm.N; ++n) cosv.push_back(std::cos(M_PI * (2.0 * n + 1.0) * k / (2.0 * dm.N)));
      uint32_t c[256];
      st = fptc_canonical_codes(&dm, c);
      if (st != FPTC_OK) return st;
      for (int s = 0; s < 256; ++s) {  // codes have <= lmax <= 16 bits
        const uint32_t l = dm.code_len[s];
        code_tab.push_back(l ? c[s] << (32u - l) | l : 0u);
      }
    }
    // the same cosines as FP32 high and low parts, transposed per domain:
    // cosf[2 (cos_off + n E + k)] = hi, [+1] = lo, hi + lo = the FP64 cosine to 2^-48
    std::vector<float> cosf(2 * cosv.size());
    for (uint32_t d = 0; d < n_domains; ++d) {
      const EncDomain &x = doms[d];
      for (uint32_t k = 0; k < x.E; ++k)
        for (uint32_t n = 0; n < x.N; ++n) {
          const double c = cosv[x.cos_off + (size_t)k * x.N + n];
          const float h = (float)c;
          const size_t j = 2 * (x.cos_off + (size_t)n * x.E + k);
          cosf[j] = h;
          cosf[j + 1] = (float)(c - (double)h);
        }
    }
    std::vector<EncSeg> segs(n_segments);
    std::vector<uint64_t> level_off(n_segments);
    std::vector<std::pair<uint64_t, uint64_t>> rooms;
    std::vector<uint32_t> block_seg, scan_seg;
    uint64_t win = 0, lv = 0, blocks = 0;
    for (uint64_t i = 0; i < n_segments; ++i) {
      const fptc_segment &s = segments[i];
      if (s.domain >= n_domains) {
        set_error("segment %llu: domain %u out of range", (unsigned long long)i, s.domain);
        return FPTC_ERR_INVALID_ARGUMENT;
      }
      const fptc_domain &dm = domains[s.domain];
      EncSeg &e = segs[i];
      e.in_offset = s.out_offset;
      e.n_samples = s.n_samples;
      e.word_offset = s.word_offset;
      e.room = s.n_words;
      e.level_offset = lv;
      e.n_windows = (s.n_samples + dm.N - 1) / dm.N;
      e.domain = s.domain;
      e.pad = 0;
      level_off[i] = lv;
      win += e.n_windows;
      lv += e.n_windows * dm.E;
      if (s.n_words) rooms.push_back({s.word_offset, s.word_offset + s.n_words});
    }
    const std::vector<uint32_t> short_seg = choose_short(segs, doms);
    {
      std::vector<bool> is_short(n_segments);
      for (uint32_t i : short_seg) is_short[i] = true;
      for (uint64_t i = 0; i < n_segments; ++i) {
        segs[i].block_base = blocks;
        if (is_short[i]) continue;
        const uint64_t nb = (segs[i].n_windows * doms[segs[i].domain].E + kPackBlock - 1) / kPackBlock;
        blocks += nb;
        block_seg.insert(block_seg.end(), nb, (uint32_t)i);
        if (!short_seg.empty()) scan_seg.push_back((uint32_t)i);
      }
    }
    std::sort(rooms.begin(), rooms.end());
    for (size_t i = 1; i < rooms.size(); ++i)
      if (rooms[i].first < rooms[i - 1].second) {
        set_error("segment rooms overlap at word %llu", (unsigned long long)rooms[i].first);
        return FPTC_ERR_INVALID_ARGUMENT;
      }
    if (lv >= (uint64_t(1) << 40) || n_segments >= (uint64_t(1) << 24)) {  // the FP64 list packs both in 64 bits
      set_error("an encoder takes at most 2^40 levels and 2^24 segments");
      return FPTC_ERR_UNSUPPORTED;
    }
    DevGuard g(device);
    if (!g.ok) return enc_cuda_fail(cudaGetLastError(), "set device");
    // the encoder under construction: released into *enc only on success, so
    // that an error return or an exception frees what it holds (destroyed
    // before g, with the encoder's device still current)
    std::unique_ptr<fptc_encoder, EncDeleter> owner(new fptc_encoder);
    fptc_encoder *const e = owner.get();
    e->device = device;
    e->n_segs = n_segments;
    e->n_windows = win;
    e->n_doms = n_domains;
    e->n_levels = lv;
    e->n_blocks = blocks;
    e->n_short = short_seg.size();
    e->n_scan = n_segments - short_seg.size();
    e->level_off = level_off;
    cudaError_t err = cudaDeviceGetAttribute(&e->sm_count, cudaDevAttrMultiProcessorCount, device);
    if (err == cudaSuccess) err = enc_upload(&e->d_segs, segs.data(), segs.size());
    if (err == cudaSuccess) err = enc_upload(&e->d_doms, doms.data(), doms.size());
    if (err == cudaSuccess) err = enc_upload(&e->d_cos, cosv.data(), cosv.size());
    if (err == cudaSuccess) err = enc_upload(&e->d_cosf, cosf.data(), cosf.size());
    if (err == cudaSuccess)
      err = cudaFuncSetAttribute(k_enc_starts<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (kStartWarps + 1) * kStartWarpBytes + kTabDomains * 1024u);
    // four CTAs an SM
    if (err == cudaSuccess)
      err = cudaFuncSetAttribute(k_enc_starts<true>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)cudaSharedmemCarveoutMaxShared);
    if (err == cudaSuccess) err = cudaMalloc(&e->d_recs, std::max<uint64_t>(blocks, 1) * sizeof(PackRec));
    if (err == cudaSuccess) err = cudaMalloc(&e->d_masks, std::max<uint64_t>(blocks, 1) * kMaskWords * 4);
    if (err == cudaSuccess) err = cudaMalloc(&e->d_first_word, std::max<uint64_t>(blocks, 1) * 8);
    if (err == cudaSuccess) err = enc_upload(&e->d_block_seg, block_seg.data(), block_seg.size());
    if (err == cudaSuccess && e->n_short) {
      err = enc_upload(&e->d_short_seg, short_seg.data(), short_seg.size());
      if (err == cudaSuccess) err = enc_upload(&e->d_scan_seg, scan_seg.data(), scan_seg.size());
    }
    if (err == cudaSuccess) err = enc_upload(&e->d_code_tab, code_tab.data(), code_tab.size());
    for (size_t i = 0; i < bounds.size(); ++i) {  // order keys (see order_key); a NaN bound: no level reached
      long long b;
      std::memcpy(&b, &bounds[i], 8);
      bound_keys[i] = std::isnan(bounds[i]) ? std::numeric_limits<long long>::max()
                                            : (b < 0 ? b ^ 0x7fffffffffffffffll : b);
    }
    if (err == cudaSuccess) err = enc_upload(&e->d_bound_keys, bound_keys.data(), bound_keys.size());
    e->w32 = true;
    for (uint32_t d = 0; d < n_domains; ++d) e->w32 = e->w32 && domains[d].N == 32 && domains[d].E == 16;
    if (err == cudaSuccess && e->w32) {  // the segment of each window kernel warp's first window
      const uint64_t per = 32u * kLvGroups, n = (win + per - 1) / per;
      std::vector<uint32_t> lvs(n);
      uint64_t sidx = 0;
      for (uint64_t c = 0; c < n; ++c) {
        const uint64_t g = c * per * 16u;  // its first level (E = 16)
        while (sidx + 1 < n_segments && segs[sidx + 1].level_offset <= g) ++sidx;
        lvs[c] = (uint32_t)sidx;
      }
      err = enc_upload(&e->d_lv_seg, lvs.data(), lvs.size());
    }
    if (err == cudaSuccess && !e->w32) {  // units of whole tiles, up to eight where that leaves the chip full
      std::vector<float> dots;
      for (uint32_t d = 0; d < n_domains; ++d) {
        const uint32_t N = doms[d].N, pairs = (N + 1) / 2, p4 = any_pairs4(N);
        e->any_warp_bytes = std::max(e->any_warp_bytes, (any_bytes(N, doms[d].E) + 15u) / 16u * 16u);
        for (uint32_t k = 0; k < doms[d].E; ++k)
          for (uint32_t n = 0; n < p4; ++n)
            dots.push_back(n < pairs ? (float)cosv[doms[d].cos_off + (size_t)k * N + n] : 0.0f);
      }
      // streams of few bins: a kernel more, so where it saves the time of one or is the only one
      uint64_t some = 0, tiny = 0;
      for (const EncSeg &sg : segs) {
        some += sg.n_windows ? 1u : 0u;
        tiny += sg.n_windows && few_bins(sg.n_windows, doms[sg.domain].E) ? 1u : 0u;
      }
      const bool by_bins = tiny && (tiny == some || tiny >= 2048);
      auto binned = [&](const EncSeg &sg) { return by_bins && few_bins(sg.n_windows, doms[sg.domain].E); };
      std::vector<EncBins> bins;
      std::vector<uint32_t> bin_first;
      for (uint64_t i = 0; i < n_segments; ++i) {
        if (!segs[i].n_windows || !binned(segs[i])) continue;
        bins.push_back(EncBins{(uint32_t)i, e->n_bins});
        e->n_bins += (uint32_t)segs[i].n_windows * doms[segs[i].domain].E;  // 2^24 streams of 128 at most
        while (bin_first.size() * 32u < e->n_bins) bin_first.push_back((uint32_t)bins.size() - 1);
      }
      e->n_bin_segs = (uint32_t)bins.size();
      if (e->n_bins) err = enc_upload(&e->d_bins, bins.data(), bins.size());
      if (err == cudaSuccess && e->n_bins) err = enc_upload(&e->d_bin_first, bin_first.data(), bin_first.size());
      uint64_t tiles = 0;
      for (const EncSeg &sg : segs) {
        if (binned(sg)) continue;
        const uint32_t t = any_tile(doms[sg.domain].N, doms[sg.domain].E);
        tiles += (sg.n_windows + t - 1) / t;
      }
      const uint64_t per = std::min<uint64_t>(8, std::max<uint64_t>(1, tiles / ((uint64_t)e->sm_count * 32u)));
      std::vector<EncUnit> units;
      for (uint64_t i = 0; i < n_segments; ++i) {
        if (binned(segs[i])) continue;
        const uint64_t step = per * any_tile(doms[segs[i].domain].N, doms[segs[i].domain].E);
        for (uint64_t w = 0; w < segs[i].n_windows; w += step)
          units.push_back(EncUnit{w, (uint32_t)i, (uint32_t)std::min<uint64_t>(step, segs[i].n_windows - w)});
      }
      e->n_units = units.size();
      if (err == cudaSuccess) err = enc_upload(&e->d_units, units.data(), units.size());
      if (err == cudaSuccess) err = enc_upload(&e->d_dots, dots.data(), dots.size());
      if (err == cudaSuccess)
        err = set_dynamic_smem_limit(reinterpret_cast<const void *>(&k_enc_levels_any), kAnyWarps * e->any_warp_bytes);
    }
    if (err == cudaSuccess) err = cudaMalloc(&e->d_seg_bad, std::max<uint64_t>(n_segments, 1) * sizeof(uint32_t));
    // room for the bins decided in FP64: 0.2 % of them on signals, a few percent when
    // decoded signals are encoded again (their levels 127 and 129 reconstruct on the
    // deadzone edge); when it fills, the level kernels decide the rest themselves
    e->fb_cap = (uint32_t)std::min<uint64_t>(std::max<uint64_t>(lv / 16, 4096), uint64_t(1) << 28);
    if (err == cudaSuccess) err = cudaMalloc(&e->d_fb_list, (size_t)e->fb_cap * sizeof(unsigned long long));
    if (err == cudaSuccess) err = cudaMalloc(&e->d_fb_count, sizeof(unsigned int));
    if (err == cudaSuccess) err = cudaMemset(e->d_fb_count, 0, sizeof(unsigned int));
    if (err == cudaSuccess) {
      const EncStatus s0{0u, 0u, ~0ull};
      err = enc_upload(&e->d_status, &s0, 1);
    }
    if (err != cudaSuccess) return enc_cuda_fail(err, "encoder upload");
    *enc = owner.release();
    return FPTC_OK;
  });
}

void fptc_encoder_destroy(fptc_encoder *enc) {
  if (!enc) return;
  DevGuard g(enc->device);
  cudaDeviceSynchronize();
  EncDeleter()(enc);
}

uint64_t fptc_encoder_levels(const fptc_encoder *enc) { return enc ? enc->n_levels : 0; }

fptc_status fptc_encoder_level_offsets(const fptc_encoder *enc, uint64_t *offsets) {
  return guarded([&]() -> fptc_status {
    clear_error();
    if (!enc || (!offsets && enc->n_segs)) {
      set_error("NULL argument");
      return FPTC_ERR_INVALID_ARGUMENT;
    }
    std::copy(enc->level_off.begin(), enc->level_off.end(), offsets);
    return FPTC_OK;
  });
}

// One encode: the level kernel (unless the levels are given) and the packing.
static fptc_status enc_run(fptc_encoder *enc, const float *d_x, bool levels_given, const uint8_t *d_levels_in,
                           uint64_t *d_words, uint8_t *d_symlen, uint64_t *d_n_words, uint8_t *d_levels,
                           fptc_stream stream) {
  clear_error();
  if (!enc) {
    set_error("NULL encoder");
    return FPTC_ERR_INVALID_ARGUMENT;
  }
  if (enc->n_segs == 0) return FPTC_OK;
  if (!d_words || !d_symlen || !d_n_words || !aligned(d_words, 8) || !aligned(d_n_words, 8)) {
    set_error("d_words, d_symlen and d_n_words are required (8-byte aligned words and counts)");
    return FPTC_ERR_INVALID_ARGUMENT;
  }
  if (levels_given && enc->n_levels && !d_levels_in) {
    set_error("d_levels is required");
    return FPTC_ERR_INVALID_ARGUMENT;
  }
  if (!levels_given && enc->n_windows && (!d_x || !aligned(d_x, 4))) {
    set_error("d_x is required (float aligned)");
    return FPTC_ERR_INVALID_ARGUMENT;
  }
  DevGuard g(enc->device);
  if (!g.ok) return enc_cuda_fail(cudaGetLastError(), "set device");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  uint8_t *lev = levels_given ? const_cast<uint8_t *>(d_levels_in) : d_levels;
  if (!lev) {
    if (!enc->d_lev_scratch) {  // first encode without a level buffer: the scratch is the encoder's
      cudaError_t e = cudaMalloc(&enc->d_lev_scratch, std::max<uint64_t>(enc->n_levels, 1));
      if (e != cudaSuccess) return enc_cuda_fail(e, "level scratch");
    }
    lev = enc->d_lev_scratch;
  }
  EncParams p = enc_params(enc, d_words, d_symlen, d_n_words, lev);
  p.x = d_x;
  cudaError_t e = cudaSuccess;
  // each kernel may start beside the one before it and waits for it where its outputs are read
  auto launch = [&](const void *kernel, uint64_t grid, uint32_t threads, size_t smem, bool overlap) {
    if (e != cudaSuccess) return;
    void *args[] = {&p};
    e = launch_after(kernel, (uint32_t)grid, threads, args, smem, s, overlap);
  };
  const bool levels = !levels_given && enc->n_levels;
  if (levels) {
    if (enc->w32) {
      // kLvGroups groups a warp, or as many as leave every warp the chip can hold (20 an SM) one
      const uint64_t all = (enc->n_windows + 31) / 32, warps = (uint64_t)enc->sm_count * 20u;
      const uint32_t groups = (uint32_t)std::min<uint64_t>(kLvGroups, (all + warps - 1) / warps);
      const uint64_t per = (uint64_t)kLvThreads * groups;
      k_enc_levels_w32<<<(unsigned)((enc->n_windows + per - 1) / per), kLvThreads, 0, s>>>(p, enc->n_windows, groups);
    } else if (enc->n_units) {
      k_enc_levels_any<<<(unsigned)((enc->n_units + kAnyWarps - 1) / kAnyWarps), kAnyWarps * 32,
                         kAnyWarps * enc->any_warp_bytes, s>>>(p, enc->n_units, enc->any_warp_bytes);
    }
    e = cudaGetLastError();
    if (enc->n_bins)
      launch(reinterpret_cast<const void *>(&k_enc_levels_bins), (enc->n_bins + 255) / 256, 256, 0, enc->n_units > 0);
    launch(reinterpret_cast<const void *>(&k_enc_fallback), (uint64_t)enc->sm_count * 8u, 256, 0, true);
  }
  const bool tab = enc->n_doms <= kTabDomains;
  bool chained = levels;  // a kernel of this call is in front
  if (enc->n_short) {
    launch(tab ? reinterpret_cast<const void *>(&k_enc_short<true>) : reinterpret_cast<const void *>(&k_enc_short<false>),
           (enc->n_short + kShortThreads - 1) / kShortThreads, kShortThreads, tab ? enc->n_doms * 1024u : 0u, chained);
    chained = true;
  }
  if (enc->n_blocks) {
    launch(tab ? reinterpret_cast<const void *>(&k_enc_starts<true>) : reinterpret_cast<const void *>(&k_enc_starts<false>),
           (enc->n_blocks + kStartWarps - 1) / kStartWarps, (kStartWarps + 1) * 32,
           (kStartWarps + 1) * kStartWarpBytes + (tab ? enc->n_doms * 1024u : 0u), chained);
    chained = true;
  }
  if (enc->n_scan) launch(reinterpret_cast<const void *>(&k_enc_scan), (enc->n_scan * 32 + 127) / 128, 128, 0, chained);
  if (enc->n_blocks)
    launch(tab ? reinterpret_cast<const void *>(&k_enc_pack<true>) : reinterpret_cast<const void *>(&k_enc_pack<false>),
           (enc->n_blocks * (kPackBlock / kPackPart) + kPackWarps - 1) / kPackWarps, kPackWarps * 32,
           tab ? enc->n_doms * 1024u : 0u, true);
  if (e != cudaSuccess) return enc_cuda_fail(e, "encode launch");
  return FPTC_OK;
}

fptc_status fptc_encode_device(fptc_encoder *enc, const float *d_x, uint64_t *d_words, uint8_t *d_symlen,
                               uint64_t *d_n_words, uint8_t *d_levels, fptc_stream stream) {
  return enc_run(enc, d_x, false, nullptr, d_words, d_symlen, d_n_words, d_levels, stream);
}

fptc_status fptc_pack_device(fptc_encoder *enc, const uint8_t *d_levels, uint64_t *d_words, uint8_t *d_symlen,
                             uint64_t *d_n_words, fptc_stream stream) {
  return enc_run(enc, nullptr, true, d_levels, d_words, d_symlen, d_n_words, nullptr, stream);
}

fptc_status fptc_encoder_status(fptc_encoder *enc, uint32_t *flags, uint64_t *first_bad) {
  clear_error();
  if (!enc) {
    set_error("NULL encoder");
    return FPTC_ERR_INVALID_ARGUMENT;
  }
  DevGuard g(enc->device);
  cudaError_t e = cudaDeviceSynchronize();
  EncStatus h{};
  if (e == cudaSuccess) e = cudaMemcpy(&h, enc->d_status, sizeof(h), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) {
    const EncStatus s0{0u, 0u, ~0ull};
    e = cudaMemcpy(enc->d_status, &s0, sizeof(s0), cudaMemcpyHostToDevice);
  }
  if (e != cudaSuccess) return enc_cuda_fail(e, "read encoder status");
  if (flags) *flags = h.flags;
  if (first_bad) *first_bad = h.flags ? (uint64_t)h.first_bad : UINT64_MAX;
  if (h.flags) {
    set_error("encoder flagged segment %llu (flags 0x%x)", (unsigned long long)h.first_bad, h.flags);
    return FPTC_ERR_CORRUPT_STREAM;
  }
  return FPTC_OK;
}

}  // extern "C"
