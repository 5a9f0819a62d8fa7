// Fused decode for window shapes other than the Table 1 default: every domain of
// the plan has a window size N in [4, 128] and any kept-bin count E <= N,
// domains of different N in one batch (Table 1 gives the ranges; Fig. 14
// measures how the throughput moves with them).
//
// The SymLen decode is that of the warp-tile kernel (stream_tiles in
// warp_tile.cuh), with tiles of one output step (several where other domains'
// steps cost more: ranges are split by tiles).  The transform is
// one of two, chosen per segment from its domain (a warp-uniform switch):
//
//  * N a power of two and at most 64 bins that reconstruct to something
//    (kz = min(E, B2)): one window per lane (32 / N consecutive windows for
//    N < 32), by the even/odd split of the DCT-III down to one bin,
//        x[n] = e[n] + o[n],  x[N - 1 - n] = e[n] - o[n],
//    e the inverse of size N / 2 on the even bins, o the sum over the odd bins,
//    compiled per N and bin count (N / 4, N / 2 or N bins) with the cosines as
//    immediate operands: no basis passes through shared memory and a
//    coefficient is dequantized once.  At N = 64, E = 32 that is 684 multiply-
//    adds and 120 additions per window, against 1024 multiply-adds and one
//    16-byte basis read per four of them in the pair form below.  The samples go
//    to two 32 x 32 tiles per warp (32 windows x 32 samples, mirrored chunks of
//    the windows together) and from there by 3-D TMA stores (the output as
//    windows x chunks x 32 floats).  (64, 32), 67 M samples: 88 us,
//    171 us in the pair form (which then had compile-time N too).
//  * otherwise (shape_pairs): a window's samples as ceil(N / 2) mirrored pairs
//        x[n] = Ev[n] + Od[n],  x[N - 1 - n] = Ev[n] - Od[n],
//    Ev / Od the sums over even / odd bins, as a small matrix product per step: the
//    step's coefficients are dequantized once into shared memory, and a lane takes
//    four windows by eight pairs, two pairs per instruction (fma.f32x2): 16 of
//    those for three 16-byte reads.  Bound by shared-memory wavefronts (a 16-byte
//    read is four of them, whatever it shares).  One lane per
//    16 pairs of one window, with a basis read for every four multiply-adds and
//    the coefficients dequantized again by each lane of a window, took 228 us for
//    33 M samples at N = 100, E = 50; this form takes 111 us (133 us with each
//    coefficient stored twice and a lane's windows side by side, when rows of 24,
//    48 or 64 samples met in the same banks: N = 24, E = 12 took 117 us, now 83).
#pragma once

#include <cuda.h>

#include "warp_tile.cuh"


namespace fptc {
namespace {

using namespace wt;

// Per-domain view of the shared tables of the shape kernel.
struct DomS {
  uint32_t lut_off;    // bytes from the start of shared memory (entries len | level << 8)
  uint32_t deq_off;    // bytes: zone rows [kZRows][kZStride] floats
  uint32_t basis_off;  // bytes: [kz][pairs8] floats (shape_pairs)
  uint32_t shift;      // 32 - lmax
  uint32_t complete;
  uint32_t E, B1, kz;  // kz = min(E, B2)
  uint32_t T;          // windows per tile
  uint32_t N;
  uint32_t form;       // compiled transform: N << 8 | bins (0: shape_pairs)
  uint32_t step;       // windows per output step
};

__host__ __device__ constexpr bool shape_pow2(uint32_t N) { return (N & (N - 1)) == 0; }
__host__ __device__ constexpr uint32_t shape_pair_count(uint32_t N) { return (N + 1) / 2; }
__host__ __device__ constexpr uint32_t shape_pairs8(uint32_t N) { return (shape_pair_count(N) + 7) / 8 * 8; }

// The compiled transform of a domain (N << 8 | bins), or 0.  N >= 64 wants two
// output tiles per warp.
__host__ __device__ constexpr uint32_t shape_form(uint32_t N, uint32_t kz, uint32_t tiles) {
  if (!shape_pow2(N) || kz > 64 || (N > 32 && tiles < 2)) return 0;
  uint32_t bins = N >= 16 ? N / 4 : N;
  while (bins < kz) bins *= 2;
  return N << 8 | bins;
}

// Windows per lane of shape_pairs: four, two with one output tile per warp (up to
// 24 warps: 80 registers a thread, half of them accumulators at two).
__host__ __device__ constexpr uint32_t shape_pair_windows(uint32_t tiles) { return tiles > 1 ? 4 : 2; }

// Places a bin's coefficients take in shape_pairs for a step of `step` windows, m a
// lane: whole lanes' worth (m is the width of their read), and no more: m times
// the lane groups of a step, of which a warp has 32 / (groups of eight pairs).
__host__ __device__ constexpr uint32_t shape_pair_places(uint32_t step, uint32_t m) { return (step + m - 1) / m * m; }

// Windows per output step.  Compiled forms: 32 lanes, 32 / N windows each for N
// < 32.  shape_pairs: as many groups of its windows as lanes for their groups
// of eight pairs, less where the coefficients or the samples would not fit the
// warp's output tiles.  Either way at most 2048 symbols.
__host__ __device__ constexpr uint32_t shape_step(uint32_t N, uint32_t E, uint32_t kz, uint32_t tiles) {
  uint32_t w = 0;
  if (shape_form(N, kz, tiles)) {
    w = N >= 32 ? 32 : 1024 / N;
  } else {
    const uint32_t bytes = tiles * (uint32_t)kOutTile;
    const uint32_t m = shape_pair_windows(tiles);
    w = 32 / (shape_pairs8(N) / 8) * m;
    const uint32_t fit_c = bytes / (4 * (kz ? kz : 1)) / 4 * 4, fit_x = bytes / (4 * N) / 4 * 4;
    w = w < fit_c ? w : fit_c;
    w = w < fit_x ? w : fit_x;
  }
  const uint32_t most = (uint32_t)kTS / E;
  if (w > most) w = most;
  // where it can be, a multiple of 16 symbols (the steps' levels then start on
  // 16-byte boundaries): 16 / gcd(E, 16) windows; always so for compiled forms
  uint32_t q = 16;
  while (q > 1 && E % 2 == 0) {
    q /= 2;
    E /= 2;
  }
  return w / q * q ? w / q * q : w;
}

// Whether every (window of a step, group of eight pairs) of shape_pairs has a lane,
// and the step's coefficients and samples their place in the warp's output
// tiles, for the window sizes [lo, hi] (a range the compiler evaluates at once).
constexpr bool shape_pairs_covered(uint32_t tiles, uint32_t lo, uint32_t hi) {
  for (uint32_t N = lo; N <= hi; ++N)
    for (uint32_t E = 1; E <= N; ++E)
      for (uint32_t kz = E; kz; kz /= 2) {
        if (shape_form(N, kz, tiles)) continue;
        const uint32_t m = shape_pair_windows(tiles), step = shape_step(N, E, kz, tiles);
        const uint32_t places = shape_pair_places(step, m), bytes = tiles * (uint32_t)kOutTile;
        if (step == 0 || places / m * (shape_pairs8(N) / 8) > 32) return false;
        if (4 * kz * places > bytes || 4 * N * step > bytes) return false;
      }
  return true;
}
template <uint32_t LO, uint32_t HI>
struct ShapePairsCheck {
  static_assert(shape_pairs_covered(1, LO, HI), "a window's pairs without a lane");
  static_assert(shape_pairs_covered(2, LO, HI), "a window's pairs without a lane");
};
template struct ShapePairsCheck<4, 48>;
template struct ShapePairsCheck<49, 68>;
template struct ShapePairsCheck<69, 84>;
template struct ShapePairsCheck<85, 100>;
template struct ShapePairsCheck<101, 115>;
template struct ShapePairsCheck<116, 128>;

// Symbols a warp's stage holds (stream_tiles): a step's and a pass's.
__host__ __device__ constexpr int shape_cap(int tiles) { return tiles > 1 ? kTS + 1024 : kMiscBytes - stream_bytes(0); }

// Tables of every domain into shared memory from byte 0 (the layout of
// shape_smem_layout).  Returns the end offset.  Contains no barrier.
template <int THREADS, int TILES>
__device__ __forceinline__ uint32_t load_shape_tables(const DecodeParams &p, uint32_t n_domains, unsigned char *smem) {
  DomS *const ds = reinterpret_cast<DomS *>(smem);
  uint32_t off = (uint32_t)align16(sizeof(DomS) * (n_domains ? n_domains : 1));
  for (uint32_t d = 0; d < n_domains; ++d) {
    const DomainDev &dm = p.domains[d];
    const uint32_t N = dm.N, p8 = shape_pairs8(N), kz = dm.B2 < dm.E ? dm.B2 : dm.E;
    const uint32_t form = shape_form(N, kz, TILES);
    const uint32_t lut_off = off;
    const uint32_t deq_off = lut_off + (uint32_t)align16((size_t)2 << dm.lmax);
    const uint32_t basis_off = deq_off + kDeqBytes;
    off = basis_off + (form ? 0u : kz * p8 * 4);
    if (threadIdx.x == 0) {
      DomS x;
      x.lut_off = lut_off;
      x.deq_off = deq_off;
      x.basis_off = basis_off;
      x.shift = 32u - dm.lmax;
      x.complete = dm.complete;
      x.E = dm.E;
      x.B1 = dm.B1;
      x.kz = kz;
      x.T = dm.tile_windows;
      x.N = N;
      x.form = form;
      x.step = shape_step(N, dm.E, kz, TILES);
      ds[d] = x;
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
    if (form) continue;
    // the half basis B[k][n], n < ceil(N / 2), zero up to the next eight; a row holds
    // the first four of every eight, then the second four (consecutive groups of
    // pairs in consecutive 16 bytes)
    float *bas = reinterpret_cast<float *>(smem + basis_off);
    const float *g_bas = p.basis + dm.basis_offset;
    const uint32_t pairs = shape_pair_count(N);
    for (uint32_t i = threadIdx.x; i < kz * p8; i += THREADS) {
      const uint32_t k = i / p8, r = i - k * p8, h = r < p8 / 2 ? 0u : 1u, q = r - h * (p8 / 2);
      const uint32_t n = q / 4 * 8 + 4 * h + q % 4;
      bas[i] = n < pairs ? __ldg(g_bas + (size_t)k * N + n) : 0.0f;
    }
  }
  return off;
}

// Where the transform of a tile writes: the warp's staging tiles, the output
// tensor maps, and whether TMA stores may be used.
struct ShapeOut {
  unsigned char *otile;  // TWO: two consecutive tiles
  uint32_t sx;           // lane & 7
  uint32_t lane;
  const CUtensorMap *map;    // the output as rows of 32 floats
  const CUtensorMap *map_n;  // as windows x chunks x 32 floats, for the domain's N >= 64
  bool tma_ok;   // the segment's output starts on a 128-byte boundary and the rows' map is valid
  bool tma_n;    // and the other map is
  bool vec32, vec16;
};

// ---- inverse transform with compile-time cosines --------------------------------
// cos(pi m / (2 N)), m < 4 N, in double by Taylor series on [0, pi/2] after the
// reflections cos(2 pi - a) = cos(a), cos(pi - a) = -cos(a); rounded to float.
template <int N>
struct CosTab {
  float v[4 * N];
};
template <int N>
__host__ __device__ constexpr CosTab<N> make_cos_tab() {
  CosTab<N> t{};
  for (int m = 0; m < 4 * N; ++m) {
    int r = m > 2 * N ? 4 * N - m : m;  // angle pi r / (2 N) in [0, pi]
    const bool neg = r > N;
    if (neg) r = 2 * N - r;
    const double x = 3.14159265358979323846 * r / (2.0 * N), x2 = x * x;
    double term = 1.0, sum = 1.0;
    for (int i = 1; i < 16; ++i) {
      term *= -x2 / ((2.0 * i - 1.0) * (2.0 * i));
      sum += term;
    }
    t.v[m] = (float)(neg ? -sum : sum);
  }
  return t;
}

// o[n] = sum over the odd bins 2 j + 1 of a window of N (co[j], j < KO).
template <int N, int KO>
__device__ __forceinline__ float odd_sum(const float (&co)[KO], int n) {
  constexpr CosTab<N> T = make_cos_tab<N>();
  float o = co[0] * T.v[(2 * n + 1) % (4 * N)];
#pragma unroll
  for (int j = 1; j < KO; ++j) o = fmaf(co[j], T.v[((2 * n + 1) * (2 * j + 1)) % (4 * N)], o);
  return o;
}

// x[0 .. N) of one window from its first K coefficients (K a power of two;
// B[0][n] = 1/2).
template <int N, int K>
__device__ __forceinline__ void idct_small(const float (&c)[K], float (&x)[N]) {
  if constexpr (K == 1) {
#pragma unroll
    for (int n = 0; n < N; ++n) x[n] = 0.5f * c[0];
  } else {
    float ce[K / 2], co[K / 2], e[N / 2];
#pragma unroll
    for (int j = 0; j < K / 2; ++j) {
      ce[j] = c[2 * j];
      co[j] = c[2 * j + 1];
    }
    idct_small<N / 2, K / 2>(ce, e);
#pragma unroll
    for (int n = 0; n < N / 2; ++n) {
      const float o = odd_sum<N, K / 2>(co, n);
      x[n] = e[n] + o;
      x[N - 1 - n] = e[n] - o;
    }
  }
}

// Coefficients FIRST, FIRST + STEP, ... of a window (COUNT of them) from its
// level bytes lv: A_z unit_z(level), 0 from bin kz on.  `fast`: rows of a
// multiple of 8 bytes, every bin in use, Table 1's first zone (B1 = 2).
template <int FIRST, int STEP, int COUNT>
__device__ __forceinline__ void load_coefs(const uint8_t *lv, const float *deq, uint32_t B1, uint32_t kz, bool fast,
                                           float (&c)[COUNT]) {
  if (fast) {
    constexpr int kLast = FIRST + STEP * (COUNT - 1);
    uint32_t w[kLast / 16 * 4 + 4];
#pragma unroll
    for (int q = 0; q <= kLast / 8; q += 2) {
      if (kLast / 8 == q) {  // the row's last (or only) 8 bytes
        const uint2 v = reinterpret_cast<const uint2 *>(lv)[q];
        w[2 * q] = v.x;
        w[2 * q + 1] = v.y;
      } else {
        const uint4 v = *reinterpret_cast<const uint4 *>(lv + 8 * q);
        w[2 * q] = v.x;
        w[2 * q + 1] = v.y;
        w[2 * q + 2] = v.z;
        w[2 * q + 3] = v.w;
      }
    }
#pragma unroll
    for (int j = 0; j < COUNT; ++j) {
      const int k = FIRST + STEP * j;
      c[j] = deq[(k < 2 ? 0 : kZStride) + ((w[k >> 2] >> (8 * (k & 3))) & 0xffu)];
    }
  } else {
#pragma unroll
    for (int j = 0; j < COUNT; ++j) {
      const uint32_t k = FIRST + STEP * j;
      c[j] = k < kz ? deq[(k < B1 ? 0 : kZStride) + lv[k]] : 0.0f;
    }
  }
}

// Waits until at most PENDING of the warp's TMA stores still read their tile.
template <int PENDING>
__device__ __forceinline__ void tma_wait_read_but() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(PENDING) : "memory");
}

// Stores the 32 windows' chunk `chunk` staged in tile to rows of 32 floats at
// (window, chunk) of the map.
__device__ __forceinline__ void tma_store_chunk(const CUtensorMap *map, const void *tile, int32_t chunk, int32_t win) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(0), "r"(chunk), "r"(win), "r"(static_cast<uint32_t>(__cvta_generic_to_shared(tile)))
               : "memory");
}

constexpr uint32_t kAllTiles = 2;  // turn: every output tile may still be read by an earlier step's stores

// Dequantization + inverse transform + reassembly of a step of n windows from
// window win (levels at lv0), N <= 32: 1024 samples, a row of 32 per lane, in the
// tile whose turn it is (TILES alternate).
template <int N, int K, int TILES>
__device__ __forceinline__ void shape_rows(const DecodeParams &p, const UnitSeg &sg, const DomS &dd,
                                           const unsigned char *smem, const uint8_t *lv0, uint64_t win, uint32_t n,
                                           const ShapeOut &o, uint32_t &turn) {
  constexpr uint32_t M = 32 / N, R = 32 * M;  // windows per lane, per step
  const uint32_t lane = o.lane;
  const float *deq = reinterpret_cast<const float *>(smem + dd.deq_off);
  const bool fast = K % 8 == 0 && dd.E == K && dd.kz == K && dd.B1 == 2;
  const uint64_t S = sg.n_samples;
  unsigned char *const tile = o.otile + (turn & 1u) * kOutTile, *const row = tile + lane * 128;
  if (lane == 0) {  // earlier steps have left this tile (kAllTiles: another transform's, which used both)
    if (turn & kAllTiles)
      tma_wait_read_but<0>();
    else
      tma_wait_read_but<TILES - 1>();
  }
  __syncwarp();
#pragma unroll
  for (uint32_t m = 0; m < M; ++m) {
    if (M * lane + m >= n) break;
    float c[K], x[N];
    load_coefs<0, 1, K>(lv0 + (M * lane + m) * dd.E, deq, dd.B1, dd.kz, fast, c);
    idct_small<N, K>(c, x);
#pragma unroll
    for (int j = 0; j < N / 4; ++j)
      *reinterpret_cast<float4 *>(row + (((m * (N / 4) + j) ^ o.sx) << 4)) =
          make_float4(x[4 * j], x[4 * j + 1], x[4 * j + 2], x[4 * j + 3]);
  }
  const uint64_t s0 = win * N;  // first sample of the step in the segment
  if (o.tma_ok && n == R && s0 + 1024 <= S) {
    fence_async_shared();
    __syncwarp();
    if (lane == 0) tma_store_rows(o.map, tile, (int32_t)((sg.out_offset + s0) >> 5));
  } else {
    const uint64_t lim = (uint64_t)n * N < S - s0 ? (uint64_t)n * N : S - s0;
    const uint64_t r0 = (uint64_t)lane * 32;
    if (r0 < lim)
      store_row(row, o.sx, p.out + sg.out_offset + s0 + r0, lim - r0 < 32 ? (uint32_t)(lim - r0) : 32u, o.vec32, o.vec16);
    if (lane == 0) asm volatile("cp.async.bulk.commit_group;" ::: "memory");  // one group a step: the turns stay in step
  }
  turn = (turn & 1u) ^ (TILES - 1);
}

// The same for N = 64, 128: a step is 32 windows, one per lane; the chunks
// (32 samples) c and N / 32 - 1 - c of the windows mirror each other and are
// staged together, one tile each.
// Two levels of the split are open at once, so that no array of N / 2 samples is
// live beside the coefficients (register spills went through L2 here: shared
// memory leaves L1 little room): with h[n] the inverse of size N / 4 on every
// fourth bin and q[n] the sum over the bins 2, 6, 10, ...,
//   e[n] = h[n] + q[n],  e[N/2 - 1 - n] = h[n] - q[n]      (n < N / 4)
//   x[j] = e[j] + o[j],  x[N - 1 - j] = e[j] - o[j]        (j < N / 2).
template <int N, int K>
__device__ __forceinline__ void shape_windows(const DecodeParams &p, const UnitSeg &sg, const DomS &dd,
                                              const unsigned char *smem, const uint8_t *lv0, uint64_t win, uint32_t n,
                                              const ShapeOut &o) {
  constexpr int kChunks = N / 32;
  const uint32_t lane = o.lane;
  const float *deq = reinterpret_cast<const float *>(smem + dd.deq_off);
  const bool fast = K % 16 == 0 && dd.E == K && dd.kz == K && dd.B1 == 2;
  const uint64_t S = sg.n_samples;
  unsigned char *const ra = o.otile + lane * 128, *const rb = ra + kOutTile;  // the lane's rows
  const uint8_t *const lv = lv0 + (lane < n ? lane : 0u) * dd.E;
  float h[N / 4];
  {
    float c4[K / 4];
    load_coefs<0, 4, K / 4>(lv, deq, dd.B1, dd.kz, fast, c4);
    idct_small<N / 4, K / 4>(c4, h);
  }
  float c2[K / 4], co[K / 2];
  load_coefs<2, 4, K / 4>(lv, deq, dd.B1, dd.kz, fast, c2);
  load_coefs<1, 2, K / 2>(lv, deq, dd.B1, dd.kz, fast, co);
  const uint64_t s0 = (win + lane) * N;  // the window's first sample in the segment
  const bool tma_step = o.tma_n && n == 32 && (win + 32) * N <= S;
  // 16-byte piece b of a lane's row
  auto put4 = [&](unsigned char *row, int b, float v0, float v1, float v2, float v3) {
    *reinterpret_cast<float4 *>(row + ((b ^ o.sx) << 4)) = make_float4(v0, v1, v2, v3);
  };
#pragma unroll
  for (int q = 0; q < kChunks / 2; ++q) {  // chunks q and kChunks - 1 - q
    if (q > 0) {  // its q[n] are the other pair's: computed again, not kept in registers meanwhile
#pragma unroll
      for (int j = 0; j < K / 4; ++j) asm volatile("" : "+f"(c2[j]));
    }
    if (lane == 0) tma_wait_read_but<0>();
    __syncwarp();
#pragma unroll
    for (int g = 0; g < (N == 64 ? 4 : 8); ++g) {
      float a[4], z[4], a2[4], z2[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int m = 4 * g + i;
        const float t = odd_sum<N / 2, K / 4>(c2, N == 128 && q == 1 ? 31 - m : m);
        if (N == 64) {  // j = m and j = 31 - m: both chunks whole
          const float e1 = h[m] + t, e2 = h[m] - t;
          const float o1 = odd_sum<N, K / 2>(co, m), o2 = odd_sum<N, K / 2>(co, 31 - m);
          a[i] = e1 + o1;       // x[m]
          z[i] = e1 - o1;       // x[63 - m]
          a2[i] = e2 + o2;      // x[31 - m]
          z2[i] = e2 - o2;      // x[32 + m]
        } else {  // j = 32 q + m
          const float e = q == 0 ? h[m % (N / 4)] + t : h[(31 - m) % (N / 4)] - t;
          const float od = odd_sum<N, K / 2>(co, 32 * q + m);
          a[i] = e + od;
          z[i] = e - od;
        }
      }
      put4(ra, g, a[0], a[1], a[2], a[3]);
      put4(rb, 7 - g, z[3], z[2], z[1], z[0]);
      if (N == 64) {
        put4(ra, 7 - g, a2[3], a2[2], a2[1], a2[0]);
        put4(rb, g, z2[0], z2[1], z2[2], z2[3]);
      }
    }
    if (tma_step) {
      fence_async_shared();
      __syncwarp();
      if (lane == 0) {
        // chunk row of the step's first window in the output: window row / (N / 32), chunk the rest
        const uint64_t r = (sg.out_offset >> 5) + win * kChunks;
        const uint64_t a = r + q, b = r + kChunks - 1 - q;
        tma_store_chunk(o.map_n, o.otile, (int32_t)(a % kChunks), (int32_t)(a / kChunks));
        tma_store_chunk(o.map_n, o.otile + kOutTile, (int32_t)(b % kChunks), (int32_t)(b / kChunks));
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      }
    } else if (lane < n) {  // each lane its own rows
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const uint64_t t = s0 + 32 * (r ? kChunks - 1 - q : q);
        if (t < S)
          store_row(r ? rb : ra, o.sx, p.out + sg.out_offset + t, S - t < 32 ? (uint32_t)(S - t) : 32u, o.vec32, o.vec16);
      }
    }
  }
}

// The compiled transform of a step's domain (uniform over the warp); false: there is none.
// ONE: the only form of the plan's domains (0: any of them).
template <int TILES, uint32_t ONE>
__device__ __forceinline__ bool shape_compiled(const DecodeParams &p, const UnitSeg &sg, const DomS &dd,
                                               const unsigned char *smem, const uint8_t *lv0, uint64_t win, uint32_t n,
                                               const ShapeOut &o, uint32_t &turn) {
#define FPTC_ROWS(N, K) \
  case (N << 8 | K): \
    if constexpr (ONE == 0 || ONE == (N << 8 | K)) shape_rows<N, K, TILES>(p, sg, dd, smem, lv0, win, n, o, turn); \
    return true;
#define FPTC_WINDOWS(N, K) \
  case (N << 8 | K): \
    if constexpr (TILES == 2 && (ONE == 0 || ONE == (N << 8 | K))) \
      shape_windows<N, K>(p, sg, dd, smem, lv0, win, n, o); \
    turn = kAllTiles; \
    return true;
  switch (ONE ? ONE : dd.form) {
    FPTC_ROWS(4, 4)
    FPTC_ROWS(8, 8)
    FPTC_ROWS(16, 4)
    FPTC_ROWS(16, 8)
    FPTC_ROWS(16, 16)
    FPTC_ROWS(32, 8)
    FPTC_ROWS(32, 16)
    FPTC_ROWS(32, 32)
    FPTC_WINDOWS(64, 16)
    FPTC_WINDOWS(64, 32)
    FPTC_WINDOWS(64, 64)
    FPTC_WINDOWS(128, 32)
    FPTC_WINDOWS(128, 64)
  }
#undef FPTC_ROWS
#undef FPTC_WINDOWS
  return false;
}

// A 1-D bulk copy of `bytes` from shared memory to dst (both 16-byte aligned, a
// multiple of 16), as a group of its own.
__device__ __forceinline__ void bulk_store(float *dst, const void *src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(__cvta_generic_to_global(dst)),
               "r"(static_cast<uint32_t>(__cvta_generic_to_shared(src))), "r"(bytes)
               : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// The pair form, any N: a step of n windows (at most dd.step), MW a lane.  The
// warp's output tiles hold the step's coefficients ([bin][place], each once) and
// then its samples (as they lie in the output).
template <int MW>
__device__ __forceinline__ void shape_pairs(const DecodeParams &p, const UnitSeg &sg, const DomS &dd,
                                            const unsigned char *smem, const uint8_t *lv0, uint64_t win, uint32_t n,
                                            const ShapeOut &o) {
  const uint32_t lane = o.lane, N = dd.N, P = shape_pair_count(N), p8 = shape_pairs8(N), kz = dd.kz;
  // lanes' windows lie G apart (rows that are multiples of 32 samples apart would
  // share their banks): place MW g + i of a bin's coefficients is window g + G i
  // (places for the step's own windows: a stream's last step, or only one, has fewer;
  // with a whole step's 200,000 streams of one window of (128, 128) took 1880 us, 1375 so)
  const uint32_t Ws = shape_pair_places(n, MW), G = Ws / MW;
  const float *deq = reinterpret_cast<const float *>(smem + dd.deq_off);
  const float *bas = reinterpret_cast<const float *>(smem + dd.basis_off);
  if (lane == 0) tma_wait_read_but<0>();  // earlier steps have left the tiles
  __syncwarp();
  // ---- coefficients, lanes along the windows
  {
    float *const cs = reinterpret_cast<float *>(o.otile);
    const uint32_t dk = 32 / Ws, dw = 32 - dk * Ws;
    uint32_t k = lane / Ws, w = lane - k * Ws;
    for (uint32_t i = lane; i < kz * Ws; i += 32) {
      const uint32_t ww = w / MW + G * (w % MW);
      cs[i] = ww < n ? deq[(k < dd.B1 ? 0 : kZStride) + lv0[ww * dd.E + k]] : 0.0f;  // i = k Ws + w
      k += dk;
      w += dw;
      if (w >= Ws) {
        w -= Ws;
        ++k;
      }
    }
  }
  __syncwarp();
  // ---- MW windows by eight pairs a lane
  const uint32_t pgs = p8 / 8, wg = lane / pgs, pg = lane - wg * pgs;
  const bool mine = wg < G;
  float2 ev[MW][4], od[MW][4];
#pragma unroll
  for (int i = 0; i < MW; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) ev[i][j] = od[i][j] = make_float2(0.0f, 0.0f);
  if (mine) {
    const float *cp = reinterpret_cast<const float *>(o.otile) + MW * wg;  // the lane's windows, bin 0
    const float4 *bp = reinterpret_cast<const float4 *>(bas) + pg;
    const uint32_t bhalf = p8 / 8, bstep = p8 / 4;
    auto bin = [&](float2(&acc)[MW][4]) {
      float2 c[MW];  // a window's coefficient in both halves
      if constexpr (MW == 4) {
        const float4 q = *reinterpret_cast<const float4 *>(cp);
        c[0] = make_float2(q.x, q.x);
        c[1] = make_float2(q.y, q.y);
        c[2] = make_float2(q.z, q.z);
        c[3] = make_float2(q.w, q.w);
      } else {
        const float2 q = *reinterpret_cast<const float2 *>(cp);
        c[0] = make_float2(q.x, q.x);
        c[1] = make_float2(q.y, q.y);
      }
      const float4 b0 = bp[0], b1 = bp[bhalf];
      cp += Ws;
      bp += bstep;
      const float2 b[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w), make_float2(b1.x, b1.y),
                           make_float2(b1.z, b1.w)};
#pragma unroll
      for (int i = 0; i < MW; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = __ffma2_rn(c[i], b[j], acc[i][j]);
    };
    uint32_t k = 0;
#pragma unroll 1
    for (; k + 2 <= kz; k += 2) {
      bin(ev);
      bin(od);
    }
    if (k < kz) bin(ev);
  }
  __syncwarp();  // the coefficients have been read: their place takes the samples
  if (mine) {
    const bool whole = N % 4 == 0 && 8 * pg + 8 <= P;
#pragma unroll
    for (int i = 0; i < MW; ++i) {
      if (wg + G * i >= n) break;
      float *const x = reinterpret_cast<float *>(o.otile) + (wg + G * i) * N;
      float f[8], m[8];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        f[2 * j] = ev[i][j].x + od[i][j].x;
        f[2 * j + 1] = ev[i][j].y + od[i][j].y;
        m[2 * j] = ev[i][j].x - od[i][j].x;
        m[2 * j + 1] = ev[i][j].y - od[i][j].y;
      }
      if (whole) {
        float4 *const a = reinterpret_cast<float4 *>(x + 8 * pg), *const b = reinterpret_cast<float4 *>(x + N - 8 - 8 * pg);
        a[0] = make_float4(f[0], f[1], f[2], f[3]);
        a[1] = make_float4(f[4], f[5], f[6], f[7]);
        b[0] = make_float4(m[7], m[6], m[5], m[4]);
        b[1] = make_float4(m[3], m[2], m[1], m[0]);
      } else {
#pragma unroll
        for (uint32_t j = 0; j < 8; ++j) {
          const uint32_t t = 8 * pg + j;
          if (t < P) {
            x[t] = f[j];
            // the middle sample of an odd N once (its odd-bin basis values are zero)
            if (N - 1 - t != t) x[N - 1 - t] = m[j];
          }
        }
      }
    }
  }
  // ---- the step's samples lie as they do in the output
  const uint64_t s0 = win * N, left = sg.n_samples - s0;
  const uint32_t total = left < (uint64_t)n * N ? (uint32_t)left : n * N;
  float *const dst = p.out + sg.out_offset + s0;
  if (((reinterpret_cast<uintptr_t>(dst) & 15u) | (total & 3u)) == 0) {
    fence_async_shared();
    __syncwarp();
    if (lane == 0) bulk_store(dst, o.otile, total * 4);
  } else {
    __syncwarp();
    const float *const x = reinterpret_cast<const float *>(o.otile);
    for (uint32_t i = lane; i < total; i += 32) __stcs(dst + i, x[i]);
    if (lane == 0) asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    __syncwarp();
  }
}

struct GeoS {
  __device__ uint32_t tile_windows(const DomS &d) const { return d.T; }
  __device__ uint32_t tile_symbols(const DomS &d) const { return d.T * d.E; }
  __device__ uint32_t step_windows(const DomS &d) const { return d.step; }
  __device__ uint32_t bins(const DomS &d) const { return d.E; }
};

// FORMS: the transforms the plan's domains use (kShapeCompiled, kShapeAny or
// both), ONE: the one compiled form they all have (0: several): an instance holds,
// and pays registers for, only those.  TILES: output tiles per warp.
// 16 warps leave 128 registers a thread; with several compiled forms in one
// kernel some of the stream's state was spilled around the larger ones, and
// spills go to L2 (shared memory leaves L1 little): (64, 32), 67 M samples, took
// 130 us in that kernel and 88 us in its own.  Plans of several forms run 12
// warps, where 44 bytes a thread are (416 at 16 warps); the instance of (128, 64)
// alone spills 24, that of the pair form alone 16, the 24-warp one (threads = 768) 132.
template <int WARPS, int TILES, int FORMS, uint32_t ONE = 0>
__global__ void __launch_bounds__(WARPS * 32, 1) k_decode_shape(const DecodeParams p, const WarpParams wp,
                                                                const __grid_constant__ ShapeMaps maps) {
  constexpr int kCapS = shape_cap(TILES);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const DomS *const ds = reinterpret_cast<const DomS *>(smem_raw);
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

  load_shape_tables<WARPS * 32, TILES>(p, wp.n_domains, smem_raw);
  __syncthreads();

  uint8_t *const stage = smem_raw + wp.warp_off + warp * stream_bytes(kCapS) + kStreamStage;
  const uintptr_t tiles0 =
      (reinterpret_cast<uintptr_t>(smem_raw + wp.warp_off + WARPS * stream_bytes(kCapS)) + 1023) & ~uintptr_t(1023);
  unsigned char *const otile = reinterpret_cast<unsigned char *>(tiles0) + warp * TILES * kOutTile;
  const bool out32 = (reinterpret_cast<uintptr_t>(p.out) & 31u) == 0;
  uint32_t turn = kAllTiles;

  dependency_wait();  // the index: from here on its outputs are read
  uint64_t tw0, tw1;
  unit_tiles(p, (uint64_t)blockIdx.x * WARPS + warp, (uint64_t)gridDim.x * WARPS, tw0, tw1);
  if (tw0 >= tw1) return;

  stream_tiles<kCapS>(
      p, tw0, tw1, ds, smem_raw, stage, lane, GeoS{},
      [&](const UnitSeg &sg, const DomS &dd, const uint8_t *levels, uint64_t win, uint32_t n) {
        if (p.levels != nullptr) {  // the step's levels are contiguous in the caller's buffer
          uint8_t *const lev = p.levels + sg.level_offset + win * dd.E;
          if (((reinterpret_cast<uintptr_t>(lev) | reinterpret_cast<uintptr_t>(levels) | (n * dd.E)) & 15u) == 0) {
            for (uint32_t j = 16 * lane; j < n * dd.E; j += 512)
              *reinterpret_cast<uint4 *>(lev + j) = *reinterpret_cast<const uint4 *>(levels + j);
          } else {
            for (uint32_t j = lane; j < n * dd.E; j += 32) lev[j] = levels[j];
          }
        }
        const uint32_t aligned = sg.out_aligned;
        const bool tma = (aligned & 4u) != 0;
        const ShapeOut o{otile, lane & 7u, lane, &maps.rows, dd.N == 64 ? &maps.n64 : &maps.n128,
                         (wp.out_tma & 1u) && tma, (wp.out_tma & (dd.N == 64 ? 2u : 4u)) && tma,
                         out32 && (aligned & 2u), (aligned & 1u) != 0};
        bool done = false;
        if constexpr (FORMS & kShapeCompiled) done = shape_compiled<TILES, ONE>(p, sg, dd, smem_raw, levels, win, n, o, turn);
        if constexpr (FORMS & kShapeAny)
          if (!done) {
            shape_pairs<(int)shape_pair_windows(TILES)>(p, sg, dd, smem_raw, levels, win, n, o);
            turn = kAllTiles;
          }
      });
  if (lane == 0) tma_wait_all();
}

}  // namespace
}  // namespace fptc
