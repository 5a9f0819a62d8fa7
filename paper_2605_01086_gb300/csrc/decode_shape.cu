// Fused decode for window shapes other than the Table 1 default: every domain of
// the plan has a window size N in [4, 128] and any kept-bin count E <= N,
// domains of different N in one batch (Table 1 gives the ranges; Fig. 14
// measures how the throughput moves with them).
//
// The SymLen decode, tile chaining, level staging and TMA output path are those
// of the warp-tile kernel (warp_tile.cuh), with tiles of T windows per domain
// (about 2048 symbols, a whole number of output steps).  The transform is one of
// two, chosen per tile from the tile's domain (a warp-uniform switch):
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
//    windows x chunks x 32 floats).  (64, 32), 67 M samples: 116 us,
//    171 us in the pair form (which then had compile-time N too).
//  * otherwise (shape_transform_any): a window's samples as ceil(N / 2) mirrored
//    pairs in groups of 16, one lane per group, with the half basis in shared
//    memory.
#include <cuda.h>

#include "warp_tile.cuh"

namespace fptc {
namespace {

using namespace wt;

// Per-domain view of the shared tables of the shape kernel.
struct DomS {
  uint32_t lut_off;    // bytes from the start of shared memory (entries len | level << 8)
  uint32_t deq_off;    // bytes: zone rows [3][kZStride] floats
  uint32_t basis_off;  // bytes: [E][brow] floats
  uint32_t shift;      // 32 - lmax
  uint32_t complete;
  uint32_t E, B1, kz;  // kz = min(E, B2)
  uint32_t T;          // windows per tile
  uint32_t N;
  uint32_t form;       // compiled transform: N << 8 | bins (0: shape_transform_any)
  uint32_t pad;
};

__host__ __device__ constexpr bool shape_pow2(uint32_t N) { return (N & (N - 1)) == 0; }
// Other N: the ceil(N / 2) sample pairs of a window in groups of 16, one lane per group.
__host__ __device__ constexpr uint32_t shape_any_pairs(uint32_t N) { return (N + 1) / 2; }
__host__ __device__ constexpr uint32_t shape_any_lanes(uint32_t N) { return (shape_any_pairs(N) + 15) / 16; }
// Windows per output step for other N: one lane group each, at most 1024 samples.
__host__ __device__ constexpr uint32_t shape_any_step(uint32_t N) {
  return 32 / shape_any_lanes(N) < 1024 / N ? 32 / shape_any_lanes(N) : 1024 / N;
}

__host__ __device__ constexpr uint32_t shape_brow(uint32_t N) { return shape_any_lanes(N) * 20; }

// The compiled transform of a domain (N << 8 | bins), or 0.  With 24 warps one
// output tile per warp is all that fits, and only N <= 32 has one.
constexpr uint32_t kMaxForm1 = 32;
__host__ __device__ constexpr uint32_t shape_form(uint32_t N, uint32_t kz, bool two_tiles) {
  if (!shape_pow2(N) || kz > 64 || (N > kMaxForm1 && !two_tiles)) return 0;
  uint32_t bins = N >= 16 ? N / 4 : N;
  while (bins < kz) bins *= 2;
  return N << 8 | bins;
}

// Windows per output step of a lane-per-window transform: 32 lanes, 32 / N
// windows each for N < 32.
__host__ __device__ constexpr uint32_t shape_lane_step(uint32_t N) { return N >= 32 ? 32 : 1024 / N; }

// Windows per tile for a domain of the shape kernel: whole steps, at most 2048
// symbols (the level staging buffer) and at most 8192 samples (the dL/dx tile of
// the block adjoint fits shared memory).
__host__ __device__ constexpr uint32_t shape_tile_windows(uint32_t N, uint32_t E) {
  const uint32_t r = shape_pow2(N) ? shape_lane_step(N) : shape_any_step(N);
  const uint32_t most = (uint32_t)kTS / E < 8192 / N ? (uint32_t)kTS / E : 8192 / N;
  return most >= r ? most / r * r : most;
}

// Tables of every domain into shared memory from byte 0 (the layout of
// shape_smem_layout).  Returns the end offset.  Contains no barrier.
template <int THREADS, bool TWO>
__device__ __forceinline__ uint32_t load_shape_tables(const DecodeParams &p, uint32_t n_domains, unsigned char *smem) {
  DomS *const ds = reinterpret_cast<DomS *>(smem);
  uint32_t off = (uint32_t)align16(sizeof(DomS) * (n_domains ? n_domains : 1));
  for (uint32_t d = 0; d < n_domains; ++d) {
    const DomainDev &dm = p.domains[d];
    const uint32_t N = dm.N, brow = shape_brow(N), kz = dm.B2 < dm.E ? dm.B2 : dm.E;
    const uint32_t form = shape_form(N, kz, TWO);
    const uint32_t lut_off = off;
    const uint32_t deq_off = lut_off + (uint32_t)align16((size_t)2 << dm.lmax);
    const uint32_t basis_off = deq_off + (uint32_t)align16(3u * kZStride * 4);
    off = basis_off + (form ? 0u : (uint32_t)align16((size_t)dm.E * brow * 4));
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
      x.pad = 0;
      ds[d] = x;
    }
    load_warp_lut<THREADS>(p.luts + dm.lut_offset, dm.lmax, smem + lut_off);
    float a0 = p.scale ? p.scale[d * 3 + 0] : dm.scale[0];
    float a1 = p.scale ? p.scale[d * 3 + 1] : dm.scale[1];
    a0 = a0 > 1e-30f ? a0 : 0.0f;
    a1 = a1 > 1e-30f ? a1 : 0.0f;
    float *deq = reinterpret_cast<float *>(smem + deq_off);
    for (uint32_t i = threadIdx.x; i < 3u * kZStride; i += THREADS) {
      const uint32_t z = i / kZStride, L = i - z * kZStride;
      deq[i] = (L < 256u && z < 2u) ? (z == 0 ? a0 : a1) * dm.unit[z][L] : 0.0f;
    }
    if (form) continue;
    // the half basis B[k][n], n < ceil(N / 2): rows of brow floats, in groups of 16 (+ 4 pad)
    float *bas = reinterpret_cast<float *>(smem + basis_off);
    const float *g_bas = p.basis + dm.basis_offset;
    const uint32_t pairs = shape_any_pairs(N);
    for (uint32_t i = threadIdx.x; i < dm.E * brow; i += THREADS) {
      const uint32_t k = i / brow, r = i - k * brow, n = 16 * (r / 20) + r % 20;
      bas[i] = r % 20 < 16 && n < pairs ? __ldg(g_bas + (size_t)k * N + n) : 0.0f;
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

__device__ __forceinline__ void put8(unsigned char *row, uint32_t sx, int b, const float (&v)[8]) {
  *reinterpret_cast<float4 *>(row + (((2 * b) ^ sx) << 4)) = make_float4(v[0], v[1], v[2], v[3]);
  *reinterpret_cast<float4 *>(row + (((2 * b + 1) ^ sx) << 4)) = make_float4(v[4], v[5], v[6], v[7]);
}

// Dequantization + inverse transform + reassembly of one decoded tile of nwin
// windows (levels at stage[0..nwin E)), N <= 32: a step is 1024 samples, a row
// of 32 per lane.  tiles: staging tiles per warp (steps alternate between two).
template <int N, int K, int TILES>
__device__ __forceinline__ void shape_rows(const DecodeParams &p, const SegDev &sg, const DomS &dd,
                                           const unsigned char *smem, const uint8_t *stage, uint64_t win0,
                                           uint32_t nwin, const ShapeOut &o) {
  constexpr uint32_t M = 32 / N, R = 32 * M;  // windows per lane, per step
  const uint32_t lane = o.lane;
  const float *deq = reinterpret_cast<const float *>(smem + dd.deq_off);
  const bool fast = K % 8 == 0 && dd.E == K && dd.kz == K && dd.B1 == 2;
  const uint64_t S = sg.n_samples;
  uint32_t turn = 0;
#pragma unroll 1
  for (uint32_t w0 = 0; w0 < nwin; w0 += R, turn ^= TILES - 1) {
    unsigned char *const tile = o.otile + turn * kOutTile, *const row = tile + lane * 128;
    if (lane == 0) {  // earlier steps have left this tile (the decoded tile's first step: both)
      if (w0 == 0)
        tma_wait_read_but<0>();
      else
        tma_wait_read_but<TILES - 1>();
    }
    __syncwarp();
    const uint32_t wl = w0 + M * lane;
#pragma unroll
    for (uint32_t m = 0; m < M; ++m) {
      if (wl + m >= nwin) break;
      float c[K], x[N];
      load_coefs<0, 1, K>(stage + (wl + m) * dd.E, deq, dd.B1, dd.kz, fast, c);
      idct_small<N, K>(c, x);
#pragma unroll
      for (int j = 0; j < N / 4; ++j)
        *reinterpret_cast<float4 *>(row + (((m * (N / 4) + j) ^ o.sx) << 4)) =
            make_float4(x[4 * j], x[4 * j + 1], x[4 * j + 2], x[4 * j + 3]);
    }
    const uint64_t s0 = (win0 + w0) * N;  // first sample of the step in the segment
    if (o.tma_ok && w0 + R <= nwin && s0 + 1024 <= S) {
      fence_async_shared();
      __syncwarp();
      if (lane == 0) tma_store_rows(o.map, tile, (int32_t)((sg.out_offset + s0) >> 5));
    } else {
      const uint64_t lim = (uint64_t)(nwin - w0) * N < S - s0 ? (uint64_t)(nwin - w0) * N : S - s0;
      const uint64_t r0 = (uint64_t)lane * 32;
      if (r0 < lim)
        store_row(row, o.sx, p.out + sg.out_offset + s0 + r0, lim - r0 < 32 ? (uint32_t)(lim - r0) : 32u, o.vec32,
                  o.vec16);
      if (TILES > 1 && lane == 0) asm volatile("cp.async.bulk.commit_group;" ::: "memory");  // the tiles' turns stay in step
    }
  }
}

// The same for N = 64, 128: a step is 32 windows, one per lane; the chunks
// (32 samples) c and N / 32 - 1 - c of the windows mirror each other and are
// staged together, one tile each.
template <int N, int K>
__device__ __forceinline__ void shape_windows(const DecodeParams &p, const SegDev &sg, const DomS &dd,
                                              const unsigned char *smem, const uint8_t *stage, uint64_t win0,
                                              uint32_t nwin, const ShapeOut &o) {
  constexpr int kChunks = N / 32;
  const uint32_t lane = o.lane;
  const float *deq = reinterpret_cast<const float *>(smem + dd.deq_off);
  const bool fast = K % 16 == 0 && dd.E == K && dd.kz == K && dd.B1 == 2;
  const uint64_t S = sg.n_samples;
  unsigned char *const ra = o.otile + lane * 128, *const rb = ra + kOutTile;  // the lane's rows
#pragma unroll 1
  for (uint32_t w0 = 0; w0 < nwin; w0 += 32) {
    const uint32_t wl = w0 + lane;
    const uint8_t *const lv = stage + (wl < nwin ? wl : w0) * dd.E;
    float e[N / 2];
    {
      float ce[K / 2];
      load_coefs<0, 2, K / 2>(lv, deq, dd.B1, dd.kz, fast, ce);
      idct_small<N / 2, K / 2>(ce, e);
    }
    float co[K / 2];
    load_coefs<1, 2, K / 2>(lv, deq, dd.B1, dd.kz, fast, co);
    const uint64_t s0 = (win0 + wl) * N;  // the window's first sample in the segment
    const bool tma_step = o.tma_n && w0 + 32 <= nwin && (win0 + w0 + 32) * N <= S;
#pragma unroll
    for (int q = 0; q < kChunks / 2; ++q) {  // chunks q and kChunks - 1 - q
      if (lane == 0) tma_wait_read_but<0>();
      __syncwarp();
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        float lo[8], hi[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int n = 32 * q + 8 * g + i;
          const float od = odd_sum<N, K / 2>(co, n);
          lo[i] = e[n] + od;
          hi[7 - i] = e[n] - od;
        }
        put8(ra, o.sx, g, lo);
        put8(rb, o.sx, 3 - g, hi);
      }
      if (tma_step) {
        fence_async_shared();
        __syncwarp();
        if (lane == 0) {
          // chunk row of the step's first window in the output: window row / (N / 32), chunk the rest
          const uint64_t r = (sg.out_offset >> 5) + (win0 + w0) * kChunks;
          const uint64_t a = r + q, b = r + kChunks - 1 - q;
          tma_store_chunk(o.map_n, o.otile, (int32_t)(a % kChunks), (int32_t)(a / kChunks));
          tma_store_chunk(o.map_n, o.otile + kOutTile, (int32_t)(b % kChunks), (int32_t)(b / kChunks));
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
      } else if (wl < nwin) {  // each lane its own rows
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const uint64_t t = s0 + 32 * (h ? kChunks - 1 - q : q);
          if (t < S)
            store_row(h ? rb : ra, o.sx, p.out + sg.out_offset + t, S - t < 32 ? (uint32_t)(S - t) : 32u, o.vec32,
                      o.vec16);
        }
      }
    }
  }
}

// The compiled transform of a tile's domain (uniform over the warp); false: there is none.
template <int TILES>
__device__ __forceinline__ bool shape_compiled(const DecodeParams &p, const SegDev &sg, const DomS &dd,
                                               const unsigned char *smem, const uint8_t *stage, uint64_t win0,
                                               uint32_t nwin, const ShapeOut &o) {
#define FPTC_ROWS(N, K) \
  case (N << 8 | K): shape_rows<N, K, TILES>(p, sg, dd, smem, stage, win0, nwin, o); return true;
#define FPTC_WINDOWS(N, K) \
  case (N << 8 | K): \
    if constexpr (TILES == 2) shape_windows<N, K>(p, sg, dd, smem, stage, win0, nwin, o); \
    return true;
  switch (dd.form) {
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

// The pair form, any N (run-time): a
// window's ceil(N / 2) sample pairs (n, N - 1 - n) in groups of 16, one lane per
// group; a step holds R = min(32 / groups, 1024 / N) windows, R N samples of the
// tile from the staging tile's start, which the lanes store row by row (vector
// stores where a row's address allows).
__device__ __forceinline__ void shape_transform_any(const DecodeParams &p, const SegDev &sg, const DomS &dd,
                                                    const unsigned char *smem, const uint8_t *stage, uint64_t win0,
                                                    uint32_t nwin, const ShapeOut &o) {
  const uint32_t N = dd.N, P = shape_any_pairs(N), L = shape_any_lanes(N), R = shape_any_step(N);
  const uint32_t brow = L * 20u;
  const uint32_t lane = o.lane;
  const float *deq0 = reinterpret_cast<const float *>(smem + dd.deq_off);
  const float *bas = reinterpret_cast<const float *>(smem + dd.basis_off);
  const uint64_t S = sg.n_samples;
  unsigned char *const row = o.otile + lane * 128;
  if (lane == 0) tma_wait_read();  // a previous tile's TMA store may still read the staging tile
  __syncwarp();
  const uint32_t wr = lane / L, q = lane % L;  // window of the step, pair group
#pragma unroll 1
  for (uint32_t w0 = 0; w0 < nwin; w0 += R) {
    const uint32_t wl = w0 + wr;
    const bool mine = wr < R && wl < nwin;
    float ev[16], od[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) ev[i] = od[i] = 0.0f;
    if (mine) {
      const uint8_t *lv = stage + wl * dd.E;
      const float *bq = bas + q * 20;
      uint32_t k = 0;
#pragma unroll 1
      for (; k + 2 <= dd.kz; k += 2) {
        const float c0 = deq0[(k < dd.B1 ? 0 : kZStride) + lv[k]];
        const float c1 = deq0[(k + 1 < dd.B1 ? 0 : kZStride) + lv[k + 1]];
        const float4 *b0 = reinterpret_cast<const float4 *>(bq + k * brow);
        const float4 *b1 = reinterpret_cast<const float4 *>(bq + (k + 1) * brow);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float4 u = b0[j], v = b1[j];
          ev[4 * j] = fmaf(c0, u.x, ev[4 * j]);
          ev[4 * j + 1] = fmaf(c0, u.y, ev[4 * j + 1]);
          ev[4 * j + 2] = fmaf(c0, u.z, ev[4 * j + 2]);
          ev[4 * j + 3] = fmaf(c0, u.w, ev[4 * j + 3]);
          od[4 * j] = fmaf(c1, v.x, od[4 * j]);
          od[4 * j + 1] = fmaf(c1, v.y, od[4 * j + 1]);
          od[4 * j + 2] = fmaf(c1, v.z, od[4 * j + 2]);
          od[4 * j + 3] = fmaf(c1, v.w, od[4 * j + 3]);
        }
      }
      if (k < dd.kz) {  // a last even bin
        const float c0 = deq0[(k < dd.B1 ? 0 : kZStride) + lv[k]];
        const float4 *b0 = reinterpret_cast<const float4 *>(bq + k * brow);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float4 u = b0[j];
          ev[4 * j] = fmaf(c0, u.x, ev[4 * j]);
          ev[4 * j + 1] = fmaf(c0, u.y, ev[4 * j + 1]);
          ev[4 * j + 2] = fmaf(c0, u.z, ev[4 * j + 2]);
          ev[4 * j + 3] = fmaf(c0, u.w, ev[4 * j + 3]);
        }
      }
      // samples n = 16 q + i and N - 1 - n of window wr at step positions wr N + ...
      // (the middle sample of an odd N once: its odd-bin basis values are zero)
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const uint32_t n = 16 * q + i;
        if (n < P) {
          const uint32_t tf = wr * N + n, tm = wr * N + (N - 1 - n);
          *reinterpret_cast<float *>(o.otile + (tf >> 5) * 128 + ((((tf & 31u) >> 2) ^ ((tf >> 5) & 7u)) << 4) +
                                     ((tf & 3u) << 2)) = ev[i] + od[i];
          if (tm != tf)
            *reinterpret_cast<float *>(o.otile + (tm >> 5) * 128 + ((((tm & 31u) >> 2) ^ ((tm >> 5) & 7u)) << 4) +
                                       ((tm & 3u) << 2)) = ev[i] - od[i];
        }
      }
    }
    __syncwarp();  // rows are written by other lanes
    const uint64_t s0 = (win0 + w0) * N;  // first sample of the step in the segment
    const uint32_t nw = nwin - w0 < R ? nwin - w0 : R;
    const uint64_t lim = (uint64_t)nw * N < S - s0 ? (uint64_t)nw * N : S - s0;
    const uint64_t r0 = (uint64_t)lane * 32;
    if (r0 < lim) {
      const uint32_t m = lim - r0 < 32 ? (uint32_t)(lim - r0) : 32u;
      float *const dst = p.out + sg.out_offset + s0 + r0;
      const uintptr_t a = reinterpret_cast<uintptr_t>(dst);
      store_row(row, o.sx, dst, m, (a & 31u) == 0, (a & 15u) == 0);
    }
    __syncwarp();  // before the next step rewrites the tile
  }
}

// FORMS: the transforms the plan's domains use (kShapeCompiled, kShapeAny or
// both): an instance holds, and pays registers for, only those.
template <int WARPS, int FORMS>
__global__ void __launch_bounds__(WARPS * 32, 1) k_decode_shape(const DecodeParams p, const WarpParams wp,
                                                                const __grid_constant__ ShapeMaps maps) {
  constexpr int TILES = WARPS > 16 ? 1 : 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const DomS *const ds = reinterpret_cast<const DomS *>(smem_raw);
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

  load_shape_tables<WARPS * 32, TILES == 2>(p, wp.n_domains, smem_raw);
  __syncthreads();

  unsigned char *const wbase = smem_raw + wp.warp_off + warp * kMiscBytes;
  uint64_t *const wbuf = reinterpret_cast<uint64_t *>(wbase);  // first-pass words
  uint8_t *const stage = wbase + kStageOff;      // tile position 0
  const uintptr_t tiles0 = (reinterpret_cast<uintptr_t>(smem_raw + wp.warp_off + WARPS * kMiscBytes) + 1023) &
                           ~uintptr_t(1023);
  unsigned char *const otile = reinterpret_cast<unsigned char *>(tiles0) + warp * TILES * kOutTile;
  const bool want_lev = p.levels != nullptr;

  dependency_wait();  // the index: from here on its outputs are read
  uint64_t tw0, tw1;
  unit_tiles(p, (uint64_t)blockIdx.x * WARPS + warp, (uint64_t)gridDim.x * WARPS, tw0, tw1);
  if (tw0 >= tw1) return;

  Ctx nxt;
  {
    const uint32_t s = warp_find_segment(p.segs, p.seg_begin, p.seg_end, tw0, lane);
    const DomS &d0 = ds[p.segs[s].domain];
    nxt = first_ctx(p, s, tw0, lane, (uint64_t)d0.T * d0.E);
  }
  uint32_t pn = fetch_pass0(p, nxt, lane, wbuf);

  for (uint64_t g = tw0; g < tw1; ++g) {
    cp_async_wait_all();
    __syncwarp();
    const Ctx cur = nxt;
    uint64_t w[kWPL];
    uint32_t n[kWPL];
#pragma unroll
    for (int u = 0; u < kWPL; ++u) {
      w[u] = wbuf[kWPL * lane + u];
      n[u] = (pn >> (8 * u)) & 0xffu;
    }
    __syncwarp();
    const uint64_t g1 = g + 1;

    const SegDev &sg = p.segs[cur.seg];
    const DomS dd = ds[sg.domain];
    const uint64_t win0 = (g - sg.tile_base) * dd.T;
    const uint64_t left = sg.n_windows - win0;
    const uint32_t nwin = left < (uint64_t)dd.T ? (uint32_t)left : dd.T;

    // ---- 1. SymLen decode into the level bytes
    TileEnd te{0u, 0u, 0u};
    if (cur.ok) {
      te = decode_tile(p, cur, nwin * dd.E, dd, smem_raw, stage, lane, w, n);
      if (te.bad && lane == 0) flag_bad(p.status, te.bad, sg.caller_index);
    }
    // ---- first words of tile g + 1 (in flight during the transform)
    if (g1 < tw1) {
      nxt = next_ctx(p, g, cur.seg, cur, te);
      pn = fetch_pass0(p, nxt, lane, wbuf);
    }
    __syncwarp();
    if (!cur.ok) continue;

    if (want_lev) {  // the tile's levels are contiguous in the caller's buffer
      uint8_t *const lev = p.levels + sg.level_offset + win0 * dd.E;
      for (uint32_t j = lane; j < nwin * dd.E; j += 32) lev[j] = stage[j];
    }

    // ---- 2./3. dequantization + inverse transform + reassembly, 1024 samples per step
    const uint32_t aligned = sg.out_aligned;
    const bool tma = (aligned & 4u) != 0;
    const ShapeOut o{otile, lane & 7u, lane, &maps.rows, dd.N == 64 ? &maps.n64 : &maps.n128, (wp.out_tma & 1u) && tma,
                     (wp.out_tma & (dd.N == 64 ? 2u : 4u)) && tma,
                     (aligned & 2u) && (reinterpret_cast<uintptr_t>(p.out) & 31u) == 0, (aligned & 1u) != 0};
    bool done = false;
    if constexpr (FORMS & kShapeCompiled) done = shape_compiled<TILES>(p, sg, dd, smem_raw, stage, win0, nwin, o);
    if constexpr (FORMS & kShapeAny)
      if (!done) shape_transform_any(p, sg, dd, smem_raw, stage, win0, nwin, o);
    __syncwarp();  // the level bytes are rewritten by the next tile
  }
  if (lane == 0) tma_wait_all();
}

template <int WARPS>
void *sptr(uint32_t forms) {
  switch (forms) {
    case kShapeCompiled: return reinterpret_cast<void *>(&k_decode_shape<WARPS, kShapeCompiled>);
    case kShapeAny: return reinterpret_cast<void *>(&k_decode_shape<WARPS, kShapeAny>);
    default: return reinterpret_cast<void *>(&k_decode_shape<WARPS, kShapeCompiled | kShapeAny>);
  }
}

void *spick(uint32_t threads, uint32_t forms) {
  switch (threads) {
    case 256: return sptr<8>(forms);
    case 512: return sptr<16>(forms);
    case 768: return sptr<24>(forms);
    default: return nullptr;
  }
}

}  // namespace

bool shape_supported(uint32_t N) { return N >= 4 && N <= 128; }

uint32_t shape_forms(uint32_t N, uint32_t kz, uint32_t threads) {
  return shape_form(N, kz, threads <= 512) ? kShapeCompiled : kShapeAny;
}

uint32_t shape_windows_per_tile(uint32_t N, uint32_t E) { return shape_tile_windows(N, E); }

size_t shape_smem_layout(uint32_t threads, const uint32_t *lmax, const uint32_t *N, const uint32_t *E,
                         const uint32_t *kz, uint32_t n_domains, WarpParams *wp) {
  const bool two = threads <= 512;  // output tiles per warp: two, one with 24 warps
  size_t o = align16(sizeof(DomS) * (n_domains ? n_domains : 1));
  for (uint32_t d = 0; d < n_domains; ++d) {
    o += align16((size_t)2 << lmax[d]);
    o += align16(3u * kZStride * 4);
    if (!shape_form(N[d], kz[d], two)) o += align16((size_t)E[d] * shape_brow(N[d]) * 4);
  }
  o = align16(o);
  *wp = WarpParams{};
  wp->n_domains = n_domains;
  wp->warp_off = (uint32_t)o;
  wp->warp_bytes = (uint32_t)kMiscBytes;
  const size_t warps = threads / 32;
  return o + warps * kMiscBytes + 1023 + warps * (two ? 2 : 1) * kOutTile;  // + alignment of the staging tiles
}

// Tensor map of an output buffer of `extent` floats as windows of N floats,
// chunks of 32: dims (32, N / 32, windows), boxes of one chunk of 32 windows.
// The last window may lie partly outside the buffer; a box only ever holds
// whole windows of a segment, so nothing there is written.
bool encode_window_map(CUtensorMap *map, float *out, uint64_t extent, uint32_t N) {
  return encode_out_map3(map, out, (extent + N - 1) / N * N, N);
}

cudaError_t shape_smem_config(uint32_t threads, uint32_t forms, size_t smem) {
  void *k = spick(threads, forms);
  if (!k) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout,
                                       (int)cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return e;
  return set_dynamic_smem_limit(k, smem);
}

cudaError_t shape_occupancy(uint32_t threads, uint32_t forms, size_t smem, int *ctas_per_sm) {
  void *k = spick(threads, forms);
  if (!k) return cudaErrorInvalidValue;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, k, (int)threads, smem);
}

cudaError_t launch_shape(const DecodeParams &p, const WarpParams &wp, const ShapeMaps &maps, uint32_t threads,
                         uint32_t forms, uint32_t grid, size_t smem, cudaStream_t stream) {
  if (p.tile_end <= p.tile_begin || grid == 0) return cudaSuccess;
  void *k = spick(threads, forms);
  if (!k) return cudaErrorInvalidValue;
  DecodeParams pp = p;
  WarpParams ww = wp;
  ShapeMaps mm = maps;
  void *args[] = {&pp, &ww, &mm};
  return launch_after(k, grid, threads, args, smem, stream, p.after_index != 0);
}

}  // namespace fptc
