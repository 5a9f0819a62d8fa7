// Fused decode for the Table 1 shape (N = 32, E = 16) with no block-wide barrier.
//
// Each warp owns a contiguous range of tiles of 32 windows (512 symbols, 1024
// samples: what its lanes transform in one step) and runs Sec. 4.2 on it as one
// stream (stream_tiles in warp_tile.cuh):
//  1. SymLen decode.  A pass gives every lane two consecutive words; a warp
//     scan of their symbol counts places each word's codewords (compaction,
//     Sec. 4.2.1).  A lane decodes a word with one decode-table lookup per
//     codeword and stores the codeword's level as one byte at its place behind
//     the symbols not yet transformed (two per 16-bit store).  Nothing else
//     happens per codeword: the dequantization waits for step 2, where the bin
//     of every value is known at compile time.  The 64-bit word is shifted
//     through hi:lo with a marker bit under it, so a word whose codewords need
//     more than 64 bits shows as an empty buffer at the end (no per-codeword
//     count).
//  2. Dequantization and inverse DCT, one window per lane, whenever 512 symbols
//     are there.  The lane reads its window's 16 levels, turns each into A_z *
//     unit_z(level) (one table read; the bin, hence the zone row, is fixed per
//     register), and evaluates the inverse of Eq. 1 by the even/odd split of the
//     DCT-III: x[n] = E[n] + O[n], x[31-n] = E[n] - O[n] with O the odd bins and
//     E the even bins, itself split the same way twice (E[15-n] = EE[n] - EO[n],
//     EE[7-n] = EEE[n] - EEO[n]); 229 FP32 operations per window with the
//     cosines as compile-time constants, so neither a basis nor coefficients
//     pass through shared memory.
//  3. Output.  Where the segment's output starts on a 128-byte boundary and
//     all 32 windows of a step are whole, the lanes write their windows into
//     the warp's shared staging tile in the 128-byte swizzled layout (chunk c
//     of row r at c ^ (r & 7): conflict-free) and one lane stores the tile
//     with a TMA tensor store (the output viewed as rows of 32 floats), so the
//     output never passes through the L1 load/store pipe.  Other windows use
//     32-byte (or 16-byte, or scalar) streaming stores.
//  The warp locates the first word of its range from the index's chunk offsets;
//  the words of a pass load while the pass before it decodes and its steps run.
// The decode tables, dequantization rows and basis of every domain stay in
// shared memory for the whole kernel.
//
// Bound by instruction issue (decode table lookups and the transform) on large
// batches.  Tiles of 128 windows decoded one by one left 11 % of the warps'
// time idle on 124 M samples (7.1 tiles a warp: some had 8), decoded the words
// at a tile's end in a pass of their own and started every tile afresh: 3,750
// warp instructions per 4096 samples, 144 us for 124 M samples (four domains,
// ragged lengths); as one stream 119 us.
#include <cuda.h>
#include <cudaTypedefs.h>

#include "warp_tile.cuh"

namespace fptc {
namespace {

using namespace wt;

// ---- compile-time cosines of the inverse transform (N = 32, E = 16) ----------
// cos(pi num / den) in double: Taylor series on [0, pi/2] after the reflections
// cos(2 pi - a) = cos(a) and cos(pi - a) = -cos(a); rounded to float.
__host__ __device__ constexpr double cos_taylor(double x) {
  double x2 = x * x, term = 1.0, sum = 1.0;
  for (int i = 1; i < 24; ++i) {
    term *= -x2 / ((2.0 * i - 1.0) * (2.0 * i));
    sum += term;
  }
  return sum;
}
__host__ __device__ constexpr float cospi_frac(int num, int den) {
  int r = num % (2 * den);
  if (r > den) r = 2 * den - r;
  const double pi = 3.14159265358979323846;
  return 2 * r <= den ? (float)cos_taylor(pi * r / den) : (float)-cos_taylor(pi * (den - r) / den);
}
// B[k][n] = cos(pi (2n+1) k / 64) grouped by the even/odd recursion:
//   eee[n]    = B[8][n]                       n < 4
//   eeo[n][j] = B[4(2j+1)][n]                 n < 4, j < 2   (bins 4, 12)
//   eo[n][j]  = B[2(2j+1)][n]                 n < 8, j < 4   (bins 2, 6, 10, 14)
//   o[n][j]   = B[2j+1][n]                    n < 16, j < 8  (odd bins)
struct IdctK {
  float eee[4];
  float eeo[4][2];
  float eo[8][4];
  float o[16][8];
};
__host__ __device__ constexpr IdctK make_idct_k() {
  IdctK K{};
  for (int n = 0; n < 4; ++n) K.eee[n] = cospi_frac(2 * n + 1, 8);
  for (int n = 0; n < 4; ++n)
    for (int j = 0; j < 2; ++j) K.eeo[n][j] = cospi_frac((2 * n + 1) * (2 * j + 1), 16);
  for (int n = 0; n < 8; ++n)
    for (int j = 0; j < 4; ++j) K.eo[n][j] = cospi_frac((2 * n + 1) * (2 * j + 1), 32);
  for (int n = 0; n < 16; ++n)
    for (int j = 0; j < 8; ++j) K.o[n][j] = cospi_frac((2 * n + 1) * (2 * j + 1), 64);
  return K;
}

// x[0..31] of one window from its 16 coefficients (inverse of Eq. 1, B[0][n] = 1/2);
// emits the samples as four blocks of 8 through put(block, v[8]).
template <class Put>
__device__ __forceinline__ void idct32(const float (&c)[16], Put put) {
  constexpr IdctK K = make_idct_k();
  const float h0 = 0.5f * c[0];
  float ee[8], eo[8];
#pragma unroll
  for (int n = 0; n < 4; ++n) {
    const float eee = fmaf(c[8], K.eee[n], h0);
    const float eeo = fmaf(c[12], K.eeo[n][1], c[4] * K.eeo[n][0]);
    ee[n] = eee + eeo;
    ee[7 - n] = eee - eeo;
  }
#pragma unroll
  for (int n = 0; n < 8; ++n) {
    float a = c[2] * K.eo[n][0];
    a = fmaf(c[6], K.eo[n][1], a);
    a = fmaf(c[10], K.eo[n][2], a);
    eo[n] = fmaf(c[14], K.eo[n][3], a);
  }
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    float lo[8], hi[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int n = 8 * j + i;
      const float e = n < 8 ? ee[n] + eo[n] : ee[15 - n] - eo[15 - n];
      float o = c[1] * K.o[n][0];
#pragma unroll
      for (int t = 1; t < 8; ++t) o = fmaf(c[2 * t + 1], K.o[n][t], o);
      lo[i] = e + o;       // x[n]
      hi[7 - i] = e - o;   // x[31 - n]
    }
    put(j, lo);
    put(3 - j, hi);
  }
}

// Symbols a warp's stage holds: a step's and a pass's (usually 600), and up to
// the bytes a warp has beside its output tile in the other warp-tile kernels.
constexpr int kCap = kMiscBytes - stream_bytes(0);
constexpr uint32_t kTileWin = 32;  // windows per tile: one step

struct GeoW {
  __device__ uint32_t tile_windows(const DomW &) const { return kTileWin; }
  __device__ uint32_t tile_symbols(const DomW &) const { return kTileWin * kE; }
  __device__ uint32_t step_windows(const DomW &) const { return kStepWin; }
  __device__ uint32_t bins(const DomW &) const { return kE; }
};

template <int WARPS>
__global__ void __launch_bounds__(WARPS * 32, WARPS > 16 ? 1 : 32 / WARPS) k_decode_warp(
    const DecodeParams p, const WarpParams wp, const __grid_constant__ CUtensorMap out_map) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const DomW *const dw = reinterpret_cast<const DomW *>(smem_raw);
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

  load_domain_tables<WARPS * 32>(p, wp.n_domains, smem_raw);
  __syncthreads();

  uint8_t *const stage = smem_raw + wp.warp_off + warp * stream_bytes(kCap) + kStreamStage;
  // output staging tile: 1024-byte aligned (the period of the 128-byte swizzle)
  const uintptr_t tiles0 =
      (reinterpret_cast<uintptr_t>(smem_raw + wp.warp_off + WARPS * stream_bytes(kCap)) + 1023) & ~uintptr_t(1023);
  unsigned char *const otile = reinterpret_cast<unsigned char *>(tiles0) + warp * kOutTile;
  // row `lane` of the staging tile, 16-byte chunk c at c ^ (lane & 7)
  unsigned char *const row = otile + lane * (kN * 4);
  const uint32_t sx = lane & 7u;
  const bool want_lev = p.levels != nullptr;
  const bool out32 = (reinterpret_cast<uintptr_t>(p.out) & 31u) == 0;

  // ---- this warp's tiles: an even split of the launch's tile range over all warps
  dependency_wait();  // the index: from here on its outputs are read
  uint64_t tw0, tw1;
  unit_tiles(p, (uint64_t)blockIdx.x * WARPS + warp, (uint64_t)gridDim.x * WARPS, tw0, tw1);
  if (tw0 >= tw1) return;

  stream_tiles<kCap>(
      p, tw0, tw1, dw, smem_raw, stage, lane, GeoW{},
      // dequantization + inverse transform + reassembly, one window per lane
      [&](const UnitSeg &sg, const DomW &dd, const uint8_t *levels, uint64_t win, uint32_t n) {
        const float *deq = reinterpret_cast<const float *>(smem_raw + dd.deq_off);
        const uint32_t aligned = sg.out_aligned;
        const uint64_t s0 = win * kN, S = sg.n_samples;  // the step's first sample
        if (lane == 0) tma_wait_read();  // the previous step has left the staging tile
        __syncwarp();
        if (lane < n) {
          const uint4 sv = *reinterpret_cast<const uint4 *>(levels + lane * kE);
          float c[16];
          window_coefs(sv, deq, dd.zmask, c);
          if (want_lev) put_levels(p.levels + sg.level_offset + (win + lane) * kE, sv);
          idct32(c, [&](int b, const float(&v)[8]) {
            *reinterpret_cast<float4 *>(row + (((2 * b) ^ sx) << 4)) = make_float4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<float4 *>(row + (((2 * b + 1) ^ sx) << 4)) = make_float4(v[4], v[5], v[6], v[7]);
          });
        }
        // all 32 windows of the step whole and inside the segment: one TMA store
        if (wp.out_tma && (aligned & 4u) && n == kStepWin && s0 + kStepWin * kN <= S) {
          fence_async_shared();
          __syncwarp();
          if (lane == 0) tma_store_rows(&out_map, otile, (int32_t)((sg.out_offset + s0) >> 5));
        } else if (lane < n) {  // each lane stores its own row
          const uint64_t r0 = s0 + lane * kN;
          store_row(row, sx, p.out + sg.out_offset + r0, r0 + kN <= S ? kN : (uint32_t)(S - r0), out32 && (aligned & 2u),
                    aligned & 1u);
        }
      });
  if (lane == 0) tma_wait_all();
}

template <int WARPS>
void *wptr() {
  return reinterpret_cast<void *>(&k_decode_warp<WARPS>);
}

void *wpick(uint32_t threads) {
  switch (threads) {
    case 128: return wptr<4>();
    case 256: return wptr<8>();
    case 512: return wptr<16>();
    case 768: return wptr<24>();
    case 896: return wptr<28>();
    case 1024: return wptr<32>();
    default: return nullptr;
  }
}

}  // namespace

uint32_t warp_tile_windows() { return kTileWin; }

// Shared-memory layout of the warp-tile kernel; returns total bytes, fills wp.
size_t warp_smem_layout(uint32_t threads, const uint32_t *lmax, uint32_t n_domains, WarpParams *wp) {
  size_t o = align16(sizeof(DomW) * (n_domains ? n_domains : 1));
  wp->n_domains = n_domains;
  for (uint32_t d = 0; d < n_domains && d < kWarpMaxDomains; ++d) {
    wp->lut_off[d] = (uint32_t)o;
    o += align16((size_t)2 << lmax[d]);
    wp->tab_off[d] = (uint32_t)o;
    o += kDeqBytes;
  }
  o = align16(o);
  wp->warp_off = (uint32_t)o;
  wp->warp_bytes = (uint32_t)stream_bytes(kCap);
  wp->out_tma = 0;
  const size_t warps = threads / 32;
  return o + warps * stream_bytes(kCap) + 1023 + warps * kOutTile;  // + alignment of the staging tiles
}

bool encode_out_map(CUtensorMap *map, float *out, uint64_t extent) {
  static const PFN_cuTensorMapEncodeTiled_v12000 encode = []() -> PFN_cuTensorMapEncodeTiled_v12000 {
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return nullptr;
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }();
  const uint64_t rows = extent / kN;
  if (!encode || !out || (reinterpret_cast<uintptr_t>(out) & 15u) || rows == 0 || rows > 0x7FFFFFFFull) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)kN, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)kN * 4};
  const cuuint32_t box[2] = {(cuuint32_t)kN, (cuuint32_t)kStepWin};
  const cuuint32_t estride[2] = {1, 1};
  return encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, out, dims, strides, box, estride, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

cudaError_t warp_smem_config(uint32_t threads, size_t smem) {
  void *k = wpick(threads);
  if (!k) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout,
                                       (int)cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return e;
  return set_dynamic_smem_limit(k, smem);
}

cudaError_t warp_occupancy(uint32_t threads, size_t smem, int *ctas_per_sm) {
  void *k = wpick(threads);
  if (!k) return cudaErrorInvalidValue;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, k, (int)threads, smem);
}

cudaError_t launch_warp(const DecodeParams &p, const WarpParams &wp, const CUtensorMap &out_map, uint32_t threads,
                        uint32_t grid, size_t smem, cudaStream_t stream) {
  if (p.tile_end <= p.tile_begin || grid == 0) return cudaSuccess;
  void *k = wpick(threads);
  if (!k) return cudaErrorInvalidValue;
  DecodeParams pp = p;
  WarpParams ww = wp;
  CUtensorMap mm = out_map;
  void *args[] = {&pp, &ww, &mm};
  return launch_after(k, grid, threads, args, smem, stream, p.after_index != 0);
}

}  // namespace fptc
