// Host side of the shape kernel (decode_shape.cuh) and its instances for plans of
// several forms; those of a single form are in decode_shape_one.cu.
#include "decode_shape.cuh"

namespace fptc {
namespace {

constexpr int kBoth = kShapeCompiled | kShapeAny;

void *spick(uint32_t threads, uint32_t tiles, uint32_t forms) {
  if (tiles == 2) {
    if (forms >> 8 && threads == (forms >> 16 == 128 ? 384u : 512u)) return shape_kernel_one(forms >> 8);
    forms &= 3u;
    switch (threads) {
      case 256: return reinterpret_cast<void *>(&k_decode_shape<8, 2, kBoth>);
      case 384:
        return forms == kShapeCompiled ? reinterpret_cast<void *>(&k_decode_shape<12, 2, kShapeCompiled>)
                                       : reinterpret_cast<void *>(&k_decode_shape<12, 2, kBoth>);
      case 512:
        return forms == kShapeAny ? reinterpret_cast<void *>(&k_decode_shape<16, 2, kShapeAny>)
                                  : reinterpret_cast<void *>(&k_decode_shape<16, 2, kBoth>);
      default: return nullptr;
    }
  }
  switch (threads) {  // one tile: where two do not fit
    case 256: return reinterpret_cast<void *>(&k_decode_shape<8, 1, kBoth>);
    case 512: return reinterpret_cast<void *>(&k_decode_shape<16, 1, kBoth>);
    case 768: return reinterpret_cast<void *>(&k_decode_shape<24, 1, kBoth>);
    default: return nullptr;
  }
}

}  // namespace

bool shape_supported(uint32_t N) { return N >= 4 && N <= 128; }

uint32_t shape_forms(uint32_t N, uint32_t kz, uint32_t tiles) {
  return shape_form(N, kz, tiles) ? kShapeCompiled : kShapeAny;
}

uint32_t shape_one_form(uint32_t N, uint32_t kz, uint32_t tiles) { return shape_form(N, kz, tiles); }

uint32_t shape_step_windows(uint32_t N, uint32_t E, uint32_t kz, uint32_t tiles) { return shape_step(N, E, kz, tiles); }

size_t shape_smem_layout(uint32_t threads, uint32_t tiles, const uint32_t *lmax, const uint32_t *N, const uint32_t *kz,
                         uint32_t n_domains, WarpParams *wp) {
  size_t o = align16(sizeof(DomS) * (n_domains ? n_domains : 1));
  for (uint32_t d = 0; d < n_domains; ++d) {
    o += align16((size_t)2 << lmax[d]);
    o += kDeqBytes;
    if (!shape_form(N[d], kz[d], tiles)) o += (size_t)kz[d] * shape_pairs8(N[d]) * 4;
  }
  o = align16(o);
  *wp = WarpParams{};
  wp->n_domains = n_domains;
  wp->warp_off = (uint32_t)o;
  wp->warp_bytes = (uint32_t)stream_bytes(shape_cap((int)tiles));
  const size_t warps = threads / 32;
  return o + warps * wp->warp_bytes + 1023 + warps * tiles * kOutTile;  // + alignment of the staging tiles
}

// Tensor map of an output buffer of `extent` floats as windows of N floats,
// chunks of 32: dims (32, N / 32, windows), boxes of one chunk of 32 windows.
// The last window may lie partly outside the buffer; a box only ever holds
// whole windows of a segment, so nothing there is written.
bool encode_window_map(CUtensorMap *map, float *out, uint64_t extent, uint32_t N) {
  return encode_out_map3(map, out, (extent + N - 1) / N * N, N);
}

cudaError_t shape_smem_config(uint32_t threads, uint32_t tiles, uint32_t forms, size_t smem) {
  void *k = spick(threads, tiles, forms);
  if (!k) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout,
                                       (int)cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return e;
  return set_dynamic_smem_limit(k, smem);
}

cudaError_t shape_occupancy(uint32_t threads, uint32_t tiles, uint32_t forms, size_t smem, int *ctas_per_sm) {
  void *k = spick(threads, tiles, forms);
  if (!k) return cudaErrorInvalidValue;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, k, (int)threads, smem);
}

cudaError_t launch_shape(const DecodeParams &p, const WarpParams &wp, const ShapeMaps &maps, uint32_t threads,
                         uint32_t tiles, uint32_t forms, uint32_t grid, size_t smem, cudaStream_t stream) {
  if (p.tile_end <= p.tile_begin || grid == 0) return cudaSuccess;
  void *k = spick(threads, tiles, forms);
  if (!k) return cudaErrorInvalidValue;
  DecodeParams pp = p;
  WarpParams ww = wp;
  ShapeMaps mm = maps;
  void *args[] = {&pp, &ww, &mm};
  return launch_after(k, grid, threads, args, smem, stream, p.after_index != 0);
}

}  // namespace fptc
