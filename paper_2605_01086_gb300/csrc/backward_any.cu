// Adjoint of the lossy decode stage (backward.cu states it) from saved levels, for
// any window shape: a warp per group of windows.
//
// As in the encoder's level kernel for other shapes, a window of gradients is
// folded once, u[n] = g[n] + g[N-1-n] and v[n] = g[n] - g[N-1-n] for n < P =
// ceil(N / 2) (the middle sample of an odd N as it is in both: its basis value is
// 0 to rounding for odd k), because
//   g_C[k] = sum_n g[n] B[k][n] = sum_{n < P} (k even ? u : v)[n] B[k][n].
// Where that is not finite (an infinity or NaN among the gradients, or two whose
// sum overflows) the plain sum over n is taken instead, as in the block kernel.
// A lane then has four windows and four bins of one parity: 32 paired multiply-
// adds (fma.f32x2, pairs along n, the halves added at the end) for four 16-byte
// reads of the folded windows and four of the basis.  g_C is staged in shared
// memory, from where consecutive lanes write consecutive values and form
// g_C * unit_z(level), added per lane and zone as an FP32 pair (two-sum) and per
// warp in FP64, one atomic per warp, domain and zone.
// A batch with fewer tiles than the chip has warps is split into parts of tiles
// (backward_any_split), and a CTA loads the tables of its own segments' domains
// only: with whole tiles per warp and every domain's tables per CTA, 40,000
// samples of eight domains (64, 64) took 60 us, longer than the 18 us of the
// block kernel (backward.cu) that this one replaced; now 17.  (One domain
// (64, 64): 33 us, the block kernel 21, now 19.)
// Bound by latency with 16 warps per SM.  One thread per (window, bin) with an
// N-term dot product from shared memory took 183 us for 16.8 M samples at N = 64,
// E = 32; this took 89 us with a level loaded at a time (the largest stall by far),
// and takes 65 us with eight of them in flight.
#include "device_util.cuh"

namespace fptc {
namespace {

constexpr uint32_t kBwWarps = 8;
constexpr uint32_t kBwLevels = 8;  // of a lane's levels, loaded together
constexpr uint32_t kBwMaxDomains = 128;  // more do not fit: a domain's unit rows are 2 KB

__host__ __device__ constexpr uint32_t bw_pitch(uint32_t n) { return ((n + 3) / 4 | 1u) * 4; }  // odd number of 16-byte pieces
__host__ __device__ constexpr uint32_t bw_pairs4(uint32_t N) { return ((N + 1) / 2 + 3) / 4 * 4; }
__host__ __device__ constexpr uint32_t bw_groups(uint32_t E) { return ((E + 1) / 2 + 3) / 4 + (E / 2 + 3) / 4; }
// Windows taken together: one item of four windows and four bins per lane,
// within 1024 samples (or 16 windows).
__host__ __device__ constexpr uint32_t bw_tile(uint32_t N, uint32_t E) {
  uint32_t t = 8;
  while (t < 64 && bw_groups(E) * t / 4 < 32 && 2 * t * N <= 1024) t *= 2;
  return t;
}
__host__ __device__ constexpr uint32_t bw_bytes(uint32_t N, uint32_t E) {
  const uint32_t t = bw_tile(N, E);
  return t * bw_pitch(N) * 4 + 2 * t * bw_pitch(bw_pairs4(N)) * 4 + (t * E * 4 + 15) / 16 * 16;
}

__device__ __forceinline__ void cp16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(__cvta_generic_to_global(src))
               : "memory");
}
__device__ __forceinline__ void cp4z(void *dst, const void *src, uint32_t bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(__cvta_generic_to_global(src)), "r"(bytes)
               : "memory");
}

// An FP32 sum with its rounding errors (which are NaN where the sum is infinite).
struct PairSum {
  float s = 0.0f, c = 0.0f;
  __device__ __forceinline__ double total() const { return isfinite(s) ? (double)s + (double)c : (double)s; }
  __device__ __forceinline__ void add(float a, float b) {  // + a * b
    const float p = __fmul_rn(a, b), e = __fmaf_rn(a, b, -p);
    const float t = __fadd_rn(s, p), z = __fsub_rn(t, s);
    c = __fadd_rn(c, __fadd_rn(__fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z)), e));
    s = t;
  }
};

// A place among the tiles: a tile and a part of it (split parts a tile).
struct BwPlace {
  uint64_t tile;
  uint32_t part;
  __device__ BwPlace(const DecodeParams &p, uint32_t split, uint64_t unit, uint64_t units) {
    const uint64_t at = (p.tile_end - p.tile_begin) * split * unit / units;
    tile = p.tile_begin + at / split;
    part = (uint32_t)(at % split);
  }
  __device__ bool before(const BwPlace &o) const { return tile < o.tile || (tile == o.tile && part < o.part); }
};

__global__ void __launch_bounds__(kBwWarps * 32, 2) k_backward_any(const BackwardParams bp, uint32_t n_domains,
                                                                  uint32_t warp_bytes, uint32_t split) {
  extern __shared__ __align__(16) unsigned char bw_smem[];
  const DecodeParams &p = bp.d;
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  uint32_t tab_bytes = 0;
  for (uint32_t d = 0; d < n_domains; ++d) tab_bytes += (512u + p.domains[d].E * bw_pairs4(p.domains[d].N)) * 4;
  float *const tabs = reinterpret_cast<float *>(bw_smem), *const xs = tabs + (tab_bytes + wid * warp_bytes) / 4;
  const uint64_t units = (uint64_t)gridDim.x * kBwWarps, unit = (uint64_t)blockIdx.x * kBwWarps + wid;
  BwPlace at(p, split, unit, units);
  const BwPlace to(p, split, unit + 1, units);
  uint32_t s = 0;
  if (at.before(to)) s = warp_find_segment(p.segs, p.seg_begin, p.seg_end, at.tile, lane);
  // ---- the domains of the CTA's segments, a bit each (in the first warp's buffers)
  uint32_t *const used = reinterpret_cast<uint32_t *>(bw_smem + tab_bytes);
  if (n_domains > 1) {
    if (threadIdx.x < kBwMaxDomains / 32) used[threadIdx.x] = 0u;
    __syncthreads();
    if (at.before(to)) {
      const uint64_t end = to.tile + (to.part ? 1u : 0u);
      for (uint32_t i = s + lane; i < p.seg_end && p.segs[i].tile_base < end; i += 32)
        atomicOr(used + p.segs[i].domain / 32u, 1u << (p.segs[i].domain & 31u));
    }
    __syncthreads();
  }
  // ---- those domains' unit rows (zeroed for a zone that is off) and basis rows of bw_pairs4(N)
  {
    uint32_t off = 0;
    for (uint32_t d = 0; d < n_domains; ++d) {
      const DomainDev &dm = p.domains[d];
      const uint32_t P = (dm.N + 1) / 2, p4 = bw_pairs4(dm.N);
      if (n_domains == 1 || (used[d / 32u] >> (d & 31u) & 1u)) {
        const float a0 = p.scale ? p.scale[d * 3 + 0] : dm.scale[0];
        const float a1 = p.scale ? p.scale[d * 3 + 1] : dm.scale[1];
        for (uint32_t i = threadIdx.x; i < 512u; i += kBwWarps * 32)
          tabs[off + i] = (i < 256u ? a0 : a1) > 1e-30f ? dm.unit[i >> 8][i & 255u] : 0.0f;
#pragma unroll 8
        for (uint32_t i = threadIdx.x; i < dm.E * p4; i += kBwWarps * 32) {
          const uint32_t k = i / p4, n = i - k * p4;
          tabs[off + 512u + i] = n < P ? __ldg(p.basis + dm.basis_offset + (size_t)k * dm.N + n) : 0.0f;
        }
      }
      off += 512u + dm.E * p4;
    }
  }
  __syncthreads();
  if (!at.before(to)) return;

  PairSum sum0, sum1;
  uint32_t dom = 0xFFFFFFFFu;
  auto flush = [&]() {
    double a0 = sum0.total(), a1 = sum1.total();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      a0 += __shfl_xor_sync(0xffffffffu, a0, o);
      a1 += __shfl_xor_sync(0xffffffffu, a1, o);
    }
    if (lane == 0 && dom != 0xFFFFFFFFu) {
      if (a0 != 0.0) atomicAdd(bp.grad_scale + dom * 3 + 0, a0);
      if (a1 != 0.0) atomicAdd(bp.grad_scale + dom * 3 + 1, a1);
    }
    sum0 = sum1 = PairSum{};
  };

  for (; at.before(to); ++s) {
    const SegDev &sg = p.segs[s];
    const uint64_t seg_end = sg.tile_base + sg.n_tiles;
    if (at.tile >= seg_end) continue;
    const DomainDev &dm = p.domains[sg.domain];
    const uint32_t N = dm.N, E = dm.E, B1 = dm.B1, B2 = dm.B2;
    if (sg.domain != dom) {
      flush();
      dom = sg.domain;
    }
    auto window = [&](const BwPlace &x) -> uint64_t {
      return (x.tile - sg.tile_base) * dm.tile_windows + dm.tile_windows * x.part / split;
    };
    const uint64_t win0 = window(at);
    const uint64_t wend = to.tile < seg_end ? min(window(to), sg.n_windows) : sg.n_windows;
    at = to;
    if (to.tile >= seg_end) {  // the range goes on, or ends, behind this segment
      at.tile = seg_end;
      at.part = 0;
    }
    if (win0 >= wend) continue;  // a part past the end of the segment's last tile
    const float *unit_tab = tabs;
    for (uint32_t d = 0; d < sg.domain; ++d) unit_tab += 512u + p.domains[d].E * bw_pairs4(p.domains[d].N);
    const float *const basis = unit_tab + 512;
    const uint32_t P = (N + 1) / 2, P4 = bw_pairs4(N), tile = bw_tile(N, E), xp = bw_pitch(N), up = bw_pitch(P4);
    const uint32_t ge = ((E + 1) / 2 + 3) / 4, go = (E / 2 + 3) / 4;
    float *const us = xs + tile * xp, *const vs = us + tile * up, *const gc = vs + tile * up;
    const uint32_t magic = (uint32_t)((0x100000000ull + N - 1) / N);  // division of numbers below 2^16 by N
    const float *const src0 = bp.grad_out + sg.out_offset;
    const bool vec = N % 4 == 0 && (reinterpret_cast<uintptr_t>(src0) & 15u) == 0;
    auto load = [&](uint64_t w0) {  // the gradients of windows w0 .., zero past the stream's end
      const uint32_t nw = wend - w0 < tile ? (uint32_t)(wend - w0) : tile, total = nw * N;
      const float *src = src0 + w0 * N;
      const uint64_t left = sg.n_samples - w0 * N;
      if (vec && left >= total) {
        for (uint32_t i = 4 * lane; i < total; i += 128) {
          const uint32_t w = __umulhi(i, magic);
          cp16(xs + w * xp + (i - w * N), src + i);
        }
      } else {
        for (uint32_t i = lane; i < total; i += 32) {
          const uint32_t w = __umulhi(i, magic);
          cp4z(xs + w * xp + (i - w * N), i < left ? src + i : src0, i < left ? 4u : 0u);
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    load(win0);
    for (uint64_t w0 = win0; w0 < wend; w0 += tile) {
      const uint32_t nw = wend - w0 < tile ? (uint32_t)(wend - w0) : tile;
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncwarp();
      // ---- fold: window and every other piece of four pairs
      for (uint32_t i = lane; i < 2 * tile; i += 32) {
        const uint32_t w = i % tile, h = i / tile;
        const float *x = xs + w * xp;
        for (uint32_t c = 4 * h; c < P4; c += 8) {
          float a[4], b[4], u[4], v[4];
          if (N % 4 == 0) {
            const float4 q = *reinterpret_cast<const float4 *>(x + c);
            const float4 r = *reinterpret_cast<const float4 *>(x + N - 4 - c);
            a[0] = q.x, a[1] = q.y, a[2] = q.z, a[3] = q.w;
            b[0] = r.w, b[1] = r.z, b[2] = r.y, b[3] = r.x;
          } else {
#pragma unroll
            for (uint32_t j = 0; j < 4; ++j) {
              a[j] = c + j < P ? x[c + j] : 0.0f;
              b[j] = c + j < P ? x[N - 1 - c - j] : 0.0f;
            }
          }
#pragma unroll
          for (uint32_t j = 0; j < 4; ++j) {
            const bool in = c + j < P, mid = 2 * (c + j) + 1 == N;
            u[j] = in ? (mid ? a[j] : a[j] + b[j]) : 0.0f;
            v[j] = in ? (mid ? a[j] : a[j] - b[j]) : 0.0f;
          }
          *reinterpret_cast<float4 *>(us + w * up + c) = make_float4(u[0], u[1], u[2], u[3]);
          *reinterpret_cast<float4 *>(vs + w * up + c) = make_float4(v[0], v[1], v[2], v[3]);
        }
      }
      __syncwarp();
      if (w0 + tile < wend) load(w0 + tile);
      // ---- g_C, four windows x four bins a lane and round
      const uint32_t wgs = tile / 4, items = wgs * (ge + go);
      float off = 0.0f;  // 0 while every g_C is finite, else NaN
      for (uint32_t item = lane; item < items; item += 32) {
        const uint32_t bg = item / wgs, wg = item - bg * wgs;
        const bool odd = bg >= ge;
        const uint32_t k0 = odd ? 8 * (bg - ge) + 1 : 8 * bg;  // bins k0, k0 + 2, + 4, + 6
        const float *rows = (odd ? vs : us) + wg * up;
        const float *cs[4];
#pragma unroll
        for (uint32_t j = 0; j < 4; ++j) cs[j] = basis + (k0 + 2 * j < E ? k0 + 2 * j : k0) * P4;
        float2 acc[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.0f, 0.0f);
        for (uint32_t c = 0; c < P4; c += 4) {
          float4 f[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) f[i] = *reinterpret_cast<const float4 *>(rows + i * wgs * up + c);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float4 g = *reinterpret_cast<const float4 *>(cs[j] + c);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              acc[i][j] = __ffma2_rn(make_float2(f[i].x, f[i].y), make_float2(g.x, g.y), acc[i][j]);
              acc[i][j] = __ffma2_rn(make_float2(f[i].z, f[i].w), make_float2(g.z, g.w), acc[i][j]);
            }
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (uint32_t j = 0; j < 4; ++j) {
            const float r = acc[i][j].x + acc[i][j].y;
            off += r - r;
            if (k0 + 2 * j < E) gc[(wg + i * wgs) * E + k0 + 2 * j] = r;
          }
      }
      __syncwarp();
      if (__any_sync(0xffffffffu, off != 0.0f)) {
        const float *const src = src0 + w0 * N;
        const uint64_t left = sg.n_samples - w0 * N;
        for (uint32_t i = lane; i < nw * E; i += 32) {
          if (isfinite(gc[i])) continue;
          const uint32_t w = i / E;
          const float *const row = p.basis + dm.basis_offset + (size_t)(i - w * E) * N;
          float acc = 0.0f;
          for (uint32_t n = 0; n < N; ++n) acc = fmaf(w * N + n < left ? src[w * N + n] : 0.0f, row[n], acc);
          gc[i] = acc;
        }
        __syncwarp();
      }
      // ---- out, and with the levels into the scale gradients
      const uint32_t total = nw * E;
      const uint64_t at = sg.level_offset + w0 * E;
      const uint8_t *const lv = bp.levels_in + at;
      if (bp.grad_coeffs) {
        float *const dst = bp.grad_coeffs + at;
        if ((reinterpret_cast<uintptr_t>(dst) & 15u) == 0 && (total & 3u) == 0) {
          for (uint32_t i = 4 * lane; i < total; i += 128)
            __stcs(reinterpret_cast<float4 *>(dst + i), *reinterpret_cast<const float4 *>(gc + i));
        } else {
          for (uint32_t i = lane; i < total; i += 32) __stcs(dst + i, gc[i]);
        }
      }
      uint32_t k = lane % E;
      const uint32_t dk = 32 % E;
      for (uint32_t i0 = lane; i0 < total; i0 += 32 * kBwLevels) {
        uint32_t L[kBwLevels];
#pragma unroll
        for (uint32_t j = 0; j < kBwLevels; ++j) L[j] = i0 + 32 * j < total ? __ldg(lv + i0 + 32 * j) : 0u;
#pragma unroll
        for (uint32_t j = 0; j < kBwLevels; ++j) {
          if (i0 + 32 * j >= total) break;
          const float g = gc[i0 + 32 * j];
          if (k < B1)
            sum0.add(g, unit_tab[L[j]]);
          else if (k < B2)
            sum1.add(g, unit_tab[256 + L[j]]);
          k += dk;
          if (k >= E) k -= E;
        }
      }
      __syncwarp();
    }
  }
  flush();
}

}  // namespace

size_t backward_any_smem(const uint32_t *N, const uint32_t *E, uint32_t n_domains, uint32_t *warp_bytes) {
  size_t tab = 0;
  *warp_bytes = 0;
  for (uint32_t d = 0; d < n_domains; ++d) {
    tab += (512 + (size_t)E[d] * bw_pairs4(N[d])) * 4;
    *warp_bytes = std::max(*warp_bytes, bw_bytes(N[d], E[d]));
  }
  return tab + (size_t)kBwWarps * *warp_bytes;
}

cudaError_t backward_any_config(size_t smem, int *ctas_per_sm) {
  const void *k = reinterpret_cast<const void *>(&k_backward_any);
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout,
                                       (int)cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess) e = set_dynamic_smem_limit(k, smem);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, k, kBwWarps * 32, smem);
  return e;
}

// Parts a tile is split in: until every warp of `ctas` has one, or a part is one
// of the kernel's own tiles (bw_tile).
uint32_t backward_any_split(uint64_t n_tiles, uint64_t ctas, const DomainDev *dd, uint32_t n_domains) {
  uint32_t most = 1;
  for (uint32_t d = 0; d < n_domains; ++d) {
    const uint32_t t = bw_tile(dd[d].N, dd[d].E);
    most = std::max(most, (dd[d].tile_windows + t - 1) / t);
  }
  return n_tiles ? (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(most, ctas * kBwWarps / n_tiles)) : 1u;
}

cudaError_t launch_backward_any(const BackwardParams &p, uint32_t n_domains, uint32_t warp_bytes, uint32_t split,
                                uint32_t grid, size_t smem, cudaStream_t stream) {
  if (p.d.tile_end <= p.d.tile_begin || grid == 0) return cudaSuccess;
  k_backward_any<<<grid, kBwWarps * 32, smem, stream>>>(p, n_domains, warp_bytes, split);
  return cudaGetLastError();
}

}  // namespace fptc
