// SymLen segment indexing (Sec. 4.2.1: an exclusive prefix sum over the symlen
// array gives every compressed word the output position of its first symbol).
//
//   1. k_index: a warp per group of 4 chunks of a segment sums each chunk's
//      symlen (and checks that none exceeds 64); the warp that counts a
//      segment's last group scans the segment's chunk sums into chunk offsets
//      and checks the total against W*E.  No CTA waits on another: the last
//      group is whichever comes last (a counter per segment, which wraps to 0).
//   2. k_tile_index: per chunk, a warp scan gives every word's symbol offset;
//      every word that holds the first symbol of a tile (tile = tile_windows
//      windows = tile_windows * E symbols) writes (word, symbols to skip).
// The decode kernels then start each tile without decoding earlier words.
//
// A few MB are read, so k_index is bound by the dependent loads of a warp:
// group, then segment and symlen (four chunks) at once.  Two kernels, one finding its
// segment by a binary search, took 16 us for the 13 M words of a mixed batch and
// 23 us for 16,384 streams of 370 words; this one 8 and 12 us, and the decode
// kernel behind it loads its tables meanwhile (launch_after).
// k_tile_index runs one warp per chunk over a contiguous chunk range per warp
// (the segment cursor advances with the chunk index), with the next chunks'
// blocks loaded while the current ones are reduced, and only for the kernels
// that read a record per tile: the warp-tile kernels locate the first word of
// their range from the chunk offsets (symbol_word).  The chunk geometry is that
// of symlen_chunks.cuh.
#include "symlen_chunks.cuh"

namespace fptc {
namespace {

// Segment (queue index) owning chunk c: the last segment whose chunk_base <= c.
__device__ __forceinline__ uint32_t chunk_segment(const SegDev *segs, uint32_t lo, uint32_t hi, uint64_t c) {
  while (hi - lo > 1) {
    const uint32_t mid = lo + (hi - lo) / 2;
    if (segs[mid].chunk_base <= c)
      lo = mid;
    else
      hi = mid;
  }
  return lo;
}

// This warp's chunk range [c0, c1) of the launch.
__device__ __forceinline__ void warp_chunks(const IndexParams &p, uint64_t &c0, uint64_t &c1) {
  const uint64_t gw = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint64_t nw = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint64_t n = p.chunk_end - p.chunk_begin;
  c0 = p.chunk_begin + n * gw / nw;
  c1 = p.chunk_begin + n * (gw + 1) / nw;
}

// Symlen blocks of chunks c .. c + P - 1 (clipped to c1) with their segments;
// the segment cursor s advances monotonically.
template <int P>
struct ChunkGroup {
  uint4 v[P];
  uint32_t seg[P];
};
template <int P>
__device__ __forceinline__ void load_group(const IndexParams &p, uint64_t c, uint64_t c1, uint32_t lane, uint32_t &s,
                                           ChunkGroup<P> &g) {
#pragma unroll
  for (int i = 0; i < P; ++i) {
    g.v[i] = make_uint4(0u, 0u, 0u, 0u);
    g.seg[i] = s;
    if (c + i < c1) {
      while (c + i >= p.segs[s].chunk_base + p.segs[s].n_chunks) ++s;
      g.seg[i] = s;
      g.v[i] = load_block(p.symlen, p.segs[s], c + i - p.segs[s].chunk_base, lane).v;
    }
  }
}

// The segment's symbol total against what its windows need, and whether a word
// claims more than 64 symbols: its flag and the plan's status.
__device__ __forceinline__ void close_segment(const IndexParams &p, uint32_t s, const SegDev &sg, uint64_t total,
                                              bool range_bad, uint32_t lane) {
  const bool count_bad = total != sg.n_symbols;
  if (lane == 0) {
    p.seg_bad[s] = (range_bad || count_bad) ? 1u : 0u;
    if (range_bad) flag_bad(p.status, kFlagSymlenRange, sg.caller_index);
    if (count_bad) flag_bad(p.status, kFlagSymbolCount, sg.caller_index);
  }
}

// Inclusive warp scan.
__device__ __forceinline__ uint32_t scan32(uint32_t x, uint32_t lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= (uint32_t)o) x += y;
  }
  return x;
}

__global__ void __launch_bounds__(256) k_index(IndexParams p) {
  dependents_may_start();
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t g = p.group_begin + (uint64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (g >= p.group_end) return;  // the whole warp
  // the group names its segment's words, so that the symlen and the segment's
  // record are requested together
  IndexGroup r;
  if (p.groups) {
    r = p.groups[g];
  } else {
    const uint32_t b = p.seg_begin;
    r.seg = b + (uint32_t)warp_last_leq(p.seg_end - b, g, lane, [&](uint64_t i) { return p.segs[b + i].group_base; });
    r.chunk = (uint32_t)(g - p.segs[r.seg].group_base) * kGroupChunks;
    r.word_offset = p.segs[r.seg].word_offset;
    r.n_words = p.segs[r.seg].n_words;
  }
  const uint32_t s = r.seg, c0 = r.chunk;
  const SegDev sg = p.segs[s];
  uint4 v[kGroupChunks];
#pragma unroll
  for (uint32_t i = 0; i < kGroupChunks; ++i)  // all zero past the segment's end
    v[i] = load_block(p.symlen, r.word_offset, r.n_words, c0 + i, lane).v;
  const uint32_t n_chunks = sg.n_chunks, n = n_chunks - c0 < kGroupChunks ? n_chunks - c0 : kGroupChunks;
  uint32_t sum = 0u, over = 0u;  // lane i: chunk i's sum and whether a word of it claims more than 64
#pragma unroll
  for (uint32_t i = 0; i < kGroupChunks; ++i) {
    const uint32_t x = __reduce_add_sync(0xffffffffu, block_sum(v[i]));
    const bool o = __any_sync(0xffffffffu, block_over64(v[i]));
    if (lane == i) {
      sum = x;
      over = o ? 1u : 0u;
    }
  }
  if (n_chunks <= kGroupChunks) {  // the whole segment
    const uint32_t incl = scan32(sum, lane);
    if (lane < n) p.chunk_off[sg.chunk_base + lane] = incl - sum;
    close_segment(p, s, sg, __shfl_sync(0xffffffffu, incl, 31), __any_sync(0xffffffffu, over != 0u), lane);
    return;
  }
  if (lane < n) __stcg(p.chunk_sum + sg.chunk_base + c0 + lane, over ? kChunkBad : sum);
  __threadfence();
  __syncwarp();
  const uint32_t groups = (uint32_t)groups_of(n_chunks);
  uint32_t before = 0u;
  if (lane == 0) before = atomicInc(p.done + s, groups - 1u);
  if (__shfl_sync(0xffffffffu, before, 0) != groups - 1u) return;
  __threadfence();
  // ---- the segment's last group: every chunk sum is there.  Four a lane and
  // round, the next round's in flight
  uint64_t run = 0;
  bool range_bad = false;
  uint32_t nx[4];
  auto fetch = [&](uint32_t j0) {
#pragma unroll
    for (uint32_t q = 0; q < 4; ++q) {
      const uint32_t j = j0 + 4 * lane + q;
      nx[q] = j < n_chunks ? __ldcg(p.chunk_sum + sg.chunk_base + j) : 0u;
    }
  };
  fetch(0);
  for (uint32_t j0 = 0; j0 < n_chunks; j0 += 128) {
    uint32_t c[4];
#pragma unroll
    for (uint32_t q = 0; q < 4; ++q) {
      range_bad = range_bad || nx[q] == kChunkBad;
      c[q] = nx[q] == kChunkBad ? 0u : nx[q];
    }
    if (n_chunks - j0 > 128) fetch(j0 + 128);
    const uint32_t tot = c[0] + c[1] + c[2] + c[3];
    const uint32_t incl = scan32(tot, lane);
    uint64_t off = run + (incl - tot);
#pragma unroll
    for (uint32_t q = 0; q < 4; ++q) {
      const uint32_t j = j0 + 4 * lane + q;
      if (j < n_chunks) p.chunk_off[sg.chunk_base + j] = off;
      off += c[q];
    }
    run += __shfl_sync(0xffffffffu, incl, 31);
  }
  close_segment(p, s, sg, run, __any_sync(0xffffffffu, range_bad), lane);
}

__global__ void __launch_bounds__(256, 3) k_tile_index(IndexParams p) {
  const uint32_t lane = threadIdx.x & 31;
  uint64_t c0, c1;
  warp_chunks(p, c0, c1);
  if (c0 >= c1) return;
  uint32_t s = chunk_segment(p.segs, p.seg_begin, p.seg_end, c0);
  constexpr int kPipe = 2;
  ChunkGroup<kPipe> cur;
  load_group(p, c0, c1, lane, s, cur);
  uint64_t off_cur[kPipe];
#pragma unroll
  for (int i = 0; i < kPipe; ++i) off_cur[i] = c0 + i < c1 ? p.chunk_off[c0 + i] : 0;
  for (uint64_t c = c0; c < c1; c += kPipe) {
    ChunkGroup<kPipe> nxt;
    load_group(p, c + kPipe, c1, lane, s, nxt);
    uint64_t off_nxt[kPipe];
#pragma unroll
    for (int i = 0; i < kPipe; ++i) off_nxt[i] = c + kPipe + i < c1 ? p.chunk_off[c + kPipe + i] : 0;
#pragma unroll
    for (int i = 0; i < kPipe; ++i) {
      if (c + i >= c1) break;
      const uint32_t si = cur.seg[i];
      if (p.seg_bad[si] != 0) continue;  // uniform over the warp
      const SegDev &sg = p.segs[si];
      const DomainDev &dm = p.domains[sg.domain];
      const uint64_t te = (uint64_t)dm.tile_windows * dm.E;  // symbols per tile
      const uint4 bv = cur.v[i];
      const uint32_t tsum = block_sum(bv);
      uint32_t x = tsum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= (uint32_t)o) x += y;
      }
      if (tsum == 0) continue;
      uint64_t off = off_cur[i] + (x - tsum);  // symbol offset (in the segment) of the block's first word
      // first tile whose start is >= off
      uint64_t tn = off < 0xFFFFFFFFull && te < 0xFFFFFFFFull ? ((uint32_t)off + (uint32_t)te - 1u) / (uint32_t)te
                                                                : (off + te - 1) / te;
      uint64_t ns = tn * te;
      if (ns >= off + tsum) continue;  // most blocks hold no tile start (a tile is thousands of symbols)
      const uint32_t wv[4] = {bv.x, bv.y, bv.z, bv.w};
      // global word index of byte 0 of this lane's block (as load_block computes it)
      const uintptr_t a0 = reinterpret_cast<uintptr_t>(p.symlen + sg.word_offset);
      const uint64_t word0 = sg.word_offset + (uint64_t)(((a0 + 15) & ~uintptr_t(15)) +
                                                         16 * (uintptr_t)(31 * (c + i - sg.chunk_base) + lane) - 16 - a0);
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const uint64_t end = off + ((wv[j >> 2] >> (8 * (j & 3))) & 0xffu);
        while (ns < end) {
          if (tn < sg.n_tiles) {
            TileRec r;
            r.first_word = word0 + j;
            r.skip = (uint32_t)(ns - off);
            r.pad = 0;
            p.tiles[sg.tile_base + tn] = r;
          }
          ++tn;
          ns += te;
        }
        off = end;
      }
    }
    cur = nxt;
#pragma unroll
    for (int i = 0; i < kPipe; ++i) off_cur[i] = off_nxt[i];
  }
}

// Symbol offset (in the segment) of every word, for the three-kernel schedule
// (Sec. 4.2.1 as the paper runs it: a global array of per-word offsets).
__global__ void __launch_bounds__(256) k_word_offsets(IndexParams p, uint32_t *word_off) {
  const uint32_t lane = threadIdx.x & 31;
  uint64_t c0, c1;
  warp_chunks(p, c0, c1);
  if (c0 >= c1) return;
  uint32_t s = chunk_segment(p.segs, p.seg_begin, p.seg_end, c0);
  for (uint64_t c = c0; c < c1; ++c) {
    while (c >= p.segs[s].chunk_base + p.segs[s].n_chunks) ++s;
    const SegDev &sg = p.segs[s];
    const LaneBlock b = load_block(p.symlen, sg, c - sg.chunk_base, lane);
    const uint32_t tsum = block_sum(b.v);
    uint32_t x = tsum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= (uint32_t)o) x += y;
    }
    if (p.seg_bad[s] != 0) continue;  // uniform over the warp
    uint32_t off = (uint32_t)p.chunk_off[c] + (x - tsum);
    const uint32_t wv[4] = {b.v.x, b.v.y, b.v.z, b.v.w};
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const uint64_t word = b.word0 + j;
      // inside the segment (block -1 wraps below word_offset and fails the test)
      if (word - sg.word_offset < sg.n_words && lane < 31) word_off[word] = off;
      off += (wv[j >> 2] >> (8 * (j & 3))) & 0xffu;
    }
  }
}

}  // namespace

cudaError_t launch_index(const IndexParams &p, cudaStream_t stream) {
  const uint64_t n_chunks = p.chunk_end - p.chunk_begin, n_groups = p.group_end - p.group_begin;
  if (p.seg_end <= p.seg_begin || n_groups == 0) return cudaSuccess;
  k_index<<<(unsigned)((n_groups + 7) / 8), 256, 0, stream>>>(p);
  // persistent warps over the chunks: at most one chunk per warp, at most p.grid CTAs of 8 warps
  const uint64_t want = (n_chunks + 7) / 8;
  const uint32_t grid = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(p.grid ? p.grid : 1024u, want));
  if (p.records) k_tile_index<<<grid, 256, 0, stream>>>(p);
  return cudaGetLastError();
}

}  // namespace fptc

namespace fptc {
cudaError_t launch_word_offsets(const IndexParams &p, uint32_t *word_off, cudaStream_t stream) {
  const uint64_t n_chunks = p.chunk_end - p.chunk_begin;
  if (n_chunks == 0 || p.seg_end <= p.seg_begin) return cudaSuccess;
  const uint64_t want = (n_chunks + 7) / 8;
  const uint32_t grid = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(p.grid ? p.grid : 1024u, want));
  k_word_offsets<<<grid, 256, 0, stream>>>(p, word_off);
  return cudaGetLastError();
}
}  // namespace fptc
