// Device helpers shared by the two binning paths: the grid-wide kernels of gs_sort.cu and the one-cluster kernel of
// gs_bin_cluster.cu.
#pragma once
#include "gs_device.cuh"

namespace gs {
namespace bin {

constexpr unsigned kFull = 0xffffffffu;

// Stable rank of a row of 32 elements inside its warp, for a radix sort: `count` and `lanes` point to the words of this
// lane's digit in arrays that belong to the warp alone, both zero at the start of a tile.  Every lane sets its bit in the
// digit's word, reads back which lanes share the digit, and takes the count so far plus the sharing lanes below it; the
// highest of them moves the count on and clears the word.  About 30 cycles of a scheduler per row, whatever the width of
// the digit - finding the sharing lanes by one ballot per digit bit takes 10 cycles a bit, the match instruction up to 250.
__device__ __forceinline__ uint32_t rank_row(uint32_t *count, uint32_t *lanes, bool valid, int lane) {
  if (valid) atomicOr(lanes, 1u << lane);
  __syncwarp();
  uint32_t m = 0, c = 0;
  if (valid) { m = *lanes; c = *count; }
  __syncwarp();
  if (valid && (m >> lane) == 1u) { *count = c + __popc(m); *lanes = 0u; }
  __syncwarp();
  return c + __popc(m & ((1u << lane) - 1u));
}

// Gaussians of more than 3 x 3 cells: their cell records worked out again by the whole warp.  The warp takes the numbers
// start, start + stride, ... below total; entry(number, g, at) gives the Gaussian and the place of its first record, and
// emit(place, g, cell, mask) is called for each record by the lane that owns it.
// A lane loads and prepares one Gaussian each; then, Gaussian by Gaussian, the lanes take the 32 tile rows of eight rows of
// cells together, and one record each.  (A row of cells at a time on four lanes, and each Gaussian's loads before its rows:
// 16.1 us for the emission of a view of 100 000 Gaussians, of which 170 are large, now 12.8.)
template <class Entry, class Emit>
__device__ __forceinline__ void big_footprints(uint32_t start, uint32_t stride, uint32_t total, const uint16_t *rect, const float *mean2d,
                                               const float *conic_opacity, int cgx, int W, int H, int lane, Entry &&entry, Emit &&emit) {
  for (uint32_t first = start; first < total; first += 32u * stride) {
    uint32_t my_g = 0, my_at = 0, my_x = 0, my_y = 0;       // columns and rows of tiles: begin | end << 16
    TileSpans mine = {};
    if (first + lane * stride < total) {
      entry(first + lane * stride, my_g, my_at);
      const ushort4 r = __ldg(reinterpret_cast<const ushort4 *>(rect) + my_g);
      const float2 m = __ldg(reinterpret_cast<const float2 *>(mean2d) + my_g);
      const float4 q = __ldg(reinterpret_cast<const float4 *>(conic_opacity) + my_g);
      mine.setup(m.x, m.y, q.x, q.y, q.z, footprint_tau(q.w), W, H);
      my_x = r.x | (uint32_t)r.z << 16;
      my_y = r.y | (uint32_t)r.w << 16;
    }
    const int held = (int)min(32u, (total - first + stride - 1) / stride);
    for (int o = 0; o < held; ++o) {
      TileSpans sp;
      sp.u = __shfl_sync(kFull, mine.u, o); sp.v = __shfl_sync(kFull, mine.v, o); sp.ila = __shfl_sync(kFull, mine.ila, o);
      sp.lb = __shfl_sync(kFull, mine.lb, o); sp.lc = __shfl_sync(kFull, mine.lc, o); sp.taup = __shfl_sync(kFull, mine.taup, o);
      sp.dys = __shfl_sync(kFull, mine.dys, o); sp.eyp = __shfl_sync(kFull, mine.eyp, o); sp.W = W; sp.H = H;
      const uint32_t g = __shfl_sync(kFull, my_g, o), x = __shfl_sync(kFull, my_x, o), y = __shfl_sync(kFull, my_y, o);
      uint32_t at = __shfl_sync(kFull, my_at, o);
      const int y0 = (int)(y & 0xffffu), y1 = (int)(y >> 16);
      for (int cy0 = y0 >> 2; 4 * cy0 < y1; cy0 += 8) {
        // lane 4 r + k: tile row k of row of cells cy0 + r
        int xa = 0, xb = 0;
        const int ty = 4 * cy0 + lane;
        const bool has = ty >= y0 && ty < y1 && sp.row(ty, (int)(x & 0xffffu), (int)(x >> 16), xa, xb);
        if (!has) xa = xb = 0;
        int lo = has ? (xa >> 2) : (1 << 30), hi = has ? ((xb - 1) >> 2) : -1;
        lo = min(lo, __shfl_xor_sync(kFull, lo, 1)); hi = max(hi, __shfl_xor_sync(kFull, hi, 1));
        lo = min(lo, __shfl_xor_sync(kFull, lo, 2)); hi = max(hi, __shfl_xor_sync(kFull, hi, 2));
        const int cells = max(hi - lo + 1, 0);
        int end = cells;                                    // records up to and including this row of cells
#pragma unroll
        for (int s = 4; s < 32; s <<= 1) {
          const int t = __shfl_up_sync(kFull, end, s);
          if (lane >= s) end += t;
        }
        const int all = __shfl_sync(kFull, end, 31);
        for (int j0 = 0; j0 < all; j0 += 32) {
          const int j = j0 + lane;
          int r = 0;                                        // record j lies in the row of cells r
#pragma unroll
          for (int s = 4; s > 0; s >>= 1) {
            const int e = __shfl_sync(kFull, end, 4 * (r + s - 1));
            if (j >= e) r += s;
          }
          r = min(r, 7);
          const int cx = __shfl_sync(kFull, lo, 4 * r) + j - __shfl_sync(kFull, end - cells, 4 * r);
          uint32_t mask = 0u;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int a0 = max(__shfl_sync(kFull, xa, 4 * r + k), 4 * cx) - 4 * cx, b0 = min(__shfl_sync(kFull, xb, 4 * r + k), 4 * cx + 4) - 4 * cx;
            if (b0 > a0) mask |= (((1u << (b0 - a0)) - 1u) << a0) << (4 * k);
          }
          if (j < all) emit(at + (uint32_t)j, g, (uint32_t)((cy0 + r) * cgx + cx), mask);
        }
        at += (uint32_t)all;
      }
    }
  }
}

// The 16 tile counts of the records a lane holds (masks of up to 8 records), as four words of four byte counters:
// one multiplication spreads the four bits of a tile row of the cell over the four bytes of a word.
__device__ __forceinline__ uint32_t spread_row(uint32_t mask, int r) { return (((mask >> (4 * r)) & 15u) * 0x00204081u) & 0x01010101u; }
__device__ __forceinline__ void count_masks(const uint32_t mask[8], uint32_t acc[4]) {
  acc[0] = acc[1] = acc[2] = acc[3] = 0u;
#pragma unroll
  for (int k = 0; k < 8; ++k)
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[r] += spread_row(mask[k], r);
}

// Sum over the warp of the byte counters, widened to 16 bits on the way (8 records x 32 lanes = 256 at most): tile
// 4 r + b of the cell ends in bits [16 (b & 1), +16) of word r * 2 + (b >> 1), in every lane.
__device__ __forceinline__ void warp_sum_counts(const uint32_t acc[4], uint32_t out[8]) {
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    out[2 * r] = (acc[r] & 0xffu) | ((acc[r] & 0xff00u) << 8);
    out[2 * r + 1] = ((acc[r] >> 16) & 0xffu) | ((acc[r] >> 8) & 0xff0000u);
  }
#pragma unroll
  for (int w = 0; w < 8; ++w)
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) out[w] += __shfl_xor_sync(kFull, out[w], s);
}
__device__ __forceinline__ uint32_t tile_count_of(const uint32_t sums[8], int t) {   // t = 4 r + b
  return (sums[2 * (t >> 2) + ((t & 3) >> 1)] >> (16 * (t & 1))) & 0xffffu;
}

__device__ __forceinline__ void store_if(uint32_t p, uint32_t *addr, uint32_t v) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %0, 0;\n\t@q st.global.u32 [%1], %2;\n\t}" :: "r"(p), "l"(addr), "r"(v) : "memory");
}

// A warp writes the instances of its 8 x 32 records (consecutive in depth order, 32 at a time).  A record's slot in the
// list of tile t is the tile's running position plus the number of lower lanes that also list t: the 16
// indicator bits of a lane's mask are spread over four words of byte counters and one warp-wide prefix sum of those
// four words ranks all 16 tiles at once (at most 32 per byte).  `mine`: lane t < 16 passes where tile t continues; every
// lane keeps all 16 running positions.  kInside: no position reaches the capacity, so that a store needs its mask bit only.
template <bool kInside>
__device__ __forceinline__ void expand_rows(const uint32_t mask[8], const uint32_t gid[8], uint32_t mine, uint32_t capacity,
                                            uint32_t *out_vals, int lane) {
  uint32_t cur[16];
#pragma unroll
  for (int t = 0; t < 16; ++t) cur[t] = __shfl_sync(kFull, mine, t);
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    // instances of the rows before, as bytes like the ranks (96 at most): the running positions move on once in four rows
    uint32_t before[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int k = 4 * half; k < 4 * half + 4; ++k) {
      const uint32_t m = mask[k];
      if (__ballot_sync(kFull, m != 0u) == 0u) continue;
      uint32_t incl[4], at[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        incl[r] = spread_row(m, r);
        at[r] = before[r] - incl[r];
      }
#pragma unroll
      for (int sft = 1; sft < 32; sft <<= 1) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const uint32_t u = __shfl_up_sync(kFull, incl[r], sft);
          if (lane >= sft) incl[r] += u;
        }
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        at[r] += incl[r];
        before[r] += __shfl_sync(kFull, incl[r], 31);
      }
#pragma unroll
      for (int t = 0; t < 16; ++t) {
        // one predicated store (no branch): the lane lists tile t and the slot lies inside the buffer
        const uint32_t pos = cur[t] + __byte_perm(at[t >> 2], 0u, 0x4440 | (t & 3));
        store_if(kInside || pos < capacity ? m & (1u << t) : 0u, out_vals + pos, gid[k]);
      }
    }
#pragma unroll
    for (int t = 0; t < 16; ++t) cur[t] += __byte_perm(before[t >> 2], 0u, 0x4440 | (t & 3));
  }
}
// `count`: instances that the warp writes for tile `lane` (lanes below 16).
__device__ __forceinline__ void expand_records(const uint32_t mask[8], const uint32_t gid[8], uint32_t mine, uint32_t count,
                                               uint32_t capacity, uint32_t *out_vals, int lane) {
  if (__all_sync(kFull, lane >= 16 || (mine <= capacity && count <= capacity - mine)))
    expand_rows<true>(mask, gid, mine, capacity, out_vals, lane);
  else
    expand_rows<false>(mask, gid, mine, capacity, out_vals, lane);
}

// By one CTA of 1024 threads: the exclusive scan of the tile counts in tile order = the tile ranges, and the launch
// order of the blend's warps (tiles by decreasing list length in log2 buckets: the long tiles start first and the short
// ones fill the tail; the order inside a bucket is whatever the atomics give, it affects scheduling only, never a result).
// A warp takes the tiles [32 w per, 32 (w + 1) per) of a strip of 1024 per, 32 neighbours at a time and all loads in flight
// together.  (With `per` neighbours per thread every store of a warp went to 32 sectors: 4161 tiles 7.3 us, now 5.3, 8160
// tiles 13.5, now 7.3.)
struct TileScan { uint32_t w[32], cnt[33], off[33], all; };
__device__ __forceinline__ void tile_scan(TileScan &s, const uint32_t *tile_counts, int num_tiles, uint32_t capacity,
                                          uint32_t *tile_starts, uint32_t *ranges, uint32_t *order) {
  constexpr int kMost = 8;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int per = min((num_tiles + 1023) / 1024, kMost), strip = 1024 * per;
  if (tid < 33) s.cnt[tid] = 0;
  __syncthreads();
  uint32_t v[kMost];
  auto tile_of = [&](int base, int k) { return base + 32 * (warp * per + k) + lane; };
  auto load = [&](int base) {
#pragma unroll
    for (int k = 0; k < kMost; ++k) {
      const int t = tile_of(base, k);
      v[k] = k < per && t < num_tiles ? __ldcg(tile_counts + t) : 0u;
    }
  };
  for (int base = 0; base < num_tiles; base += strip) {
    load(base);
#pragma unroll
    for (int k = 0; k < kMost; ++k)
      if (k < per && tile_of(base, k) < num_tiles) atomicAdd(&s.cnt[32 - __clz(v[k])], 1u);
  }
  __syncthreads();
  if (warp == 0) {                             // lane l: bucket 32 - l, the longest lists first
    const uint32_t c = s.cnt[32 - lane], inc = warp_inclusive(c, lane);
    s.off[32 - lane] = inc - c;
    if (lane == 31) s.off[0] = inc;
  }
  uint32_t carry = 0;
  for (int base = 0; base < num_tiles; base += strip) {
    if (strip < num_tiles) load(base);
    uint32_t sum = 0, before[kMost];             // of the warp; of it before the tile
#pragma unroll
    for (int k = 0; k < kMost; ++k) {
      before[k] = 0u;
      if (k >= per) continue;
      const uint32_t inc = warp_inclusive(v[k], lane);
      before[k] = sum + inc - v[k];
      sum += __shfl_sync(kFull, inc, 31);
    }
    if (lane == 0) s.w[warp] = sum;
    __syncthreads();
    if (warp == 0) {
      const uint32_t w = s.w[lane], winc = warp_inclusive(w, lane);
      s.w[lane] = winc - w;
      if (lane == 31) s.all = winc;
    }
    __syncthreads();
    const uint32_t first = carry + s.w[warp];
    carry += s.all;
#pragma unroll
    for (int k = 0; k < kMost; ++k) {
      const int t = tile_of(base, k);
      if (k >= per || t >= num_tiles) continue;
      const uint32_t start = first + before[k];
      tile_starts[t] = start;
      // a tile without instances: (0, 0); never past the capacity of the instance buffers (a device-side count may
      // exceed it: the lists are then cut off and the host is told)
      const uint32_t s0 = min(start, capacity), e0 = start + v[k] < start ? capacity : min(start + v[k], capacity);
      reinterpret_cast<uint2 *>(ranges)[t] = e0 > s0 ? make_uint2(s0, e0) : make_uint2(0u, 0u);
      order[atomicAdd(&s.off[32 - __clz(v[k])], 1u)] = (uint32_t)t;
    }
    __syncthreads();
  }
}

}  // namespace bin
}  // namespace gs
