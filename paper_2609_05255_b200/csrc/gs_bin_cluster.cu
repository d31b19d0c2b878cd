// Binning of scenes that do not fill the chip: the whole chain - Gaussians ordered by depth, cell records emitted in that
// order, records ordered by cell, instances counted per tile, tile ranges - in ONE kernel of one thread-block cluster,
// and a second one that writes the instance lists.
//
// For such scenes the grid-wide chain of gs_sort.cu (12 launches) is bound by the launches: each of its kernels has a
// few microseconds of work at most.  Here the up to 16 CTAs of a cluster, 1024 threads each on an SM of its own, meet at
// hardware barriers instead, and exchange digit histograms through distributed shared memory.  Keys and records go
// through global memory between the passes (a few MB that stay in L2).
// The results are the same bits as those of the grid-wide chain: both are stable sorts.
// The same kernel as a cooperative grid of one CTA per SM, for larger scenes, was no faster than the chain (barriers of
// 2 us, and every CTA reads every other's digits): a step on 100 000 Gaussians 212 against 217 us, on a million 642 against 604.
#include <mutex>

#include "gs_bin.cuh"

namespace gs {
namespace {

using namespace bin;

constexpr int kThreads = 1024, kWarps = 32;
constexpr int kRows = 8;                       // elements per thread and tile
constexpr int kTile = kThreads * kRows;        // elements a CTA ranks at a time
constexpr int kBins = 1 << kClusterDigit;
constexpr int kCountRow = kWarps + 1;           // (odd: a digit's warps, and a warp's digits, lie in different banks)
constexpr int kCountMax = 2048;                // up to this many Gaussians the depth order is found by counting

struct Shared {
  uint32_t keys[kTile], vals[kTile];           // a tile in digit order
  uint32_t count[kBins * kCountRow];           // per digit and warp
  uint32_t lanes[kBins * kCountRow];           // per digit and warp: lanes of the row being ranked that have it
  uint32_t digits[kBins];                      // digits of this CTA's elements (read by the others)
  uint32_t start[kBins + 1];                   // of every digit in the output
  uint32_t base[kBins];                        // where this CTA's next element of a digit goes
  uint32_t tile_count[kBins], tile_start[kBins];
  uint32_t piece_first[kBins + 1];
  uint32_t warp_sum[kWarps];
  uint32_t lowest, highest, records;           // (read by the others)
  uint32_t all_lowest, all_highest, records_before, all_records;
  TileScan scan;
};

// ---- the CTAs of the cluster -----------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_rank() { uint32_t r; asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ uint32_t cluster_size() { uint32_t r; asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r)); return r; }
// All have come here and see each other's writes.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// A word of another CTA's shared memory, at the place it has in this one's.
__device__ __forceinline__ uint32_t remote_word(const uint32_t *p, uint32_t rank) {
  uint32_t v;
  asm volatile("{\n\t.reg .u32 a;\n\tmapa.shared::cluster.u32 a, %1, %2;\n\tld.shared::cluster.u32 %0, [a];\n\t}"
               : "=r"(v) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank) : "memory");
  return v;
}

// Exclusive prefix sum over the CTA; `total` comes out in every thread.
__device__ __forceinline__ uint32_t block_exclusive(Shared &s, uint32_t v, uint32_t &total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t inc = warp_inclusive(v, lane);
  __syncthreads();                             // the last use of warp_sum is over
  if (lane == 31) s.warp_sum[warp] = inc;
  __syncthreads();
  const uint32_t w = s.warp_sum[lane], winc = warp_inclusive(w, lane);
  total = __shfl_sync(kFull, winc, 31);
  return inc - v + __shfl_sync(kFull, winc - w, warp);
}

// ---- one pass of the stable radix sort over this CTA's elements [begin, end) ----------------------------------------
// Digits of `bits` bits at `shift`; load(i, key, val) fetches element i.  Every CTA counts its digits, the counts are
// exchanged, and the elements go where all smaller digits everywhere, the same digit in the CTAs before, and the same
// digit earlier in this CTA leave them.  Where the elements fit one tile, the ranks found on the way are the count.
struct Tile { uint32_t key[kRows], val[kRows], place[kRows]; };

// Ranks a tile: place = elements of the same digit before in this warp; s.count [digit][warp] becomes the elements of the
// digit in the warps before, s.tile_count the digit's total.
template <class Load>
__device__ __forceinline__ void rank_tile(Shared &s, Tile &t, uint32_t first, int len, int shift, int bits, Load &&load) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nb = 1 << bits;
  const uint32_t mask = (uint32_t)nb - 1u;
  const int rows = (len + kThreads - 1) / kThreads, span = rows * 32;
  for (int k = tid; k < nb * kCountRow; k += kThreads) s.count[k] = s.lanes[k] = 0u;
#pragma unroll
  for (int r = 0; r < kRows; ++r) {
    const int local = warp * span + r * 32 + lane;
    if (r < rows && local < len) load(first + local, t.key[r], t.val[r]);
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kRows; ++r) {
    if (r >= rows) break;
    const int at = (int)((t.key[r] >> shift) & mask) * kCountRow + warp;
    t.place[r] = rank_row(s.count + at, s.lanes + at, warp * span + r * 32 + lane < len, lane);
  }
  __syncthreads();
  // per digit, four threads scan the counts of eight warps each
  for (int d0 = 0; d0 < nb; d0 += kThreads / 4) {
    const int d = d0 + (tid >> 2), q = tid & 3;
    uint32_t *c = s.count + min(d, nb - 1) * kCountRow + 8 * q, v[8], sum = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) { v[i] = sum; sum += c[i]; }
    uint32_t inc = sum, u = __shfl_up_sync(kFull, inc, 1, 4);
    if (q >= 1) inc += u;
    u = __shfl_up_sync(kFull, inc, 2, 4);
    if (q >= 2) inc += u;
    if (d < nb) {
#pragma unroll
      for (int i = 0; i < 8; ++i) c[i] = v[i] + inc - sum;
      if (q == 3) s.tile_count[d] = inc;
    }
  }
  __syncthreads();
}

// Writes a ranked tile: through shared memory in digit order, so that neighbouring threads write neighbouring places.
__device__ __forceinline__ void write_tile(Shared &s, const Tile &t, int len, int shift, int bits, uint32_t *keys_out, uint32_t *vals_out) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nb = 1 << bits;
  const uint32_t mask = (uint32_t)nb - 1u;
  const int rows = (len + kThreads - 1) / kThreads, span = rows * 32;
  uint32_t total;
  const uint32_t begins = block_exclusive(s, tid < nb ? s.tile_count[tid] : 0u, total);
  if (tid < nb) s.tile_start[tid] = begins;
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kRows; ++r) {
    if (r >= rows) break;
    if (warp * span + r * 32 + lane < len) {
      const uint32_t d = (t.key[r] >> shift) & mask, at = s.tile_start[d] + s.count[d * kCountRow + warp] + t.place[r];
      s.keys[at] = t.key[r];
      s.vals[at] = t.val[r];
    }
  }
  __syncthreads();
#pragma unroll 4
  for (int j = tid; j < len; j += kThreads) {
    const uint32_t k = s.keys[j], d = (k >> shift) & mask, to = s.base[d] + ((uint32_t)j - s.tile_start[d]);
    keys_out[to] = k;
    vals_out[to] = s.vals[j];
  }
  __syncthreads();
  if (tid < nb) s.base[tid] += s.tile_count[tid];
}

// From the digits of all CTAs: where every digit starts in the output (s.start), and where this CTA's elements
// go (s.base).
__device__ __forceinline__ void place_digits(Shared &s, int bits) {
  const int tid = threadIdx.x, nb = 1 << bits;
  if (tid < nb) s.start[tid] = s.base[tid] = 0u;
  cluster_sync();
  const uint32_t rank = cluster_rank(), ctas = cluster_size();
  // kThreads / nb threads per digit share the CTAs out, eight loads in flight
  const int parts = kThreads >> bits, d = tid & (nb - 1);
  uint32_t before = 0, all = 0;
  for (uint32_t c0 = tid >> bits; c0 < ctas; c0 += 8 * parts) {
    uint32_t v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = c0 + k * parts < ctas ? remote_word(&s.digits[d], c0 + k * parts) : 0u;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      all += v[k];
      before += c0 + k * parts < rank ? v[k] : 0u;
    }
  }
  if (all) atomicAdd(&s.start[d], all);
  if (before) atomicAdd(&s.base[d], before);
  __syncthreads();
  uint32_t total;
  all = tid < nb ? s.start[tid] : 0u;
  const uint32_t start = block_exclusive(s, all, total);
  if (tid < nb) { s.start[tid] = start; s.base[tid] += start; }
  if (tid == 0) s.start[nb] = total;
  __syncthreads();
}

template <class Load>
__device__ __forceinline__ void radix_pass(Shared &s, uint32_t begin, uint32_t end, int shift, int bits, uint32_t *keys_out,
                                           uint32_t *vals_out, Load &&load) {
  const int tid = threadIdx.x, nb = 1 << bits;
  const uint32_t mask = (uint32_t)nb - 1u, count = end - begin;
  Tile t;
  if (count <= kTile) {
    rank_tile(s, t, begin, (int)count, shift, bits, load);
    if (tid < nb) s.digits[tid] = s.tile_count[tid];
    place_digits(s, bits);
    write_tile(s, t, (int)count, shift, bits, keys_out, vals_out);
  } else {
    // sixteen histograms, shared by two warps each
    for (int k = tid; k < 16 << bits; k += kThreads) s.count[k] = 0u;
    __syncthreads();
    for (uint32_t i = begin + tid; i < end; i += kThreads) {
      uint32_t k, v;
      load(i, k, v);
      atomicAdd(&s.count[(((tid >> 5) & 15) << bits) + ((k >> shift) & mask)], 1u);
    }
    __syncthreads();
    if (tid < nb) {
      uint32_t c = 0;
#pragma unroll
      for (int w = 0; w < 16; ++w) c += s.count[(w << bits) + tid];
      s.digits[tid] = c;
    }
    place_digits(s, bits);
    for (uint32_t first = begin; first < end; first += kTile) {
      const int len = (int)min((uint32_t)kTile, end - first);
      rank_tile(s, t, first, len, shift, bits, load);
      write_tile(s, t, len, shift, bits, keys_out, vals_out);
      __syncthreads();
    }
  }
  cluster_sync();
}

// Depth order of up to kCountMax Gaussians: every CTA holds all keys and finds the ranks of its own by counting those that
// come before them, eight threads to a Gaussian.
__device__ __forceinline__ void order_by_counting(Shared &s, const uint32_t *depth_key, uint32_t n, uint32_t begin, uint32_t end, uint32_t *order) {
  const int tid = threadIdx.x;
  for (uint32_t i = tid; i < (n + 31u & ~31u); i += kThreads) s.keys[i] = i < n ? __ldg(depth_key + i) : 0xffffffffu;
  __syncthreads();
  for (uint32_t i0 = begin; i0 < end; i0 += kThreads / 8) {
    const uint32_t i = i0 + (tid >> 3), mine = s.keys[min(i, n - 1u)];
    uint32_t before = 0;
    for (uint32_t j = 4 * (tid & 7); j < n; j += 32) {
      const uint4 k = *reinterpret_cast<const uint4 *>(s.keys + j);
      before += (k.x < mine || (k.x == mine && j < i)) + (k.y < mine || (k.y == mine && j + 1 < i)) +
                (k.z < mine || (k.z == mine && j + 2 < i)) + (k.w < mine || (k.w == mine && j + 3 < i));
    }
#pragma unroll
    for (int sft = 1; sft < 8; sft <<= 1) before += __shfl_xor_sync(kFull, before, sft);
    if ((tid & 7) == 0 && i < end) order[before] = i;
  }
}

// The stored records of a warp's 32 Gaussians (3 x 3 cells at most each; count 0: none) to their places `at`: a lane per
// record, so that neighbouring lanes read neighbouring words of a row and write neighbouring places.  (With a lane per
// Gaussian every load and store touches 32 rows: the emission of 20 000 Gaussians took 6.5 us, now 4.7.)  `owners`: 288 bytes of the warp's shared memory.
__device__ __forceinline__ void copy_records(const uint32_t *cell_records, uint32_t g, uint32_t count, uint32_t at, uint32_t capacity,
                                             uint32_t *rec_keys, uint32_t *rec_vals, unsigned char *owners, int lane) {
  const uint32_t inc = warp_inclusive(count, lane), total = __shfl_sync(kFull, inc, 31), first = inc - count;
  for (uint32_t k = 0; k < count; ++k) owners[first + k] = (unsigned char)lane;
  __syncwarp();
  for (uint32_t j0 = 0; j0 < total; j0 += 64) {    // two loads in flight
    uint32_t id[2], to[2], rec[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t j = j0 + 32 * h + lane;
      const int o = j < total ? owners[j] : 0;
      const uint32_t k = j - __shfl_sync(kFull, first, o);
      id[h] = __shfl_sync(kFull, g, o);
      const uint32_t place = __shfl_sync(kFull, at, o) + k;
      to[h] = j < total ? place : 0xffffffffu;
      rec[h] = j < total ? __ldg(cell_records + (size_t)id[h] * kCellSlots + k) : 0u;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (to[h] < capacity) {                      // never past the buffers, even if the count was taken on the device
        rec_keys[to[h]] = rec[h];
        rec_vals[to[h]] = id[h];
      }
  }
  __syncwarp();
}

__global__ void __launch_bounds__(kThreads, 1) k_bin_cluster(ClusterBinArgs a) {
  dependency_wait();
  extern __shared__ __align__(16) unsigned char cluster_smem[];
  Shared &s = *reinterpret_cast<Shared *>(cluster_smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t rank = cluster_rank(), ctas = cluster_size();
  const uint32_t n = a.n, per = (n + ctas - 1) / ctas;
  const uint32_t begin = min(n, rank * per), end = min(n, begin + per), count = end - begin;
  if (tid == 0) {
    if (rank == 0) { a.report.send(); *a.num_big = 0u; }
    s.lowest = s.all_lowest = 0xffffffffu;
    s.highest = s.all_highest = s.records_before = s.all_records = 0u;
  }
  __syncthreads();

  // ---- depth order
  if (n <= kCountMax) {
    order_by_counting(s, a.depth_key, n, begin, end, a.order);
    cluster_sync();
  } else {
    // Keys are taken relative to the smallest one, culled Gaussians after the largest one: a view's depths differ in some
    // 24 to 27 bits, three passes of digits of nine bits or less
    {
      uint32_t lo = 0xffffffffu, hi = 0u;
#pragma unroll 4
      for (uint32_t i = begin + tid; i < end; i += kThreads) {
        const uint32_t k = __ldg(a.depth_key + i);
        if (k != 0xffffffffu) { lo = min(lo, k); hi = max(hi, k); }
      }
      lo = __reduce_min_sync(kFull, lo); hi = __reduce_max_sync(kFull, hi);
      if (lane == 0) { atomicMin(&s.lowest, lo); atomicMax(&s.highest, hi); }
    }
    cluster_sync();
    if (tid < ctas) { atomicMin(&s.all_lowest, remote_word(&s.lowest, tid)); atomicMax(&s.all_highest, remote_word(&s.highest, tid)); }
    __syncthreads();
    const uint32_t lowest = min(s.all_lowest, s.all_highest), culled = s.all_highest - lowest + 1u;
    const int key_bits = 32 - __clz(culled), passes = (key_bits + kClusterDigit - 1) / kClusterDigit, width = (key_bits + passes - 1) / passes;
    for (int p = 0; p < passes; ++p) {
      const bool odd = (passes - p) & 1;       // the last pass ends in the caller's arrays
      const uint32_t *keys_in = odd ? a.tmp_keys : a.keys, *vals_in = odd ? a.tmp_vals : a.order;
      radix_pass(s, begin, end, p * width, width, odd ? a.keys : a.tmp_keys, odd ? a.order : a.tmp_vals,
                 [&](uint32_t i, uint32_t &k, uint32_t &v) {
                   if (p) { k = __ldcg(keys_in + i); v = __ldcg(vals_in + i); return; }
                   k = __ldg(a.depth_key + i);
                   k = k == 0xffffffffu ? culled : k - lowest;
                   v = i;
                 });
    }
  }

  // ---- one record per (Gaussian, cell of 4 x 4 tiles), in depth order: a thread per Gaussian for the places
  static_assert(kClusterMax <= 16 * kThreads, "a thread has one Gaussian at most");
  const uint32_t g = tid < count ? __ldcg(a.order + begin + tid) : 0u, cc = tid < count ? __ldg(a.cell_count + g) : 0u, cnt = cc & ~kCellBig;
  uint32_t own_records;
  const uint32_t place = block_exclusive(s, cnt, own_records);
  if (tid == 0) s.records = own_records;
  cluster_sync();
  if (tid < ctas) {
    const uint32_t v = remote_word(&s.records, tid);
    atomicAdd(&s.all_records, v);
    if (tid < rank) atomicAdd(&s.records_before, v);
  }
  __syncthreads();
  const uint32_t capacity = a.capacity, first_record = s.records_before;
  if (rank == 0 && tid == 0 && s.all_records > capacity) *a.overflow = 1u;      // more records than the buffers hold
  if (cc & kCellBig) {                         // large footprints wait for a warp, below
    const uint32_t slot = atomicAdd(a.num_big, 1u);
    a.tmp_vals[slot] = g; a.tmp_keys[slot] = first_record + place;
  }
  copy_records(a.cell_records, g, (cc & kCellBig) ? 0u : cnt, first_record + place, capacity, a.rec_keys, a.rec_vals,
               reinterpret_cast<unsigned char *>(s.count) + warp * 32 * kCellSlots, lane);
  // large footprints are worked out by a warp each; the near ones are the large ones, so they are shared out over the cluster
  cluster_sync();
  {
    const uint32_t waiting = __ldcg(a.num_big);
    big_footprints(rank + ctas * warp, ctas * kWarps, waiting, a.rect, a.mean2d, a.conic_opacity, a.cgx, a.W, a.H, lane,
                   [&](uint32_t b, uint32_t &bg, uint32_t &place) { bg = __ldcg(a.tmp_vals + b); place = __ldcg(a.tmp_keys + b); },
                   [&](uint32_t dst, uint32_t bg, uint32_t cell, uint32_t tiles) {
                     if (dst < capacity) {
                       a.rec_keys[dst] = (cell << 16) | tiles;
                       a.rec_vals[dst] = bg;
                     }
                   });
    if (waiting) cluster_sync();
  }
  // ---- records by cell
  radix_pass(s, min(capacity, first_record), min(capacity, first_record + own_records), 16, a.cell_bits, a.sorted_rec_keys,
             a.sorted_rec_vals, [&](uint32_t i, uint32_t &k, uint32_t &v) { k = __ldcg(a.rec_keys + i); v = __ldcg(a.rec_vals + i); });

  // ---- instances per tile, by pieces of kBinPiece records of one cell
  const int cells = a.num_cells;
  {
    const uint32_t len = tid < cells ? s.start[tid + 1] - s.start[tid] : 0u;
    uint32_t total;
    const uint32_t first = block_exclusive(s, (len + kBinPiece - 1) / kBinPiece, total);
    if (tid < cells) s.piece_first[tid] = first;
    if (tid == 0) s.piece_first[cells] = total;
    __syncthreads();
    if (rank == 0) {
      if (tid <= cells) a.piece_first[tid] = s.piece_first[tid];
      if (tid < cells) { a.cell_ranges[2 * tid] = s.start[tid]; a.cell_ranges[2 * tid + 1] = s.start[tid + 1]; }
    }
  }
  for (uint32_t q = rank * kWarps + warp; q < s.piece_first[cells]; q += ctas * kWarps) {
    int lo = 0, hi = cells - 1;                // largest cell with piece_first <= q
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (s.piece_first[mid] <= q) lo = mid; else hi = mid - 1;
    }
    const uint32_t from = s.start[lo] + (q - s.piece_first[lo]) * kBinPiece, to = min(from + kBinPiece, s.start[lo + 1]);
    uint32_t tiles[8], acc[4], sums[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const uint32_t i = from + 32 * k + lane;
      tiles[k] = i < to ? __ldcg(a.sorted_rec_keys + i) & 0xffffu : 0u;
    }
    count_masks(tiles, acc);
    warp_sum_counts(acc, sums);
    if (lane < 16) a.piece_counts[(size_t)q * 16 + lane] = tile_count_of(sums, lane);
  }
  cluster_sync();
  // per cell (one warp each): where each piece's instances of a tile begin inside the tile's list, and how long that is;
  // a lane takes the sixteen counts of a piece, 32 pieces at a time
  for (int c = rank * kWarps + warp; c < cells; c += ctas * kWarps) {
    const uint32_t q0 = s.piece_first[c], q1 = s.piece_first[c + 1];
    uint32_t carry = 0;                        // of tile lane (lanes 0..15)
    for (uint32_t q = q0; q < q1; q += 32) {
      uint4 v[4] = {};
      if (q + lane < q1)
#pragma unroll
        for (int r = 0; r < 4; ++r) v[r] = __ldcg(reinterpret_cast<const uint4 *>(a.piece_counts) + (size_t)(q + lane) * 4 + r);
      uint32_t *w = reinterpret_cast<uint32_t *>(v);
      uint32_t sum = 0;
#pragma unroll
      for (int t = 0; t < 16; t += 2) {        // two tiles per word: 32 pieces hold at most 8192 instances of a tile
        const uint32_t both = w[t] | w[t + 1] << 16, inc = warp_inclusive(both, lane), all = __shfl_sync(kFull, inc, 31), before = inc - both;
        w[t] = __shfl_sync(kFull, carry, t) + (before & 0xffffu);
        w[t + 1] = __shfl_sync(kFull, carry, t + 1) + (before >> 16);
        sum = lane == t ? all & 0xffffu : lane == t + 1 ? all >> 16 : sum;
      }
      carry += sum;
      if (q + lane < q1)
#pragma unroll
        for (int r = 0; r < 4; ++r) reinterpret_cast<uint4 *>(a.piece_bases)[(size_t)(q + lane) * 4 + r] = v[r];
    }
    const int tx = 4 * (c % a.cgx) + (lane & 3), ty = 4 * (c / a.cgx) + (lane >> 2);
    if (lane < 16 && tx < a.gx && ty < a.gy) a.tile_counts[ty * a.gx + tx] = carry;
  }
  cluster_sync();
  if (rank == 0) tile_scan(s.scan, a.tile_counts, a.gx * a.gy, a.pair_capacity32, a.tile_starts, a.tile_ranges, a.tile_order);
}

// The instance lists: one warp per piece.
constexpr int kExpandThreads = 128;
__global__ void __launch_bounds__(kExpandThreads) k_expand_pieces(ClusterBinArgs a) {
  dependency_wait();
  const int lane = threadIdx.x & 31;
  const uint32_t pieces = __ldg(a.piece_first + a.num_cells);
  for (uint32_t q = blockIdx.x * (kExpandThreads / 32) + (threadIdx.x >> 5); q < pieces; q += gridDim.x * (kExpandThreads / 32)) {
    int lo = 0, hi = a.num_cells - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (__ldg(a.piece_first + mid) <= q) lo = mid; else hi = mid - 1;
    }
    const uint32_t from = __ldg(a.cell_ranges + 2 * lo) + (q - __ldg(a.piece_first + lo)) * kBinPiece;
    const uint32_t to = min(from + kBinPiece, __ldg(a.cell_ranges + 2 * lo + 1));
    uint32_t tiles[8], gid[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const uint32_t i = from + 32 * k + lane;
      tiles[k] = i < to ? __ldg(a.sorted_rec_keys + i) & 0xffffu : 0u;
      gid[k] = i < to ? __ldg(a.sorted_rec_vals + i) : 0u;
    }
    const int tx = 4 * (lo % a.cgx) + (lane & 3), ty = 4 * (lo / a.cgx) + (lane >> 2);
    uint32_t mine = 0;                         // (a tile of the cell outside the image has no instances)
    if (lane < 16 && tx < a.gx && ty < a.gy) mine = __ldg(a.tile_starts + ty * a.gx + tx) + __ldg(a.piece_bases + (size_t)q * 16 + lane);
    expand_records(tiles, gid, mine, kBinPiece, a.pair_capacity32, a.out_vals, lane);    // (kBinPiece at most)
  }
}

}  // namespace

namespace {
// Dependent launch of `ctas` CTAs as one cluster; attr has room for two.
cudaLaunchConfig_t cluster_config(int ctas, cudaLaunchAttribute attr[2], cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = ctas; cfg.blockDim = kThreads; cfg.dynamicSmemBytes = sizeof(Shared); cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = ctas; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 2;
  return cfg;
}
}  // namespace

int bin_cluster_limit(int device) {
  // asked once per process and device, whose share of a GPU does not change (the question takes 2 ms)
  static std::once_flag asked[64];
  static int limits[64] = {};
  if (device < 0 || device >= 64) return 0;
  std::call_once(asked[device], [device] {
    if (cudaFuncSetAttribute(k_bin_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Shared)) == cudaSuccess &&
        cudaFuncSetAttribute(k_bin_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
      for (int ctas = kClusterCtas; ctas >= 1 && !limits[device]; ctas /= 2) {
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cfg = cluster_config(ctas, attr, nullptr);
        cfg.numAttrs = 1;
        int active = 0;
        if (cudaOccupancyMaxActiveClusters(&active, k_bin_cluster, &cfg) == cudaSuccess && active > 0) limits[device] = ctas;
      }
    }
    cudaGetLastError();                        // a refusal is an answer
  });
  return limits[device];
}

int launch_bin_cluster(const ClusterBinArgs &a, int ctas, int64_t record_bound, cudaStream_t st) {
  cudaLaunchAttribute attr[2];
  const cudaLaunchConfig_t cfg = cluster_config(ctas, attr, st);
  if (cudaLaunchKernelEx(&cfg, k_bin_cluster, a) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  const int64_t warps = (record_bound + kBinPiece - 1) / kBinPiece + a.num_cells, blocks = (warps + 3) / 4;
  launch_chained(k_expand_pieces, (int)(blocks < 148 * 12 ? blocks : 148 * 12), kExpandThreads, 0, st, a);
  return 2;
}

}  // namespace gs
