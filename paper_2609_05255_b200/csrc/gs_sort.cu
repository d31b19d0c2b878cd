// Ordering and binning: a stable LSD radix sort (digits of 4 to 9 bits, keys staged and ranked in shared
// memory, no inter-block waiting) and the kernels that turn its output into per-tile lists.
//
// (1) The Gaussians are sorted once by their 32-bit depth key (ties keep the index order), by buckets (gs_depth_sort.cu) or, beyond 4M
//     and where the near plane lets depths be zero or negative, by the radix sort; culled ones
//     leaving after the first of the four passes.
// (2) In that order every Gaussian emits one record per CELL of 4 x 4 tiles that its footprint reaches - the cell id
//     and a 16-bit mask of the tiles met inside the cell, as the preprocess left them - and the records are sorted by
//     cell id alone (a quarter of the elements and fewer bits than a sort of the (Gaussian, tile) instances).
// (3) A cell's records, still in depth order, are expanded into the lists of its 16 tiles: counts per chunk of 2048
//     records, one scan for the start of every tile and of every chunk inside it, then each chunk writes its
//     instances, a warp ranking 32 records for all 16 tiles with one prefix sum of byte counters.
// The result is the instance list ordered by (tile, depth key, index), with its per-tile ranges.
#include <algorithm>
#include "gs_bin.cuh"

namespace gs {
namespace {

using namespace bin;

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kItems = 16;
constexpr int kSortTile = kSortThreads * kItems;   // 4096 elements per block iteration
constexpr int kMaxSortBlocks = 444;                // 3 resident CTAs x 148 SMs: one full wave
constexpr int kMaxDigitBits = 9;   // widest radix digit: 512 bins
constexpr int kScanBlock = 256;   // Gaussians per block of the tiles-touched prefix sum and per CTA of the instance emission


// Block b sorts one contiguous range of the input, worked through in tiles of at most kSortTile elements.  While one
// tile per block is enough (count <= blocks x kSortTile) the ranges are equal, rounded up to a multiple of the block
// size, so that a full wave of CTAs shares the work evenly and every warp of a CTA ranks the same number of items.
// Beyond that, whole tiles are dealt out as evenly as they go: a pass costs a fixed latency per tile, and two full
// tiles in a few blocks measured faster than two half tiles in every block (0.40 against 0.45 ms per 8 views on
// 2 M records).  The grid is sized by the host's bound on the count; the ranges follow the count the kernels see
// (which may live on the device), so the work stays balanced either way.
constexpr int kMinPerBlock = 1024;
int sort_blocks(int64_t count) {
  const int64_t b = (count + kMinPerBlock - 1) / kMinPerBlock;
  return (int)(b < 1 ? 1 : b < kMaxSortBlocks ? b : kMaxSortBlocks);
}

struct BlockRange {
  int64_t begin, end;   // this block's elements
  int tiles, tile_len;  // worked through as `tiles` pieces of `tile_len` (the last one may be short)
};

__device__ __forceinline__ BlockRange block_range(int64_t count) {
  const int64_t nb = (int64_t)gridDim.x;
  BlockRange r;
  if (count <= nb * kSortTile) {
    int64_t per = (count + nb - 1) / nb;
    per = (per + kSortThreads - 1) / kSortThreads * kSortThreads;
    r.begin = min(count, (int64_t)blockIdx.x * per);
    r.end = min(count, r.begin + per);
    r.tiles = r.end > r.begin ? 1 : 0;
    r.tile_len = (int)per;
  } else {
    const int64_t tiles = (count + kSortTile - 1) / kSortTile;
    const int b = (int)blockIdx.x;
    const int each = (int)(tiles / nb), extra = (int)(tiles - (int64_t)each * nb);
    r.tiles = each + (b < extra ? 1 : 0);
    r.begin = ((int64_t)b * each + min(b, extra)) * kSortTile;
    r.end = min(count, r.begin + (int64_t)r.tiles * kSortTile);
    r.tile_len = kSortTile;
  }
  return r;
}

// The depth keys are sorted with their bits rotated: the sign bit, which only culled Gaussians have set, comes last.  The
// first of the four passes then has the culled ones in a digit of their own (visible ones have even digits), the largest,
// and puts them where they belong for good; the other passes and the record emission see the visible ones only (1.2 of 3 million in a view from inside a
// scene: the four passes 147 us before, 107 now, the emission 68 and 50).
// What the emission needs to know of a Gaussian first, how many records it has (nine at most, unless its footprint is large),
// travels with its id in the upper bits of the sorted value, where ids leave room: read in order by the first pass, where the
// last pass and the emission fetched it from random rows (emission of 1M Gaussians 33.4 us before, 30.3 now, of 1.5M 46.2
// and 41.6; the sort itself takes as long as before).
constexpr int kIdBits = 28;
constexpr uint32_t kCountUnknown = 15u;        // a large footprint: to be looked up
static_assert(kCellSlots < (int)kCountUnknown, "counts of the stored records fit");
__device__ __forceinline__ uint32_t rotated(uint32_t key) { return __funnelshift_l(key, key, 1); }

// Where a block's elements of a digit go follows from the digits of all blocks before it.  Blocks are taken in groups of
// about the square root of their number: a block adds its digits to its group's sums, and the scatter adds up the groups
// before its own and the blocks before it in its group - 43 loads at most, where a kernel of its own scanned the
// rows before (444 blocks: 4.4 us, and a launch in each pass).
constexpr int kMaxGroups = 22;                   // ceil(sqrt(kMaxSortBlocks)), also the largest group
constexpr int kGroupTables = 6;                  // four passes of the depth sort, two of the record sort
static_assert(kMaxGroups * kMaxGroups >= kMaxSortBlocks, "groups");
int group_size(int blocks) { int g = 1; while (g * g < blocks) ++g; return g; }

// Digit histogram of each block's contiguous range: table[block][digit], added to groups[block / group][digit] unless
// `groups` is null (it is not cleared yet: the first pass, whose block clears the tables of the passes to come).
template <bool ROTATE>
__global__ void __launch_bounds__(kSortThreads) k_radix_hist(const uint32_t *__restrict__ keys, int64_t count,
                                                             const unsigned long long *__restrict__ count_dev,
                                                             int shift, int bits, uint32_t *__restrict__ table,
                                                             uint32_t *__restrict__ groups, int group,
                                                             uint32_t *__restrict__ clear, int clear_words, SortEpilogue ep,
                                                             CountReport report) {
  dependency_wait();
  if (blockIdx.x == 0 && threadIdx.x == 0) report.send();
  for (int i = blockIdx.x * kSortThreads + threadIdx.x; i < clear_words; i += gridDim.x * kSortThreads) clear[i] = 0u;
  // the arrays the scatter of this pass accumulates into start from their neutral values
  if (ep.block_sums)
    for (int i = blockIdx.x * kSortThreads + threadIdx.x; i < ep.num_block_sums; i += gridDim.x * kSortThreads) ep.block_sums[i] = 0u;
  if (ep.ranges && !ep.chunk_first)
    for (int i = blockIdx.x * kSortThreads + threadIdx.x; i < 2 * ep.num_ranges; i += gridDim.x * kSortThreads)
      ep.ranges[i] = (i & 1) ? 0u : 0xffffffffu;
  if (count_dev) count = min(count, (int64_t)__ldg(count_dev));     // the true length lives on the device
  // up to 256 digits: one histogram per warp (fewer collisions); more: four shared by the warps
  __shared__ uint32_t s_hist[kSortWarps << 8];
  const int tid = threadIdx.x, warp = tid >> 5;
  const int nb = 1 << bits, copies = nb <= 256 ? kSortWarps : kSortWarps / 2;
  const uint32_t mask = (uint32_t)nb - 1u;
  for (int k = tid; k < copies * nb; k += kSortThreads) s_hist[k] = 0;
  __syncthreads();
  const BlockRange r = block_range(count);
  uint32_t *mine = s_hist + (warp % copies) * nb;
  // eight loads in flight, also of the last ones (four, and the last ones singly: 7.1 us for 2.0M records, now 5.8)
  const uint32_t *own = keys + r.begin;
  const uint32_t length = (uint32_t)(r.end - r.begin);
  auto put = [&](uint32_t k) { atomicAdd(mine + (((ROTATE ? rotated(k) : k) >> shift) & mask), 1u); };
  constexpr uint32_t kLoads = 8, kStep = kLoads * kSortThreads;
  uint32_t i = tid;
  for (; i - tid + kStep <= length; i += kStep) {
    uint32_t k[kLoads];
#pragma unroll
    for (int h = 0; h < (int)kLoads; ++h) k[h] = __ldg(own + i + h * kSortThreads);
#pragma unroll
    for (int h = 0; h < (int)kLoads; ++h) put(k[h]);
  }
  if (i - tid < length) {
    uint32_t k[kLoads];
#pragma unroll
    for (int h = 0; h < (int)kLoads; ++h) k[h] = i + h * kSortThreads < length ? __ldg(own + i + h * kSortThreads) : 0u;
#pragma unroll
    for (int h = 0; h < (int)kLoads; ++h)
      if (i + h * kSortThreads < length) put(k[h]);
  }
  __syncthreads();
  for (int d = tid; d < nb; d += kSortThreads) {
    uint32_t t = 0;
    for (int w = 0; w < copies; ++w) t += s_hist[w * nb + d];
    table[(blockIdx.x << bits) + d] = t;
    if (groups && t) atomicAdd(groups + ((blockIdx.x / group) << bits) + d, t);
  }
}

// The groups' sums of the first pass: one CTA per group.
__global__ void __launch_bounds__(1 << 8) k_group_sums(const uint32_t *__restrict__ table, int nblocks, int group,
                                                       uint32_t *__restrict__ groups) {
  dependency_wait();
  const int first = blockIdx.x * group, last = min(nblocks, first + group);
  uint32_t t = 0;
#pragma unroll 8
  for (int b = first; b < last; ++b) t += __ldg(table + (b << 8) + threadIdx.x);
  groups[(blockIdx.x << 8) + threadIdx.x] = t;
}

// Exclusive prefix sums over kSortThreads * DPT values in thread-major order (thread t holds values t * DPT ..): each
// thread scans its own values, the thread totals are scanned across the block.
template <int DPT>
__device__ __forceinline__ void block_exclusive_scan(const uint32_t v[DPT], uint32_t out[DPT], uint32_t *s_warp_tot, int tid) {
  const int lane = tid & 31, warp = tid >> 5;
  uint32_t sum = 0;
#pragma unroll
  for (int j = 0; j < DPT; ++j) { out[j] = sum; sum += v[j]; }
  const uint32_t inc = warp_inclusive(sum, lane);
  if (lane == 31) s_warp_tot[warp] = inc;
  __syncthreads();
  uint32_t off = inc - sum;
#pragma unroll
  for (int w = 0; w < kSortWarps; ++w) off += (w < warp) ? s_warp_tot[w] : 0u;
  __syncthreads();
#pragma unroll
  for (int j = 0; j < DPT; ++j) out[j] += off;
}

template <int BITS> constexpr size_t scatter_smem_bytes() {
  return sizeof(uint32_t) * (2 * kSortTile + (size_t)(kSortWarps + 2) * (BITS <= 8 ? 256 : (1 << BITS)) + kSortWarps + 1);
}

// One pass: stable scatter of this block's range by the BITS-wide digit at `shift` (BITS up to kMaxDigitBits; the
// digit arrays hold max(256, 2^BITS) entries, thread t looking after digits t * DPT ..).  Slots past the
// end of the input carry the largest digit and sit at the end of the last tile, so they rank after
// every real key and are never written.
// EP selects the epilogue: 0 none, 1 the last pass of the depth sort: leaves the Gaussians' record counts in place of the
// keys, and their sums per block of sorted positions, 2 ranges of
// equal ids = key >> key_shift (last pass of the record sort: inside a block's run of one digit the keys are
// non-decreasing, because the earlier passes ordered the lower bits, so a change of id between neighbours of a run
// is a boundary; the two ends of a run may continue in another block and enter with an atomic min / max), 3 the first
// pass of the depth sort: keys come as they are, the largest digit's elements go to their final place and are counted out,
// 4 the record sort in a single pass: the digits' totals are the ranges, and the chunks of the expansion follow from them.
template <int BITS, int EP>
__global__ void __launch_bounds__(kSortThreads, 3) k_radix_scatter(
    const uint32_t *__restrict__ keys_in, const uint32_t *__restrict__ vals_in, uint32_t *__restrict__ keys_out,
    uint32_t *__restrict__ vals_out, int64_t count, const unsigned long long *__restrict__ count_dev, int shift,
    const uint32_t *__restrict__ table, const uint32_t *__restrict__ groups, int group, SortEpilogue ep) {
  dependency_wait();
  constexpr int NB = BITS <= 8 ? 256 : (1 << BITS);   // entries of the digit arrays
  constexpr int DPT = NB / kSortThreads;              // digits per thread
  extern __shared__ __align__(16) uint32_t s_dyn[];
  uint32_t *s_keys = s_dyn, *s_vals = s_keys + kSortTile;
  uint32_t *s_warp_cnt = s_vals + kSortTile;          // [kSortWarps][NB]
  uint32_t *s_digit_start = s_warp_cnt + kSortWarps * NB, *s_base = s_digit_start + NB, *s_warp_tot = s_base + NB;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t lt_mask = (1u << lane) - 1u;
  if (count_dev) count = min(count, (int64_t)__ldg(count_dev));
  constexpr uint32_t kDigitMask = (1u << BITS) - 1u;

  // global base of every digit for this block: all smaller digits everywhere + the same digit in the blocks before
  {
    uint32_t tot[DPT] = {}, before[DPT] = {}, start[DPT];
    if (tid * DPT <= (int)kDigitMask) {
      const int own = (int)blockIdx.x / group, num = ((int)gridDim.x + group - 1) / group, in_group = (int)blockIdx.x - own * group;
      uint32_t v[kMaxGroups][DPT], u[kMaxGroups][DPT];     // all in flight together: in two halves the pass took 3 us more
#pragma unroll
      for (int g = 0; g < kMaxGroups; ++g)
#pragma unroll
        for (int j = 0; j < DPT; ++j) {
          v[g][j] = g < num ? __ldg(groups + (g << BITS) + tid * DPT + j) : 0u;
          u[g][j] = g < in_group ? __ldg(table + ((own * group + g) << BITS) + tid * DPT + j) : 0u;
        }
#pragma unroll
      for (int g = 0; g < kMaxGroups; ++g)
#pragma unroll
        for (int j = 0; j < DPT; ++j) {
          tot[j] += v[g][j];
          before[j] += u[g][j] + (g < own ? v[g][j] : 0u);
        }
    }
    block_exclusive_scan<DPT>(tot, start, s_warp_tot, tid);
#pragma unroll
    for (int j = 0; j < DPT; ++j) {
      const int d = tid * DPT + j;
      s_base[d] = start[j] + before[j];
      if (EP == 3 && blockIdx.x == 0 && d == (int)kDigitMask) *ep.visible = start[j];
    }
    if (EP == 4 && blockIdx.x == gridDim.x - 1) {       // (its range is the shortest)
      uint32_t chunks[DPT], first[DPT];
#pragma unroll
      for (int j = 0; j < DPT; ++j) chunks[j] = (tot[j] + kCellChunk - 1) / kCellChunk;
      block_exclusive_scan<DPT>(chunks, first, s_warp_tot, tid);
#pragma unroll
      for (int j = 0; j < DPT; ++j) {
        const int d = tid * DPT + j;
        if (d < ep.num_ranges) {
          ep.ranges[2 * d] = start[j]; ep.ranges[2 * d + 1] = start[j] + tot[j];
          ep.chunk_first[d] = first[j];
        }
        s_warp_cnt[d] = first[j]; s_warp_cnt[NB + d] = start[j]; s_warp_cnt[2 * NB + d] = start[j] + tot[j];
        if (d == NB - 1) s_warp_tot[0] = ep.chunk_first[ep.num_ranges] = first[j] + chunks[j];
      }
      __syncthreads();
      for (uint32_t q = tid; q < s_warp_tot[0]; q += kSortThreads) {
        int lo = 0;                                     // the last digit whose chunks begin at q or before
        for (int step = NB / 2; step > 0; step /= 2) lo += s_warp_cnt[lo + step] <= q ? step : 0;
        const uint32_t begin = s_warp_cnt[NB + lo] + (q - s_warp_cnt[lo]) * kCellChunk;
        ep.chunks[q] = make_uint4(begin, min(begin + kCellChunk, s_warp_cnt[2 * NB + lo]), (uint32_t)lo, 0u);
      }
      __syncthreads();
    }
  }

  const BlockRange r = block_range(count);
  const int span = r.tile_len / kSortWarps;           // consecutive elements of a tile that one warp ranks
  const int items = span / 32;                        // ... as this many rows of 32 (at most kItems)
  for (int t = 0; t < r.tiles; ++t) {
    const int64_t tile_begin = r.begin + (int64_t)t * r.tile_len;
    if (tile_begin >= r.end) break;
    const int valid_count = (int)min((int64_t)r.tile_len, r.end - tile_begin);
    for (int k = tid; k < kSortWarps * NB; k += kSortThreads) s_warp_cnt[k] = 0;
    __syncthreads();
    uint32_t key[kItems], val[kItems];
    unsigned short rank[kItems];
    // all loads first (independent, in flight together), then the serial ranking chain
#pragma unroll
    for (int it = 0; it < kItems; ++it) {
      const int local = warp * span + it * 32 + lane;
      const bool ok = it < items && local < valid_count;
      const int64_t idx = tile_begin + local;
      key[it] = ok ? (EP == 3 ? rotated(__ldg(keys_in + idx)) : __ldg(keys_in + idx)) : 0xffffffffu;
      val[it] = ok ? (vals_in ? __ldg(vals_in + idx) : (uint32_t)idx) : 0u;
      if (EP == 3 && ok && ep.id_mask != ~0u) {
        const uint32_t c = __ldg(ep.counts + idx);
        val[it] |= min(c, kCountUnknown) << kIdBits;    // (a large footprint's count has its top bit set)
      }
    }
#pragma unroll
    for (int it = 0; it < kItems; ++it) {
      if (it >= items) break;                         // the same for every thread of the CTA
      const int local = warp * span + it * 32 + lane;
      const bool ok = local < valid_count;
      const uint32_t d = ok ? ((key[it] >> shift) & kDigitMask) : kDigitMask;
      // lanes with the same digit form a group; its first lane bumps the warp's counter once and
      // hands the old value to the group.  A warp's shared-memory atomics execute in program order,
      // so the 16 items need no barrier between them and their latencies overlap.
      // The group comes from one ballot per digit bit: a fixed cost, where the match instruction
      // takes time in proportion to the number of different digits in the warp.
      uint32_t peers = kFull;
#pragma unroll
      for (int b = 0; b < BITS; ++b) {
        const bool bit = (d >> b) & 1u;
        const uint32_t m = __ballot_sync(kFull, bit);
        peers &= bit ? m : ~m;
      }
      const int leader = __ffs(peers) - 1;
      uint32_t prior = 0;
      if (lane == leader) prior = atomicAdd(&s_warp_cnt[warp * NB + d], (uint32_t)__popc(peers));
      prior = __shfl_sync(kFull, prior, leader);
      rank[it] = (unsigned short)(prior + __popc(peers & lt_mask));
    }
    __syncthreads();
    // per digit: exclusive scan over warps, then over digits
    uint32_t cnt[DPT], dstart[DPT];
#pragma unroll
    for (int j = 0; j < DPT; ++j) {
      const int d = tid * DPT + j;
      uint32_t c = 0;
#pragma unroll
      for (int w = 0; w < kSortWarps; ++w) {
        const uint32_t x = s_warp_cnt[w * NB + d];
        s_warp_cnt[w * NB + d] = c;
        c += x;
      }
      cnt[j] = c;
    }
    block_exclusive_scan<DPT>(cnt, dstart, s_warp_tot, tid);
#pragma unroll
    for (int j = 0; j < DPT; ++j) s_digit_start[tid * DPT + j] = dstart[j];
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kItems; ++it) {
      if (it >= items) break;
      const int local = warp * span + it * 32 + lane;
      const uint32_t d = (local < valid_count) ? ((key[it] >> shift) & kDigitMask) : kDigitMask;
      const uint32_t pos = s_digit_start[d] + s_warp_cnt[warp * NB + d] + rank[it];
      s_keys[pos] = key[it];
      s_vals[pos] = val[it];
    }
    __syncthreads();
    constexpr int kOut = 4;                             // rows written together, so that what they wait for overlaps
    for (int j0 = 0; j0 < valid_count; j0 += kOut * kSortThreads) {
      uint32_t gpos[kOut], count_of[kOut];
#pragma unroll
      for (int h = 0; h < kOut; ++h) {
        const int j = j0 + h * kSortThreads + tid;
        const bool ok = j < valid_count;
        gpos[h] = count_of[h] = 0u;
        if (!ok) continue;
        const uint32_t k = s_keys[j], d = (k >> shift) & kDigitMask, v = s_vals[j], run_first = s_digit_start[d];
        gpos[h] = s_base[d] + ((uint32_t)j - run_first);
        if (EP == 1) {
          const uint32_t id = v & ep.id_mask, c = ep.id_mask != ~0u && v >> kIdBits != kCountUnknown ? v >> kIdBits : __ldg(ep.counts + id);
          keys_out[gpos[h]] = c;
          vals_out[gpos[h]] = id;
          count_of[h] = c & ~kCellBig;
        } else if (EP == 3 && d == kDigitMask) {
          ep.final_vals[gpos[h]] = v & ep.id_mask;
        } else {
          keys_out[gpos[h]] = k;
          vals_out[gpos[h]] = v;
        }
        if (EP == 2) {
          const uint32_t run_end = d == kDigitMask ? (uint32_t)valid_count : s_digit_start[d + 1];   // slots past the input hold no run
          const uint32_t id = k >> ep.key_shift;
          if ((uint32_t)j == run_first) atomicMin(ep.ranges + 2 * id, gpos[h]);
          else if ((s_keys[j - 1] >> ep.key_shift) != id) ep.ranges[2 * id] = gpos[h];
          if ((uint32_t)j + 1 == run_end) atomicMax(ep.ranges + 2 * id + 1, gpos[h] + 1);
          else if ((s_keys[j + 1] >> ep.key_shift) != id) ep.ranges[2 * id + 1] = gpos[h] + 1;
        }
      }
      if (EP == 1) {
#pragma unroll
        for (int h = 0; h < kOut; ++h) {
          // the Gaussian's count, added to the sum of its block of kScanBlock sorted positions: once per warp for the first
          // lane's block and once for the last one's (runs of this digit are long, so that hardly any lane has another)
          const bool ok = j0 + h * kSortThreads + tid < valid_count;
          const uint32_t any = __ballot_sync(kFull, ok);
          if (!any) continue;
          const int last = 31 - __clz(any);
          const uint32_t blk = gpos[h] / kScanBlock, blk0 = __shfl_sync(kFull, blk, 0), blk1 = __shfl_sync(kFull, blk, last);
          const bool in0 = blk == blk0, in1 = !in0 && blk == blk1;
          const uint32_t sum0 = __reduce_add_sync(kFull, in0 && ok ? count_of[h] : 0u), sum1 = __reduce_add_sync(kFull, in1 && ok ? count_of[h] : 0u);
          if (lane == 0 && sum0) atomicAdd(ep.block_sums + blk0, sum0);
          if (lane == last && sum1) atomicAdd(ep.block_sums + blk1, sum1);
          if (ok && !in0 && !in1 && count_of[h]) atomicAdd(ep.block_sums + blk, count_of[h]);
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < DPT; ++j) s_base[tid * DPT + j] += cnt[j];
    __syncthreads();
  }
}

__global__ void k_iota(uint32_t *__restrict__ out, int n, CountReport report) {
  if (blockIdx.x == 0 && threadIdx.x == 0) report.send();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = (uint32_t)i;
}

// The stored records of a Gaussian (3 x 3 cells at most) to their places: all loads first, they are one cache line.
// (A lane per record instead, as the one-cluster kernel has it, measured the same at 1M Gaussians and 6 % more at 3M: the rows
// of a depth order lie anywhere, and that is what it waits for.)
__device__ __forceinline__ void copy_records(const uint32_t *cell_records, uint32_t g, uint32_t count, uint32_t at, uint32_t capacity,
                                             uint32_t *rec_keys, uint32_t *rec_vals) {
  const uint32_t *src = cell_records + (size_t)g * kCellSlots;
  uint32_t rec[kCellSlots];
#pragma unroll
  for (int k = 0; k < kCellSlots; ++k) rec[k] = k < (int)count ? __ldg(src + k) : 0u;
#pragma unroll
  for (int k = 0; k < kCellSlots; ++k)
    if (k < (int)count && at + k < capacity) {   // never past the buffers, even if the count was taken on the device
      rec_keys[at + k] = rec[k];
      rec_vals[at + k] = g;
    }
}

// ---- cell records in depth order ---------------------------------------------------------------
// Every Gaussian, in depth order, writes its records (cell id << 16 | tile mask) and its id.  A Gaussian of at most
// 3 x 3 cells copies what the preprocess stored; a larger one is worked out again by a warp.  The large ones are the near
// ones, side by side in this order, so a CTA collects its own and shares them out over its warps.
// Eight CTAs per SM, although the large ones' path then spills: the copies wait for random rows (at five CTAs 55 instead of
// 50 us in a view of 1.2 million).
__global__ void __launch_bounds__(kScanBlock, 8) k_emit_records(
    const uint32_t *__restrict__ order, const uint32_t *__restrict__ sorted_count, const uint32_t *__restrict__ cell_records,
    const uint16_t *__restrict__ rect, const float *__restrict__ mean2d, const float *__restrict__ conic_opacity,
    const uint32_t *__restrict__ block_sums, const unsigned long long *__restrict__ visible, int64_t n, int cgx, int W, int H, uint32_t capacity,
    uint32_t *__restrict__ rec_keys, uint32_t *__restrict__ rec_vals, unsigned long long *__restrict__ rec_total,
    uint32_t *__restrict__ overflow) {
  dependency_wait();
  __shared__ uint32_t s_w[kScanBlock / 32], s_before[kScanBlock / 32];
  __shared__ uint32_t s_big[kScanBlock], s_big_at[kScanBlock], s_num_big;
  if (visible) n = min(n, (int64_t)__ldg(visible)); // culled Gaussians have no record
  const int last_block = max((int)((n + kScanBlock - 1) / kScanBlock) - 1, 0);
  if ((int)blockIdx.x > last_block) return;
  if (threadIdx.x == 0) s_num_big = 0u;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t i = (int64_t)blockIdx.x * kScanBlock + tid;
  uint32_t g = 0, cc = 0;
  if (i < n) {
    g = __ldg(order + i);
    cc = __ldg(sorted_count + i);
  }
  const uint32_t cnt = cc & ~kCellBig;
  const uint32_t inc = warp_inclusive(cnt, lane);
  if (lane == 31) s_w[warp] = inc;
  // records of all CTAs before this one: the sums per kScanBlock Gaussians come from the last pass of the depth
  // sort; every CTA adds up its own prefix (a few loads per thread) instead of a scan kernel doing it for all
  uint32_t before = 0;
  for (int k = tid; k < (int)blockIdx.x; k += kScanBlock) before += __ldg(block_sums + k);
#pragma unroll
  for (int sft = 16; sft > 0; sft >>= 1) before += __shfl_xor_sync(kFull, before, sft);
  if (lane == 0) s_before[warp] = before;
  __syncthreads();
  uint32_t off = 0;
#pragma unroll
  for (int k = 0; k < kScanBlock / 32; ++k) off += s_before[k] + ((k < warp) ? s_w[k] : 0u);
  off += inc - cnt;
  if ((int)blockIdx.x == last_block && tid == kScanBlock - 1) {   // the last thread of all: its end is the number of records
    *rec_total = (unsigned long long)off + cnt;
    if (off + cnt > capacity) *overflow = 1u;                    // more records than the buffers hold: tell the host
  }
  if (cnt && !(cc & kCellBig)) copy_records(cell_records, g, cnt, off, capacity, rec_keys, rec_vals);
  if (cc & kCellBig) {
    const uint32_t slot = atomicAdd(&s_num_big, 1u);
    s_big[slot] = g;
    s_big_at[slot] = off;
  }
  __syncthreads();
  big_footprints(warp, kScanBlock / 32, s_num_big, rect, mean2d, conic_opacity, cgx, W, H, lane,
                 [&](uint32_t b, uint32_t &bg, uint32_t &at) { bg = s_big[b]; at = s_big_at[b]; },
                 [&](uint32_t dst, uint32_t bg, uint32_t cell, uint32_t mask) {
                   if (dst < capacity) {
                     rec_keys[dst] = (cell << 16) | mask;
                     rec_vals[dst] = bg;
                   }
                 });
}

// ---- from the sorted records of a cell to the lists of its tiles ----------------------------------
// Chunks: the records of cell c, [range_c.start, range_c.end), in pieces of kCellChunk; chunk_first[c] = number of
// chunks of the cells before c.  A cell without records comes in as (0xffffffff, 0), the neutral values of the
// range epilogue.
__global__ void __launch_bounds__(1024) k_cell_chunks(const uint32_t *__restrict__ cell_ranges, int num_cells,
                                                      uint32_t *__restrict__ chunk_first) {
  dependency_wait();
  __shared__ uint32_t s_w[32];
  __shared__ uint32_t s_carry;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) s_carry = 0;
  __syncthreads();
  for (int base = 0; base < num_cells; base += 1024) {
    const int c = base + tid;
    uint32_t v = 0;
    if (c < num_cells) {
      const uint32_t s0 = cell_ranges[2 * c], e0 = cell_ranges[2 * c + 1];
      v = e0 > s0 ? (e0 - s0 + kCellChunk - 1) / kCellChunk : 0u;
    }
    const uint32_t inc = warp_inclusive(v, lane);
    if (lane == 31) s_w[warp] = inc;
    __syncthreads();
    if (warp == 0) {
      const uint32_t w = s_w[lane];
      s_w[lane] = warp_inclusive(w, lane) - w;
    }
    __syncthreads();
    const uint32_t carry = s_carry;
    if (c < num_cells) chunk_first[c] = carry + s_w[warp] + inc - v;
    __syncthreads();
    if (tid == 1023) s_carry = carry + s_w[warp] + inc;
    __syncthreads();
  }
  if (tid == 0) chunk_first[num_cells] = s_carry;
}

// ... and which records they are: (begin, end, cell) of every chunk.  One warp per cell.
__global__ void __launch_bounds__(256) k_chunk_list(const uint32_t *__restrict__ cell_ranges, const uint32_t *__restrict__ chunk_first,
                                                    int num_cells, uint4 *__restrict__ chunks) {
  dependency_wait();
  const int lane = threadIdx.x & 31, cell = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (cell >= num_cells) return;
  const uint32_t s0 = __ldg(cell_ranges + 2 * cell), e0 = __ldg(cell_ranges + 2 * cell + 1);
  const uint32_t q0 = __ldg(chunk_first + cell), q1 = __ldg(chunk_first + cell + 1);
  for (uint32_t q = q0 + lane; q < q1; q += 32) {
    const uint32_t begin = s0 + (q - q0) * kCellChunk;
    chunks[q] = make_uint4(begin, min(begin + (uint32_t)kCellChunk, e0), (uint32_t)cell, 0u);
  }
}

// The two kernels below work on chunks.  Their number is known on the device only, and the host's bound (a record for every
// instance) is several times too high: a wave of CTAs goes through the chunks there are.
constexpr int kExpandThreads = 256;
constexpr int kExpandWarps = kExpandThreads / 32;

// Per chunk: how many instances it holds for each of the 16 tiles of its cell.
constexpr int kCountBlocks = 148 * 6;
__global__ void __launch_bounds__(kExpandThreads, 6) k_chunk_counts(const uint32_t *__restrict__ rec_keys, const uint4 *__restrict__ chunks,
                                                                    const uint32_t *__restrict__ num_chunks, uint32_t *__restrict__ chunk_counts) {
  dependency_wait();
  __shared__ uint32_t s_cnt[2][kExpandWarps][16];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t num = __ldg(num_chunks);
  int round = 0;                       // (two sets of counters: one barrier per chunk)
  for (uint32_t q = blockIdx.x; q < num; q += gridDim.x, round ^= 1) {
    const uint4 c = __ldg(chunks + q);
    // warp w holds records [begin + 256 w, + 256): lane l the records 256 w + 32 k + l, k = 0..7
    uint32_t mask[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const uint32_t idx = c.x + (uint32_t)(256 * warp + 32 * k + lane);
      mask[k] = idx < c.y ? (__ldg(rec_keys + idx) & 0xffffu) : 0u;
    }
    uint32_t acc[4], sums[8];
    count_masks(mask, acc);
    warp_sum_counts(acc, sums);
    if (lane < 16) s_cnt[round][warp][lane] = tile_count_of(sums, lane);
    __syncthreads();
    if (tid < 16) {
      uint32_t t = 0;
#pragma unroll
      for (int w = 0; w < kExpandWarps; ++w) t += s_cnt[round][w][tid];
      chunk_counts[(size_t)q * 16 + tid] = t;
    }
  }
}

// Per cell (one warp each, lanes 0..15 = its tiles): where each chunk's instances of a tile begin inside the tile's
// list (the running sum of the chunks' counts, in chunk order) and the length of that list.
__global__ void __launch_bounds__(256) k_cell_prefix(const uint32_t *__restrict__ chunk_first, const uint32_t *__restrict__ chunk_counts,
                                                     int gx, int gy, int cgx, int num_cells, uint32_t *__restrict__ chunk_bases,
                                                     uint32_t *__restrict__ tile_counts) {
  dependency_wait();
  const int lane = threadIdx.x & 31, cell = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (cell >= num_cells || lane >= 16) return;
  const uint32_t q0 = __ldg(chunk_first + cell), q1 = __ldg(chunk_first + cell + 1);
  uint32_t run = 0;
  uint32_t q = q0;
  for (; q + 4 <= q1; q += 4) {   // four independent loads in flight
    const uint32_t v0 = __ldg(chunk_counts + (size_t)q * 16 + lane), v1 = __ldg(chunk_counts + (size_t)(q + 1) * 16 + lane);
    const uint32_t v2 = __ldg(chunk_counts + (size_t)(q + 2) * 16 + lane), v3 = __ldg(chunk_counts + (size_t)(q + 3) * 16 + lane);
    chunk_bases[(size_t)q * 16 + lane] = run; run += v0;
    chunk_bases[(size_t)(q + 1) * 16 + lane] = run; run += v1;
    chunk_bases[(size_t)(q + 2) * 16 + lane] = run; run += v2;
    chunk_bases[(size_t)(q + 3) * 16 + lane] = run; run += v3;
  }
  for (; q < q1; ++q) {
    chunk_bases[(size_t)q * 16 + lane] = run;
    run += __ldg(chunk_counts + (size_t)q * 16 + lane);
  }
  const int tx = 4 * (cell % cgx) + (lane & 3), ty = 4 * (cell / cgx) + (lane >> 2);
  if (tx < gx && ty < gy) tile_counts[ty * gx + tx] = run;
}

__global__ void __launch_bounds__(1024) k_tile_scan(const uint32_t *__restrict__ tile_counts, int num_tiles, uint32_t capacity,
                                                    uint32_t *__restrict__ tile_starts, uint32_t *__restrict__ ranges,
                                                    uint32_t *__restrict__ order) {
  dependency_wait();
  __shared__ TileScan s;
  tile_scan(s, tile_counts, num_tiles, capacity, tile_starts, ranges, order);
}

// Per chunk: write its instances.  The running positions of the tiles start from the tile's range, the chunk's offset
// inside it and what the warps before this one hold.
// Bound by the instructions of the ranking (issue 67 %, ALU pipe 57 % busy): a warp whose positions all lie inside the
// buffers stores by the mask bits alone.  Before, a CTA also searched its chunk's cell (eight dependent loads), and two of
// three CTAs found that they had no chunk.  1M Gaussians, 2.0M records, 7.9M instances: the expansion 55 us, with the chunk
// list 50, with the stores 44.5.
constexpr int kExpandBlocks = 148 * 4;
__global__ void __launch_bounds__(kExpandThreads, 4) k_expand(const uint32_t *__restrict__ rec_keys, const uint32_t *__restrict__ rec_vals,
                                                              const uint4 *__restrict__ chunks, const uint32_t *__restrict__ num_chunks,
                                                              const uint32_t *__restrict__ chunk_bases,
                                                              const uint32_t *__restrict__ tile_starts, int gx, int gy, int cgx,
                                                              uint32_t capacity, uint32_t *__restrict__ out_vals) {
  dependency_wait();
  __shared__ uint32_t s_cnt[2][kExpandWarps][16];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t num = __ldg(num_chunks);
  int round = 0;
  for (uint32_t q = blockIdx.x; q < num; q += gridDim.x, round ^= 1) {
    const uint4 c = __ldg(chunks + q);
    uint32_t mask[8], gid[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const uint32_t idx = c.x + (uint32_t)(256 * warp + 32 * k + lane);
      const bool ok = idx < c.y;
      mask[k] = ok ? (__ldg(rec_keys + idx) & 0xffffu) : 0u;
      gid[k] = ok ? __ldg(rec_vals + idx) : 0u;
    }
    // lane t < 16 works out where tile t of the cell continues
    const int tx = 4 * ((int)c.z % cgx) + (lane & 3), ty = 4 * ((int)c.z / cgx) + (lane >> 2);
    uint32_t mine = 0;
    if (lane < 16 && tx < gx && ty < gy)      // (a tile of the cell outside the image has no instances)
      mine = __ldg(tile_starts + ty * gx + tx) + __ldg(chunk_bases + (size_t)q * 16 + lane);
    uint32_t acc[4], sums[8];
    count_masks(mask, acc);
    warp_sum_counts(acc, sums);
    if (lane < 16) s_cnt[round][warp][lane] = tile_count_of(sums, lane);
    __syncthreads();
    if (lane < 16)
      for (int w = 0; w < warp; ++w) mine += s_cnt[round][w][lane];
    expand_records(mask, gid, mine, tile_count_of(sums, lane & 15), capacity, out_vals, lane);
  }
}

}  // namespace

size_t sort_scratch_bytes(int64_t n, int64_t records) {
  constexpr size_t kTable = (1 << kMaxDigitBits) * sizeof(uint32_t);
  return kGroupTables * kMaxGroups * kTable + std::max(2 * sort_blocks(std::max(n, records)) * kTable, bucket_scratch_bytes(n));
}

namespace {
// The groups' sums of pass `p` of a view (the four of the depth sort, then the record sort's).
uint32_t *group_table(void *scratch, int p) { return static_cast<uint32_t *>(scratch) + ((size_t)p * kMaxGroups << kMaxDigitBits); }
uint32_t *block_table(void *scratch) { return group_table(scratch, kGroupTables); }

template <int BITS, int EP>
void launch_scatter(int blocks, const uint32_t *src_k, const uint32_t *src_v, uint32_t *dst_k, uint32_t *dst_v, int64_t count,
                    const unsigned long long *count_dev, int shift, const uint32_t *table, const uint32_t *groups,
                    const SortEpilogue &ep, cudaStream_t st) {
  constexpr size_t smem = scatter_smem_bytes<BITS>();
  static bool opted[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (smem > 48 * 1024 && dev >= 0 && dev < 64 && !opted[dev]) {
    cudaFuncSetAttribute(k_radix_scatter<BITS, EP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    opted[dev] = true;
  }
  launch_chained(k_radix_scatter<BITS, EP>, blocks, kSortThreads, smem, st, src_k, src_v, dst_k, dst_v, count, count_dev, shift, table,
                 groups, group_size(blocks), ep);
}
}  // namespace

int radix_passes(int num_bits) { return num_bits <= kMaxDigitBits ? 1 : 2; }

int launch_record_sort(uint32_t *keys, uint32_t *vals, uint32_t *other_keys, uint32_t *other_vals, int64_t count,
                       const unsigned long long *count_dev, int cell_bits, void *scratch, const SortEpilogue &epilogue, cudaStream_t st) {
  const int passes = radix_passes(cell_bits);
  int bits = (cell_bits + passes - 1) / passes;    // digits of equal width: 13 bits sort as 7 + 6
  if (bits < 4) bits = 4;                          // (bits above the keys' range are zero: sorting on them changes nothing)
  const int blocks = sort_blocks(count), group = group_size(blocks);
  uint32_t *table = block_table(scratch);
  for (int p = 0; p < passes; ++p) {
    const uint32_t *src_k = p ? other_keys : keys, *src_v = p ? other_vals : vals;
    uint32_t *dst_k = p ? keys : other_keys, *dst_v = p ? vals : other_vals, *groups = group_table(scratch, 4 + p);
    const int mode = p < passes - 1 ? 0 : passes == 1 ? 4 : 2, shift = 16 + bits * p;
    SortEpilogue ep = {};
    if (mode) ep = epilogue;
    if (mode == 2) ep.chunk_first = nullptr;
    launch_chained(k_radix_hist<false>, blocks, kSortThreads, 0, st, src_k, count, count_dev, shift, bits, table, groups, group,
                   (uint32_t *)nullptr, 0, ep, CountReport{});
#define GS_SCATTER(B, EP) launch_scatter<B, EP>(blocks, src_k, src_v, dst_k, dst_v, count, count_dev, shift, table, groups, ep, st)
#define GS_SCATTER_TWO(B) if (mode == 2) GS_SCATTER(B, 2); else if (mode == 4) GS_SCATTER(B, 4); else GS_SCATTER(B, 0); break;
    switch (bits) {
      case 4: GS_SCATTER(4, 4); break;             // (one pass; two passes have digits of five to eight bits)
      case 9: GS_SCATTER(9, 4); break;
      case 5: GS_SCATTER_TWO(5)
      case 6: GS_SCATTER_TWO(6)
      case 7: GS_SCATTER_TWO(7)
      default: GS_SCATTER_TWO(8)
    }
#undef GS_SCATTER_TWO
#undef GS_SCATTER
  }
  return 2 * passes;
}

int launch_depth_sort(const uint32_t *depth_key, uint32_t *keys, uint32_t *order, uint32_t *tmp_keys, uint32_t *tmp_vals, int64_t n,
                      unsigned long long *visible, void *scratch, const SortEpilogue &epilogue, const CountReport &report, cudaStream_t st) {
  if (visible && bucket_sort_takes(n))             // (the record sort's groups are cleared by the way)
    return launch_bucket_sort(depth_key, keys, order, reinterpret_cast<unsigned long long *>(tmp_keys), n, visible, block_table(scratch),
                              group_table(scratch, 4), 2 * kMaxGroups << kMaxDigitBits, epilogue, report, st);
  const int blocks = sort_blocks(n), group = group_size(blocks);
  uint32_t *table = block_table(scratch);
  SortEpilogue ep[4] = {};
  ep[3] = epilogue;
  ep[3].id_mask = ~0u;
  if (visible) {
    ep[0].visible = visible;
    ep[0].final_vals = order;
    ep[0].counts = epilogue.counts;
    ep[0].id_mask = ep[3].id_mask = n <= (int64_t)1 << kIdBits ? (1u << kIdBits) - 1u : ~0u;
  }
  for (int p = 0; p < 4; ++p) {
    const uint32_t *src_k = p == 0 ? depth_key : p & 1 ? tmp_keys : keys, *src_v = p == 0 ? nullptr : p & 1 ? tmp_vals : order;
    uint32_t *dst_k = p & 1 ? keys : tmp_keys, *dst_v = p & 1 ? order : tmp_vals, *groups = group_table(scratch, p);
    const unsigned long long *count = p == 0 ? nullptr : visible;
    uint32_t *clear = group_table(scratch, 1);
    const int clear_words = p == 0 ? (int)(table - clear) : 0;
    launch_chained(p == 0 && visible ? k_radix_hist<true> : k_radix_hist<false>, blocks, kSortThreads, 0, st, src_k, n, count, 8 * p, 8, table,
                   p == 0 ? (uint32_t *)nullptr : groups, group, clear, clear_words, ep[p], p == 0 ? report : CountReport{});
    if (p == 0) launch_chained(k_group_sums, (blocks + group - 1) / group, 256, 0, st, table, blocks, group, groups);
#define GS_SCATTER(EP) launch_scatter<8, EP>(blocks, src_k, src_v, dst_k, dst_v, n, count, 8 * p, table, groups, ep[p], st)
    if (p == 0 && visible) GS_SCATTER(3); else if (p < 3) GS_SCATTER(0); else GS_SCATTER(1);
#undef GS_SCATTER
  }
  return 9;
}

size_t scan_scratch_bytes(int64_t n) { return (size_t)((n + kScanBlock - 1) / kScanBlock + 1) * sizeof(uint32_t); }
int num_scan_blocks(int64_t n) { return (int)((n + kScanBlock - 1) / kScanBlock); }

int launch_emit_records(const uint32_t *depth_order, const uint32_t *sorted_count, const uint32_t *cell_records,
                        const uint16_t *rect, const float *mean2d, const float *conic_opacity, const uint32_t *block_sums,
                        const unsigned long long *visible, uint32_t *rec_keys, uint32_t *rec_vals, unsigned long long *rec_total, uint32_t *overflow, int64_t n,
                        int cgx, int W, int H, int64_t capacity, cudaStream_t st) {
  if (n <= 0) return 0;
  const uint32_t cap = capacity > 0xffffffffll ? 0xffffffffu : (uint32_t)capacity;
  launch_chained(k_emit_records, num_scan_blocks(n), kScanBlock, 0, st, depth_order, sorted_count, cell_records, rect, mean2d, conic_opacity,
                 block_sums, visible, n, cgx, W, H, cap, rec_keys, rec_vals, rec_total, overflow);
  return 1;
}

int max_pieces(int64_t record_capacity, int num_cells) { return (int)((record_capacity + kBinPiece - 1) / kBinPiece) + num_cells; }

int launch_expand(const uint32_t *rec_keys, const uint32_t *rec_vals, const uint32_t *cell_ranges, const CellScratch &cs, bool chunks_known,
                  int64_t record_capacity, int64_t pair_capacity, int gx, int gy, int cgx, int cgy,
                  uint32_t *sorted_vals, uint32_t *tile_ranges, uint32_t *tile_order, cudaStream_t st) {
  const int num_cells = cgx * cgy, chunks = (int)((record_capacity + kCellChunk - 1) / kCellChunk) + num_cells;
  const uint32_t cap = pair_capacity > 0xffffffffll ? 0xffffffffu : (uint32_t)pair_capacity, *num_chunks = cs.chunk_first + num_cells;
  if (!chunks_known) {
    launch_chained(k_cell_chunks, 1, 1024, 0, st, cell_ranges, num_cells, cs.chunk_first);
    launch_chained(k_chunk_list, (num_cells + 7) / 8, 256, 0, st, cell_ranges, cs.chunk_first, num_cells, cs.chunks);
  }
  launch_chained(k_chunk_counts, std::min(chunks, kCountBlocks), kExpandThreads, 0, st, rec_keys, cs.chunks, num_chunks, cs.chunk_counts);
  launch_chained(k_cell_prefix, (num_cells + 7) / 8, 256, 0, st, cs.chunk_first, cs.chunk_counts, gx, gy, cgx, num_cells, cs.chunk_bases,
                 cs.tile_counts);
  launch_chained(k_tile_scan, 1, 1024, 0, st, cs.tile_counts, gx * gy, cap, cs.tile_starts, tile_ranges, tile_order);
  launch_chained(k_expand, std::min(chunks, kExpandBlocks), kExpandThreads, 0, st, rec_keys, rec_vals, cs.chunks, num_chunks, cs.chunk_bases,
                 cs.tile_starts, gx, gy, cgx, cap, sorted_vals);
  return chunks_known ? 4 : 6;
}

// No record is sorted (no Gaussian, none that reaches a tile, or no room for an instance): every tile is empty.
int launch_empty_binning(uint32_t *tile_ranges, uint32_t *tile_order, int num_tiles, const CountReport &report, cudaStream_t st) {
  cudaMemsetAsync(tile_ranges, 0, (size_t)num_tiles * 2 * sizeof(uint32_t), st);
  k_iota<<<(num_tiles + 255) / 256, 256, 0, st>>>(tile_order, num_tiles, report);
  return 1;
}

}  // namespace gs
