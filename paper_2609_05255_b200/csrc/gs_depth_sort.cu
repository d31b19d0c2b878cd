// Depth order of the visible Gaussians by buckets: a sample of the keys gives splitters, one pass over the keys counts and one
// moves them into buckets of up to about 2048, and a CTA per bucket sorts it in shared memory.  Four or five launches and two
// trips through memory, where the radix sort of gs_sort.cu makes four trips in nine launches.
//
// An element is one word of 64 bits: the depth key, then the Gaussian's index, then (4 bits, not part of the order) its record
// count.  No two are equal, so the order - key, ties by index - needs no stable step, and the splitters balance the buckets
// whatever the keys are: a plane of Gaussians at one depth is split by index.
//
// Sum of the kernels' times, us (the radix sort before -> this one; of it: sample, count, scatter, buckets):
//     20 011     25.8 -> 18.2     5.4   4.4   4.2   4.2        1M (878 000 visible)     76 -> 50     12.3   9.4  10.9  17.8
//    100 000     31.5 -> 22.4     6.7   5.3   4.9   5.5        1.5M (1.26 visible)      93 -> 65     14.4  11.5  16.8  22.6
//    300 007     48.5 -> 30.3     7.1   6.3   6.4  10.5        3M (1.1 visible)        114 -> 74     16.7  15.4  19.1  23.0
// Where the keys do not spread, crowded bins cost a second split or a sort by digits, us in all (the radix sort; evenly spread;
// 95 % in a tenth of a depth unit, the others from 0.3 to 300; 42 depths and a few far ones; 3, 1000, 20 000 planes):
//    100 000     37   26   36   37   38   30   27                3M         160  119  155  158  128  161  161
//    300 007     44   33   47   49   42   41   34                4.2M       201  159  219  214  168  210  211
//         1M     72   55   76   76   70   72   79
// and a bucket that the sample missed (its places depend on the indices alone, so an order in memory can hide from it) is shared
// by all CTAs: of 65 000 elements 80, of 260 000 155 (the radix sort 51, 58), of 1M 700, of 4.2M, all there can be, 5400.
// What bounds them: the sample one SM's shared memory, the passes the latency of their few loads per thread (two CTAs per SM, the
// first loads sent ahead of the prologue) and the scattered stores of 8 bytes, the buckets the chain of load, bins, scan, place,
// rank and write (two CTAs of 81 KB per SM, 1.7 waves at 1M).
#include <algorithm>
#include "gs_bin.cuh"

namespace gs {
namespace {

using namespace bin;
typedef unsigned long long u64;

constexpr int kOversample = 8;                   // samples per bucket: 3.75 times the mean, what a CTA sorts, is exceeded once in 2 10^6 buckets
constexpr int kMeanLeast = 256, kMeanMost = 2048;
constexpr int kSamplesMost = 16384;              // shared memory of k_splitters
constexpr int kBucketsMost = kSamplesMost / kOversample + 1;
constexpr int kSampleThreads = 1024, kSampleBins = 8192;
constexpr int kGuideBins = kSampleBins / 2;
constexpr int kThreads = 512, kWarps = kThreads / 32;
constexpr int kBlocksMost = 148 * 2;             // CTAs of the two passes over the keys
constexpr int kPer = 15, kBucketMost = kPer * kThreads;    // elements that a CTA sorts in shared memory, of which two CTAs leave 92 KB of L1
constexpr int kBins = 4096;
constexpr int kCrowded = 48;                     // elements of one bin
constexpr uint32_t kCountUnknown = 15u;          // a large footprint: to be looked up
constexpr uint32_t kCulled = 0xffffffffu;
static_assert(kCellSlots < (int)kCountUnknown, "counts of the stored records fit");

// Elements of an average bucket of n Gaussians: a bucket per SM, within limits.  (256 buckets of 390 for 100 000: the sample takes 3 us
// more; buckets of 1024 from 524 288 on: the sample 6 to 10 us more, the buckets 1 less.)
int bucket_mean(int64_t n) { return (int)std::min<int64_t>(kMeanMost, std::max<int64_t>(kMeanLeast, n / 148)); }
int sample_stride(int64_t n) { return bucket_mean(n) / kOversample; }
int block_elements(int64_t n) {
  const int64_t per = (n + kBlocksMost - 1) / kBlocksMost;
  return (int)((per + kThreads - 1) / kThreads * kThreads);
}

// Elements to bins in the order of their keys (both conversions are monotonic).
struct BinMap {
  uint32_t lo;
  float scale;
  __device__ __forceinline__ BinMap(uint32_t least, uint32_t largest, int bins)
      : lo(least), scale(0.999f * (float)bins / ((float)(largest - least) + 1.f)) {}
  __device__ __forceinline__ uint32_t operator()(uint32_t v) const { return (uint32_t)((float)(v - lo) * scale); }
};

// Sample and blocks of up to n Gaussians, at most: sizes that never fall as n grows, so that a workspace also serves smaller scenes.
// (Between 39 072 and 303 104 the stride is n / 1184 rounded down, 33 and more: at most 1184 + 1184 / 33 samples.)
int samples_most(int64_t n) { return (int)std::max<int64_t>(std::min<int64_t>((n + 31) / 32, 1232), (n + 255) / 256); }
int blocks_most(int64_t n) { return (int)std::min<int64_t>(kBlocksMost, (n + kThreads - 1) / kThreads); }

struct Scratch {
  u64 *splitters;                                // [buckets]
  uint32_t *head;                                // number of splitters; smallest and largest sampled key; are they the same?
  uint32_t *sampled;                             // keys of the sample
  uint16_t *guide;                               // [kGuideBins + 1]: splitters in the bins before
  uint32_t *totals, *starts;                     // [buckets + 1]: elements of a bucket, elements before it
  uint32_t *before;                              // [blocks, buckets]: elements of the bucket from blocks served earlier
  uint32_t *culled, *culled_before;              // [blocks]; [blocks, kWarps]: those of the block's warps before
  uint32_t *large;                               // number of the buckets of more than kBucketMost elements, then which
  uint32_t buckets;                              // at most
  size_t bytes;
};
Scratch carve(void *base, int64_t n) {
  n = std::min<int64_t>(n, kBucketSortMost);
  Scratch s;
  char *p = static_cast<char *>(base);
  auto take = [&](size_t bytes) { char *q = p; p += (bytes + 255) & ~(size_t)255; return q; };
  const size_t samples = samples_most(n), buckets = samples / kOversample + 1, blocks = blocks_most(n);
  s.buckets = (uint32_t)buckets;
  s.splitters = reinterpret_cast<u64 *>(take(sizeof(u64) * buckets));
  s.head = reinterpret_cast<uint32_t *>(take(16));
  s.sampled = reinterpret_cast<uint32_t *>(take(4 * samples));
  s.guide = reinterpret_cast<uint16_t *>(take(2 * (kGuideBins + 8)));
  s.totals = reinterpret_cast<uint32_t *>(take(4 * (buckets + 1)));
  s.starts = reinterpret_cast<uint32_t *>(take(4 * (buckets + 1)));
  s.before = reinterpret_cast<uint32_t *>(take(4 * blocks * buckets));
  s.culled = reinterpret_cast<uint32_t *>(take(4 * blocks));
  s.culled_before = reinterpret_cast<uint32_t *>(take(4 * blocks * kWarps));
  s.large = reinterpret_cast<uint32_t *>(take(4 * (1 + (n / kBucketMost))));
  s.bytes = (size_t)(p - static_cast<char *>(base));
  return s;
}

__device__ __forceinline__ u64 element(uint32_t key, uint32_t id) { return (u64)key << 32 | (u64)(id << 4); }

// In place, exclusive: thread t holds values [t per, (t + 1) per).  Returns the total.
template <int T, int PER>
__device__ __forceinline__ uint32_t scan_in_place(uint32_t *v, uint32_t *s_warp, int tid) {
  const int lane = tid & 31, warp = tid >> 5;
  uint32_t x[PER], sum = 0;
  static_assert(PER % 4 == 0, "vectors");
#pragma unroll
  for (int j = 0; j < PER; j += 4) {
    const uint4 q = *reinterpret_cast<const uint4 *>(v + tid * PER + j);
    x[j] = q.x; x[j + 1] = q.y; x[j + 2] = q.z; x[j + 3] = q.w;
  }
#pragma unroll
  for (int j = 0; j < PER; ++j) { const uint32_t c = x[j]; x[j] = sum; sum += c; }
  const uint32_t inc = warp_inclusive(sum, lane);
  if (lane == 31) s_warp[warp] = inc;
  __syncthreads();
  const uint32_t w = lane < T / 32 ? s_warp[lane] : 0u, winc = warp_inclusive(w, lane);
  const uint32_t off = inc - sum + __shfl_sync(kFull, winc - w, warp), all = __shfl_sync(kFull, winc, 31);
#pragma unroll
  for (int j = 0; j < PER; j += 4)
    *reinterpret_cast<uint4 *>(v + tid * PER + j) = make_uint4(off + x[j], off + x[j + 1], off + x[j + 2], off + x[j + 3]);
  __syncthreads();
  return all;
}

// For what the bins below do not spread (planes of Gaussians at one depth, a narrow range of depths with a few far ones): m <= T PER
// elements in shared memory by digits of seven bits, in stable passes whose time does not depend on the keys.  Key, less the
// smallest, and index are one number without the bits between them (id_bits of index), of which the bits [from, to) count.
// Not inlined: the kernels' own paths keep their registers.
constexpr int kDigitBits = 7, kDigits = 1 << kDigitBits;
struct DigitArea { uint32_t elements, tables, sums; };   // byte offsets; tables: [2, T / 32, kDigits] words; sums: kDigitSums words
constexpr int kDigitSums = kDigits + 32;
template <int T, int PER>
__device__ __noinline__ void sort_by_digits(DigitArea area, uint32_t m, uint32_t least, int id_bits, int from, int to) {
  extern __shared__ __align__(16) unsigned char raw[];
  constexpr int W = T / 32;
  typedef uint32_t Table[kDigits];
  u64 *a = reinterpret_cast<u64 *>(raw + area.elements);
  Table *counts = reinterpret_cast<Table *>(raw + area.tables), *all_lanes = counts + W;
  uint32_t *base = reinterpret_cast<uint32_t *>(raw + area.sums), *sums = base + kDigits;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, rows = (int)((m + T - 1) / T);
  uint32_t *count = counts[warp], *lanes = all_lanes[warp];       // see rank_row
#pragma unroll 1
  for (int shift = from; shift < to; shift += kDigitBits) {
#pragma unroll
    for (int d = 0; d < kDigits; d += 32) { count[d + lane] = 0u; lanes[d + lane] = 0u; }
    u64 x[PER];
    uint32_t at[PER];
#pragma unroll
    for (int h = 0; h < PER; ++h) {
      if (h >= rows) break;
      const uint32_t i = (warp * rows + h) * 32 + lane;
      x[h] = i < m ? a[i] : 0ull;
    }
    __syncwarp();
#pragma unroll
    for (int h = 0; h < PER; ++h) {
      if (h >= rows) break;
      const u64 v = (u64)((uint32_t)(x[h] >> 32) - least) << id_bits | (uint32_t)x[h] >> 4;
      const uint32_t d = (uint32_t)(v >> shift) & (kDigits - 1u);
      at[h] = d << 16 | rank_row(count + d, lanes + d, (warp * rows + h) * 32 + lane < m, lane);
    }
    __syncthreads();
    uint32_t total = 0;                          // of the digit tid; the warps' counts become what is in the warps before
    if (tid < kDigits) {
      uint32_t c[W];
#pragma unroll
      for (int w = 0; w < W; ++w) c[w] = counts[w][tid];
#pragma unroll
      for (int w = 0; w < W; ++w) { counts[w][tid] = total; total += c[w]; }
    }
    const uint32_t inc = warp_inclusive(total, lane);
    if (lane == 31) sums[warp] = inc;
    __syncthreads();
    const uint32_t before = __reduce_add_sync(kFull, lane < warp && lane < kDigits / 32 ? sums[lane] : 0u);
    if (tid < kDigits) base[tid] = before + inc - total;
    __syncthreads();
#pragma unroll
    for (int h = 0; h < PER; ++h) {
      if (h >= rows) break;
      const uint32_t d = at[h] >> 16;
      if ((warp * rows + h) * 32 + lane < m) a[base[d] + count[d] + (at[h] & 0xffffu)] = x[h];
    }
    __syncthreads();
  }
}
__device__ __forceinline__ int bits_of(uint32_t v) { return 32 - __clz(v); }

// Where sample j lies: one in every `stride` elements, at a place that varies.
__device__ __forceinline__ uint32_t sample_place(uint32_t j, uint32_t stride) { return j * stride + __umulhi(j * 2654435761u, stride); }

// The sampled keys by a launch of their own where they are many: what one SM can have in flight makes the fetching of 5800
// scattered words 10 us; 2000 are as fast without the launch.
constexpr int kFetchThreads = 256, kFetchFrom = 2 * kSampleThreads + 1;
__global__ void __launch_bounds__(kFetchThreads) k_fetch_samples(const uint32_t *__restrict__ keys, uint32_t n, uint32_t stride, uint32_t samples,
                                                                 uint32_t *__restrict__ sampled) {
  dependency_wait();
  const uint32_t j = blockIdx.x * kFetchThreads + threadIdx.x, i = sample_place(j, stride);
  if (j < samples) sampled[j] = i < n ? __ldg(keys + i) : kCulled;
}

// One CTA: the sample sorted; every kOversample-th is a splitter.  The sample's bins become the guide by which the next kernel
// finds an element's splitters.  It also clears what that kernel adds to.
struct SampleArea {
  uint32_t *bins, *key, *sorted_key;             // sorted: by bin
  uint16_t *sorted;                              // which sample
  uint8_t *slot;                                 // place in the bin
  // (the digit passes have 64-bit elements over both arrays of keys, their tables in the bins and their sums past the elements)
  static constexpr size_t bytes(int samples) {
    const size_t padded = (samples + 15) & ~15;
    return kSampleBins * 4 + std::max(padded * 11, padded * 8 + kDigitSums * 4);
  }
  __device__ __forceinline__ SampleArea(unsigned char *raw, uint32_t samples) {
    samples = (samples + 15) & ~15u;
    bins = reinterpret_cast<uint32_t *>(raw);
    key = bins + kSampleBins;
    sorted_key = key + samples;
    sorted = reinterpret_cast<uint16_t *>(sorted_key + samples);
    slot = reinterpret_cast<uint8_t *>(sorted + samples);
  }
};
__global__ void __launch_bounds__(kSampleThreads) k_splitters(const uint32_t *__restrict__ keys, uint32_t n, uint32_t stride, uint32_t samples,
                                                              Scratch s, int fetched, int id_bits, CountReport report) {
  dependency_wait();
  extern __shared__ __align__(16) unsigned char raw[];
  __shared__ uint32_t s_least[kSampleThreads / 32], s_largest[kSampleThreads / 32], s_warp[kSampleThreads / 32];
  const SampleArea m(raw, samples);
  const int tid = threadIdx.x, lane = tid & 31;
  auto place = [&](uint32_t j) { return sample_place(j, stride); };
  if (tid == 0) report.send();
  for (int i = tid; i < kSampleBins / 4; i += kSampleThreads) reinterpret_cast<uint4 *>(m.bins)[i] = make_uint4(0u, 0u, 0u, 0u);
  for (uint32_t i = tid; i <= s.buckets; i += kSampleThreads) s.totals[i] = 0u;
  uint32_t least = 0xffffffffu, largest = 0u;
#pragma unroll 4
  for (uint32_t j = tid; j < samples; j += kSampleThreads) {
    const uint32_t i = place(j), k = fetched ? __ldg(s.sampled + j) : i < n ? __ldg(keys + i) : kCulled;
    m.key[j] = k;
    least = min(least, k);
    if (k != kCulled) largest = max(largest, k);
  }
  least = __reduce_min_sync(kFull, least); largest = __reduce_max_sync(kFull, largest);
  if (lane == 0) { s_least[tid >> 5] = least; s_largest[tid >> 5] = largest; }
  __syncthreads();
  least = __reduce_min_sync(kFull, s_least[lane]); largest = __reduce_max_sync(kFull, s_largest[lane]);
  const bool by_place = least == largest;        // all keys are the same
  const BinMap bin(by_place ? 0u : least, by_place ? samples - 1 : largest, kSampleBins);
  uint32_t most = 0;
#pragma unroll 4
  for (uint32_t j = tid; j < samples; j += kSampleThreads) {
    const uint32_t k = m.key[j];
    if (k == kCulled) continue;
    const uint32_t slot = atomicAdd(&m.bins[bin(by_place ? j : k)], 1u);
    m.slot[j] = (uint8_t)min(slot, 255u);
    most = max(most, slot);
  }
  const bool crowded = __syncthreads_or(most >= kCrowded);
  const uint32_t count = scan_in_place<kSampleThreads, kSampleBins / kSampleThreads>(m.bins, s_warp, tid);
  for (int i = tid; i <= kGuideBins; i += kSampleThreads)
    s.guide[i] = (uint16_t)((i < kGuideBins ? m.bins[2 * i] : count) / kOversample);
  if (crowded) {
    uint32_t key[kSamplesMost / kSampleThreads];
#pragma unroll
    for (int h = 0; h < kSamplesMost / kSampleThreads; ++h) key[h] = h * kSampleThreads + tid < (int)samples ? m.key[h * kSampleThreads + tid] : 0u;
    u64 *a = reinterpret_cast<u64 *>(m.key);
    __syncthreads();
#pragma unroll
    for (int h = 0; h < kSamplesMost / kSampleThreads; ++h) {           // (culled ones last; the places rise as they stand)
      const uint32_t j = h * kSampleThreads + tid;
      if (j < samples) a[j] = element(min(key[h], largest + 1), place(j));
    }
    __syncthreads();
    static_assert(kSampleBins >= 2 * kSampleThreads / 32 * kDigits, "the tables fit the bins");
    const uint32_t elements = kSampleBins * 4;
    sort_by_digits<kSampleThreads, kSamplesMost / kSampleThreads>({elements, 0u, elements + ((samples + 15) & ~15u) * 8}, samples, least, id_bits,
                                                                  id_bits, id_bits + bits_of(largest + 1 - least));
    for (uint32_t j = tid; j < count / kOversample; j += kSampleThreads) s.splitters[j] = a[(j + 1) * kOversample - 1];
  } else {
#pragma unroll 4
    for (uint32_t j = tid; j < samples; j += kSampleThreads) {
      const uint32_t k = m.key[j];
      if (k == kCulled) continue;
      const uint32_t at = m.bins[bin(by_place ? j : k)] + m.slot[j];
      m.sorted_key[at] = k;
      m.sorted[at] = (uint16_t)j;
    }
    __syncthreads();
    // rank among the few of the bin, in the order of the bins: neighbours read neighbouring words
    for (uint32_t at = tid; at < count; at += kSampleThreads) {
      const uint32_t k = m.sorted_key[at], j = m.sorted[at], b = bin(by_place ? j : k);
      const uint32_t begin = m.bins[b], end = b + 1 < kSampleBins ? m.bins[b + 1] : count;
      uint32_t rank = begin;
      for (uint32_t q = begin; q < end; ++q) {
        const uint32_t other = m.sorted_key[q];
        rank += other < k || (other == k && m.sorted[q] < j);
      }
      if (rank % kOversample == kOversample - 1) s.splitters[rank / kOversample] = element(k, place(j));
    }
  }
  if (tid == 0) *reinterpret_cast<uint4 *>(s.head) = make_uint4(count / kOversample, least, largest, by_place ? 1u : 0u);
}

// Bucket of every element, and its number among those of its CTA there; per CTA and bucket how many elements earlier CTAs (in
// the order of the atomics: any will do) put there; the culled ones of every warp.
__global__ void __launch_bounds__(kThreads, 2) k_bucket_count(const uint32_t *__restrict__ keys, uint32_t n, int per, Scratch s,
                                                              uint32_t *__restrict__ codes, uint32_t *__restrict__ block_sums, int num_block_sums,
                                                              uint32_t *__restrict__ clear, int clear_words) {
  dependency_wait();
  __shared__ u64 s_split[kBucketsMost];
  __shared__ uint32_t s_hist[kBucketsMost + 1], s_warp[kWarps];
  __shared__ __align__(16) uint16_t s_guide[kGuideBins + 8];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = blockIdx.x * kThreads + tid; i < num_block_sums; i += gridDim.x * kThreads) block_sums[i] = 0u;
  for (int i = blockIdx.x * kThreads + tid; i < clear_words; i += gridDim.x * kThreads) clear[i] = 0u;
  constexpr int kRows = 4;
  const uint32_t span = (uint32_t)per / kWarps;    // a multiple of 32
  const uint32_t begin = blockIdx.x * (uint32_t)per + warp * span, end = min(n, begin + span);
  uint32_t next[kRows];
  auto load = [&](uint32_t i0) {
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const uint32_t i = i0 + 32 * r + lane;
      next[r] = i < end ? __ldg(keys + i) : kCulled;
    }
  };
  load(begin);
  const uint4 head = __ldg(reinterpret_cast<const uint4 *>(s.head));
  const int num = (int)head.x;
  for (int i = tid; i < num; i += kThreads) s_split[i] = __ldg(s.splitters + i);
  for (int i = tid; i <= num; i += kThreads) s_hist[i] = 0u;
  for (int i = tid; i < kGuideBins / 8 + 1; i += kThreads) reinterpret_cast<uint4 *>(s_guide)[i] = __ldg(reinterpret_cast<const uint4 *>(s.guide) + i);
  __syncthreads();
  const BinMap bin(head.y, head.z, kSampleBins);
  uint32_t culled = 0;
  for (uint32_t i0 = begin; i0 < end; i0 += 32 * kRows) {
    uint32_t key[kRows], at[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r) key[r] = next[r];
    load(i0 + 32 * kRows);
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      // the splitters of the element's bin, then a search among them (rarely more than one)
      const u64 x = element(key[r], i0 + 32 * r + lane);
      const uint32_t b = bin(min(max(key[r], head.y), head.z)) >> 1;
      uint32_t lo = head.w ? 0u : s_guide[b], hi = head.w ? head.x : s_guide[b + 1];
      while (lo < hi) {
        const uint32_t mid = (lo + hi) / 2;
        if (s_split[mid] <= x) lo = mid + 1; else hi = mid;
      }
      at[r] = lo;
    }
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const uint32_t i = i0 + 32 * r + lane;
      const bool ok = key[r] != kCulled;
      const uint32_t live = __ballot_sync(kFull, ok);
      culled += __popc(__ballot_sync(kFull, !ok && i < end));
      if (!ok) {
        if (i < end) codes[i] = kCulled;
        continue;
      }
      // neighbours in memory that lie in one bucket are counted together
      const int leader = __ffs(live) - 1;
      const uint32_t first = __shfl_sync(live, at[r], leader);
      uint32_t slot;
      if (__all_sync(live, at[r] == first)) {
        uint32_t base = 0;
        if (lane == leader) base = atomicAdd(&s_hist[first], (uint32_t)__popc(live));
        slot = __shfl_sync(live, base, leader) + __popc(live & ((1u << lane) - 1u));
      } else {
        slot = atomicAdd(&s_hist[at[r]], 1u);
      }
      codes[i] = at[r] << 16 | slot;
    }
  }
  if (lane == 0) s_warp[warp] = culled;
  __syncthreads();
  if (warp == 0) {
    const uint32_t c = lane < kWarps ? s_warp[lane] : 0u, inc = warp_inclusive(c, lane);
    if (lane < kWarps) s.culled_before[blockIdx.x * kWarps + lane] = inc - c;
    if (lane == 31) s.culled[blockIdx.x] = inc;
  }
  uint32_t *row = s.before + (size_t)blockIdx.x * s.buckets;
  for (int i = tid; i <= num; i += kThreads) {
    const uint32_t c = s_hist[i];
    if (c) row[i] = atomicAdd(s.totals + i, c);
  }
}

// Elements to their buckets; culled Gaussians to the end of the order, by index.
__global__ void __launch_bounds__(kThreads, 2) k_bucket_scatter(const uint32_t *__restrict__ keys, const uint32_t *__restrict__ codes,
                                                                const uint32_t *__restrict__ counts, uint32_t n, int per, Scratch s,
                                                                u64 *__restrict__ out, uint32_t *__restrict__ order, u64 *__restrict__ visible) {
  dependency_wait();
  constexpr int kScan = (kBucketsMost + kThreads * 4 - 1) / (kThreads * 4) * 4;
  __shared__ __align__(16) uint32_t s_base[kScan * kThreads];
  __shared__ uint32_t s_warp[kWarps], s_culled, s_large;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kRows = 4;
  const uint32_t span = (uint32_t)per / kWarps;
  const uint32_t begin = blockIdx.x * (uint32_t)per + warp * span, end = min(n, begin + span);
  uint32_t key[kRows], code[kRows], cnt[kRows];
  auto load = [&](uint32_t i0) {
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const uint32_t i = i0 + 32 * r + lane;
      key[r] = i < end ? __ldg(keys + i) : 0u;
      code[r] = i < end ? __ldg(codes + i) : 0u;
      cnt[r] = i < end ? __ldg(counts + i) : 0u;
    }
  };
  load(begin);
  const int num = (int)__ldg(s.head);
  if (tid == 0) s_culled = s_large = 0u;
  for (int i = tid; i < kScan * kThreads; i += kThreads) s_base[i] = i <= num ? __ldg(s.totals + i) : 0u;
  __syncthreads();
  uint32_t culled = 0;
  for (int i = tid; i < (int)blockIdx.x; i += kThreads) culled += __ldg(s.culled + i);
  culled = __reduce_add_sync(kFull, culled);
  if (lane == 0 && culled) atomicAdd(&s_culled, culled);
  const uint32_t all = scan_in_place<kThreads, kScan>(s_base, s_warp, tid);
  if (blockIdx.x == 0) {
    for (int i = tid; i <= num + 1; i += kThreads) {
      s.starts[i] = s_base[i];
      if (i <= num && s_base[i + 1] - s_base[i] > kBucketMost) s.large[1 + atomicAdd(&s_large, 1u)] = (uint32_t)i;
    }
    __syncthreads();
    if (tid == 0) { *visible = all; s.large[0] = s_large; }
  }
  const uint32_t *row = s.before + (size_t)blockIdx.x * s.buckets;
  for (int i = tid; i <= num; i += kThreads) s_base[i] += __ldg(row + i);     // (of a bucket without elements here: not read)
  __syncthreads();
  uint32_t last = all + s_culled + __ldg(s.culled_before + blockIdx.x * kWarps + warp);
  for (uint32_t i0 = begin; i0 < end; i0 += 32 * kRows) {
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const uint32_t i = i0 + 32 * r + lane;
      const bool gone = i < end && code[r] == kCulled;
      const uint32_t away = __ballot_sync(kFull, gone);
      if (gone) order[last + __popc(away & ((1u << lane) - 1u))] = i;
      else if (i < end) out[s_base[code[r] >> 16] + (code[r] & 0xffffu)] = element(key[r], i) | min(cnt[r], kCountUnknown);
      last += __popc(away);
    }
    load(i0 + 32 * kRows);
  }
}

// One CTA per bucket: its elements into bins by their keys (by their indices where the keys are all the same), two
// bins or more per element, and each to its place among the few of its bin.  Leaves the Gaussians' ids and record counts in order, and
// the counts' sums per 256 positions.
constexpr int kSegmentsMost = kBucketMost / kCrowded + 1;
struct __align__(16) BucketArea {
  u64 a[kBucketMost];
  uint32_t bins[kBins], sums[kDigitSums], warp[kWarps], range[4];
  uint32_t segment[4][kSegmentsMost];            // complements of the smallest key and index, largest key and index
};
static_assert(2 * (sizeof(BucketArea) + 1024) <= 164 * 1024, "two CTAs in the carve-out of 164 KB");
static_assert(kBins >= 2 * kWarps * kDigits, "the tables fit the bins");
constexpr DigitArea kBucketDigits = {0u, kBucketMost * 8, kBucketMost * 8 + kBins * 4};

// Where bins hold many elements (few different depths, or a few far from the others): m.a[0, count) stands in the order of the
// bins, which begin at m.bins.  A crowded bin is split once more between its own smallest and largest key, or index where the
// keys are the same, two elements to a part; what is crowded even then goes by digits.
// 1M Gaussians in 1000 planes, every bucket crowded: the kernel 35 us, by digits alone 62, evenly spread 22.
__device__ __noinline__ void sort_crowded(uint32_t count, u64 first, u64 last, int id_bits) {
  extern __shared__ __align__(16) unsigned char raw[];
  BucketArea &m = *reinterpret_cast<BucketArea *>(raw);
  constexpr int T = kThreads;
  const int tid = threadIdx.x, lane = tid & 31, shift = first >> 32 == last >> 32 ? 0 : 32;
  const BinMap bin((uint32_t)(first >> shift), (uint32_t)(last >> shift), kBins);
  for (int i = tid; i < 4 * kSegmentsMost; i += T) m.segment[0][i] = 0u;
  __syncthreads();
  u64 x[kPer];
  uint32_t at[kPer];                             // begin of the bin, elements in it; then part, place in the part
#pragma unroll
  for (int h = 0; h < kPer; ++h) {
    if (h * T >= (int)count) break;
    const bool ok = h * T + tid < (int)count;
    x[h] = ok ? m.a[h * T + tid] : 0ull;
    at[h] = 0u;
    if (ok) {
      const uint32_t b = bin((uint32_t)(x[h] >> shift)), begin = m.bins[b], end = b + 1 < kBins ? m.bins[b + 1] : count;
      at[h] = begin << 16 | (end - begin);
    }
    const bool split = (at[h] & 0xffffu) > (uint32_t)kCrowded;
    const uint32_t key = (uint32_t)(x[h] >> 32), id = (uint32_t)x[h], slot = (at[h] >> 16) / kCrowded;
    const uint32_t v[4] = {~key, ~id, key, id};
    const uint32_t voters = __ballot_sync(kFull, split);
    if (voters == 0u) continue;
    const uint32_t one = __shfl_sync(kFull, slot, __ffs(voters) - 1);
    if (__all_sync(kFull, !split || slot == one)) {               // (most warps lie inside one bin)
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t most = __reduce_max_sync(kFull, split ? v[k] : 0u);
        if (lane == 0) atomicMax(&m.segment[k][one], most);
      }
    } else if (split) {
#pragma unroll
      for (int k = 0; k < 4; ++k) atomicMax(&m.segment[k][slot], v[k]);
    }
  }
  __syncthreads();
  for (int i = tid; i < kBins / 4; i += T) reinterpret_cast<uint4 *>(m.bins)[i] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  uint32_t most = 0;
#pragma unroll
  for (int h = 0; h < kPer; ++h) {
    if (h * T >= (int)count) break;
    if (h * T + tid < (int)count) {
      const uint32_t begin = at[h] >> 16, size = at[h] & 0xffffu;
      uint32_t part = begin;
      if (size > (uint32_t)kCrowded) {
        const uint32_t seg = begin / kCrowded, k0 = ~m.segment[0][seg], k1 = m.segment[2][seg];
        const bool same = k0 == k1;
        const BinMap inner(same ? ~m.segment[1][seg] : k0, same ? m.segment[3][seg] : k1, (int)size);
        part += inner(same ? (uint32_t)x[h] : (uint32_t)(x[h] >> 32));
      }
      part /= 2;
      const uint32_t slot = atomicAdd(&m.bins[part], 1u);
      most = max(most, slot);
      at[h] = part << 16 | slot;
    }
  }
  if (__syncthreads_or(most >= 2 * kCrowded)) {
    const uint32_t least = (uint32_t)(first >> 32);
    sort_by_digits<T, kPer>(kBucketDigits, count, least, id_bits, 0, bits_of((uint32_t)(last >> 32) - least) + id_bits);
    return;
  }
  scan_in_place<T, kBins / T>(m.bins, m.warp, tid);
#pragma unroll
  for (int h = 0; h < kPer; ++h) {
    if (h * T >= (int)count) break;
    if (h * T + tid < (int)count) m.a[m.bins[at[h] >> 16] + (at[h] & 0xffffu)] = x[h];
  }
  __syncthreads();
#pragma unroll
  for (int h = 0; h < kPer; ++h) {
    if (h * T >= (int)count) break;
    if (h * T + tid < (int)count) {
      const uint32_t part = at[h] >> 16, end = part + 1 < kBins ? m.bins[part + 1] : count;
      uint32_t rank = m.bins[part];
      for (uint32_t q = rank; q < end; ++q) rank += m.a[q] < x[h];
      at[h] = rank;
    }
  }
  __syncthreads();
#pragma unroll
  for (int h = 0; h < kPer; ++h) {
    if (h * T >= (int)count) break;
    if (h * T + tid < (int)count) m.a[at[h]] = x[h];
  }
  __syncthreads();
}

// Ids, record counts and the counts' sums of the elements m.a[0, count), which come at `start` in the order.
__device__ __forceinline__ void leave(const BucketArea &m, uint32_t start, uint32_t count, const uint32_t *counts, uint32_t *counts_out,
                                      uint32_t *order, uint32_t *block_sums, int tid) {
  for (uint32_t j0 = 0; j0 < count; j0 += kThreads) {
    const uint32_t j = j0 + tid, pos = start + j;
    uint32_t c = 0;
    if (j < count) {
      const uint32_t v = (uint32_t)m.a[j], id = v >> 4;
      c = v & 15u;
      if (c == kCountUnknown) c = __ldg(counts + id);
      counts_out[pos] = c;
      order[pos] = id;
      c &= ~kCellBig;
    }
    // a warp's 32 positions lie in two blocks of 256 at most
    const uint32_t first = __shfl_sync(kFull, pos, 0) / 256u;
    const uint32_t sum0 = __reduce_add_sync(kFull, pos / 256u == first ? c : 0u), sum1 = __reduce_add_sync(kFull, pos / 256u == first ? 0u : c);
    if ((tid & 31) == 0 && sum0) atomicAdd(block_sums + first, sum0);
    if ((tid & 31) == 0 && sum1) atomicAdd(block_sums + first + 1, sum1);
  }
}

// Buckets beyond shared memory (the sample missed what the bucket holds): all CTAs take parts of them.  A part lies between two
// samples of the bucket; a CTA reads the whole bucket, keeps what is in its part and counts what comes before.  What is more
// than it can keep it takes in several turns, each up to the middle of those that it kept.
constexpr uint32_t kPartMean = 2048, kPartsMost = 512, kPartOversample = kBucketMost / kPartsMost;
__device__ __noinline__ void sort_large_buckets(const u64 *in, const Scratch &s, uint32_t large, const uint32_t *counts, uint32_t *counts_out,
                                                uint32_t *order, uint32_t *block_sums, int id_bits) {
  extern __shared__ __align__(16) unsigned char raw[];
  BucketArea &m = *reinterpret_cast<BucketArea *>(raw);
  const int tid = threadIdx.x, lane = tid & 31;
  uint32_t part = blockIdx.x;
  for (uint32_t e = 0; e < large; ++e) {
    const uint32_t bucket = s.large[1 + e], start = s.starts[bucket], total = s.starts[bucket + 1] - start;
    const uint32_t parts = min((total + kPartMean - 1) / kPartMean, kPartsMost), samples = parts * kPartOversample;
    for (; part < parts; part += gridDim.x) {
      __syncthreads();
      for (uint32_t j = tid; j < samples; j += kThreads) m.a[j] = in[start + (uint32_t)((u64)j * total / samples)];
      __syncthreads();
      sort_by_digits<kThreads, kPer>(kBucketDigits, samples, 0u, id_bits, 0, 32 + id_bits);
      u64 lo = part == 0 ? 0ull : m.a[part * kPartOversample];
      const u64 end = part + 1 == parts ? ~0ull : m.a[(part + 1) * kPartOversample];
      u64 hi = end;
      while (lo < end) {
        __syncthreads();
        if (tid < 2) m.range[tid] = 0u;
        __syncthreads();
        uint32_t before = 0;
        constexpr int kLoads = 8;
        for (uint32_t i0 = tid; i0 < total; i0 += kLoads * kThreads) {
          u64 x[kLoads];
#pragma unroll
          for (int h = 0; h < kLoads; ++h) x[h] = i0 + h * kThreads < total ? in[start + i0 + h * kThreads] : ~0ull;
#pragma unroll
          for (int h = 0; h < kLoads; ++h) {
            before += x[h] < lo;
            if (x[h] >= lo && x[h] < hi) {
              const uint32_t at = atomicAdd(&m.range[0], 1u);
              if (at < (uint32_t)kBucketMost) m.a[at] = x[h];
            }
          }
        }
        before = __reduce_add_sync(kFull, before);
        if (lane == 0) atomicAdd(&m.range[1], before);
        __syncthreads();
        const uint32_t found = m.range[0], have = min(found, (uint32_t)kBucketMost);
        sort_by_digits<kThreads, kPer>(kBucketDigits, have, 0u, id_bits, 0, 32 + id_bits);
        if (found > have) {
          hi = m.a[kBucketMost / 2];
        } else {
          leave(m, start + m.range[1], have, counts, counts_out, order, block_sums, tid);
          lo = hi;
          hi = end;
        }
      }
    }
    part -= parts;
  }
}

__global__ void __launch_bounds__(kThreads, 2) k_bucket_sort(const u64 *__restrict__ in, Scratch s, const uint32_t *__restrict__ counts,
                                                             uint32_t *__restrict__ counts_out, uint32_t *__restrict__ order,
                                                             uint32_t *__restrict__ block_sums, int id_bits) {
  dependency_wait();
  extern __shared__ __align__(16) unsigned char raw[];
  BucketArea &m = *reinterpret_cast<BucketArea *>(raw);
  constexpr int T = kThreads;
  const int tid = threadIdx.x, lane = tid & 31;
  const uint4 head = __ldg(reinterpret_cast<const uint4 *>(s.head));
  const uint32_t start = __ldg(s.starts + blockIdx.x), count = __ldg(s.starts + blockIdx.x + 1) - start, large = __ldg(s.large);
  u64 first = __ldg(s.splitters + max((int)blockIdx.x, 1) - 1), last = __ldg(s.splitters + blockIdx.x);
  if (blockIdx.x <= head.x && count - 1u < (uint32_t)kBucketMost) {
    u64 x[kPer];
    uint32_t at[kPer];
#pragma unroll
    for (int h = 0; h < kPer; ++h) {
      if (h * T >= (int)count) break;
      x[h] = h * T + tid < (int)count ? in[start + h * T + tid] : ~0ull;
    }
    for (int i = tid; i < kBins / 4; i += T) reinterpret_cast<uint4 *>(m.bins)[i] = make_uint4(0u, 0u, 0u, 0u);
    // the bucket lies between two splitters, the first and the last one where their elements do
    if (blockIdx.x == 0 || blockIdx.x == head.x) {
      uint32_t range[4] = {0u, 0u, 0u, 0u};          // complements of the smallest key and index, largest key and index
#pragma unroll
      for (int h = 0; h < kPer; ++h) {
        if (h * T >= (int)count) break;
        const uint32_t k = (uint32_t)(x[h] >> 32), i = (uint32_t)x[h];
        if (h * T + tid < (int)count) {
          range[0] = max(range[0], ~k); range[1] = max(range[1], ~i); range[2] = max(range[2], k); range[3] = max(range[3], i);
        }
      }
      if (tid < 4) m.range[tid] = 0u;
      __syncthreads();
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        range[k] = __reduce_max_sync(kFull, range[k]);
        if (lane == 0) atomicMax(&m.range[k], range[k]);
      }
      __syncthreads();
      first = (u64)~m.range[0] << 32 | ~m.range[1];
      last = (u64)m.range[2] << 32 | m.range[3];
    }
    const bool by_id = first >> 32 == last >> 32;
    const int shift = by_id ? 0 : 32;
    const uint32_t lo = (uint32_t)(first >> shift), hi = (uint32_t)(last >> shift);
    const BinMap bin(lo, hi, kBins);
    __syncthreads();
    uint32_t most = 0;
#pragma unroll
    for (int h = 0; h < kPer; ++h) {
      if (h * T >= (int)count) break;
      at[h] = 0u;
      if (h * T + tid < (int)count) {
        const uint32_t b = bin((uint32_t)(x[h] >> shift)), slot = atomicAdd(&m.bins[b], 1u);
        most = max(most, slot);
        at[h] = b << 16 | slot;
      }
    }
    const bool crowded = __syncthreads_or(most >= kCrowded);
    scan_in_place<T, kBins / T>(m.bins, m.warp, tid);
#pragma unroll
    for (int h = 0; h < kPer; ++h) {
      if (h * T >= (int)count) break;
      if (h * T + tid < (int)count) m.a[m.bins[at[h] >> 16] + (at[h] & 0xffffu)] = x[h];
    }
    __syncthreads();
    if (crowded) {
      sort_crowded(count, first, last, id_bits);
    } else {
#pragma unroll
      for (int h = 0; h < kPer; ++h) {
        if (h * T >= (int)count) break;
        if (h * T + tid < (int)count) {
          x[h] = m.a[h * T + tid];               // in the order of the bins, so that neighbours read neighbouring words
          const uint32_t b = bin((uint32_t)(x[h] >> shift)), begin = m.bins[b], end = b + 1 < kBins ? m.bins[b + 1] : count;
          uint32_t rank = begin;
          if (end - begin > 1)
            for (uint32_t q = begin; q < end; ++q) rank += m.a[q] < x[h];
          at[h] = rank;
        }
      }
      __syncthreads();
#pragma unroll
      for (int h = 0; h < kPer; ++h) {
        if (h * T >= (int)count) break;
        if (h * T + tid < (int)count) m.a[at[h]] = x[h];
      }
      __syncthreads();
    }
    leave(m, start, count, counts, counts_out, order, block_sums, tid);
  }
  if (large > 0) sort_large_buckets(in, s, large, counts, counts_out, order, block_sums, id_bits);
}

template <auto Kernel>
void allow_smem(size_t bytes) {
  static bool opted[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && opted[dev]) return;
  cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (dev >= 0 && dev < 64) opted[dev] = true;
}
}  // namespace

bool bucket_sort_takes(int64_t n) { return n <= kBucketSortMost; }

size_t bucket_scratch_bytes(int64_t n) { return carve(nullptr, n).bytes; }

int launch_bucket_sort(const uint32_t *depth_key, uint32_t *counts_out, uint32_t *order, unsigned long long *pairs, int64_t n,
                       unsigned long long *visible, void *scratch, uint32_t *clear, int clear_words, const SortEpilogue &ep,
                       const CountReport &report, cudaStream_t st) {
  static_assert((int64_t)kBucketSortMost * kOversample <= (int64_t)kSamplesMost * kMeanMost, "samples fit");
  const int per = block_elements(n), blocks = (int)((n + per - 1) / per), stride = sample_stride(n);
  const int samples = (int)((n + stride - 1) / stride);
  const Scratch s = carve(scratch, n);
  allow_smem<k_splitters>(SampleArea::bytes(kSamplesMost));
  const bool fetch = samples >= kFetchFrom;
  int id_bits = 1;
  while ((n - 1) >> id_bits) ++id_bits;
  if (fetch)
    launch_chained(k_fetch_samples, (samples + kFetchThreads - 1) / kFetchThreads, kFetchThreads, 0, st, depth_key, (uint32_t)n, (uint32_t)stride,
                   (uint32_t)samples, s.sampled);
  launch_chained(k_splitters, 1, kSampleThreads, SampleArea::bytes(samples), st, depth_key, (uint32_t)n, (uint32_t)stride, (uint32_t)samples, s,
                 (int)fetch, id_bits, report);
  launch_chained(k_bucket_count, blocks, kThreads, 0, st, depth_key, (uint32_t)n, per, s, counts_out, ep.block_sums, ep.num_block_sums, clear,
                 clear_words);
  launch_chained(k_bucket_scatter, blocks, kThreads, 0, st, depth_key, counts_out, ep.counts, (uint32_t)n, per, s, pairs, order, visible);
  allow_smem<k_bucket_sort>(sizeof(BucketArea));
  launch_chained(k_bucket_sort, samples / kOversample + 1, kThreads, sizeof(BucketArea), st, pairs, s, ep.counts, counts_out, order, ep.block_sums,
                 id_bits);
  return fetch ? 5 : 4;
}

}  // namespace gs
