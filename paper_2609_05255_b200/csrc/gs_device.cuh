// Internal declarations shared by the translation units of libgs_b200 (not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include "gs.h"

namespace gs {

constexpr float kAlphaMin = 1.0f / 255.0f;
constexpr float kAlphaMax = 0.99f;
constexpr float kTmin = 1e-4f;
constexpr float kDilation = 0.3f;
constexpr float kExtentPad = 1.00001f;  // keeps fp32 rounding from dropping an edge pixel
constexpr float kLog2e = 1.4426950408889634f;
constexpr int kMlpW1 = 0, kMlpW2 = 512, kMlpW3 = 768;

// Camera as the kernels see it (passed by value).
// Cells: 4 x 4 tiles.  The binning sorts one record per (Gaussian, cell) instead of one per (Gaussian, tile).
constexpr int kCellSlots = 9;                 // records kept per Gaussian by the preprocess (3 x 3 cells)
constexpr uint32_t kCellBig = 0x80000000u;    // flag in cell_count: records not stored, derive them again
constexpr int kCellChunk = 2048;              // records of one cell that one CTA expands

struct CamDev {
  int W, H, gx, gy;
  int cgx, cgy;         // cells per row / column: ceil(gx / 4), ceil(gy / 4)
  float fx, fy, cx, cy;
  float R[9], t[3];
  float oc[3];          // camera centre in world space
  float near_plane, far_plane;
  float limx, limy;     // 1.3 x half field of view, as tan
  float bg[3];
};

// ---- launches (all enqueue on `st`; none synchronises; each returns the number of kernels it
// launched) ---------------------------------------------------------------------------------
// Appearance "model" of the preprocess kernels in the separate-pass (unfused) step: no colour is decoded; the
// forward leaves the view directions of the visible Gaussians where the colours go, the backward takes dL/dd
// from a buffer.  The appearance kernels run as launches of their own around them.
constexpr int kAppExternal = 3;
// The neural model with the decoder's products taken on plain fp16 operands (the paper's precision) instead of
// split ones: GsScene.decoder_precision = GS_DECODER_HALF.  Same kernels, same weights, same layout.
constexpr int kAppNeuralHalf = 4;

// Instances of a view: below 2^31 Gaussians with at most 2^20 tiles each (65536 cells of 16).  The 13 bits left in a word
// of 64 count the warps of the preprocess (888 CTAs of four on a B200).
constexpr int kSumBits = 51;
struct PreprocessArgs {
  int64_t n;
  const float *means, *log_scales, *quats, *logits, *base_color, *sh_rest;
  const __half *features, *weights;
  int deg, act;
  float *mean2d, *conic_opacity, *color, *extent;
  uint32_t *depth_key, *tiles_touched, *cell_count, *cell_records;
  uint16_t *rect;
  unsigned long long *pair_counter;   // [0] receives the instance count; [1] zero before and after: the sum so far (kSumBits)
                                      // and, above it, the warps that have added to it
  unsigned long long *timeout; // set to 1 if a bounded wait on a bulk copy ran out (never expected)
};
int launch_preprocess_fwd(int app, const PreprocessArgs &a, const CamDev &cam, cudaStream_t st);

// Who received a gradient in a view: a bit per Gaussian, set by the warps of the blend backward.  With few Gaussians in a large
// image all warps are at the same few words, which the L2 serves one after another: the blend backward of 5000 Gaussians at
// 1280 x 720 took 242 us (8 x 8 pixels per warp), 118 without the bits.  So the bits of less than 65 536 Gaussians exist up to 16 times, if there is a tile for every 20 of them; a warp sets
// those of one copy, and a reader takes the copies together: 120 us; 1000 Gaussians at 640 x 480 45 -> 24, 5000 at 3840 x 2160
// 1000 -> 668, 20 011 at 640 x 480 79 -> 67.  (A byte per Gaussian, stored, is no better than the atomics on bits; looking at
// what an addition to the Gaussian's row finds there waits for the answer, 10 to 30 % more below 1000 tiles.)
struct GradFlags {
  uint32_t *words;              // [copies, stride]
  uint32_t stride;
  int copies;                   // 1, 4 or 16
  void layout(int64_t n) {
    copies = n < 16384 ? 16 : n < 65536 ? 4 : 1;
    stride = (uint32_t)((n + 31) / 32 + 31) & ~31u;      // whole lines of 128 bytes
  }
  // Words for the copies of up to n Gaussians: never less than a smaller scene's.
  static size_t room(int64_t n) {
    const size_t stride = (size_t)((n + 31) / 32 + 31) & ~(size_t)31, copied = 16 * stride;
    return copied < 8192 ? copied : stride < 8192 ? 8192 : stride;
  }
#ifdef __CUDACC__
  template <bool kCopies>
  __device__ __forceinline__ void set(uint32_t warp, uint32_t id) const {
    atomicOr(words + (kCopies ? (warp & (uint32_t)(copies - 1)) * stride : 0u) + (id >> 5), 1u << (id & 31u));
  }
  __device__ __forceinline__ uint32_t word(int64_t w) const {
    uint32_t v = __ldg(words + w);
    for (int c = 1; c < copies; c += 3) {              // (more at a time is more code, which costs where there are no copies)
      const uint32_t *p = words + c * stride + w;
      v |= __ldg(p) | __ldg(p + stride) | __ldg(p + 2 * stride);
    }
    return v;
  }
#endif
};
struct PreprocessBwdArgs {
  int64_t n;
  const float *means, *log_scales, *quats, *logits, *base_color, *sh_rest;
  const __half *features, *weights;
  int deg, act;
  const float *g2d;            // [n,12]: dL/dcolor(3), dL/dopacity, dL/dconic(3), dL/dmean2d(2), pad
  const float *gd_in;          // kAppExternal only: [n,3] dL/dd from the separate appearance backward
  GradFlags flags;             // who received a gradient in this view (only their rows are written)
  float *g_means, *g_log_scales, *g_quats, *g_logits, *g_base, *g_sh_rest, *g_features;
  float *w_partials;           // [kWgradBlocks, 816]
  float *g_weights;            // [816]
  unsigned long long *timeout; // set to 1 if a bounded wait on a bulk copy ran out (never expected)
};
int launch_preprocess_bwd(int app, const PreprocessBwdArgs &a, const CamDev &cam, cudaStream_t st);

struct AppearanceArgs {
  int64_t n;
  int deg, act;
  const float *base_color, *sh_rest, *dirs;
  const __half *features, *weights;
  float *color;                // forward
  const float *g_color;        // backward
  float *g_base, *g_sh_rest, *g_features, *g_dirs;
  float *w_partials, *g_weights;
  unsigned long long *timeout; // optional: set to 1 if a bounded wait on a bulk copy ran out (never expected)
  int engine;                  // GsDecoderEngine for the default neural decoder: warp-level MMA, tcgen05, or per kernel the faster
  const uint32_t *mask;        // optional [n]: Gaussians with a zero here are skipped (no colour written; zero
                               // gradient rows written); the tiles-touched array in the unfused step
  GradFlags flags;             // optional, backward of the decoder variants on tcgen05: only the
                               // flagged ones are worked on (gathered into full tiles) and written
  const float *means, *g2d;    // optional, with flags (the unfused step): view directions from the means and the camera
  float oc[3];                 // centre oc, dL/dcolor from columns 0..2 of the [n,12] rows g2d, instead of dirs / g_color
};
int launch_appearance_fwd(int app, const AppearanceArgs &a, cudaStream_t st);
int launch_appearance_bwd(int app, const AppearanceArgs &a, cudaStream_t st);

// Decoder variants (1-3 hidden layers of 16 or 32 neurons, 8 encoded or 16 raw features): tcgen05 kernels unless
// a.engine is GS_ENGINE_WARP_MMA or the active degree is 0, fp32 FMA kernels then.
int variant_num_weights(int hidden, int layers);
size_t variant_partials_floats();   // floats of per-block weight-gradient partials the backward needs
int launch_variant_fwd(int hidden, int layers, int nfeat, const AppearanceArgs &a, cudaStream_t st);
int launch_variant_bwd(int hidden, int layers, int nfeat, const AppearanceArgs &a, cudaStream_t st);

// Unfused step, backward: view directions of the masked-in Gaussians and their dL/dcolor (columns 0..2 of the
// [n,12] rows) as dense [n,3] arrays for the separate appearance backward.
int launch_unfused_prepare(int64_t n, const float *means, const CamDev &cam, const float *g2d, const uint32_t *mask,
                           float *dirs, float *g_color, cudaStream_t st);

// What the first kernel after a device-counted preprocess does with the instance count: it tells the host - `host` is a
// word of pinned memory that receives the view's number (24 bits) above the count (40 bits): one store, nothing to wait for
// - and raises the flag if the lists will be cut off.  A count that the 40 bits cannot hold goes as their largest value, at
// which the host reads the word on the device instead.
constexpr int kCountBits = 40;
constexpr unsigned long long kCountMost = (1ull << kCountBits) - 1, kViewMask = (1ull << (64 - kCountBits)) - 1;
struct CountReport {
  const unsigned long long *count;             // null: nothing to report
  unsigned long long capacity;
  uint32_t *overflow;
  unsigned long long *host, view;              // host null: no report
#ifdef __CUDACC__
  __device__ __forceinline__ void send() const {
    if (!count) return;
    const unsigned long long c = *count;
    if (c > capacity) *overflow = 1u;
    if (host) *reinterpret_cast<volatile unsigned long long *>(host) = view << kCountBits | (c < kCountMost ? c : kCountMost);
  }
#endif
};

constexpr int kWgradBlocks = 592;   // persistent blocks of the decoder-gradient kernels (4 x 148)

// Sorting / binning.
// What the scatter of the last pass of a sort adds on its way out (nothing where the pointers are null).
struct SortEpilogue {
  // depth sort: sums of the Gaussians' record counts (counts[id], without the flag of a large footprint) per 256
  // consecutive Gaussians of the sorted order, from which the record emission takes its offsets; cleared by the same pass
  const uint32_t *counts;
  uint32_t id_mask;             // bits of a sorted value that are the id (all: no count travels with it)
  uint32_t *block_sums;
  int num_block_sums;
  // record sort: [start, end) of every id = key >> key_shift in the sorted list (an id that does not occur has an empty
  // range), and the chunks of the expansion: the number of those of the ids before each, and (begin, end, id) of them all
  uint32_t *ranges;
  int num_ranges;
  int key_shift;
  uint32_t *chunk_first;
  uint4 *chunks;
  // depth sort: the number of visible Gaussians, and the place of the culled ones behind them, found by the first pass
  unsigned long long *visible;
  uint32_t *final_vals;
};
size_t sort_scratch_bytes(int64_t n, int64_t records);
// Stable sort of the cell records (keys: cell << 16 | tile mask) by cell, in radix_passes() passes: an odd number ends in
// other_keys / other_vals, an even one in keys / vals.  `count` bounds the number of records (and sizes the grid), the true
// number is read on the device.  With one pass it also leaves the chunks of the expansion.  Comes after launch_depth_sort,
// which prepares the scratch it shares with it.
int launch_record_sort(uint32_t *keys, uint32_t *vals, uint32_t *other_keys, uint32_t *other_vals, int64_t count,
                       const unsigned long long *count_dev, int cell_bits, void *scratch, const SortEpilogue &epilogue, cudaStream_t st);
int radix_passes(int num_bits);
// The depth order: ids by (key, id) ascending, where a key is the bits of a float, or 0xffffffff: culled Gaussians, behind
// all others.  tmp_keys / tmp_vals [n] are scratch, keys [n] receives the record counts in that order.  With visible != nullptr all floats are positive; it receives
// the number of Gaussians that are not culled, and the epilogue's block sums cover those.
int launch_depth_sort(const uint32_t *depth_key, uint32_t *keys, uint32_t *order, uint32_t *tmp_keys, uint32_t *tmp_vals, int64_t n,
                      unsigned long long *visible, void *scratch, const SortEpilogue &epilogue, const CountReport &report, cudaStream_t st);
// The same by buckets (gs_depth_sort.cu), for cameras that cull every depth of zero and below: pairs [n] is scratch, `clear` is
// cleared on the way.
constexpr int64_t kBucketSortMost = 1 << 22;  // Gaussians
bool bucket_sort_takes(int64_t n);
size_t bucket_scratch_bytes(int64_t n);
int launch_bucket_sort(const uint32_t *depth_key, uint32_t *counts_out, uint32_t *order, unsigned long long *pairs, int64_t n,
                       unsigned long long *visible, void *scratch, uint32_t *clear, int clear_words, const SortEpilogue &ep,
                       const CountReport &report, cudaStream_t st);
size_t scan_scratch_bytes(int64_t n);
int num_scan_blocks(int64_t n);   // entries of the block sums that launch_emit_records reads
int launch_emit_records(const uint32_t *depth_order, const uint32_t *sorted_count, const uint32_t *cell_records,
                        const uint16_t *rect, const float *mean2d, const float *conic_opacity, const uint32_t *block_sums,
                        const unsigned long long *visible, uint32_t *rec_keys, uint32_t *rec_vals, unsigned long long *rec_total, uint32_t *overflow, int64_t n,
                        int cgx, int W, int H, int64_t capacity, cudaStream_t st);
// Scratch of the expansion: chunk_first [cells + 1], chunks, chunk_counts and chunk_bases [max_pieces, 16], tile_counts and
// tile_starts [tiles].
struct CellScratch { uint32_t *chunk_first, *chunk_counts, *chunk_bases, *tile_counts, *tile_starts; uint4 *chunks; };
int max_pieces(int64_t record_capacity, int num_cells);   // of kBinPiece records (the grid-wide expansion works in larger chunks)
int launch_expand(const uint32_t *rec_keys, const uint32_t *rec_vals, const uint32_t *cell_ranges, const CellScratch &cs, bool chunks_known,
                  int64_t record_capacity, int64_t pair_capacity, int gx, int gy, int cgx, int cgy,
                  uint32_t *sorted_vals, uint32_t *tile_ranges, uint32_t *tile_order, cudaStream_t st);
// The whole binning in one cluster of CTAs and one expansion kernel (gs_bin_cluster.cu), for scenes that do not fill the
// chip.  Up to 2^kClusterDigit cells.
constexpr int kClusterDigit = 9;              // widest digit of its sorts
constexpr int kClusterMax = 8192;             // Gaussians (512 per CTA of the largest cluster)
constexpr int kBinPiece = 256;                // records of one cell that a warp counts and expands
struct ClusterBinArgs {
  uint32_t n, capacity;                        // Gaussians; records the buffers hold
  uint32_t pair_capacity32;
  CountReport report;
  uint32_t *overflow;
  const uint32_t *depth_key, *cell_count, *cell_records;
  const uint16_t *rect;
  const float *mean2d, *conic_opacity;
  uint32_t *keys, *order, *tmp_keys, *tmp_vals;                            // [n]
  uint32_t *rec_keys, *rec_vals, *sorted_rec_keys, *sorted_rec_vals;       // [capacity]
  uint32_t *cell_ranges, *piece_first, *piece_counts, *piece_bases, *tile_counts, *tile_starts;
  uint32_t *tile_ranges, *tile_order, *out_vals;
  uint32_t *num_big;                           // scratch: Gaussians whose records wait for a warp
  int num_cells, cell_bits, cgx, gx, gy, W, H;
};
// CTAs of the cluster for n Gaussians, one for every 64 up to 16 (1000 Gaussians: 33 us on 16 CTAs, 36 on 4), each alone on
// its SM; 0: the grid-wide kernels.  `limit`: the largest cluster that the device, or the share of it that the process has,
// can hold at all (bin_cluster_limit, with that device current).
constexpr int kClusterCtas = 16;
inline int cluster_ctas(int64_t n, int num_cells, int limit) {
  if (n > kClusterMax || num_cells > (1 << kClusterDigit)) return 0;
  int ctas = 1;
  while (ctas < kClusterCtas && (int64_t)ctas * 64 < n) ctas *= 2;
  return ctas <= limit ? ctas : 0;
}
int bin_cluster_limit(int device);
// Returns 0, with nothing launched, if the cluster is refused (a stream with fewer SMs than the context had).
int launch_bin_cluster(const ClusterBinArgs &a, int ctas, int64_t record_bound, cudaStream_t st);
int launch_empty_binning(uint32_t *tile_ranges, uint32_t *tile_order, int num_tiles, const CountReport &report, cudaStream_t st);

// Blend.
// (sorted_tiles: the tile id of every instance of the sorted list, written by the tile's CTA on its way in)
int launch_blend_fwd(const CamDev &cam, const uint32_t *ranges, const uint32_t *order, const uint32_t *vals,
                      const float *mean2d, const float *conic_opacity, const float *color, uint32_t *sorted_tiles,
                      float *image, float *final_T, uint32_t *n_contrib, cudaStream_t st);
// Gradient arrays whose rows start as zeros (16-byte aligned): the backward then writes the rows of the Gaussians that
// received a gradient.
struct ZeroRows {
  static constexpr int kMost = 8;
  float *ptr[kMost];
  uint64_t floats[kMost];
  uint32_t slice[kMost];        // groups of four floats that one warp writes (set by the launch)
  int count;
  void add(float *p, uint64_t n) { if (n) { ptr[count] = p; floats[count++] = n; } }
};
// Zeros, 16-byte aligned and a multiple of 16 bytes, for the blend backward that follows.
int launch_clear(void *p, size_t bytes, cudaStream_t st);
// Also sets the flag bit of every Gaussian (of n) that received a gradient, and fills `zeros`.
int launch_blend_bwd(int64_t n, const CamDev &cam, const uint32_t *ranges, const uint32_t *order, const uint32_t *vals,
                      const float *mean2d, const float *conic_opacity, const float *color,
                      const float *final_T, const uint32_t *n_contrib, const float *dL_dimage,
                      float *g2d, const GradFlags &flags, const ZeroRows &zeros, cudaStream_t st);

int launch_neural_fold(int64_t n, const __half *features, const __half *weights, __half *preact, cudaStream_t st);
int launch_neural_prepass(int64_t n, int deg, int act, const float *means, const float *logits, const float *base_color,
                          const __half *preact, const __half *weights, const float eye[3], uint8_t *rgba, float *color,
                          cudaStream_t st);
int launch_adam(const GsAdamTensor *tensors, int num_tensors, int64_t step, int num_sms, cudaStream_t st);
int launch_blend_count(const CamDev &cam, const uint32_t *ranges, const uint32_t *vals, const float *mean2d,
                       const float *conic_opacity, const float *color, unsigned long long *counts, cudaStream_t st);

// ---- device helpers -------------------------------------------------------------------------
#ifdef __CUDACC__

// Real orthonormal SH basis, degrees 0..3, order m = -l..l.
__device__ __forceinline__ void sh_basis(float x, float y, float z, float Y[16]) {
  const float xx = x * x, yy = y * y, zz = z * z;
  Y[0] = 0.28209479177387814f;
  Y[1] = -0.4886025119029199f * y;
  Y[2] = 0.4886025119029199f * z;
  Y[3] = -0.4886025119029199f * x;
  Y[4] = 1.0925484305920792f * x * y;
  Y[5] = -1.0925484305920792f * y * z;
  Y[6] = 0.31539156525252005f * (2.f * zz - xx - yy);
  Y[7] = -1.0925484305920792f * x * z;
  Y[8] = 0.5462742152960396f * (xx - yy);
  Y[9] = -0.5900435899266435f * y * (3.f * xx - yy);
  Y[10] = 2.890611442640554f * x * y * z;
  Y[11] = -0.4570457994644658f * y * (4.f * zz - xx - yy);
  Y[12] = 0.3731763325901154f * z * (2.f * zz - 3.f * xx - 3.f * yy);
  Y[13] = -0.4570457994644658f * x * (4.f * zz - xx - yy);
  Y[14] = 1.445305721320277f * z * (xx - yy);
  Y[15] = -0.5900435899266435f * x * (xx - 3.f * yy);
}

// Accumulate g_d += w * grad Y_k(d) for one basis function (k is a compile-time constant after
// unrolling).
__device__ __forceinline__ void sh_grad_acc(int k, float x, float y, float z, float w, float &gx,
                                            float &gy, float &gz) {
  const float c1 = 0.4886025119029199f, c2a = 1.0925484305920792f, c2b = 0.31539156525252005f,
              c2c = 0.5462742152960396f, c3a = 0.5900435899266435f, c3b = 2.890611442640554f,
              c3c = 0.4570457994644658f, c3d = 0.3731763325901154f, c3e = 1.445305721320277f;
  switch (k) {
    case 1: gy -= c1 * w; break;
    case 2: gz += c1 * w; break;
    case 3: gx -= c1 * w; break;
    case 4: gx += c2a * y * w; gy += c2a * x * w; break;
    case 5: gy -= c2a * z * w; gz -= c2a * y * w; break;
    case 6: gx -= 2.f * c2b * x * w; gy -= 2.f * c2b * y * w; gz += 4.f * c2b * z * w; break;
    case 7: gx -= c2a * z * w; gz -= c2a * x * w; break;
    case 8: gx += 2.f * c2c * x * w; gy -= 2.f * c2c * y * w; break;
    case 9: gx -= 6.f * c3a * x * y * w; gy -= 3.f * c3a * (x * x - y * y) * w; break;
    case 10: gx += c3b * y * z * w; gy += c3b * x * z * w; gz += c3b * x * y * w; break;
    case 11: gx += 2.f * c3c * x * y * w; gy -= c3c * (4.f * z * z - x * x - 3.f * y * y) * w;
             gz -= 8.f * c3c * y * z * w; break;
    case 12: gx -= 6.f * c3d * x * z * w; gy -= 6.f * c3d * y * z * w;
             gz += 3.f * c3d * (2.f * z * z - x * x - y * y) * w; break;
    case 13: gx -= c3c * (4.f * z * z - 3.f * x * x - y * y) * w; gy += 2.f * c3c * x * y * w;
             gz -= 8.f * c3c * x * z * w; break;
    case 14: gx += 2.f * c3e * x * z * w; gy -= 2.f * c3e * y * z * w; gz += c3e * (x * x - y * y) * w; break;
    case 15: gx -= 3.f * c3a * (x * x - y * y) * w; gy += 6.f * c3a * x * y * w; break;
    default: break;
  }
}

// tau = 2 ln(255 o): the alpha >= 1/255 ellipse is conic-form <= tau.  One function, so that the
// preprocess and the instance emission get identical bits.
__device__ __forceinline__ float footprint_tau(float o) { return 2.f * logf(255.f * o); }

// Exact tile overlap of the alpha >= 1/255 ellipse, row of tiles by row of tiles.  The ellipse is
// (la dx + lb dy)^2 + (lc dy)^2 <= tau with (la, lb, lc) the Cholesky factor of the conic.  Over a
// band of pixel-centre rows dy in [da, db] the set is convex, so the tiles it meets in that row are
// exactly those between its leftmost and rightmost point; the rightmost point over the band is at
// the band end nearest to dy_r = -lb sqrt(tau / C) / lc (C = lb^2 + lc^2), the leftmost at the one
// nearest to -dy_r.  Every operation is rounded once, in a fixed order (no contraction), so the
// same integers come out of any IEEE fp32 evaluation; tau and the band are padded by 2e-5 / 1e-5
// so that rounding can only add a tile, never drop a pixel the blend would accept.
struct TileSpans {
  float u, v, ila, lb, lc, taup, dys, eyp;
  int W, H;
  __device__ __forceinline__ void setup(float u_, float v_, float la, float lb_, float lc_, float tau, int W_, int H_) {
    u = u_; v = v_; lb = lb_; lc = lc_; W = W_; H = H_;
    taup = __fmul_rn(tau, 1.00002f);
    const float rl = __frcp_rn(lc);
    ila = __frcp_rn(la);
    const float C = __fadd_rn(__fmul_rn(lb, lb), __fmul_rn(lc, lc));
    dys = __fmul_rn(__fmul_rn(lb, rl), __fsqrt_rn(__fdiv_rn(taup, C)));
    eyp = __fmul_rn(__fmul_rn(__fsqrt_rn(taup), rl), 1.00001f);
  }
  // Tiles [xa, xb) of tile row ty, clipped to the bounding rectangle's columns [tx0, tx1).
  __device__ __forceinline__ bool row(int ty, int tx0, int tx1, int &xa, int &xb) const {
    const float ylo = (float)(16 * ty) + 0.5f, yhi = fminf((float)(16 * ty) + 15.5f, (float)H - 0.5f);
    const float da = fmaxf(__fsub_rn(ylo, v), -eyp), db = fminf(__fsub_rn(yhi, v), eyp);
    if (!(da <= db)) return false;
    const float dyR = fminf(fmaxf(-dys, da), db), dyL = fminf(fmaxf(dys, da), db);
    const float tR = __fmul_rn(lc, dyR), tL = __fmul_rn(lc, dyL);
    const float sR = __fsqrt_rn(fmaxf(__fsub_rn(taup, __fmul_rn(tR, tR)), 0.f));
    const float sL = __fsqrt_rn(fmaxf(__fsub_rn(taup, __fmul_rn(tL, tL)), 0.f));
    const float xr = __fmul_rn(__fsub_rn(sR, __fmul_rn(lb, dyR)), ila);
    const float xl = __fmul_rn(__fsub_rn(-sL, __fmul_rn(lb, dyL)), ila);
    const float ihi = floorf(__fsub_rn(__fadd_rn(u, xr), 0.5f)), ilo = ceilf(__fsub_rn(__fadd_rn(u, xl), 0.5f));
    if (!(ilo <= ihi) || ihi < 0.f || ilo > (float)(W - 1)) return false;
    const int pa = (int)fmaxf(ilo, 0.f), pb = (int)fminf(ihi, (float)(W - 1));
    xa = max(pa >> 4, tx0);
    xb = min((pb >> 4) + 1, tx1);
    return xa < xb;
  }
  __device__ __forceinline__ unsigned count(int tx0, int ty0, int tx1, int ty1) const {
    unsigned c = 0;
    for (int ty = ty0; ty < ty1; ++ty) {
      int xa, xb;
      if (row(ty, tx0, tx1, xa, xb)) c += (unsigned)(xb - xa);
    }
    return c;
  }
};

// Colour activations (Sec. 3.1) of z = c0 + 0.5 + A(d) and their derivatives: 0 ReLU(z), 1 softplus(z) with
// beta = 10, 2 sigmoid(4 (z - 0.5)), 3 clamp(z, 0, 1).  The derivative at a kink is 0.
__device__ __forceinline__ float color_act_z(int act, float z) {
  if (act == GS_ACT_SOFTPLUS) { const float t = 10.f * z; return t > 15.f ? z : 0.1f * log1pf(expf(t)); }
  if (act == GS_ACT_SIGMOID) return 1.f / (1.f + expf(fmaf(-4.f, z, 2.f)));
  if (act == GS_ACT_HARD_SIGMOID) return fminf(fmaxf(z, 0.f), 1.f);
  return fmaxf(z, 0.f);
}
__device__ __forceinline__ float color_act_grad_z(int act, float z) {
  if (act == GS_ACT_SOFTPLUS) return 1.f / (1.f + expf(-10.f * z));
  if (act == GS_ACT_SIGMOID) { const float y = 1.f / (1.f + expf(fmaf(-4.f, z, 2.f))); return 4.f * y * (1.f - y); }
  if (act == GS_ACT_HARD_SIGMOID) return (z > 0.f && z < 1.f) ? 1.f : 0.f;
  return z > 0.f ? 1.f : 0.f;
}

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// ---- the neural decoder's inputs and residual squashing, shared by every kernel that evaluates it
__device__ __forceinline__ void unpack_features(const uint4 &raw, float f[8]) {
  const __half2 *h = reinterpret_cast<const __half2 *>(&raw);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float2 v = __half22float2(h[j]);
    f[2 * j] = v.x; f[2 * j + 1] = v.y;
  }
}
__device__ __forceinline__ void load_features(const __half *features, int64_t i, float f[8]) {
  unpack_features(__ldg(reinterpret_cast<const uint4 *>(features) + i), f);
}

// Decoder inputs of one Gaussian (Eq. 5, Eq. 6 with k = 1): SH basis of the direction masked by the
// active degree, then (sin f_j, cos f_j).  The fast sincos is used inside [-pi, pi] (absolute error
// below 4e-7 there), the accurate one outside.
__device__ __forceinline__ void decoder_inputs(float dx, float dy, float dz, const float f[8], int deg, float x[32]) {
  sh_basis(dx, dy, dz, x);
  const int na = (deg + 1) * (deg + 1);
  if (na < 16) {
#pragma unroll
    for (int k = 0; k < 16; ++k) x[k] = k < na ? x[k] : 0.f;
  }
  float big = 0.f;
#pragma unroll
  for (int j = 0; j < 8; ++j) big = fmaxf(big, fabsf(f[j]));
  if (big <= 3.14159265f) {   // one decision for the eight of them: features are O(0.1 .. 1)
#pragma unroll
    for (int j = 0; j < 8; ++j) __sincosf(f[j], &x[16 + 2 * j], &x[17 + 2 * j]);
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j) sincosf(f[j], &x[16 + 2 * j], &x[17 + 2 * j]);
  }
}

// tanh(y) = 1 - 2 / (e^{2y} + 1) on the exponential and reciprocal units: absolute error of a few 1e-7 over the
// whole range (the residual is an absolute colour offset, so that is the error that counts), saturating to +-1.
__device__ __forceinline__ float tanh_fast(float y) {
  const float e = ex2_approx(y * 2.885390081777927f);    // 2 log2(e)
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(e + 1.f));
  return fmaf(-2.f, r, 1.f);
}

// Inclusive prefix sum over a warp.
template <class T>
__device__ __forceinline__ T warp_inclusive(T v, int lane) {
#pragma unroll
  for (int s = 1; s < 32; s <<= 1) {
    const T t = __shfl_up_sync(0xffffffffu, v, s);
    if (lane >= s) v += t;
  }
  return v;
}

// A float on its own way into shared memory, no register held.
__device__ __forceinline__ void copy_async4(void *dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Programmatic dependent launch.  A step is a chain of short, dependent launches (8 to 18 per view), a decode or a viewer frame one or
// two, repeated.
// Launched with the attribute below, a kernel may be placed on the SMs as soon as the CTAs of its predecessor in the
// stream have exited, without waiting for the predecessor's completion to be processed; dependency_wait() returns once
// the predecessor has completed and its writes are visible, and every kernel here calls it before its first access to
// global memory, so the order of all reads and writes is the stream's.  Launched without the attribute it is a no-op.
// When it came in, the binning of a view of 1M took 214 instead of 248 us on one stream (180 by now).  Letting the successor in earlier
// (griddepcontrol.launch_dependents at the top of every kernel) gained no more on one stream and cost 4 % with
// several views in flight: the successor's CTAs then sit on the SMs for the whole run of the predecessor, in the
// places of the other streams' kernels.
// With the blend backward and the kernels outside the step launched like this too, between repeated calls: the forward and backward decode of 1M
// Gaussians 108.5 -> 103.5 us, a viewer frame of 3M 55.4 -> 53.6, steps 71.1 -> 67.4 (1000 Gaussians) and 587.9 -> 581.9 (1M SH).
__device__ __forceinline__ void dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <class... KArgs, class... Args>
void launch_chained(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

#endif  // __CUDACC__

}  // namespace gs
