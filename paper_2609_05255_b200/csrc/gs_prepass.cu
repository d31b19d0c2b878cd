// Viewer-side evaluation of the neural appearance model (App. C.3, "Neural"), as CUDA kernels instead
// of fragment shaders.  Export: the 17 view-independent columns of the first layer (16 encoded
// features + the constant degree-0 input) are folded into 16 half-precision pre-activations per
// Gaussian.  Per frame: the 15 direction-dependent columns (padded to 16) and the two later layers,
// 560 multiply-accumulates per Gaussian, in half precision on tensor cores with fp32 accumulation,
// and one 8-bit RGBA texel per Gaussian as the result.
#include <cuda_fp16.h>

#include <algorithm>

#include "gs_device.cuh"
#include "gs_mlp_mma.cuh"

namespace gs {
namespace {

constexpr int kFoldThreads = 128;
constexpr int kPrepassThreads = 128;
constexpr int kPrepassWarps = kPrepassThreads / 32;
constexpr int kPrepassBlocks = 7;   // resident CTAs per SM (3M: four 51.2 us, six 49.4, seven 48.9, eight 50.1, nine 53.1)
constexpr int kXRow = 12;   // 32-bit words per staged input row: 8 half pairs + 4 pad (conflict-free fragment reads)

__global__ void __launch_bounds__(kFoldThreads) k_neural_fold(int64_t n, const __half *__restrict__ features,
                                                              const __half *__restrict__ weights,
                                                              __half *__restrict__ preact) {
  __shared__ float s_w[GS_MLP_HIDDEN][17];   // column 0 and the 16 feature columns of the first layer
  dependency_wait();
  for (int k = threadIdx.x; k < GS_MLP_HIDDEN * 17; k += kFoldThreads) {
    const int o = k / 17, c = k % 17;
    s_w[o][c] = __half2float(weights[kMlpW1 + o * GS_MLP_IN + (c == 0 ? 0 : 15 + c)]);
  }
  __syncthreads();
  const int64_t i = (int64_t)blockIdx.x * kFoldThreads + threadIdx.x;
  if (i >= n) return;
  const uint4 raw = __ldg(reinterpret_cast<const uint4 *>(features) + i);
  const __half2 *h = reinterpret_cast<const __half2 *>(&raw);
  float enc[16];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float2 f = __half22float2(h[j]);
    sincosf(f.x, &enc[4 * j], &enc[4 * j + 1]);
    sincosf(f.y, &enc[4 * j + 2], &enc[4 * j + 3]);
  }
  uint32_t out[8];
#pragma unroll
  for (int o = 0; o < GS_MLP_HIDDEN; o += 2) {
    float a0 = s_w[o][0] * 0.28209479177387814f, a1 = s_w[o + 1][0] * 0.28209479177387814f;
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      a0 = fmaf(s_w[o][1 + c], enc[c], a0);
      a1 = fmaf(s_w[o + 1][1 + c], enc[c], a1);
    }
    const __half2 p = __floats2half2_rn(a0, a1);
    out[o / 2] = *reinterpret_cast<const uint32_t *>(&p);
  }
  uint4 *dst = reinterpret_cast<uint4 *>(preact + 16 * i);
  dst[0] = make_uint4(out[0], out[1], out[2], out[3]);
  dst[1] = make_uint4(out[4], out[5], out[6], out[7]);
}

__device__ __forceinline__ uint32_t pack_half2(float a, float b) {
  const __half2 p = __floats2half2_rn(a, b);
  return *reinterpret_cast<const uint32_t *>(&p);
}
__device__ __forceinline__ uint32_t pack_relu(float a, float b) {              // (rounding keeps the sign)
  const __half2 p = __hmax2(__floats2half2_rn(a, b), __float2half2_rn(0.f));
  return *reinterpret_cast<const uint32_t *>(&p);
}
__device__ __forceinline__ uint32_t pack_weights(const __half *w, int idx) {   // w[idx], w[idx + 1]; idx is even
  return __ldg(reinterpret_cast<const uint32_t *>(w + idx));
}

// The next 32 rows of a warp, on their way into shared memory while it works on the current ones: 120 pieces of 16 bytes, four
// for most lanes, which hold no registers on the way.
struct __align__(16) PrepassRows {
  float mean[96], base[96], logit[32];
  uint32_t pre[32 * 8];
};
struct RowCopies {
  const char *src[4];           // of the lane's pieces, in the rows to fetch next
  uint32_t step[4], off[4];     // bytes of a row in its array; of the piece from the first row on
  __device__ __forceinline__ RowCopies(const float *means, const float *base, const float *logits, const __half *preact, int64_t row0, int lane) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int c = lane + 32 * k;
      const void *p = c < 24 ? (const void *)means : c < 48 ? (const void *)base : c < 56 ? (const void *)logits : (const void *)preact;
      step[k] = c < 48 ? 12u : c < 56 ? 4u : 32u;
      off[k] = 16u * (uint32_t)(c - (c < 24 ? 0 : c < 48 ? 24 : c < 56 ? 48 : 56));
      src[k] = static_cast<const char *>(p) + row0 * step[k] + off[k];
    }
  }
  // `left`: rows from the first one to the end of the arrays; `stride`: from here to the next fetch.
  __device__ __forceinline__ void fetch(PrepassRows &to, int64_t left, uint32_t stride, int lane) {
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&to) + 16u * (uint32_t)lane;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (k == 3 && lane >= 24) break;
      if (left >= 32) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 512u * k), "l"(src[k]) : "memory");
      } else {                                   // what is past the end reads as zero
        const uint32_t have = (uint32_t)left * step[k], size = have > off[k] ? min(have - off[k], 16u) : 0u;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + 512u * k), "l"(src[k]), "r"(size) : "memory");
      }
      src[k] += stride * step[k];
    }
  }
};
static_assert(sizeof(PrepassRows) == 120 * 16, "pieces");

// One warp per 32 Gaussians at a time.  Lane L prepares row L (direction, SH basis, base colour, alpha byte);
// the rows reach the tensor-core fragment layout through a small shared-memory tile; the weights
// live in ten registers per lane for the whole kernel.
// Bound by instruction issue (192 MB need 29 us): the warps are persistent, so that the weights are read once, the rectifiers
// work on packed halves, degree 3 has an instance without the selects of the others, the rows come in asynchronous copies a
// trip ahead and reach the fragments through ldmatrix, and the activation is chosen once.  3M Gaussians: 61.3 us at first,
// 53.2 with loads at the start of every trip (62 % of the issue slots) and fragments word by word, 52.5 with the copies alone,
// 50.7 with ldmatrix and vector stores, 48.1 with one branch for the activation (75 % of the slots).
template <bool kFull3>   // degree 3: all direction inputs in use
__global__ void __launch_bounds__(kPrepassThreads, kPrepassBlocks) k_neural_prepass(int64_t n, int deg, int act, const float *__restrict__ means,
                                                                    const float *__restrict__ logits,
                                                                    const float *__restrict__ base_color,
                                                                    const __half *__restrict__ preact,
                                                                    const __half *__restrict__ weights, float ex, float ey,
                                                                    float ez, uchar4 *__restrict__ rgba,
                                                                    float *__restrict__ color) {
  __shared__ __align__(16) uint32_t s_x[kPrepassWarps][32][kXRow];
  __shared__ float s_y[kPrepassWarps][32][3];
  __shared__ PrepassRows s_rows[kPrepassWarps][2];
  dependency_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  // B fragments: B[k][nn] = W[nn][k]; b0 holds k = 2t, 2t+1 and b1 k = 2t+8, 2t+9 of column nn = 8 nt + g.
  // Layer 1 keeps only the direction columns 1..15 (column 0 is the folded constant: its weight is dropped).
  uint32_t w1b0[2], w1b1[2], w2b0[2], w2b1[2], w3b0, w3b1;
#pragma unroll
  for (int nt = 0; nt < 2; ++nt) {
    const int nn = nt * 8 + g;
    w1b0[nt] = pack_weights(weights, kMlpW1 + nn * GS_MLP_IN + 2 * t);
    if (t == 0) w1b0[nt] &= 0xffff0000u;
    w1b1[nt] = pack_weights(weights, kMlpW1 + nn * GS_MLP_IN + 2 * t + 8);
    w2b0[nt] = pack_weights(weights, kMlpW2 + nn * GS_MLP_HIDDEN + 2 * t);
    w2b1[nt] = pack_weights(weights, kMlpW2 + nn * GS_MLP_HIDDEN + 2 * t + 8);
  }
  w3b0 = g < 3 ? pack_weights(weights, kMlpW3 + g * GS_MLP_HIDDEN + 2 * t) : 0u;
  w3b1 = g < 3 ? pack_weights(weights, kMlpW3 + g * GS_MLP_HIDDEN + 2 * t + 8) : 0u;
  const int na = (deg + 1) * (deg + 1);

  const int64_t row_first = ((int64_t)blockIdx.x * kPrepassWarps + warp) * 32;
  RowCopies copies(means, base_color, logits, preact, row_first, lane);
  const uint32_t stride = gridDim.x * kPrepassThreads;
  if (row_first < n) copies.fetch(s_rows[warp][0], n - row_first, stride, lane);
  // where ldmatrix finds the lane's row of a fragment of 16 rows
  const uint32_t x_at = mlp::smem_u32(&s_x[warp][lane & 15][4 * (lane >> 4)]), pre_at = mlp::smem_u32(s_rows[warp][0].pre + 8 * (lane & 15) + 4 * (lane >> 4));
  int turn = 0;
#pragma unroll 1
  for (int64_t row0 = row_first; row0 < n; row0 += stride, turn ^= 1) {
    const int rows = (int)min(n - row0, (int64_t)32);     // of this warp; what lies at row0 is addressed by 32-bit offsets
    const bool in = lane < rows;
    const PrepassRows &own = s_rows[warp][turn];
    copies_wait();
    __syncwarp();                                         // (the other buffer has been read, too)
    if (row0 + stride < n) copies.fetch(s_rows[warp][turn ^ 1], n - row0 - stride, stride, lane);
    // ---- this lane's Gaussian: direction, direction inputs, base colour, alpha
    float4 c = make_float4(0.f, 0.f, 0.f, 0.f);   // base colour and the alpha texel value
    {
      float Y[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) Y[k] = 0.f;
      if (in) {
        const float *mean = own.mean + 3 * lane, *base = own.base + 3 * lane;
        const float dx = mean[0] - ex, dy = mean[1] - ey, dz = mean[2] - ez;
        const float inv = rsqrtf(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
        sh_basis(dx * inv, dy * inv, dz * inv, Y);
        const float o = 1.f / (1.f + __expf(-own.logit[lane]));
        c = make_float4(base[0], base[1], base[2],
                        fmaf(fminf(fmaxf(o, 0.f), 1.f), 255.f, 0.5f));
      }
      Y[0] = 0.f;   // folded into the pre-activations
      uint32_t x[8];
#pragma unroll
      for (int k = 0; k < 8; ++k)
        x[k] = kFull3 ? pack_half2(Y[2 * k], Y[2 * k + 1]) : pack_half2(2 * k < na ? Y[2 * k] : 0.f, 2 * k + 1 < na ? Y[2 * k + 1] : 0.f);
      uint4 *row = reinterpret_cast<uint4 *>(s_x[warp][lane]);
      row[0] = make_uint4(x[0], x[1], x[2], x[3]);
      row[1] = make_uint4(x[4], x[5], x[6], x[7]);
    }
    __syncwarp();
    float y[2][4];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
      uint32_t a[4], pre[4];                     // pre: rows g and g + 8 of the first eight columns, then of the others
      mlp::ldsm_x4(a, x_at + mt * 16 * kXRow * 4);
      mlp::ldsm_x4(pre, pre_at + turn * (uint32_t)sizeof(PrepassRows) + mt * 16 * 32);
      // ---- layer 1, accumulators start at the folded pre-activations
      float h[2][4];
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) {
        const float2 f0 = __half22float2(*reinterpret_cast<const __half2 *>(&pre[2 * nt]));
        const float2 f1 = __half22float2(*reinterpret_cast<const __half2 *>(&pre[2 * nt + 1]));
        h[nt][0] = f0.x; h[nt][1] = f0.y; h[nt][2] = f1.x; h[nt][3] = f1.y;
        if (kFull3 || deg > 0) mlp::mma16816(h[nt], a, w1b0[nt], w1b1[nt]);
      }
      // ---- layer 2: the ReLU'd outputs of two column tiles are one A fragment
      a[0] = pack_relu(h[0][0], h[0][1]); a[1] = pack_relu(h[0][2], h[0][3]);
      a[2] = pack_relu(h[1][0], h[1][1]); a[3] = pack_relu(h[1][2], h[1][3]);
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) {
        h[nt][0] = h[nt][1] = h[nt][2] = h[nt][3] = 0.f;
        mlp::mma16816(h[nt], a, w2b0[nt], w2b1[nt]);
      }
      // ---- layer 3 (three outputs, padded to eight columns)
      a[0] = pack_relu(h[0][0], h[0][1]); a[1] = pack_relu(h[0][2], h[0][3]);
      a[2] = pack_relu(h[1][0], h[1][1]); a[3] = pack_relu(h[1][2], h[1][3]);
      y[mt][0] = y[mt][1] = y[mt][2] = y[mt][3] = 0.f;
      mlp::mma16816(y[mt], a, w3b0, w3b1);
    }
    // ---- the three outputs go back from the fragment layout (lanes t = 0 hold outputs 0, 1 of rows g and
    // g + 8, lanes t = 1 output 2) to one row per lane, so that every lane finishes its own Gaussian
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
      if (t == 0) {
        s_y[warp][mt * 16 + g][0] = y[mt][0]; s_y[warp][mt * 16 + g][1] = y[mt][1];
        s_y[warp][mt * 16 + g + 8][0] = y[mt][2]; s_y[warp][mt * 16 + g + 8][1] = y[mt][3];
      } else if (t == 1) {
        s_y[warp][mt * 16 + g][2] = y[mt][0];
        s_y[warp][mt * 16 + g + 8][2] = y[mt][2];
      }
    }
    __syncwarp();
    if (in) {
      float col[3];
      unsigned q[3];
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) {
        // tanh(a) = 1 - 2 / (exp(2a) + 1); the fast exponential and division are far inside the texel's step
        const float res = kFull3 || deg > 0 ? 1.f - __fdividef(2.f, __expf(2.f * s_y[warp][lane][ch]) + 1.f) : 0.f;
        col[ch] = (ch == 0 ? c.x : ch == 1 ? c.y : c.z) + 0.5f + res;
      }
      if (act == GS_ACT_RELU) {                  // (one branch for the three)
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) col[ch] = color_act_z(GS_ACT_RELU, col[ch]);
      } else {
#pragma unroll 1
        for (int ch = 0; ch < 3; ++ch) {
          const float z = color_act_z(act, col[0]);
          col[0] = col[1]; col[1] = col[2]; col[2] = z;
        }
      }
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) q[ch] = (unsigned)fmaf(fminf(col[ch], 1.f), 255.f, 0.5f);   // (rounds down)
      reinterpret_cast<uint32_t *>(rgba + row0)[lane] = q[0] | q[1] << 8 | q[2] << 16 | (unsigned)c.w << 24;
      if (color) {
        float *out = color + 3 * row0 + (uint32_t)(3 * lane);
        out[0] = col[0]; out[1] = col[1]; out[2] = col[2];
      }
    }
  }
}

}  // namespace

int launch_neural_fold(int64_t n, const __half *features, const __half *weights, __half *preact, cudaStream_t st) {
  if (n <= 0) return 0;
  launch_chained(k_neural_fold, (unsigned)((n + kFoldThreads - 1) / kFoldThreads), kFoldThreads, 0, st, n, features, weights, preact);
  return 1;
}

int launch_neural_prepass(int64_t n, int deg, int act, const float *means, const float *logits, const float *base_color,
                          const __half *preact, const __half *weights, const float eye[3], uint8_t *rgba, float *color,
                          cudaStream_t st) {
  if (n <= 0) return 0;
  const int64_t blocks = std::min<int64_t>((n + kPrepassThreads - 1) / kPrepassThreads, 148 * kPrepassBlocks);
  launch_chained(deg >= 3 ? k_neural_prepass<true> : k_neural_prepass<false>, (unsigned)blocks, kPrepassThreads, 0, st, n, deg, act, means, logits,
                 base_color, preact, weights, eye[0], eye[1], eye[2], reinterpret_cast<uchar4 *>(rgba), color);
  return 1;
}

}  // namespace gs
