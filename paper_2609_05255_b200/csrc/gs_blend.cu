// Per-tile alpha blending, forward and backward.  Every warp works on its own (CTAs of one warp): it owns a region of a
// tile, 8 x 8 pixels in the forward, 16 x 8, 8 x 8 or 4 x 8 in the backward, walks the tile's depth-ordered list 32
// entries at a time with the next ones on their way, drops those that cannot reach its region, and composites the rest
// without a branch or a vote per entry.
//
// What bounds both kernels is the register file, not the arithmetic pipes: a packed fp32 multiply-add with three
// different register pairs takes three cycles of a scheduler, one with two pairs two, so the time goes with the operands
// read.  Hence predicates instead of 0 / 1 factors in the forward and, in the backward, no shuffles or selects per entry:
// what crosses lanes is parked in shared memory and summed later.
#include <algorithm>

#include "gs_device.cuh"

namespace gs {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr float kLn2 = 0.6931471805599453f;

// ---- vectors of pixels ----------------------------------------------------------------------------------------
// A lane's pixels travel as packed fp32 pairs (one instruction, two IEEE operations) or, with one pixel per lane, as
// plain floats; the overloads below let one body serve both.
template <class V> __device__ __forceinline__ V bc(float x);
template <> __device__ __forceinline__ float bc<float>(float x) { return x; }
template <> __device__ __forceinline__ float2 bc<float2>(float x) { return make_float2(x, x); }
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float2 mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float2 add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float mad(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float2 mad(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float neg(float a) { return -a; }
__device__ __forceinline__ float2 neg(float2 a) { return make_float2(-a.x, -a.y); }
template <bool B> struct Flag { static constexpr bool value = B; };
__device__ __forceinline__ float hsum(float a) { return a; }
__device__ __forceinline__ float hsum(float2 a) { return a.x + a.y; }

// ---- how a tile is shared out ------------------------------------------------------------------------------------
// A warp owns a region of 4 NPX x 8 pixels of one tile and works through the tile's list on its own: lane (g, t) =
// (lane / 4, lane % 4) has NPX pixels in row g from column NPX t on.
template <int NPX> struct Share;
template <> struct Share<4> { using V = float2; static constexpr int kVecs = 2, kWarps = 2, kColumns = 1; };
template <> struct Share<2> { using V = float2; static constexpr int kVecs = 1, kWarps = 4, kColumns = 2; };
template <> struct Share<1> { using V = float; static constexpr int kVecs = 1, kWarps = 8, kColumns = 4; };
// First pixel of the warp's region.
template <int NPX>
__device__ __forceinline__ void region_of(int tile, int gx, int warp, int &rx, int &ry) {
  rx = (tile % gx) * GS_TILE + (warp % Share<NPX>::kColumns) * 4 * NPX;
  ry = (tile / gx) * GS_TILE + (warp / Share<NPX>::kColumns) * 8;
}
__device__ __forceinline__ float get(float v, int) { return v; }
__device__ __forceinline__ float get(float2 v, int k) { return k ? v.y : v.x; }
__device__ __forceinline__ void put(float &v, int, float x) { v = x; }
__device__ __forceinline__ void put(float2 &v, int k, float x) { if (k) v.y = x; else v.x = x; }
template <class V> struct Lanes;
template <> struct Lanes<float> { static constexpr int value = 1; };
template <> struct Lanes<float2> { static constexpr int value = 2; };

// ---- the list, 32 entries at a time ------------------------------------------------------------------------------
// Lane l fetches the parameters of entry l of the next 32 with asynchronous copies while the warp works on the current
// ones (the id was loaded one round earlier still), so neither the gather nor the two dependent loads are waited for.
struct __align__(16) RawEntries {
  float4 conic[32];
  float2 mean[32];
  float color[3][32];
};
// Entries the warp works on.
constexpr int kStaged = 32;
struct __align__(16) StagedEntries {
  float4 shape[kStaged];      // -x, -y, la, lb
  float4 rest[kStaged];       // lc, o, position in the list, -
  float4 rgb[kStaged];
};

__device__ __forceinline__ void copy_async16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async8(void *dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

__device__ __forceinline__ void fetch_entry(RawEntries &raw, int lane, uint32_t g, const float *mean2d, const float *conic_opacity,
                                            const float *color) {
  copy_async16(&raw.conic[lane], conic_opacity + 4 * (size_t)g);
  copy_async8(&raw.mean[lane], mean2d + 2 * (size_t)g);
#pragma unroll
  for (int c = 0; c < 3; ++c) copy_async4(&raw.color[c][lane], color + 3 * (size_t)g + c);
}

// Can the entry reach alpha = 1/255 somewhere in the box [x0, x1] x [y0, y1] (offsets from its centre)?  The exponent
// f = (la x + lb y)^2 + (lc y)^2 is convex, so its minimum over the box lies at the centre if the box holds it, else on
// the vertical or the horizontal edge facing it, where it is a clamped one-dimensional minimum.  All candidates are
// points of the box, so an error in where they lie moves the value by its square only; `slack` covers the rounding of
// the pixels' own evaluation (|la x| below 2^15 with an error of 2^-24 each, times 2 |la x + lb y| < 6).
__device__ __forceinline__ bool may_touch(float x0, float x1, float y0, float y1, float la, float lb, float lc, float limit) {
  const float kSlack = 0.02f;
  const float xn = fminf(fmaxf(0.f, x0), x1), yn = fminf(fmaxf(0.f, y0), y1);
  const float ye = fminf(fmaxf(-xn * la * lb * rcp_approx(fmaf(lb, lb, lc * lc)), y0), y1);
  const float xe = fminf(fmaxf(-yn * lb * rcp_approx(la), x0), x1);
  const float u1 = fmaf(la, xn, lb * ye), v1 = lc * ye, u2 = fmaf(la, xe, lb * yn), v2 = lc * yn;
  const float f = fminf(fmaf(u1, u1, v1 * v1), fmaf(u2, u2, v2 * v2));
  return !(f > limit + kSlack);     // (a NaN stays in)
}

// Turns the lane's fetched entry into a staged one if it can touch the warp's region, closing ranks; returns how many
// there are, rounded up to whole groups of kGroup with neutral entries.  `clamp`: one of them has an opacity above the alpha clamp.
// (la, lb, lc) is the Cholesky factor of the conic, scaled by sqrt(0.5 log2 e), so that alpha = o exp(power) =
// o 2^-((la dx + lb dy)^2 + (lc dy)^2): a sum of two squares has no cancellation, which keeps alpha accurate to a
// few ulp even for footprints hundreds of pixels wide (the expanded quadratic form loses 1e-4 there).
// `pos` and `id` go with the entry (its position in the list, its Gaussian).  NPX = 0 keeps every entry.
template <int NPX, int kGroup>
__device__ __forceinline__ int stage_entries(const RawEntries &raw, StagedEntries &st, int lane, bool valid, uint32_t pos, uint32_t id,
                                             float rx0, float ry0, bool &clamp) {
  const float kS = 0.8493218002880191f;   // sqrt(0.5 * log2(e))
  float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
  float2 m = make_float2(0.f, 0.f);
  float la = 0.f, lb = 0.f, lc = 0.f;
  if (valid) {
    q = raw.conic[lane]; m = raw.mean[lane];
    la = kS * q.x; lb = kS * q.y; lc = kS * q.z;
    const float x0 = rx0 - m.x, y0 = ry0 - m.y;
    valid = NPX == 0 || may_touch(x0, x0 + (float)(4 * NPX - 1), y0, y0 + 7.f, la, lb, lc, __log2f(255.f * q.w));
  }
  const uint32_t taken = __ballot_sync(kFull, valid);
  clamp = __any_sync(kFull, valid && !(q.w <= kAlphaMax));
  const int count = __popc(taken);
  if (valid) {
    const int slot = __popc(taken & ((1u << lane) - 1u));
    st.shape[slot] = make_float4(-m.x, -m.y, la, lb);
    st.rest[slot] = make_float4(lc, q.w, __uint_as_float(pos), 0.f);
    st.rgb[slot] = make_float4(raw.color[0][lane], raw.color[1][lane], raw.color[2][lane], __uint_as_float(id));
  }
  if (lane < (-count & (kGroup - 1))) {          // neutral: alpha = 0
    st.shape[count + lane] = st.rest[count + lane] = st.rgb[count + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __syncwarp();
  return (count + kGroup - 1) & ~(kGroup - 1);
}

// Alphas of a lane's pixels (fx: the centres of its columns, fy: that of its row), not yet clamped.  One explicit
// operation order, shared by the forward, the backward and the pair counter, so that all take identical decisions.
// (lb dy belongs to all pixels of a lane: it must not be rounded before the sum, or their errors have one sign - with
// that, three times as many gradients of a 100k scene miss 1e-3.)
template <int NPX>
__device__ __forceinline__ void alphas(const float4 &shape, const float4 &rest, const typename Share<NPX>::V fx[Share<NPX>::kVecs],
                                       float fy, typename Share<NPX>::V alpha[Share<NPX>::kVecs]) {
  using V = typename Share<NPX>::V;
  const float dy = __fadd_rn(fy, shape.y), c = __fmul_rn(rest.x, dy), s = __fmul_rn(c, c);
#pragma unroll
  for (int k = 0; k < Share<NPX>::kVecs; ++k) {
    const V u = mad(bc<V>(shape.w), bc<V>(dy), mul(bc<V>(shape.z), add(fx[k], bc<V>(shape.x)))), f = mad(u, u, bc<V>(s));
#pragma unroll
    for (int i = 0; i < Lanes<V>::value; ++i) put(alpha[k], i, ex2_approx(-get(f, i)));
    alpha[k] = mul(bc<V>(rest.y), alpha[k]);
  }
}

// One pixel of the forward composites one entry, all by predicates.  It takes the entry if alpha >= 1/255 (q) and
// the transmittance behind the entry, n, stays at 1e-4 or more (p); then the entry's colour is added with weight w and
// its position noted.  T follows n either way: once it has fallen below 1e-4 no later n can pass, so the pixel has
// stopped for good, and F keeps the transmittance it stopped with.
__device__ __forceinline__ void composite(float alpha, float n, float w, const float4 &c, uint32_t pos1, float &T, float &F, float &R,
                                          float &G, float &B, uint32_t &last) {
  asm("{\n\t.reg .pred q, p;\n\t"
      "setp.geu.f32 q, %6, %7;\n\t"
      "setp.ge.and.f32 p, %8, %9, q;\n\t"
      "@p fma.rn.f32 %2, %10, %11, %2;\n\t"
      "@p fma.rn.f32 %3, %10, %12, %3;\n\t"
      "@p fma.rn.f32 %4, %10, %13, %4;\n\t"
      "@p mov.f32 %1, %8;\n\t"
      "@p mov.u32 %5, %14;\n\t"
      "@q mov.f32 %0, %8;\n\t}"
      : "+f"(T), "+f"(F), "+f"(R), "+f"(G), "+f"(B), "+r"(last)
      : "f"(alpha), "f"(kAlphaMin), "f"(n), "f"(kTmin), "f"(w), "f"(c.x), "f"(c.y), "f"(c.z), "r"(pos1));
}

// Forward.  Entries are taken four at a time: their alphas do not depend on one another, only the chain through T does.
// 8 x 8 pixels per warp measured best from 16 tiles to 8160 (16 x 8 ties at 8160, 5 us more at 4108 tiles, 11 at 2550; two
// entries at a time: 1 to 2 us more where a launch is only a few warps per scheduler).
// 1M Gaussians, 1256 x 828: 152 -> 105 us; 92 M -> 81 M warp instructions, 76 % of the issue slots.  With 32 warps per SM, the
// most there can be of one-warp CTAs, instead of 28 -> 101, and 201 -> 193 in a view of 3M: one word spilled, before the loop.
constexpr int kFwdPixels = 2, kFwdGroup = 4;
__global__ void __launch_bounds__(32, 32) k_blend_fwd(
    CamDev cam, const uint32_t *__restrict__ ranges, const uint32_t *__restrict__ order, const uint32_t *__restrict__ vals,
    const float *__restrict__ mean2d, const float *__restrict__ conic_opacity, const float *__restrict__ color,
    uint32_t *__restrict__ sorted_tiles, float *__restrict__ image, float *__restrict__ final_T, uint32_t *__restrict__ n_contrib) {
  dependency_wait();
  constexpr int NPX = kFwdPixels;
  using V = Share<NPX>::V;
  constexpr int kVecs = Share<NPX>::kVecs, kWarps = Share<NPX>::kWarps, kLanes = Lanes<V>::value;
  __shared__ RawEntries raw;
  __shared__ StagedEntries st;
  const int lane = threadIdx.x, warp = (int)(blockIdx.x % kWarps), tile = (int)__ldg(order + blockIdx.x / kWarps);
  int rx, ry;
  region_of<NPX>(tile, cam.gx, warp, rx, ry);
  const int px = rx + NPX * (lane & 3), py = ry + (lane >> 2);
  const uint32_t start = __ldg(ranges + 2 * tile), end = __ldg(ranges + 2 * tile + 1);
  // the key of every instance of this tile's stretch of the sorted list is the tile id: stores that nothing here waits for
  if (sorted_tiles)
    for (uint32_t p = start + 32u * warp + lane; p < end; p += 32 * kWarps) sorted_tiles[p] = (uint32_t)tile;
  const float fy = (float)py + 0.5f, rx0 = (float)rx + 0.5f, ry0 = (float)ry + 0.5f;
  // T, F: transmittance (see composite); pixels outside the image start stopped
  V fx[kVecs];
  float T[NPX], F[NPX], R[NPX], G[NPX], B[NPX];
  uint32_t last[NPX];                       // position + 1 of the last composited entry
#pragma unroll
  for (int k = 0; k < NPX; ++k) {
    put(fx[k / kLanes], k % kLanes, (float)(px + k) + 0.5f);
    T[k] = px + k < cam.W && py < cam.H ? 1.f : 0.f;
    F[k] = 1.f;
    R[k] = G[k] = B[k] = 0.f;
    last[k] = 0u;
  }
  auto any_live = [&]() {
    float t = T[0];
#pragma unroll
    for (int k = 1; k < NPX; ++k) t = fmaxf(t, T[k]);
    return __any_sync(kFull, t >= kTmin);
  };
  const uint32_t len = end - start;
  uint32_t id = 0;
  if ((uint32_t)lane < len) fetch_entry(raw, lane, __ldg(vals + start + lane), mean2d, conic_opacity, color);
  if (32u + (uint32_t)lane < len) id = __ldg(vals + start + 32u + lane);
  for (uint32_t base = 0; base < len; base += 32) {
    if (!any_live()) break;                 // every pixel of the region has stopped
    copies_wait();
    bool clamp;
    const int count = stage_entries<NPX, kFwdGroup>(raw, st, lane, base + lane < len, base + lane + 1u, 0u, rx0, ry0, clamp);
    if (base + 32u + lane < len) fetch_entry(raw, lane, id, mean2d, conic_opacity, color);
    if (base + 64u + lane < len) id = __ldg(vals + start + base + 64u + lane);
    auto work = [&](auto clamped) {
      for (int j0 = 0; j0 < count; j0 += 8) {
        if (j0 && !any_live()) break;
        const int j1 = min(j0 + 8, count);
        for (int j = j0; j < j1; j += kFwdGroup) {
          V al[kFwdGroup][kVecs];
#pragma unroll
          for (int e = 0; e < kFwdGroup; ++e) {
            alphas<NPX>(st.shape[j + e], st.rest[j + e], fx, fy, al[e]);
            if (decltype(clamped)::value)
#pragma unroll
              for (int k = 0; k < kVecs; ++k)
#pragma unroll
                for (int i = 0; i < kLanes; ++i) put(al[e][k], i, fminf(kAlphaMax, get(al[e][k], i)));
          }
#pragma unroll
          for (int e = 0; e < kFwdGroup; ++e) {
            const float4 c = st.rgb[j + e];
            const uint32_t pos1 = __float_as_uint(st.rest[j + e].z);
#pragma unroll
            for (int k = 0; k < kVecs; ++k) {
              // transmittance behind the entry as T (1 - alpha), both roundings included: the backward takes T in front as T + w with
              // w = T alpha / (1 - alpha), the same 1 - alpha, and drifts if the forward rounds another expression (T - alpha T in one
              // rounding: 2.4 times as many gradients of a 1M scene missed 1e-3 when the backward divided by 1 - alpha)
              V t;
#pragma unroll
              for (int i = 0; i < kLanes; ++i) put(t, i, T[kLanes * k + i]);
              const V w = mul(al[e][k], t), n = mul(t, add(bc<V>(1.f), neg(al[e][k])));
#pragma unroll
              for (int i = 0; i < kLanes; ++i) {
                const int p = kLanes * k + i;
                composite(get(al[e][k], i), get(n, i), get(w, i), c, pos1, T[p], F[p], R[p], G[p], B[p], last[p]);
              }
            }
          }
        }
      }
    };
    if (clamp) work(Flag<true>()); else work(Flag<false>());
    __syncwarp();                            // the staged entries have been read
  }
  copies_wait();
  const size_t plane = (size_t)cam.W * cam.H;
#pragma unroll
  for (int k = 0; k < NPX; ++k)
    if (px + k < cam.W && py < cam.H) {
      const size_t pix = (size_t)py * cam.W + px + k;
      const float t = F[k];
      image[pix] = fmaf(t, cam.bg[0], R[k]);
      image[plane + pix] = fmaf(t, cam.bg[1], G[k]);
      image[2 * plane + pix] = fmaf(t, cam.bg[2], B[k]);
      final_T[pix] = t;
      n_contrib[pix] = last[k];
    }
}

// ---- backward ----------------------------------------------------------------------------------------------------
__device__ __forceinline__ void red_add4(float *p, float a, float b, float c, float d) {
  asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

// v if alpha >= 1/255 and the entry lies inside the pixel's walk, else 0
__device__ __forceinline__ float select_alpha(float alpha, uint32_t pos, uint32_t nc, float v) {
  float r;
  asm("{\n\t.reg .pred q, p;\n\tsetp.lt.u32 q, %1, %2;\n\tsetp.geu.and.f32 p, %3, %4, q;\n\tselp.f32 %0, %5, 0f00000000, p;\n\t}"
      : "=f"(r) : "r"(pos), "r"(nc), "f"(alpha), "f"(kAlphaMin), "f"(v));
  return r;
}

// The 2D gradients and flags start from zero.  (As a memset, which neither neighbour can be chained to, 2 to 5 us of the stream
// passed around it.  Letting the blend backward in early, to overlap its first loads, is no gain and a trap: the few warps of a
// small image then pile up on the SMs that this kernel leaves first, 49 -> 60 to 160 us for 30 tiles.)
constexpr int kClearThreads = 256, kClearBlocks = 148 * 4;
__global__ void __launch_bounds__(kClearThreads) k_clear(float4 *__restrict__ rows, size_t quads) {
  dependency_wait();
#pragma unroll 4
  for (size_t i = (size_t)blockIdx.x * kClearThreads + threadIdx.x; i < quads; i += (size_t)gridDim.x * kClearThreads)
    rows[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// One warp's slice of the rows that start as zeros.
constexpr int kZeroWarps = 148 * 2;           // at least; see launch_blend_bwd
__device__ __forceinline__ void zero_rows(const ZeroRows &z, int lane) {
#pragma unroll 1
  for (int k = 0; k < z.count; ++k) {
    float4 *p = reinterpret_cast<float4 *>(z.ptr[k]) + (uint64_t)blockIdx.x * z.slice[k];
    const uint64_t quads = z.floats[k] >> 2, from = (uint64_t)blockIdx.x * z.slice[k];
    const uint32_t count = from < quads ? (uint32_t)min(quads - from, (uint64_t)z.slice[k]) : 0u;
    for (uint32_t i = lane; i < count; i += 32) __stcs(p + i, make_float4(0.f, 0.f, 0.f, 0.f));
    if (blockIdx.x == 0 && lane < (int)(z.floats[k] & 3u)) z.ptr[k][4 * quads + lane] = 0.f;
  }
}

// What the lanes leave of an entry: dp of their pixels and their colour sums, kBatch entries at a time.  Strides chosen
// so that the reads of sum_entries meet no bank conflict: four lanes read neighbouring values of one entry, and the
// eight (float4), sixteen (float2) or thirty-two (float) lanes that are served together cover all banks.
constexpr int kBatch = 8, kParkStride = 36;
template <int NPX> struct Dp;
template <> struct Dp<4> { using T = float4; };
template <> struct Dp<2> { using T = float2; };
template <> struct Dp<1> { using T = float; };
template <int NPX>
struct __align__(16) Parked {
  typename Dp<NPX>::T dp[kBatch * kParkStride];
  float2 rg[kBatch * kParkStride];
  float b[kBatch * kParkStride];
};

__device__ __forceinline__ float4 pack(const float2 v[2]) { return make_float4(v[0].x, v[0].y, v[1].x, v[1].y); }
template <int NPX, class V>
__device__ __forceinline__ void park(Parked<NPX> &p, int e, int lane, const V dp[Share<NPX>::kVecs], float r, float g, float b) {
  if constexpr (NPX == 4) p.dp[e * kParkStride + lane] = pack(dp); else p.dp[e * kParkStride + lane] = dp[0];
  p.rg[e * kParkStride + lane] = make_float2(r, g);
  p.b[e * kParkStride + lane] = b;
}
// Sums over the region of entry e, in all of its four lanes: dp times 1, x, y, x^2, xy, y^2 (about the region's middle) and
// the colours.  Lane t takes the strips of the eight lanes (g, t).
struct Sums { float m, mx, my, mxx, mxy, myy, r, g, b; };
__device__ __forceinline__ float sum4(float v) {
  v += __shfl_xor_sync(kFull, v, 1);
  return v + __shfl_xor_sync(kFull, v, 2);
}
template <int NPX>
__device__ __forceinline__ Sums sum_entries(const Parked<NPX> &p, int e, int t) {
  using V = typename Share<NPX>::V;
  constexpr int kVecs = Share<NPX>::kVecs, kLanes = Lanes<V>::value;
  V m[kVecs], my[kVecs], myy[kVecs];          // per column of the strip
  float2 rg = make_float2(0.f, 0.f);
  float b = 0.f;
#pragma unroll
  for (int g = 0; g < 8; ++g) {
    const int at = e * kParkStride + 4 * g + t;
    V v[kVecs];
    if constexpr (NPX == 4) { const float4 q = p.dp[at]; v[0] = make_float2(q.x, q.y); v[1] = make_float2(q.z, q.w); } else v[0] = p.dp[at];
    const float y = (float)g - 3.5f;
#pragma unroll
    for (int k = 0; k < kVecs; ++k) {
      m[k] = g ? add(m[k], v[k]) : v[k];
      my[k] = g ? mad(bc<V>(y), v[k], my[k]) : mul(bc<V>(y), v[k]);
      myy[k] = g ? mad(bc<V>(y * y), v[k], myy[k]) : mul(bc<V>(y * y), v[k]);
    }
    rg = __fadd2_rn(rg, p.rg[at]);
    b += p.b[at];
  }
  Sums s = {};
#pragma unroll
  for (int k = 0; k < NPX; ++k) {
    const float x = (float)(NPX * t + k) + 0.5f - 2.f * NPX, c = get(m[k / kLanes], k % kLanes), cy = get(my[k / kLanes], k % kLanes);
    s.m += c; s.mx = fmaf(x, c, s.mx); s.mxx = fmaf(x * x, c, s.mxx);
    s.my += cy; s.mxy = fmaf(x, cy, s.mxy);
    s.myy += get(myy[k / kLanes], k % kLanes);
  }
  s.m = sum4(s.m); s.mx = sum4(s.mx); s.my = sum4(s.my); s.mxx = sum4(s.mxx); s.mxy = sum4(s.mxy); s.myy = sum4(s.myy);
  s.r = sum4(rg.x); s.g = sum4(rg.y); s.b = sum4(b);
  return s;
}
template <int NPX>
struct __align__(16) BwdArea {
  RawEntries raw;
  StagedEntries st;
  Parked<NPX> parked;
};

// Backward: walk each pixel's composited entries back to front.  The transmittance in front of
// an entry is recovered by dividing out (1 - alpha); the light arriving from behind it is summed
// up on the way (both stay relatively accurate: a front-to-back replay that forms that light as
// "final pixel - prefix" cancels badly for deep entries).  Only its product with the pixel's
// upstream gradient is needed, so one scalar per pixel carries it.
//
// What a pixel sends to a Gaussian's conic and mean is linear in dp = dL/d(power) times (1, dx, dy, dx^2, dx dy, dy^2),
// and the opacity gradient needs no sum of its own: alpha = o exp(power) where it is not clamped, so dL/do = (sum of
// dp) / o.  Per entry nine sums over the region's pixels are due, six moments of dp and three colours.  A lane parks its
// pixels' dp and its three colour sums in shared memory as they are; after every eight entries four lanes per entry add
// them up, with the weights x and y (tile-local half-integers: exact) as constants, shift the moments to the Gaussian's
// own centre and send them off with three vector reductions to the g2d row:
// (d colour r, g, b, d opacity) (d conic A, B, C, d mean u) (d mean v, -, -, -).
// Per entry that is 3 stores and about 20 instructions, where a butterfly of the nine sums over the warp took 19 shuffles
// (4 cycles each), as many adds and 14 selects, and the same sums as products on the tensor cores (tf32 operands in two
// terms) took fewer instructions but 105 register operands instead of 55: 215 against 181 us (neither writing zero rows, below).
//
// The kernel leaves the memory idle, so its warps also write what needs no arithmetic: every gradient row that is zero
// because its Gaussian received nothing (in a scene with occlusion most of them: 94 % of the listed Gaussians of a view of
// 1M).  All rows are zeroed here, each warp a slice on its way out (on its way in, the first wave writes them all at once
// and the others' reads wait behind that: 23 us more at 1M); a bit per Gaussian says who received a gradient, and the
// projection and appearance backward works on those alone.  1M Gaussians, 1256 x 828: 259 us without the zero rows -> 207
// with those of the neural model, 62 % of the issue slots, FMA pipe 55 % busy.
//
// What does not depend on the carried state is worked out for four entries at a time, so that the reciprocals, exponentials and
// products of one entry fill the waits of another: 209 -> 199 us at 1M (4108 tiles), 436 -> 381 in a view of 3M over depths of
// 1 to 50 (8160), with 16 warps per SM.  More warps do not help: 24 of 80 registers take as long as 19 of 96, and so do 15
// (padded shared memory); batches of four entries, which would make room for 28, cost 15 to 30 % for their longer sums.
//
// 16 x 8 pixels per warp is best where the launch fills the chip; smaller regions give more warps and cull more where it
// does not, and where a few long lists make the time.  Measured with all three (4 x 8, 8 x 8, 16 x 8; us, zero rows
// included) for scenes of 5000 to 100 000 Gaussians in a box, 300 000 and 1M in clusters and 2M over depths of 1 to 50:
//     tiles    box of 5000     box of 100 000      clusters of 300 000   of 1M             deep
//       64     32  39  69       54  52  84
//      100     33  36  59       83  75 118
//      256     30  31  44       58  55  87
//      576     43  34  40       67  53  75         109 127 195           135 127 227
//     1024     58  40  44       94  69  67         114  98 160           141 110 173
//     1600     78  53  49      133  89  84         139 106 141           169 123 132
//     2500    113  73  64      183 121 108         177 120 128           214 147 153       334 336 642
//     3025    132  84  71      213 138 119         202 134 147           239 159 164       358 395 663
//     3600    154  97  80      248 157 133         228 149 148           268 175 173       361 348 681
//     4225    176 110  89      282 179 151         256 164 157           299 193 185       394 291 579
//     5625                                         317 203 182           370 235 216       475 305 501
// So 4 x 8 up to 64 tiles, and up to 100 with 50 Gaussians per tile; 8 x 8 up to 1000, where the boxes change over, up to 3200
// with 50 per tile, for the clusters (154 000 in 2632: 105 against 122), and up to 6000 with 350, for the deep scenes (3M in
// 8160: 415 against 381).  With
// four views in flight, which fill the chip together, 16 x 8 does less work in all of them: 2126 against 2176 us for an
// iteration on 300 000 in clusters, 2500 tiles.
// kCopies: the flags exist several times (0.6 us more for 300 000 Gaussians, where they do not, if it is asked here).
template <int NPX, bool kCopies>
__global__ void __launch_bounds__(32, NPX == 1 ? 28 : 16) k_blend_bwd(
    CamDev cam, const uint32_t *__restrict__ ranges, const uint32_t *__restrict__ order, const uint32_t *__restrict__ vals,
    const float *__restrict__ mean2d, const float *__restrict__ conic_opacity, const float *__restrict__ color,
    const float *__restrict__ final_T, const uint32_t *__restrict__ n_contrib, const float *__restrict__ dL_dimage,
    float *__restrict__ g2d, GradFlags flags, ZeroRows zeros) {
  using V = typename Share<NPX>::V;
  constexpr int kVecs = Share<NPX>::kVecs, kLanes = Lanes<V>::value, kWarps = Share<NPX>::kWarps, kGroup = 4;
  dependency_wait();
  __shared__ BwdArea<NPX> area;
  const int lane = threadIdx.x;
  if (blockIdx.x >= (unsigned)(cam.gx * cam.gy * kWarps)) {      // a warp without a region, see launch_blend_bwd
    zero_rows(zeros, lane);
    return;
  }
  const int warp = (int)(blockIdx.x % kWarps), tile = (int)__ldg(order + blockIdx.x / kWarps);
  RawEntries &raw = area.raw;
  StagedEntries &st = area.st;
  const int g = lane >> 2, t = lane & 3;
  int rx, ry;
  region_of<NPX>(tile, cam.gx, warp, rx, ry);
  const int px = rx + NPX * t, py = ry + g;
  const uint32_t start = __ldg(ranges + 2 * tile);
  const float fy = (float)py + 0.5f, rx0 = (float)rx + 0.5f, ry0 = (float)ry + 0.5f;
  const size_t plane = (size_t)cam.W * cam.H;
  uint32_t nc[NPX], wmax = 0;
  V fx[kVecs], T[kVecs], Gr[kVecs], Gg[kVecs], Gb[kVecs], S[kVecs];   // S: G . (light from behind)
#pragma unroll
  for (int k = 0; k < NPX; ++k) {
    float tr = 1.f, gr = 0.f, gg = 0.f, gb = 0.f;
    nc[k] = 0u;
    if (px + k < cam.W && py < cam.H) {
      const size_t pix = (size_t)py * cam.W + px + k;
      nc[k] = __ldg(n_contrib + pix);
      tr = __ldg(final_T + pix);
      gr = __ldg(dL_dimage + pix); gg = __ldg(dL_dimage + plane + pix); gb = __ldg(dL_dimage + 2 * plane + pix);
    }
    const int v = k / kLanes, i = k % kLanes;
    put(fx[v], i, (float)(px + k) + 0.5f);
    put(T[v], i, tr); put(Gr[v], i, gr); put(Gg[v], i, gg); put(Gb[v], i, gb);
    put(S[v], i, tr * fmaf(gb, cam.bg[2], fmaf(gg, cam.bg[1], gr * cam.bg[0])));
    wmax = max(wmax, nc[k]);
  }
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) wmax = max(wmax, __shfl_xor_sync(kFull, wmax, s));
  if (wmax == 0 || wmax > __ldg(ranges + 2 * tile + 1) - start) {   // nothing composited in this region
    zero_rows(zeros, lane);
    return;
  }
  uint32_t base = (wmax - 1u) & ~31u;          // first entry of the last piece of 32
  uint32_t id = 0;
  if (base + lane < wmax) {
    id = __ldg(vals + start + base + lane);
    fetch_entry(raw, lane, id, mean2d, conic_opacity, color);
  }
  uint32_t id_next = base >= 32u ? __ldg(vals + start + base - 32u + lane) : 0u;
  for (;; base -= 32u) {
    copies_wait();
    bool clamp;
    const int count = stage_entries<NPX, kGroup>(raw, st, lane, base + lane < wmax, base + lane, id, rx0, ry0, clamp);
    if (base >= 32u) {
      id = id_next;
      fetch_entry(raw, lane, id, mean2d, conic_opacity, color);
      if (base >= 64u) id_next = __ldg(vals + start + base - 64u + lane);
    }
    for (int top = count; top > 0; top = (top - 1) & ~(kBatch - 1)) {
      const int bottom = (top - 1) & ~(kBatch - 1);
      auto work = [&](auto clamped) {
        constexpr bool kClamp = decltype(clamped)::value;
        for (int j = top - kGroup; j >= bottom; j -= kGroup) {
          // What does not depend on the carried state, for a group of entries.  A pixel that did not composite an entry (it
          // lies beyond the pixel's walk, or alpha < 1/255) enters with alpha = 0, for which the reciprocal is 1, every
          // product below is 0 and its carried state is unchanged.
          V a[kGroup][kVecs], odds[kGroup][kVecs], gc[kGroup][kVecs], free[kGroup][kVecs];   // odds: alpha / (1 - alpha)
#pragma unroll
          for (int e = kGroup - 1; e >= 0; --e) {
            const float4 b = st.rest[j + e], c = st.rgb[j + e];
            const uint32_t pos = __float_as_uint(b.z);
            alphas<NPX>(st.shape[j + e], b, fx, fy, a[e]);
#pragma unroll
            for (int k = 0; k < kVecs; ++k) {
#pragma unroll
              for (int i = 0; i < kLanes; ++i) {
                const float x = get(a[e][k], i);
                put(a[e][k], i, select_alpha(x, pos, nc[kLanes * k + i], kClamp ? fminf(kAlphaMax, x) : x));
                if (kClamp) put(free[e][k], i, x > kAlphaMax ? 0.f : 1.f);
              }
              const V d = add(bc<V>(1.f), neg(a[e][k]));
#pragma unroll
              for (int i = 0; i < kLanes; ++i) put(odds[e][k], i, rcp_approx(get(d, i)));
              odds[e][k] = mul(a[e][k], odds[e][k]);
              gc[e][k] = mad(Gb[k], bc<V>(c.z), mad(Gg[k], bc<V>(c.y), mul(Gr[k], bc<V>(c.x))));
            }
          }
          V dp[kGroup][kVecs], cr[kGroup], cg[kGroup], cb[kGroup];
#pragma unroll
          for (int e = kGroup - 1; e >= 0; --e)
#pragma unroll
            for (int k = 0; k < kVecs; ++k) {
              const V w = mul(T[k], odds[e][k]);                // the entry's weight: alpha T / (1 - alpha), T behind it
              if (k == 0) { cr[e] = mul(w, Gr[k]); cg[e] = mul(w, Gg[k]); cb[e] = mul(w, Gb[k]); }
              else { cr[e] = mad(w, Gr[k], cr[e]); cg[e] = mad(w, Gg[k], cg[e]); cb[e] = mad(w, Gb[k], cb[e]); }
              // alpha times d pixel / d alpha = (T c - S) / (1 - alpha), S = everything composited behind this entry.  (The difference
              // first, in one rounding: as w c - odds S it loses what the two have in common, ten times as much in the 3M view.)
              dp[e][k] = mul(odds[e][k], mad(T[k], gc[e][k], neg(S[k])));
              if (kClamp) dp[e][k] = mul(dp[e][k], free[e][k]);     // clamped at 0.99: alpha does not depend on opacity and power
              S[k] = mad(w, gc[e][k], S[k]);
              T[k] = add(T[k], w);                       // in front of it: T / (1 - alpha) = T + w
            }
#pragma unroll
          for (int e = kGroup - 1; e >= 0; --e) park<NPX>(area.parked, j + e - bottom, lane, dp[e], hsum(cr[e]), hsum(cg[e]), hsum(cb[e]));
        }
      };
      if (clamp) work(Flag<true>()); else work(Flag<false>());
      __syncwarp();
      // four lanes per entry
      const int e = lane >> 2, slot = bottom + e;
      const Sums s = sum_entries<NPX>(area.parked, e, t);
      if (slot < top) {
        // moments about the Gaussian's centre from those about the region's: d = (X + ox, Y + oy)
        const float4 sh = st.shape[slot], re = st.rest[slot];
        const float ox = (float)rx + 2.f * NPX + sh.x, oy = (float)ry + 4.f + sh.y;
        const float sx = fmaf(ox, s.m, s.mx), sy = fmaf(oy, s.m, s.my);
        const float sxx = fmaf(ox, s.mx + sx, s.mxx);
        const float sxy = fmaf(oy, sx, fmaf(ox, s.my, s.mxy));
        const float syy = fmaf(oy, s.my + sy, s.myy);
        // the staged factor is the conic's Cholesky factor times sqrt(0.5 log2 e)
        const float A = 2.f * kLn2 * sh.z * sh.z, B = 2.f * kLn2 * sh.z * sh.w, C = 2.f * kLn2 * fmaf(sh.w, sh.w, re.x * re.x);
        const uint32_t gid = __float_as_uint(st.rgb[slot].w);
        float *dst = g2d + (size_t)gid * 12;
        const bool touched = s.m != 0.f || s.mx != 0.f || s.my != 0.f || s.mxx != 0.f || s.mxy != 0.f || s.myy != 0.f || s.r != 0.f ||
                             s.g != 0.f || s.b != 0.f;
        if (touched) {
          if (t == 0) red_add4(dst, s.r, s.g, s.b, __fdividef(s.m, re.y));
          if (t == 1) red_add4(dst + 4, -0.5f * sxx, -sxy, -0.5f * syy, fmaf(A, sx, B * sy));
          if (t == 2) atomicAdd(dst + 8, fmaf(B, sx, C * sy));
          if (t == 3) flags.set<kCopies>(blockIdx.x, gid);
        }
      }
      __syncwarp();                              // the parked values have been read
    }
    if (base == 0u) break;
  }
  zero_rows(zeros, lane);
}

// Measurement only: replay the forward's decisions for regions of 16 x 8 pixels and count, over all pixels, the list
// entries evaluated (until each pixel stopped) and the pairs composited; and per region the entries walked until all of
// its pixels stopped and those among them that none of its live pixels accepted.
// counts[0] += evaluated, counts[1] += composited, counts[2] += (region, entry) steps, counts[3] += steps without a taker.
__global__ void __launch_bounds__(32) k_blend_count(CamDev cam, const uint32_t *__restrict__ ranges, const uint32_t *__restrict__ vals,
                                                    const float *__restrict__ mean2d, const float *__restrict__ conic_opacity,
                                                    const float *__restrict__ color, unsigned long long *__restrict__ counts) {
  constexpr int NPX = 4;
  __shared__ RawEntries raw;
  __shared__ StagedEntries st;
  const int lane = threadIdx.x, tile = blockIdx.x / 2;
  int rx, ry;
  region_of<NPX>(tile, cam.gx, blockIdx.x % 2, rx, ry);
  const int px = rx + NPX * (lane & 3), py = ry + (lane >> 2);
  const float2 fx[2] = {make_float2((float)px + 0.5f, (float)px + 1.5f), make_float2((float)px + 2.5f, (float)px + 3.5f)};
  const uint32_t start = __ldg(ranges + 2 * tile), end = __ldg(ranges + 2 * tile + 1);
  float T[NPX];
  unsigned live = 0;
  unsigned long long evaluated = 0, composited = 0, steps = 0, idle = 0;
#pragma unroll
  for (int k = 0; k < NPX; ++k) {
    T[k] = 1.f;
    if (px + k < cam.W && py < cam.H) live |= 1u << k;
  }
  for (uint32_t base = start; base < end && __any_sync(kFull, live != 0u); base += 32) {
    const int cnt = (int)min(32u, end - base);
    if (lane < cnt) fetch_entry(raw, lane, __ldg(vals + base + lane), mean2d, conic_opacity, color);
    copies_wait();
    bool clamp;
    stage_entries<0, 1>(raw, st, lane, lane < cnt, 0u, 0u, 0.f, 0.f, clamp);
    for (int j = 0; j < cnt; ++j) {
      if (!__any_sync(kFull, live != 0u)) break;
      float2 alpha[2];
      alphas<NPX>(st.shape[j], st.rest[j], fx, (float)py + 0.5f, alpha);
      evaluated += __popc(live);
      bool taken = false;
#pragma unroll
      for (int k = 0; k < NPX; ++k) {
        const float al = get(alpha[k / 2], k % 2);
        if (!((live >> k) & 1u) || al < kAlphaMin) continue;
        taken = true;
        const float n = __fmul_rn(T[k], __fadd_rn(1.f, -fminf(kAlphaMax, al)));
        if (!(n >= kTmin)) { live &= ~(1u << k); continue; }
        T[k] = n;
        ++composited;
      }
      ++steps;
      if (!__any_sync(kFull, taken)) ++idle;
    }
    __syncwarp();
  }
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) {
    evaluated += __shfl_xor_sync(kFull, evaluated, s);
    composited += __shfl_xor_sync(kFull, composited, s);
  }
  if (lane == 0) {
    atomicAdd(counts, evaluated); atomicAdd(counts + 1, composited);
    atomicAdd(counts + 2, steps); atomicAdd(counts + 3, idle);     // the same in every lane
  }
}

}  // namespace

int launch_blend_count(const CamDev &cam, const uint32_t *ranges, const uint32_t *vals, const float *mean2d,
                       const float *conic_opacity, const float *color, unsigned long long *counts, cudaStream_t st) {
  k_blend_count<<<2 * cam.gx * cam.gy, 32, 0, st>>>(cam, ranges, vals, mean2d, conic_opacity, color, counts);
  return 1;
}

int launch_blend_fwd(const CamDev &cam, const uint32_t *ranges, const uint32_t *order, const uint32_t *vals,
                     const float *mean2d,
                     const float *conic_opacity, const float *color, uint32_t *sorted_tiles, float *image, float *final_T,
                     uint32_t *n_contrib, cudaStream_t st) {
  launch_chained(k_blend_fwd, cam.gx * cam.gy * Share<kFwdPixels>::kWarps, 32, 0, st, cam, ranges, order, vals, mean2d, conic_opacity,
                 color, sorted_tiles, image, final_T, n_contrib);
  return 1;
}

int launch_clear(void *p, size_t bytes, cudaStream_t st) {
  const size_t quads = bytes / 16;
  const int blocks = (int)std::min<size_t>(kClearBlocks, (quads + 4 * kClearThreads - 1) / (4 * kClearThreads));
  launch_chained(k_clear, blocks, kClearThreads, 0, st, static_cast<float4 *>(p), quads);
  return 1;
}

int launch_blend_bwd(int64_t n, const CamDev &cam, const uint32_t *ranges, const uint32_t *order, const uint32_t *vals,
                     const float *mean2d,
                     const float *conic_opacity, const float *color, const float *final_T,
                     const uint32_t *n_contrib, const float *dL_dimage, float *g2d, const GradFlags &flags, const ZeroRows &zeros,
                     cudaStream_t st) {
  const int tiles = cam.gx * cam.gy;
  // The rows that start as zeros are shared out over all warps of the grid.  An image of few tiles does not have the warps
  // for that - 16 x 16 pixels of a scene of 3M have 8, and 708 MB of SH gradients: 1473 us, now 120 - so warps without a
  // region make up what is missing to two per SM, each with 4 KB at least.  (One per SM: 121 us for 16 x 16 pixels, 134 for
  // 64 x 64 of the same scene; two 120 and 120, four 121 and 123, eight 126 and 126, sixteen 129 and 137.)
  uint64_t quads = 0;
  for (int k = 0; k < zeros.count; ++k) quads += zeros.floats[k] >> 2;
  const int zero_warps = (int)std::min<uint64_t>(kZeroWarps, quads / 256);
  auto launch = [&](auto kernel, int warps) {
    ZeroRows z = zeros;
    const int ctas = std::max(tiles * warps, zero_warps);
    for (int k = 0; k < z.count; ++k) z.slice[k] = (uint32_t)(((z.floats[k] >> 2) + ctas - 1) / ctas);
    launch_chained(kernel, ctas, 32, 0, st, cam, ranges, order, vals, mean2d, conic_opacity, color, final_T, n_contrib, dL_dimage, g2d, flags, z);
  };
  // (the measurements behind the lines are at the kernel)
  auto pick = [&](auto copies) {
    constexpr bool kCopies = decltype(copies)::value;
    const auto per_tile = [&](int64_t least) { return n >= least * tiles; };
    if (tiles <= 64 || (tiles <= 100 && per_tile(50))) launch(k_blend_bwd<1, kCopies>, Share<1>::kWarps);
    else if (tiles <= 1000 || (tiles <= 3200 && per_tile(50)) || (tiles <= 6000 && per_tile(350))) launch(k_blend_bwd<2, kCopies>, Share<2>::kWarps);
    else launch(k_blend_bwd<4, kCopies>, Share<4>::kWarps);
  };
  if (flags.copies > 1) pick(Flag<true>()); else pick(Flag<false>());
  return 1;
}

}  // namespace gs
