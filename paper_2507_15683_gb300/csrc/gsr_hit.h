// Which warps of a tile a Gaussian can reach: the alpha-floor test of a pixel and
// its conservative form for a block of pixels. Plain C++ too, so that the second
// can be checked against the first without a GPU.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#ifdef __CUDACC__
#define GSR_FN __device__ __forceinline__
#else
#define GSR_FN inline
// rounded operations of the host (to be compiled without contraction)
inline float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __fdividef(float a, float b) { return a / b; }
inline float __logf(float a) { return logf(a); }
#endif

namespace gsr {

constexpr int kWarps = 8;  // of a tile

// -0.5 (A dx^2 + C dy^2) - B dx dy with one fixed rounding sequence, shared by
// the forward and backward kernels so that both take identical skip decisions.
GSR_FN float gs_power(float A, float B, float C, float dx, float dy) {
  const float q = __fmaf_rn(C, __fmul_rn(dy, dy), __fmul_rn(A, __fmul_rn(dx, dx)));
  return __fmaf_rn(-B, __fmul_rn(dx, dy), __fmul_rn(-0.5f, q));
}

// Threshold of the alpha-floor test as an ellipse: o exp(power) >= 1/255 with
// power = -q/2, q(d) = A dx^2 + 2 B dx dy + C dy^2, needs q <= 2 ln(255 o).
// Margins (1 % + 0.01 on the log, 0.1 % + 1e-3 on the threshold) cover the
// fp32 evaluation of the per-pixel test; -1 marks a Gaussian whose opacity
// cannot reach the floor anywhere.
GSR_FN float floor_threshold(float o) {
  const float Lp = __logf(255.0f * o) * 1.01f + 0.01f;
  return Lp > 0.0f ? 2.0f * Lp * 1.001f + 1e-3f : -1.0f;
}

// Bit w set when a staged Gaussian (centre a.xy in tile-local pixels, conic
// A = a.z, B = a.w, C) can reach the floor at some pixel centre of warp w's 8 x 4
// block, for the warps w0 <= w < w1: the minimum over the block of the
// positive-definite quadratic q is at most thr. If not, every pixel of the warp
// would skip the Gaussian, so the warp skips it without changing any result.
// The minimum is q at the centre (0) when the centre is inside, and otherwise
// lies on an edge that faces the centre: moving from any other point of the
// block towards the centre lowers q. So a block takes at most two edges, the
// facing vertical one (whose terms are shared by the four blocks of a column of
// blocks) and the facing horizontal one (shared by the two of a row). Computed
// once per staged Gaussian and warp block by a staging thread. Taking the best
// of all four edges per block, behind a bounding-box test, cost about 450 warp
// instructions for 32 entries, 12 % of the forward pass: with this and the
// exponential beside it, 162 -> 155 us (1080p forward), 452 -> 425 us (tangent pass).
//
// binary32: q is a sum of terms that cancel, here and in gs_power. With u = 2^-24
// and S = A dx^2 + C dy^2 (>= 2 |B dx dy|), each evaluation is within 10 u S of
// the exact q of the staged numbers (offset, products and sums rounded once
// each), and a form that the determinant test passes although it is slightly
// indefinite is within 2 u S of a semidefinite one. So thr is raised by 2^-19
// times S at the tile's farthest point, 32 u S for 22. Without it, long thin
// splats (minor sigma 0.55 to 2) lost blending blocks: 0.006 % at a major sigma
// of 300 to 1,000 pixels, 0.35 % at 1,000 to 3,000. Up to 20 pixels the margin
// adds 0.003 % to the blocks that are walked.
template <int W0 = 0, int W1 = kWarps>
GSR_FN uint32_t warp_hit_mask(float4 a, float C, float thr, int w0 = W0, int w1 = W1) {
  if (!(thr > 0.0f)) return 0u;
  const float A = a.z, B = a.w;
  const float ex = fabsf(a.x - 8.0f) + 7.5f, ey = fabsf(a.y - 8.0f) + 7.5f;  // to the tile's farthest pixel centre
  thr = fmaxf(thr, fmaf(A * ex * ex + C * ey * ey, 0x1p-19f, thr));
  if (!(A > 0.0f) || !(C > 0.0f) || !(A * C - B * B > 0.0f)) return (1u << w1) - (1u << w0);
  const float kx = -__fdividef(B, C), ky = -__fdividef(B, A);  // best dy on a vertical edge per dx, best dx on a horizontal one per dy
  uint32_t mask = 0u;
#pragma unroll
  for (int cx = 0; cx < 2; ++cx) {
    const float dxl = (float)(8 * cx) + 0.5f - a.x, dxh = dxl + 7.0f;
    const float fx = dxl > 0.0f ? dxl : fminf(dxh, 0.0f);  // facing vertical edge, 0: the centre is between the edges
    const float vy = kx * fx, va = A * fx * fx, vb = 2.0f * B * fx;
#pragma unroll
    for (int ry = 0; ry < 4; ++ry) {
      const int wv = 2 * ry + cx;
      if (wv < w0 || wv >= w1) continue;
      const float dyl = (float)(4 * ry) + 0.5f - a.y, dyh = dyl + 3.0f;
      const float fy = dyl > 0.0f ? dyl : fminf(dyh, 0.0f);
      // on the vertical edge (for fx = 0 this is q at dx = 0: an upper bound of the minimum, and 0 inside)
      const float y = fminf(fmaxf(vy, dyl), dyh);
      float best = fmaf(fmaf(C, y, vb), y, va);
      // on the horizontal edge
      const float x = fminf(fmaxf(ky * fy, dxl), dxh);
      best = fminf(best, fmaf(fmaf(A, x, 2.0f * B * fy), x, C * fy * fy));
      if (best <= thr) mask |= 1u << wv;
    }
  }
  return mask;
}

}  // namespace gsr
