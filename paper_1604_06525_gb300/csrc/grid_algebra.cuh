// Per-pixel arithmetic of applyJTJ on the grids, one pixel per thread, in the
// roundings and the order of the packed 128-pixel-tile kernels (grid_kernels.cu):
// whichever kernel computes a pixel's row, it computes the same bits.
#pragma once

#include "opt_internal.cuh"

namespace optgb {

// What a neighbour pair of the warp needs of a pixel: direction, cos / sin of
// theta, UrShape.
struct WarpPix {
  float px, py, pt, c, s, ux, uy;
};

// Adds the grouped own + incoming rows of the pair (i, j) (the scalar form of
// pair2): with v = U_i - U_j, a = p_i - p_j and G_k = (s_k v_x + c_k v_y,
// s_k v_y - c_k v_x),
//   q_d,i += 2 a + G_i p_t,i + G_j p_t,j,  q_t,i += G_i . (a + G_i p_t,i).
__device__ __forceinline__ void warp_pair(const WarpPix& o, const WarpPix& n, float& ax, float& ay, float& at) {
  const float vx = __fsub_rn(o.ux, n.ux), vy = __fsub_rn(o.uy, n.uy), nvx = __fsub_rn(n.ux, o.ux);
  const float a = __fsub_rn(o.px, n.px), b = __fsub_rn(o.py, n.py);
  const float gix = __fmaf_rn(o.s, vx, __fmul_rn(o.c, vy)), giy = __fmaf_rn(o.c, nvx, __fmul_rn(o.s, vy));
  const float gjx = __fmaf_rn(n.s, vx, __fmul_rn(n.c, vy)), gjy = __fmaf_rn(n.c, nvx, __fmul_rn(n.s, vy));
  const float tx = __fmaf_rn(gix, o.pt, a), ty = __fmaf_rn(giy, o.pt, b);
  ax = __fadd_rn(__fadd_rn(tx, __fmaf_rn(gjx, n.pt, a)), ax);
  ay = __fadd_rn(__fadd_rn(ty, __fmaf_rn(gjy, n.pt, b)), ay);
  at = __fadd_rn(__fmaf_rn(gix, tx, __fmul_rn(giy, ty)), at);
}

// Poisson: S_i p_i - 2 (p_L + (p_R + (p_U + p_D))) with one rounding of the product
// and difference, the directions zero off the free pixels.
__device__ __forceinline__ float pois_row(float S, float p, float l, float r, float u, float d) {
  const float n = __fadd_rn(l, __fadd_rn(r, __fadd_rn(u, d)));
  return __fmaf_rn(S, p, __fmul_rn(-2.f, n));
}

}  // namespace optgb
