// Device algebra of the warp on a graph (see graph2d_kernels.cu), shared by the
// per-launch kernels and the resident PCG loop (resident.cu).
#pragma once

#include "mesh_algebra.cuh"

namespace optgb {

// Terms of one neighbour in applyJTJ / w_reg at a vertex with direction pi = (dx,
// dy, theta) and geometry gi = (U, cos, sin), added up in the order of the
// neighbour list by every kernel.  With v = U_i - U_j, d = p_i - p_j and G_k = (s_k
// v_x + c_k v_y, s_k v_y - c_k v_x): own J p / s_w = d + G_i p_t,i, the incoming
// one, negated, d + G_j p_t,j.
__device__ __forceinline__ void wg_terms(const float4& pi, const float4& gi, const float4& pj, const float4& gj,
                                         bool own, bool in, float (&f)[3]) {
  const float vx = gi.x - gj.x, vy = gi.y - gj.y;
  const float dx = pi.x - pj.x, dy = pi.y - pj.y;
  f[0] = f[1] = f[2] = 0.f;
  if (own) {
    const float Gx = fmaf(gi.w, vx, __fmul_rn(gi.z, vy)), Gy = fmaf(gi.w, vy, __fmul_rn(-gi.z, vx));
    f[0] = fmaf(Gx, pi.z, dx);
    f[1] = fmaf(Gy, pi.z, dy);
    f[2] = fmaf(Gx, f[0], __fmul_rn(Gy, f[1]));
  }
  if (in) {
    const float Gx = fmaf(gj.w, vx, __fmul_rn(gj.z, vy)), Gy = fmaf(gj.w, vy, __fmul_rn(-gj.z, vx));
    f[0] += fmaf(Gx, pj.z, dx);
    f[1] += fmaf(Gy, pj.z, dy);
  }
}

// The edge rows of applyJTJ / w_reg at vertex i.  Edges given both ways (pr.sym)
// are visited once.  lst: the out-edge targets; load(j): vertex j's direction.
template <typename Load>
__device__ __forceinline__ void wg_gather(const MeshProb& pr, int i, const int* lst, int o0, int o1, const float4& pi,
                                          const float4& gi, Load load, float (&f)[3]) {
  const bool sym = pr.sym != 0;
  auto edge = [&](int j, bool own, bool in) {
    float t[3];
    wg_terms(pi, gi, load(j), __ldg(pr.grec + j), own, in, t);
#pragma unroll
    for (int c = 0; c < 3; ++c) f[c] += t[c];
  };
  int j4[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) j4[t] = o0 + t < o1 ? lst[o0 + t] : 0;
#pragma unroll
  for (int t = 0; t < 4; ++t)
    if (o0 + t < o1) edge(j4[t], true, sym);
  for (int k = o0 + 4; k < o1; ++k) edge(lst[k], true, sym);
  if (!sym)
    for (int k = pr.irow[i]; k < pr.irow[i + 1]; ++k) edge(pr.isrc[k], false, true);
}

// The rows without damping from the edge sums.
__device__ __forceinline__ void wg_rows(const MeshProb& pr, const float (&f)[3], const float (&p)[3], bool handle,
                                        float (&q)[3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    q[k] = __fmul_rn(pr.w_reg, f[k]);
    if (k < 2 && handle) q[k] = fmaf(pr.w_fit, p[k], q[k]);
  }
}

}  // namespace optgb
