// Device algebra of the embedded deformation (see embedded_kernels.cu), shared by
// the per-launch kernels and the resident PCG loop (resident.cu).
#pragma once

#include "mesh_algebra.cuh"

namespace optgb {

constexpr int NXE = 12;   // unknowns per vertex
constexpr int NME = 10;   // distinct-diagonal planes
constexpr int KBE = 6;    // neighbour indices fetched ahead per vertex (icosphere degree 5 / 6)

// Visits the out-edge targets e1[o0 .. o1) (or in-edge sources) of a vertex:
// the first KBE indices are loaded together before any neighbour record is
// needed, the rest of a longer row one by one.
template <typename F>
__device__ __forceinline__ void for_list(const int* __restrict__ idx, int o0, int o1, F&& f) {
  int j[KBE];
#pragma unroll
  for (int t = 0; t < KBE; ++t) j[t] = o0 + t < o1 ? __ldg(idx + o0 + t) : 0;
#pragma unroll
  for (int t = 0; t < KBE; ++t)
    if (o0 + t < o1) f(j[t]);
  for (int k = o0 + KBE; k < o1; ++k) f(__ldg(idx + k));
}

__device__ __forceinline__ int mplane_e(int c) { return c < 3 ? 0 : c - 2; }

__device__ __forceinline__ void load12(const float4* rec, int v, float (&o)[NXE]) {
  const float4 a = rec[3 * (size_t)v], b = rec[3 * (size_t)v + 1], c = rec[3 * (size_t)v + 2];
  o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w;
  o[4] = b.x; o[5] = b.y; o[6] = b.z; o[7] = b.w;
  o[8] = c.x; o[9] = c.y; o[10] = c.z; o[11] = c.w;
}
__device__ __forceinline__ void store12(float4* rec, int v, const float (&o)[NXE]) {
  rec[3 * (size_t)v] = make_float4(o[0], o[1], o[2], o[3]);
  rec[3 * (size_t)v + 1] = make_float4(o[4], o[5], o[6], o[7]);
  rec[3 * (size_t)v + 2] = make_float4(o[8], o[9], o[10], o[11]);
}

// The six constraint values (c0.c1, c0.c2, c1.c2, c0.c0 - 1, c1.c1 - 1,
// c2.c2 - 1) of the matrix m[9] (row-major), unscaled.
__device__ __forceinline__ void col_constraints(const float* m, float (&f)[6]) {
  float d01 = 0.f, d02 = 0.f, d12 = 0.f, d00 = 0.f, d11 = 0.f, d22 = 0.f;
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const float c0 = m[3 * r], c1 = m[3 * r + 1], c2 = m[3 * r + 2];
    d01 += c0 * c1; d02 += c0 * c2; d12 += c1 * c2;
    d00 += c0 * c0; d11 += c1 * c1; d22 += c2 * c2;
  }
  f[0] = d01; f[1] = d02; f[2] = d12; f[3] = d00 - 1.f; f[4] = d11 - 1.f; f[5] = d22 - 1.f;
}

// Linearised constraints J_rot t of a matrix direction t[9] at m[9], unscaled
// (explicit multiply-adds: the same bits in every kernel).
__device__ __forceinline__ void col_constraints_lin(const float* m, const float* t, float (&f)[6]) {
  float a01 = 0.f, a02 = 0.f, a12 = 0.f, a00 = 0.f, a11 = 0.f, a22 = 0.f;
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const float c0 = m[3 * r], c1 = m[3 * r + 1], c2 = m[3 * r + 2];
    const float t0 = t[3 * r], t1 = t[3 * r + 1], t2 = t[3 * r + 2];
    a01 = fmaf(c1, t0, fmaf(c0, t1, a01));
    a02 = fmaf(c2, t0, fmaf(c0, t2, a02));
    a12 = fmaf(c2, t1, fmaf(c1, t2, a12));
    a00 = fmaf(c0, t0, a00);
    a11 = fmaf(c1, t1, a11);
    a22 = fmaf(c2, t2, a22);
  }
  f[0] = a01; f[1] = a02; f[2] = a12; f[3] = 2.f * a00; f[4] = 2.f * a11; f[5] = 2.f * a22;
}

// out[9] += J_rot^T y for the six constraint values y (unscaled).
__device__ __forceinline__ void col_constraints_t(const float* m, const float (&y)[6], float* out) {
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const float c0 = m[3 * r], c1 = m[3 * r + 1], c2 = m[3 * r + 2];
    out[3 * r] = fmaf(c1, y[0], fmaf(c2, y[1], fmaf(2.f * c0, y[3], out[3 * r])));
    out[3 * r + 1] = fmaf(c0, y[0], fmaf(c2, y[2], fmaf(2.f * c1, y[4], out[3 * r + 1])));
    out[3 * r + 2] = fmaf(c0, y[1], fmaf(c1, y[2], fmaf(2.f * c2, y[5], out[3 * r + 2])));
  }
}

// Terms of one neighbour in applyJTJ at a vertex (direction pi, rest position
// ui), added up in the order of the neighbour list by every kernel: with w = U_i -
// U_j and P the matrix part, f = [(p_i - p_j) - P_i w] (own residual) + [(p_i -
// p_j) - P_j w] (incoming, negated), and g, the matrix rows w_reg J p w^T of the
// own one.
__device__ __forceinline__ void ed_terms(float wreg, const float (&pi)[NXE], const float4& ui, const float (&pj)[NXE],
                                         const float4& uj, bool own, bool in, float (&f)[3], float (&g)[9]) {
  const float wv[3] = {ui.x - uj.x, ui.y - uj.y, ui.z - uj.z};
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const float d = pi[r] - pj[r];
    f[r] = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) g[3 * r + c] = 0.f;
    if (own) {
      const float jp = d - fmaf(pi[3 + 3 * r], wv[0], fmaf(pi[4 + 3 * r], wv[1], __fmul_rn(pi[5 + 3 * r], wv[2])));
      f[r] = jp;
      const float t = __fmul_rn(wreg, jp);
#pragma unroll
      for (int c = 0; c < 3; ++c) g[3 * r + c] = __fmul_rn(t, wv[c]);
    }
    if (in)
      f[r] += d - fmaf(pj[3 + 3 * r], wv[0], fmaf(pj[4 + 3 * r], wv[1], __fmul_rn(pj[5 + 3 * r], wv[2])));
  }
}

// The edge rows of applyJTJ at vertex i: f (displacement rows / w_reg) and g
// (matrix rows, to be subtracted).  Where every edge is given both ways (pr.sym) a
// neighbour is visited once for both its residuals.  lst: the out-edge targets
// (pr.e1 or a copy of a run of it); load(j, p): vertex j's direction.
template <typename Load>
__device__ __forceinline__ void ed_gather(const MeshProb& pr, int i, const int* lst, int o0, int o1,
                                          const float (&pi)[NXE], const float4& ui, Load load, float (&f)[3],
                                          float (&g)[9]) {
  const bool sym = pr.sym != 0;
  auto edge = [&](int j, bool own, bool in) {
    float pj[NXE], tf[3], tg[9];
    load(j, pj);
    ed_terms(pr.w_reg, pi, ui, pj, __ldg(pr.grec + j), own, in, tf, tg);
#pragma unroll
    for (int c = 0; c < 3; ++c) f[c] += tf[c];
#pragma unroll
    for (int c = 0; c < 9; ++c) g[c] += tg[c];
  };
  for (int k = o0; k < o1; ++k) edge(lst[k], true, sym);
  if (!sym)
    for (int k = pr.irow[i]; k < pr.irow[i + 1]; ++k) edge(pr.isrc[k], false, true);
}

// The rows of applyJTJ without damping from the edge sums: q = w_reg f (+ w_fit p
// on a handle), -g, and the constraint rows w_rot J_rot^T J_rot p.
__device__ __forceinline__ void ed_rows(const MeshProb& pr, int i, const float (&pi)[NXE], const float (&f)[3],
                                        const float (&g)[9], bool handle, float (&q)[NXE]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    q[c] = __fmul_rn(pr.w_reg, f[c]);
    if (handle) q[c] = fmaf(pr.w_fit, pi[c], q[c]);
  }
  float m9[9], y[6], t[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    m9[k] = pr.x[(3 + k) * (long long)pr.Vp + i];
    t[k] = 0.f;
  }
  col_constraints_lin(m9, pi + 3, y);
#pragma unroll
  for (int k = 0; k < 6; ++k) y[k] *= pr.w_rot;
  col_constraints_t(m9, y, t);
#pragma unroll
  for (int k = 0; k < 9; ++k) q[3 + k] = t[k] - g[k];
}

}  // namespace optgb
