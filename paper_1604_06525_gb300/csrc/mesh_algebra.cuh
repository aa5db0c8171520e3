// Device algebra of the ARAP mesh and volume energies (see graph_kernels.cu for
// the derivation): rotations, per-vertex records, neighbour walks and the
// gather of one applyJTJ, shared by the per-launch kernels and the resident
// PCG loop (resident.cu).
#pragma once

#include "opt_internal.cuh"

namespace optgb {

__device__ __forceinline__ int handle_of(const MeshProb& pr, int v) {
  const int t = v / VT;
  for (int h = pr.hbeg[t]; h < pr.hbeg[t + 1]; ++h)
    if (pr.hpix[h] == v) return h;
  return -1;
}

constexpr int KB = 6;             // neighbour indices fetched ahead per vertex (icosphere degree 5 / 6)
// The 7-point stencil of a W x H x D voxel grid (volumetric problems): the
// six neighbour offsets in ascending order -- the order the sorted edge lists
// give -- and which of them lie inside the grid.
struct Stencil3 {
  int off[6];
  bool ok[6];
};
__device__ __forceinline__ Stencil3 stencil3(const MeshProb& pr, int i) {
  const int W = pr.gw, H = pr.gh, WH = W * H;
  const int x = i % W, y = (i / W) % H, z = i / WH;
  Stencil3 st;
  st.off[0] = -WH; st.ok[0] = z > 0;
  st.off[1] = -W;  st.ok[1] = y > 0;
  st.off[2] = -1;  st.ok[2] = x > 0;
  st.off[3] = 1;   st.ok[3] = x + 1 < W;
  st.off[4] = W;   st.ok[4] = y + 1 < H;
  st.off[5] = WH;  st.ok[5] = z + 1 < pr.gd;
  return st;
}

// --- rotations -------------------------------------------------------------
struct GeoRec {
  float U[3];
  float q[4];       // unit quaternion (w, x, y, z) of R(A)
};
__device__ __forceinline__ GeoRec load_geo(const float4* __restrict__ grec, int v) {
  const float4 a = __ldg(grec + 2 * (size_t)v), b = __ldg(grec + 2 * (size_t)v + 1);
  GeoRec g;
  g.U[0] = a.x; g.U[1] = a.y; g.U[2] = a.z;
  g.q[0] = a.w; g.q[1] = b.x; g.q[2] = b.y; g.q[3] = b.z;
  return g;
}
// (cos a_y, sin a_y, cos a_z, sin a_z) of a vertex: what its axes beta_m need
__device__ __forceinline__ float4 load_axes(const MeshProb& pr, int v) {
  return __ldg(pr.grec + 2 * (size_t)pr.V + v);
}
// Quaternion and axes of Rz(az) Ry(ay) Rx(ax), from the half angles.
__device__ __forceinline__ void angles_to_quat(const float* a, float (&q)[4], float4& axes) {
  float sx, cx, sy, cy, sz, cz;
  sincosf(0.5f * a[0], &sx, &cx);
  sincosf(0.5f * a[1], &sy, &cy);
  sincosf(0.5f * a[2], &sz, &cz);
  const float cc = cy * cz, ss = sy * sz, sc = sy * cz, cs = cy * sz;
  q[0] = fmaf(cx, cc, sx * ss);
  q[1] = fmaf(sx, cc, -cx * ss);
  q[2] = fmaf(cx, sc, sx * cs);
  q[3] = fmaf(cx, cs, -sx * sc);
  axes = make_float4(fmaf(-2.f * sy, sy, 1.f), 2.f * sy * cy, fmaf(-2.f * sz, sz, 1.f), 2.f * sz * cz);
}
// D = R - I (no cancellation for small angles)
__device__ __forceinline__ void quat_delta_matrix(const float (&q)[4], float (&D)[3][3]) {
  const float w = q[0], x2 = 2.f * q[1], y2 = 2.f * q[2], z2 = 2.f * q[3];
  const float xx = __fmul_rn(x2, q[1]), yy = __fmul_rn(y2, q[2]), zz = __fmul_rn(z2, q[3]);
  D[0][0] = -(yy + zz);                 D[0][1] = fmaf(x2, q[2], -z2 * w);  D[0][2] = fmaf(x2, q[3], y2 * w);
  D[1][0] = fmaf(x2, q[2], z2 * w);     D[1][1] = -(xx + zz);               D[1][2] = fmaf(y2, q[3], -x2 * w);
  D[2][0] = fmaf(x2, q[3], -y2 * w);    D[2][1] = fmaf(y2, q[3], x2 * w);   D[2][2] = -(xx + yy);
}
__device__ __forceinline__ void mat_vec(const float (&D)[3][3], const float (&v)[3], float (&o)[3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i) o[i] = fmaf(D[i][0], v[0], fmaf(D[i][1], v[1], D[i][2] * v[2]));
}
// (R - I) v of a quaternion used once: t = 2 u x v, then w t + u x t
__device__ __forceinline__ void quat_delta(const float (&q)[4], const float (&v)[3], float (&o)[3]) {
  const float x2 = 2.f * q[1], y2 = 2.f * q[2], z2 = 2.f * q[3];
  const float t0 = fmaf(y2, v[2], -z2 * v[1]), t1 = fmaf(z2, v[0], -x2 * v[2]), t2 = fmaf(x2, v[1], -y2 * v[0]);
  o[0] = fmaf(q[0], t0, fmaf(q[2], t2, -q[3] * t1));
  o[1] = fmaf(q[0], t1, fmaf(q[3], t0, -q[1] * t2));
  o[2] = fmaf(q[0], t2, fmaf(q[1], t1, -q[2] * t0));
}
// o -= a x b
__device__ __forceinline__ void sub_cross(float (&o)[3], const float (&a)[3], const float (&b)[3]) {
  o[0] = fmaf(-a[1], b[2], fmaf(a[2], b[1], o[0]));
  o[1] = fmaf(-a[2], b[0], fmaf(a[0], b[2], o[1]));
  o[2] = fmaf(-a[0], b[1], fmaf(a[1], b[0], o[2]));
}
// o += a x b
__device__ __forceinline__ void add_cross(float (&o)[3], const float (&a)[3], const float (&b)[3]) {
  o[0] = fmaf(a[1], b[2], fmaf(-a[2], b[1], o[0]));
  o[1] = fmaf(a[2], b[0], fmaf(-a[0], b[2], o[1]));
  o[2] = fmaf(a[0], b[1], fmaf(-a[1], b[0], o[2]));
}
// w = sum_m p_m beta_m
__device__ __forceinline__ void angular_velocity(const float4& ax, float pa, float pb, float pc, float (&w)[3]) {
  const float h = pa * ax.x;
  w[0] = fmaf(ax.z, h, -ax.w * pb);
  w[1] = fmaf(ax.w, h, ax.z * pb);
  w[2] = fmaf(-ax.y, pa, pc);
}
// (beta_x . t, beta_y . t, beta_z . t)
__device__ __forceinline__ void axis_rows(const float4& ax, const float (&t)[3], float (&o)[3]) {
  const float t1 = fmaf(ax.z, t[0], ax.w * t[1]);
  o[0] = fmaf(ax.x, t1, -ax.y * t[2]);
  o[1] = fmaf(ax.z, t[1], -ax.w * t[0]);
  o[2] = t[2];
}
// o_m += |beta_m x y|^2
__device__ __forceinline__ void axis_squares(const float4& ax, const float (&y)[3], float (&o)[3]) {
  const float y1 = fmaf(ax.z, y[0], ax.w * y[1]), y2 = fmaf(ax.z, y[1], -ax.w * y[0]);
  const float t = fmaf(ax.y, y1, ax.x * y[2]);
  o[0] = fmaf(t, t, fmaf(y2, y2, o[0]));
  o[1] = fmaf(y1, y1, fmaf(y[2], y[2], o[1]));
  o[2] = fmaf(y1, y1, fmaf(y2, y2, o[2]));
}

// Records written in the same launch chain (plain loads, not the read-only
// path): a displacement, or (p_d, w).
__device__ __forceinline__ void load_vec3(const float4* vrec, int v, float (&o)[3]) {
  const float4 a = vrec[2 * (size_t)v];
  o[0] = a.x; o[1] = a.y; o[2] = a.z;
}
__device__ __forceinline__ void load_pw(const float4* vrec, int v, float (&p)[3], float (&w)[3]) {
  const float4 a = vrec[2 * (size_t)v], b = vrec[2 * (size_t)v + 1];
  p[0] = a.x; p[1] = a.y; p[2] = a.z;
  w[0] = a.w; w[1] = b.x; w[2] = b.y;
}

// Runs edge(j, own, in) for the neighbours j of vertex i: own for the far end of
// every out-edge, in for the source of every in-edge.  Where both lists are
// equal (every undirected edge given both ways: pr.sym, and the voxel stencil)
// each neighbour is visited once with both; the first KB neighbour indices are
// loaded together.
// lst: the out-edge targets (a copy of a run of them in shared memory, or
// pr.e1), of which vertex i has [o0, o1).
template <bool G3, typename Edge>
__device__ __forceinline__ void for_neighbours(const MeshProb& pr, int i, const int* lst, int o0, int o1, Edge edge) {
  if (G3) {
    const Stencil3 st = stencil3(pr, i);
#pragma unroll
    for (int t = 0; t < 6; ++t)
      if (st.ok[t]) edge(i + st.off[t], true, true);
    return;
  }
  const bool sym = pr.sym != 0;
  int jo[KB];
#pragma unroll
  for (int t = 0; t < KB; ++t) jo[t] = o0 + t < o1 ? lst[o0 + t] : 0;
#pragma unroll
  for (int t = 0; t < KB; ++t)
    if (o0 + t < o1) edge(jo[t], true, sym);
  // longer rows; then, one-way edges, the in-edge list
  const int lists = sym ? 1 : 2;
  for (int l = 0; l < lists; ++l) {
    const int k1 = l ? pr.irow[i + 1] : o1;
    const int* src = l ? pr.isrc : lst;
#pragma unroll 1
    for (int k = l ? pr.irow[i] : o0 + KB; k < k1; ++k) edge(src[k], l == 0, sym || l == 1);
  }
}

// Terms of one neighbour in applyJTJ at a vertex (direction pd, w; geometry U and
// D = R - I), added up in the order of the neighbour list by every kernel, so
// that they compute the same bits: f, J_e p / s_w of the out-edge minus that of
// the in-edge, and tq, the torque of the out-edge.  The neighbour: direction (pj,
// wj), geometry gj.
__device__ __forceinline__ void mesh_terms(const float (&pd)[3], const float (&w)[3], const float (&U)[3],
                                           const float (&D)[3][3], const float (&pj)[3], const float (&wj)[3],
                                           const GeoRec& gj, bool own, bool in, float (&f)[3], float (&tq)[3]) {
  float d[3], v[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    d[c] = pd[c] - pj[c];
    v[c] = U[c] - gj.U[c];
    f[c] = 0.f;
    tq[c] = 0.f;
  }
  if (own) {
    // d - w x y, y = R_i v
    float y[3], t[3] = {d[0], d[1], d[2]};
    mat_vec(D, v, y);
#pragma unroll
    for (int c = 0; c < 3; ++c) y[c] += v[c];
    sub_cross(t, w, y);
#pragma unroll
    for (int c = 0; c < 3; ++c) f[c] = t[c];
    add_cross(tq, y, t);
  }
  if (in) {
    // the in-edge's residual, negated: d - w_j x (R_j v)
    float y[3], t[3] = {d[0], d[1], d[2]};
    quat_delta(gj.q, v, y);
#pragma unroll
    for (int c = 0; c < 3; ++c) y[c] += v[c];
    sub_cross(t, wj, y);
#pragma unroll
    for (int c = 0; c < 3; ++c) f[c] += t[c];
  }
}

// The edge rows of applyJTJ at vertex i.  load(j, p, w): vertex j's direction.
template <bool G3, typename Load>
__device__ __forceinline__ void mesh_gather(const MeshProb& pr, int i, const int* lst, int o0, int o1,
                                            const float (&pd)[3], const float (&wi)[3], const GeoRec& gi, Load load,
                                            float (&f)[3], float (&tq)[3]) {
  float D[3][3];
  quat_delta_matrix(gi.q, D);
  for_neighbours<G3>(pr, i, lst, o0, o1, [&](int j, bool own, bool in) {
    const GeoRec gj = load_geo(pr.grec, j);
    float pj[3], wj[3], tf[3], tt[3];
    load(j, pj, wj);
    mesh_terms(pd, wi, gi.U, D, pj, wj, gj, own, in, tf, tt);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      f[c] += tf[c];
      tq[c] += tt[c];
    }
  });
}

}  // namespace optgb
