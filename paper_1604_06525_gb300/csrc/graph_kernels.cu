// Matrix-free graph kernels (Sec. 4.1 "Graph-based Array Access", Sec. 5.3.2).
//
// The paper maps one thread to one edge residual and scatters its
// contributions to the rows of the two vertices with atomics (Fig. 11).  Here
// every row of J^T F, diag(J^T J) and J^T J p is gathered instead: one thread
// owns one vertex i and walks
//   * its out-edges (i, j) (edges sorted by (v0, v1) -> CSR rows): the
//     residual's own rows at i (displacement and angles), and
//   * its in-edges (j, i) (a transposed list built at planning): the
//     residual's rows at its far end, the displacement rows of i,
// so each edge residual is evaluated twice (once from each end) and no
// atomic or cross-thread sum is needed; every row is summed in a fixed
// order.  What a thread reads of a neighbour sits in two per-vertex records
// (array of structures, a few 32-byte sectors per gather instead of one
// sector per plane):
//   grec[v] = (U_x, U_y, U_z, q_w), (q_x, q_y, q_z, 0): rest position and the
//             rotation R(A_v) as a unit quaternion; behind the 2 V of them, own
//             vertex only, (cos a_y, sin a_y, cos a_z, sin a_z)
//                                                   written by PCGInit's vertex pass
//   vrec[v] = x's displacement in PCGInit; (p_d, w) in applyJTJ, 2 float4;
//             (x_d, U, delta_d but for its last component) in the energies, 2 float4
//
// ARAP mesh algebra per edge e = (a, b), v = U_a - U_b, d = O - U:
//   r_e       = s_w [(d_a - d_b) + (v - R(A_a) v)]              (= Fig. 25)
//   dr/dd_a   = s_w I,  dr/dd_b = -s_w I.
// R = Rz(az) Ry(ay) Rx(ax), so dR/dA_m = [beta_m]x R with the unit axes
//   beta_z = e_z, beta_y = Rz e_y, beta_x = Rz Ry e_x, and with y = R(A_a) v
//   dr/dA_a,m = -s_w beta_m x y.
// A direction's angles therefore enter a residual only through the angular
// velocity w_a = sum_m p_a,m beta_m, formed once per vertex:
//   J_e p = s_w [(p_a,d - p_b,d) - w_a x y],
// and the angle rows of J^T t are -s_w beta_m . sum_e y x t_e: one torque per
// vertex.  (Three derivative vectors per edge end, as the rows are printed,
// cost three times the arithmetic: 128^3 volume, gather 110 -> 90 us, energies
// 186 -> 120 us, LM 3 x 10 solve 7.88 -> 7.37 ms; the gather is now bound by the
// records it moves through L1 / L2, 64 B per neighbour.)
//
// Per outer iteration (PCGInit): k_mesh_init_v (quaternions, axes, records),
// k_mesh_init_pull (J^T F, diag, M^-1, r, delta, float64 r.z and E).
// Per PCG iteration: k_mesh_apply_v (p = z + beta p into the planes, p_d and w
// into the records), k_mesh_apply_pull (J^T J p + fit + damping, p.q ->
// alpha), k_mesh_update (vector update -> beta).
#include "opt_internal.cuh"
#include "mesh_algebra.cuh"
#include "opt_launch.h"

namespace optgb {

namespace {

#ifndef MESH_PULL_MIN_BLOCKS
#define MESH_PULL_MIN_BLOCKS 4    // resident blocks per SM the gather apply is compiled for
#endif

__device__ __forceinline__ float4 ld4g(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ float c4(const float4& a, int k) {
  return k == 0 ? a.x : (k == 1 ? a.y : (k == 2 ? a.z : a.w));
}

// ---------------------------------------------------------------------------
// PCGInit
// ---------------------------------------------------------------------------
// Vertex pass: the quaternion and axes of every vertex and both records.
__global__ void __launch_bounds__(NT) k_mesh_init_v(const MeshProb* __restrict__ probs,
                                                    const Chunk* __restrict__ chunks) {
  const Chunk ch = chunks[blockIdx.x];
  const MeshProb pr = probs[ch.prob];
  pdl_begin();
  if (pr.s->done) return;
  const long long pl = pr.Vp;
  for (int v = ch.begin + threadIdx.x; v < ch.end; v += NT) {
    float x[6], U[3], q[4];
#pragma unroll
    for (int c = 0; c < 6; ++c) x[c] = pr.x[c * pl + v];
#pragma unroll
    for (int c = 0; c < 3; ++c) U[c] = __ldg(pr.U + c * pl + v);
    float4 axes;
    angles_to_quat(x + 3, q, axes);
    pr.grec[2 * (size_t)v] = make_float4(U[0], U[1], U[2], q[0]);
    pr.grec[2 * (size_t)v + 1] = make_float4(q[1], q[2], q[3], 0.f);
    pr.grec[2 * (size_t)pr.V + v] = axes;
    pr.vrec[2 * (size_t)v] = make_float4(x[0], x[1], x[2], 0.f);
  }
}

// Gather pass: per vertex i the rows of J^T F (fit, own edge residuals with
// their angle rows, incoming edge residuals), diag(J^T J) (displacement:
// planned w_reg * degree + w_fit; angles: w_reg sum |beta_m x y|^2 over the
// out-edges), the energy of the own residuals, then b = -J^T F, M^-1, r = b,
// delta = 0.
// resident blocks per SM the gather PCGInit is compiled for (85 registers;
// measured against 2 and 4: level-9 PCGInit 330 -> 316 us, level 7 39.8 -> 36.1 us)
#ifndef MESH_INIT_MIN_BLOCKS
#define MESH_INIT_MIN_BLOCKS 3
#endif
template <bool G3>
__global__ void __launch_bounds__(NT, MESH_INIT_MIN_BLOCKS) k_mesh_init_pull(const MeshProb* __restrict__ probs,
                                                       const Chunk* __restrict__ chunks,
                                                       double* __restrict__ part, int k_outer, float dmin,
                                                       float dmax) {
  const Chunk ch = chunks[blockIdx.x];
  const MeshProb pr = probs[ch.prob];
  pdl_begin();
  Scalars* s = pr.s;
  if (s->done) return;
  const long long pl = pr.Vp;
  const float lam = pr.lm ? s->lambda_f : 0.0f;
  F2 acc_rz = f2_zero(), acc_E = f2_zero();
  for (int i = ch.begin + threadIdx.x; i < ch.end; i += NT) {
    float xi[3];
    load_vec3(pr.vrec, i, xi);
    const GeoRec gi = load_geo(pr.grec, i);
    const float4 axes = load_axes(pr, i);
    float D[3][3];
    quat_delta_matrix(gi.q, D);
    float g[6];                                    // J^T F
    float f[3] = {0.f, 0.f, 0.f};                  // sum of the residuals / s_w, in-edges negative
    float tq[3] = {0.f, 0.f, 0.f};                 // torque
    float da[3] = {0.f, 0.f, 0.f};                 // angle diagonal / w_reg
    float es = 0.f, e = 0.f;
    auto own_edge = [&](const float (&d)[3], const float (&v)[3]) {
      float dv[3], r[3], y[3];
      mat_vec(D, v, dv);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        r[c] = d[c] - dv[c];
        y[c] = v[c] + dv[c];
        f[c] += r[c];
        es = fmaf(r[c], r[c], es);
      }
      add_cross(tq, y, r);
      axis_squares(axes, y, da);
    };
    // residual of (j, i) / s_w: -(d + (R_j - I) (U_j - U_i)) with d = x_i - x_j
    auto in_edge = [&](const GeoRec& gj, const float (&d)[3], const float (&v)[3]) {
      float dv[3];
      quat_delta(gj.q, v, dv);
#pragma unroll
      for (int c = 0; c < 3; ++c) f[c] += d[c] - dv[c];
    };
    const int o0 = G3 ? 0 : pr.orow[i], o1 = G3 ? 0 : pr.orow[i + 1];
    for_neighbours<G3>(pr, i, pr.e1, o0, o1, [&](int j, bool own, bool in) {
      const GeoRec gj = load_geo(pr.grec, j);
      float xj[3], d[3], v[3];
      load_vec3(pr.vrec, j, xj);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        d[c] = xi[c] - xj[c];
        v[c] = gi.U[c] - gj.U[c];
      }
      if (own) own_edge(d, v);
      if (in) in_edge(gj, d, v);
    });
    {
      float ga[3];
      axis_rows(axes, tq, ga);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        g[c] = pr.w_reg * f[c];
        g[3 + c] = -pr.w_reg * ga[c];
        da[c] *= pr.w_reg;
      }
    }
    const int h = handle_of(pr, i);
    if (h >= 0) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float fh = pr.s_f * (xi[c] - pr.htgt[3 * h + c]);
        g[c] = fmaf(pr.s_f, fh, g[c]);
        e = fmaf(fh, fh, e);
      }
    }
    e = fmaf(pr.w_reg, es, e);
    const float dg[4] = {pr.degw[i], da[0], da[1], da[2]};
    float mv[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float dcv;
      mv[k] = minv_entry(dg[k], lam, dmin, dmax, pr.use_precond, &dcv);
      pr.m[k * pl + i] = mv[k];
      if (pr.lm) pr.dc[k * pl + i] = dcv;
      if (pr.diag_out) pr.diag_out[k * pl + i] = dg[k];
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const float b = -g[c];
      pr.r[c * pl + i] = b;
      pr.d[c * pl + i] = 0.f;
      if (pr.jtf_out) pr.jtf_out[c * pl + i] = g[c];
      f2_add_prod(acc_rz, b, __fmul_rn(mv[c < 3 ? 0 : c - 2], b));
    }
    f2_add(acc_E, e);
  }
  pdl_trigger();
  if (publish_partials(part, blockIdx.x, acc_rz, acc_E, &s->counter, pr.vchunk_end - pr.vchunk_begin)) {
    double rz, E;
    gather_partials(part, pr.vchunk_begin, pr.vchunk_end, &s->counter, rz, E);
    if (threadIdx.x == 0) {
      set_rz(s, rz);
      s->E = E;
      if (pr.Ehist && k_outer >= 0) pr.Ehist[k_outer] = E;
      s->beta_f = 0.f;
      s->pcg_active = (rz != 0.0) && isfinite(rz);
      if (!isfinite(rz) || !isfinite(E)) s->nonfinite = 1;
    }
  }
}

// ---------------------------------------------------------------------------
// PCGStep: applyJTJ
// ---------------------------------------------------------------------------
// Direction update p = z + beta p (or p = p_override), four vertices per
// thread from the planes (every load of a quad before any store), written to
// the planes and to the 6-vector records.  Vertex ranges start at multiples
// of 256 and the planes are padded to 32 (zeros), so a quad never leaves the
// plane; records are written for real vertices only.
__global__ void __launch_bounds__(NT) k_mesh_apply_v(const MeshProb* __restrict__ probs,
                                                     const Chunk* __restrict__ chunks,
                                                     const float* __restrict__ p_override, int par,
                                                     int update) {
  const Chunk ch = chunks[blockIdx.x];
  const MeshProb pr = probs[ch.prob];
  pdl_begin();
  Scalars* s = pr.s;
  if (s->done || !s->pcg_active) return;
  const long long pl = pr.Vp;
  const float beta = s->beta_f;
  const float* __restrict__ pin = p_override ? p_override : pr.p + (long long)(par & 1) * 6 * pl;
  float* __restrict__ pout = pr.p + (long long)((par + 1) & 1) * 6 * pl;
  const int q0 = ch.begin / 4, q1 = (ch.end + 3) / 4;
  for (int qi = q0 + threadIdx.x; qi < q1; qi += NT) {
    const int v0 = 4 * qi;
    float4 pv[6];
    if (update) {
      float4 rr[6], mm[4], po[6];
#pragma unroll
      for (int c = 0; c < 6; ++c) rr[c] = ld4g(pr.r + c * pl + v0);
#pragma unroll
      for (int k = 0; k < 4; ++k) mm[k] = ld4g(pr.m + k * pl + v0);
      if (beta != 0.0f) {
#pragma unroll
        for (int c = 0; c < 6; ++c) po[c] = ld4g(pin + c * pl + v0);
      }
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        const float4 m = mm[c < 3 ? 0 : c - 2];
        pv[c] = make_float4(m.x * rr[c].x, m.y * rr[c].y, m.z * rr[c].z, m.w * rr[c].w);
        if (beta != 0.0f) {
          pv[c].x = fmaf(beta, po[c].x, pv[c].x); pv[c].y = fmaf(beta, po[c].y, pv[c].y);
          pv[c].z = fmaf(beta, po[c].z, pv[c].z); pv[c].w = fmaf(beta, po[c].w, pv[c].w);
        }
      }
#pragma unroll
      for (int c = 0; c < 6; ++c) *reinterpret_cast<float4*>(pout + c * pl + v0) = pv[c];
    } else {
#pragma unroll
      for (int c = 0; c < 6; ++c) pv[c] = ld4g(pin + c * pl + v0);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int v = v0 + k;
      if (v < pr.V) {
        float w[3];
        angular_velocity(load_axes(pr, v), c4(pv[3], k), c4(pv[4], k), c4(pv[5], k), w);
        pr.vrec[2 * (size_t)v] = make_float4(c4(pv[0], k), c4(pv[1], k), c4(pv[2], k), w[0]);
        pr.vrec[2 * (size_t)v + 1] = make_float4(w[1], w[2], 0.f, 0.f);
      }
    }
  }
}

// Gather pass: q_i = (fit + damping) p_i + sum over out-edges (i, j) of the
// own rows s_w J_e p (displacement) and the torque rows (angles) + sum over
// in-edges (j, i) of -s_w J_e p (displacement); p.q -> alpha.  The
// kernel is bound by its dependent index -> record loads, so it is compiled for
// MESH_PULL_MIN_BLOCKS resident blocks per SM.
template <bool G3>
__global__ void __launch_bounds__(NT, MESH_PULL_MIN_BLOCKS) k_mesh_apply_pull(const MeshProb* __restrict__ probs,
                                                                             const Chunk* __restrict__ chunks,
                                                                             double* __restrict__ part,
                                                                             const float* __restrict__ p_override,
                                                                             int pcur) {
  const Chunk ch = chunks[blockIdx.x];
  const MeshProb pr = probs[ch.prob];
  pdl_begin();
  Scalars* s = pr.s;
  if (s->done || !s->pcg_active) return;
  const long long pl = pr.Vp;
  const float lam = pr.lm ? s->lambda_f : 0.0f;
  const float* __restrict__ pa = (p_override ? p_override : pr.p + (long long)(pcur & 1) * 6 * pl) + 3 * pl;
  F2 acc = f2_zero();
  for (int i = ch.begin + threadIdx.x; i < ch.end; i += NT) {
    float pd[3], wi[3];
    load_pw(pr.vrec, i, pd, wi);
    const GeoRec gi = load_geo(pr.grec, i);
    float f[3] = {0.f, 0.f, 0.f}, tq[3] = {0.f, 0.f, 0.f};
    mesh_gather<G3>(
        pr, i, pr.e1, G3 ? 0 : pr.orow[i], G3 ? 0 : pr.orow[i + 1], pd, wi, gi,
        [&](int j, float (&pj)[3], float (&wj)[3]) { load_pw(pr.vrec, j, pj, wj); }, f, tq);
    float q[6], ga[3];
    axis_rows(load_axes(pr, i), tq, ga);
    const float pi[6] = {pd[0], pd[1], pd[2], pa[i], pa[pl + i], pa[2 * pl + i]};
    const bool hit = handle_of(pr, i) >= 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      q[c] = pr.w_reg * f[c];
      if (hit) q[c] = fmaf(pr.w_fit, pd[c], q[c]);
      q[3 + c] = -pr.w_reg * ga[c];
    }
    if (pr.lm) {
#pragma unroll
      for (int c = 0; c < 6; ++c) q[c] = fmaf(lam * pr.dc[(c < 3 ? 0 : c - 2) * pl + i], pi[c], q[c]);
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      pr.q[c * pl + i] = q[c];
      f2_add_prod(acc, pi[c], q[c]);
    }
  }
  pdl_trigger();
  const F2 sums[1] = {acc};
  if (publish_sums<1>(part, blockIdx.x, sums, &s->counter, pr.vchunk_end - pr.vchunk_begin)) {
    Sum pq[1];
    gather_sums<1>(part, pr.vchunk_begin, pr.vchunk_end, &s->counter, pq);
    if (threadIdx.x == 0) finish_alpha(s, pq[0]);
  }
}

// ---------------------------------------------------------------------------
// PCGStep: applyJTJ fused with the direction update, ARAP mesh (tiled)
// ---------------------------------------------------------------------------
// One block per vertex tile of VT vertices (the tile-chunk table), one vertex
// per thread.  The block stages the tile's vertices and its halo (the
// out-of-tile neighbours, a table built at planning) in shared memory: the
// displacement rows of the direction p = M^-1 r + beta p_old (formed here,
// halo included, with the same roundings everywhere) and the rest position U.
// With R_i and w_i formed once per vertex, the linearized residual of an
// out-edge e = (i, j) is
//   t_e = J_e p = s_w [(p_i,d - p_j,d) - w_i x y],   y = R_i (U_i - U_j);
// it adds s_w t_e to i's displacement rows and y x t_e to i's torque.  Each t_e goes to a shared-memory slot; in-edges that start
// outside the tile are evaluated edge-parallel from their source's data into
// further slots; every vertex then subtracts s_w t_e of its in-edges, read
// from their slots (a slot table built at planning).  So each residual is
// evaluated once inside a tile and once more per tile border it crosses, no
// atomic is used, and every row is summed in a fixed order.

// The direction of vertex v, components [0, NC): p = M^-1 r + beta p_old
// (update) or the given p; the same roundings wherever it is formed.
template <int NC>
__device__ __forceinline__ void mesh_direction(const MeshProb& pr, int v, long long pl, int update, float beta,
                                               const float* __restrict__ pin, float (&o)[NC]) {
  if (update) {
    float m[NC < 4 ? 1 : 4];
#pragma unroll
    for (int k = 0; k < (NC < 4 ? 1 : 4); ++k) m[k] = __ldg(pr.m + k * pl + v);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      o[c] = __fmul_rn(m[c < 3 ? 0 : c - 2], pr.r[c * pl + v]);
      if (beta != 0.0f) o[c] = __fmaf_rn(beta, pin[c * pl + v], o[c]);
    }
  } else {
#pragma unroll
    for (int c = 0; c < NC; ++c) o[c] = pin[c * pl + v];
  }
}

#ifndef MESH_TILED_MIN_BLOCKS
#define MESH_TILED_MIN_BLOCKS 4   // resident blocks per SM the tiled apply is compiled for
#endif

__global__ void __launch_bounds__(NT, MESH_TILED_MIN_BLOCKS) k_mesh_apply_tiled(
    const MeshProb* __restrict__ probs, const Chunk* __restrict__ tchunks, double* __restrict__ part,
    const float* __restrict__ p_override, int par, int update) {
  const Chunk ch = tchunks[blockIdx.x];
  const MeshProb pr = probs[ch.prob];
  pdl_begin();
  Scalars* s = pr.s;
  if (s->done || !s->pcg_active) return;
  __shared__ float spu[6][VT + MT_HALO];   // the tile's vertices, then its halo: p_d (3), U (3)
  __shared__ float st[3][MT_SLOTS];        // J_e p of the tile's out-edges, then of the remote in-edges
  const long long pl = pr.Vp;
  const float sw = pr.s_w;
  const float beta = s->beta_f;
  const float* __restrict__ pin = p_override ? p_override : pr.p + (long long)(par & 1) * 6 * pl;
  float* __restrict__ pout = pr.p + (long long)((par + 1) & 1) * 6 * pl;
  const int tid = threadIdx.x;
  const int vb = ch.begin, ve = ch.end, T = vb / VT;
  const int i = vb + tid;
  const bool own = i < ve;
  const int ebase = pr.orow[vb], nout = pr.orow[ve] - ebase;
  const int ibase = pr.irow[vb];
  // A: this vertex's direction and geometry, its edge tables fetched ahead
  int o0 = 0, o1 = 0, n0 = 0, n1 = 0;
  int ln[KB], sl[KB];
  float pi[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  float ui[3] = {0.f, 0.f, 0.f}, qi[4] = {1.f, 0.f, 0.f, 0.f};
  float4 axes = make_float4(1.f, 0.f, 1.f, 0.f);
  if (own) {
    o0 = pr.orow[i]; o1 = pr.orow[i + 1];
    n0 = pr.irow[i]; n1 = pr.irow[i + 1];
#pragma unroll
    for (int t = 0; t < KB; ++t) {
      ln[t] = o0 + t < o1 ? pr.lnbr[o0 + t] : 0;
      sl[t] = n0 + t < n1 ? pr.itslot[n0 + t] : 0;
    }
    mesh_direction<6>(pr, i, pl, update, beta, pin, pi);
    if (update) {
#pragma unroll
      for (int c = 0; c < 6; ++c) pout[c * pl + i] = pi[c];
    }
    const GeoRec g = load_geo(pr.grec, i);
#pragma unroll
    for (int c = 0; c < 3; ++c) ui[c] = g.U[c];
#pragma unroll
    for (int c = 0; c < 4; ++c) qi[c] = g.q[c];
    axes = load_axes(pr, i);
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) { spu[c][tid] = pi[c]; spu[3 + c][tid] = ui[c]; }
  {
    const int h0 = pr.hptr[T], nh = pr.hptr[T + 1] - h0;
    for (int l = tid; l < nh; l += NT) {
      const int j = pr.hvtx[h0 + l];
      float pj[3];
      mesh_direction<3>(pr, j, pl, update, beta, pin, pj);
      const float4 g = __ldg(pr.grec + 2 * (size_t)j);
      spu[0][VT + l] = pj[0]; spu[1][VT + l] = pj[1]; spu[2][VT + l] = pj[2];
      spu[3][VT + l] = g.x; spu[4][VT + l] = g.y; spu[5][VT + l] = g.z;
    }
  }
  __syncthreads();
  // B: own edges (displacement rows, S_i), their J_e p into the slots
  float q[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  float tq[3] = {0.f, 0.f, 0.f};
  if (own) {
    float D[3][3], w[3];
    angular_velocity(axes, pi[3], pi[4], pi[5], w);
    quat_delta_matrix(qi, D);
    auto own_edge = [&](int k, int l) {
      const float v[3] = {ui[0] - spu[3][l], ui[1] - spu[4][l], ui[2] - spu[5][l]};
      float t[3] = {pi[0] - spu[0][l], pi[1] - spu[1][l], pi[2] - spu[2][l]}, y[3];
      mat_vec(D, v, y);
#pragma unroll
      for (int a = 0; a < 3; ++a) y[a] += v[a];
      sub_cross(t, w, y);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        t[a] *= sw;
        q[a] = fmaf(sw, t[a], q[a]);
        st[a][k - ebase] = t[a];
      }
      add_cross(tq, y, t);
    };
#pragma unroll
    for (int t = 0; t < KB; ++t)
      if (o0 + t < o1) own_edge(o0 + t, ln[t]);
    for (int k = o0 + KB; k < o1; ++k) own_edge(k, pr.lnbr[k]);
  }
  {
    // in-edges arriving from outside the tile, edge-parallel, from the source's data
    const int r0 = pr.rptr[T], nr = pr.rptr[T + 1] - r0, h0 = pr.hptr[T];
    for (int r = tid; r < nr; r += NT) {
      const int w = pr.rin[r0 + r];
      const int dl = w & 0xffff;
      const int j = pr.hvtx[h0 + (w >> 16) - VT];
      float pj[6];
      mesh_direction<6>(pr, j, pl, update, beta, pin, pj);
      const GeoRec gj = load_geo(pr.grec, j);
      float wj[3], y[3];
      angular_velocity(load_axes(pr, j), pj[3], pj[4], pj[5], wj);
      const float v[3] = {gj.U[0] - spu[3][dl], gj.U[1] - spu[4][dl], gj.U[2] - spu[5][dl]};
      float t[3] = {pj[0] - spu[0][dl], pj[1] - spu[1][dl], pj[2] - spu[2][dl]};
      quat_delta(gj.q, v, y);
#pragma unroll
      for (int a = 0; a < 3; ++a) y[a] += v[a];
      sub_cross(t, wj, y);
#pragma unroll
      for (int a = 0; a < 3; ++a) st[a][nout + r] = sw * t[a];
    }
  }
  __syncthreads();
  // C: angle rows, in-edge displacement rows, fit, damping; p.q
  F2 acc = f2_zero();
  if (own) {
    float ga[3];
    axis_rows(axes, tq, ga);
#pragma unroll
    for (int m = 0; m < 3; ++m) q[3 + m] = -sw * ga[m];
    auto in_edge = [&](int slot) {
#pragma unroll
      for (int a = 0; a < 3; ++a) q[a] = fmaf(-sw, st[a][slot], q[a]);
    };
#pragma unroll
    for (int t = 0; t < KB; ++t)
      if (n0 + t < n1) in_edge(sl[t]);
    for (int k = n0 + KB; k < n1; ++k) in_edge(pr.itslot[k]);
    if (handle_of(pr, i) >= 0) {
#pragma unroll
      for (int c = 0; c < 3; ++c) q[c] = fmaf(pr.w_fit, pi[c], q[c]);
    }
    if (pr.lm) {
      const float lam = s->lambda_f;
#pragma unroll
      for (int c = 0; c < 6; ++c) q[c] = fmaf(lam * pr.dc[(c < 3 ? 0 : c - 2) * pl + i], pi[c], q[c]);
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      pr.q[c * pl + i] = q[c];
      f2_add_prod(acc, pi[c], q[c]);
    }
  }
  (void)ibase;
  pdl_trigger();
  const F2 sums[1] = {acc};
  if (publish_sums<1>(part, blockIdx.x, sums, &s->counter, pr.tchunk_end - pr.tchunk_begin)) {
    Sum pq[1];
    gather_sums<1>(part, pr.tchunk_begin, pr.tchunk_end, &s->counter, pq);
    if (threadIdx.x == 0) finish_alpha(s, pq[0]);
  }
}

// delta += alpha p, r -= alpha q, z = M^-1 r, r.z -> beta; four
// vertices per thread, all loads first.
__global__ void __launch_bounds__(NT) k_mesh_update(const MeshProb* __restrict__ probs,
                                                    const Chunk* __restrict__ chunks,
                                                    double* __restrict__ part, int par) {
  const Chunk ch = chunks[blockIdx.x];
  const MeshProb pr = probs[ch.prob];
  pdl_begin();
  Scalars* s = pr.s;
  if (s->done || !s->pcg_active) return;
  const long long pl = pr.Vp;
  const float alpha = s->alpha_f;
  const float* __restrict__ pn = pr.p + (long long)((par + 1) & 1) * 6 * pl;
  F2x2 acc = f2x2_zero();
  const int q0 = ch.begin / 4, q1 = (ch.end + 3) / 4;
  for (int qi = q0 + threadIdx.x; qi < q1; qi += NT) {
    const int v0 = 4 * qi;
    float4 pv[6], qv[6], dv[6], rv[6], mv[4];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      pv[c] = ld4g(pn + c * pl + v0);
      qv[c] = ld4g(pr.q + c * pl + v0);
      dv[c] = *reinterpret_cast<const float4*>(pr.d + c * pl + v0);
      rv[c] = *reinterpret_cast<const float4*>(pr.r + c * pl + v0);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) mv[k] = ld4g(pr.m + k * pl + v0);
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const float4 m = mv[c < 3 ? 0 : c - 2];
      dv[c].x += alpha * pv[c].x; dv[c].y += alpha * pv[c].y;
      dv[c].z += alpha * pv[c].z; dv[c].w += alpha * pv[c].w;
      rv[c].x -= alpha * qv[c].x; rv[c].y -= alpha * qv[c].y;
      rv[c].z -= alpha * qv[c].z; rv[c].w -= alpha * qv[c].w;
      const float2 r01 = make_float2(rv[c].x, rv[c].y), r23 = make_float2(rv[c].z, rv[c].w);
      f2x2_add_prod(acc, r01, pk_mul(make_float2(m.x, m.y), r01));
      f2x2_add_prod(acc, r23, pk_mul(make_float2(m.z, m.w), r23));
      *reinterpret_cast<float4*>(pr.d + c * pl + v0) = dv[c];
      *reinterpret_cast<float4*>(pr.r + c * pl + v0) = rv[c];
    }
  }
  pdl_trigger();
  const F2 sums[1] = {f2x2_fold(acc)};
  if (publish_sums<1>(part, blockIdx.x, sums, &s->counter, pr.vchunk_end - pr.vchunk_begin)) {
    Sum rz[1];
    gather_sums<1>(part, pr.vchunk_begin, pr.vchunk_end, &s->counter, rz);
    if (threadIdx.x == 0) finish_beta(s, rz[0]);
  }
}

// ---------------------------------------------------------------------------
// energies and the outer update
// ---------------------------------------------------------------------------
// Vertex pass of the energies on edge lists: what the gather reads of a
// neighbour, its displacement, rest position and (mode 1) the first two components of
// its displacement step, in one record; the third is read from its plane (a sector of its
// own either way).  (A voxel's neighbours lie next to it in the planes.)
__global__ void __launch_bounds__(NT) k_mesh_energy_v(const MeshProb* __restrict__ probs,
                                                      const Chunk* __restrict__ chunks, int mode) {
  const Chunk ch = chunks[blockIdx.x];
  const MeshProb pr = probs[ch.prob];
  pdl_begin();
  if (mode == 1 && pr.s->done) return;
  const long long pl = pr.Vp;
  for (int v = ch.begin + threadIdx.x; v < ch.end; v += NT) {
    float x[3], U[3], d[2] = {0.f, 0.f};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      x[c] = pr.x[c * pl + v];
      U[c] = __ldg(pr.U + c * pl + v);
      if (mode == 1 && c < 2) d[c] = pr.d[c * pl + v];
    }
    pr.vrec[2 * (size_t)v] = make_float4(x[0], x[1], x[2], U[0]);
    pr.vrec[2 * (size_t)v + 1] = make_float4(U[1], U[2], d[0], d[1]);
  }
}

// Energy of every vertex's fit residual and out-edge residuals.  mode 0: at x;
// mode 1: at x + delta, and the model value |F(x) + J(x) delta|^2 (the fit
// residual is linear: one value serves both).  The rotations and the angular
// velocity of delta are formed once per vertex, not per edge (edge-parallel
// with sincosf at both ends: 166 us on the 128^3 volume).
template <bool G3>
__global__ void __launch_bounds__(NT) k_mesh_energy(const MeshProb* __restrict__ probs,
                                                    const Chunk* __restrict__ chunks,
                                                    double* __restrict__ part, int mode, int hist_idx) {
  const Chunk ch = chunks[blockIdx.x];
  const MeshProb pr = probs[ch.prob];
  pdl_begin();
  Scalars* s = pr.s;
  if (mode == 1 && s->done) return;
  const long long pl = pr.Vp;
  F2 e0 = f2_zero(), e1 = f2_zero();
  for (int i = ch.begin + threadIdx.x; i < ch.end; i += NT) {
    float xi[3], ui[3], di[3], w[3] = {0.f, 0.f, 0.f}, D[3][3], D2[3][3];
    {
      float a[3], q[4];
      float4 axes;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        xi[c] = pr.x[c * pl + i];
        ui[c] = __ldg(pr.U + c * pl + i);
        a[c] = pr.x[(3 + c) * pl + i];
      }
      angles_to_quat(a, q, axes);
      quat_delta_matrix(q, D);
      if (mode == 1) {
        float t[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          di[c] = pr.d[c * pl + i];
          t[c] = pr.d[(3 + c) * pl + i];
          a[c] += t[c];
        }
        angular_velocity(axes, t[0], t[1], t[2], w);
        float4 unused;
        angles_to_quat(a, q, unused);
        quat_delta_matrix(q, D2);
      }
    }
    float fit = 0.f;
    const int h = handle_of(pr, i);
    if (h >= 0) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        float dv = xi[c];
        if (mode == 1) dv += di[c];
        const float f = pr.s_f * (dv - pr.htgt[3 * h + c]);
        fit = fmaf(f, f, fit);
      }
    }
    auto edge = [&](int j) {
      float d[3], v[3], dd[3];
      if (G3) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          d[c] = xi[c] - pr.x[c * pl + j];
          v[c] = ui[c] - __ldg(pr.U + c * pl + j);
          if (mode == 1) dd[c] = di[c] - pr.d[c * pl + j];
        }
      } else {
        const float4 ra = pr.vrec[2 * (size_t)j], rb = pr.vrec[2 * (size_t)j + 1];
        d[0] = xi[0] - ra.x; d[1] = xi[1] - ra.y; d[2] = xi[2] - ra.z;
        v[0] = ui[0] - ra.w; v[1] = ui[1] - rb.x; v[2] = ui[2] - rb.y;
        if (mode == 1) {
          dd[0] = di[0] - rb.z; dd[1] = di[1] - rb.w;
          dd[2] = di[2] - pr.d[2 * pl + j];
        }
      }
      float y[3], r[3];
      mat_vec(D, v, y);
#pragma unroll
      for (int c = 0; c < 3; ++c) r[c] = d[c] - y[c];
      float se = 0.f, sm = 0.f;
      if (mode == 0) {
#pragma unroll
        for (int c = 0; c < 3; ++c) se = fmaf(r[c], r[c], se);
        f2_add_prod(e0, pr.w_reg, se);
        return;
      }
      float y2[3];
      mat_vec(D2, v, y2);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float u = (d[c] + dd[c]) - y2[c];
        se = fmaf(u, u, se);
        r[c] += dd[c];
        y[c] += v[c];
      }
      sub_cross(r, w, y);
#pragma unroll
      for (int c = 0; c < 3; ++c) sm = fmaf(r[c], r[c], sm);
      f2_add_prod(e0, pr.w_reg, se);
      f2_add_prod(e1, pr.w_reg, sm);
    };
    if (G3) {
      const Stencil3 st = stencil3(pr, i);
#pragma unroll
      for (int t = 0; t < 6; ++t)
        if (st.ok[t]) edge(i + st.off[t]);
    } else {
      for (int k = pr.orow[i]; k < pr.orow[i + 1]; ++k) edge(pr.e1[k]);
    }
    if (h >= 0) {
      f2_add(e0, fit);
      if (mode == 1) f2_add(e1, fit);
    }
  }
  pdl_trigger();
  if (publish_partials(part, blockIdx.x, e0, e1, &s->counter, pr.vchunk_end - pr.vchunk_begin)) {
    double a, b;
    gather_partials(part, pr.vchunk_begin, pr.vchunk_end, &s->counter, a, b);
    if (threadIdx.x == 0) {
      if (mode == 0) {
        s->E = a;
        const int k = hist_idx >= 0 ? hist_idx : (hist_idx == -1 ? s->outer_done : -1);
        if (pr.Ehist && k >= 0) pr.Ehist[k] = a;
        if (!isfinite(a)) s->nonfinite = 1;
      } else {
        s->E_trial = a;
        s->model = b;
      }
    }
  }
}

__global__ void __launch_bounds__(NT) k_mesh_step(const MeshProb* __restrict__ probs,
                                                  const Chunk* __restrict__ chunks, int cond) {
  const Chunk ch = chunks[blockIdx.x];
  const MeshProb pr = probs[ch.prob];
  pdl_begin();
  if (cond && !pr.s->accept) return;
  if (!cond && pr.s->done) return;
  const long long pl = pr.Vp;
  float* __restrict__ x = pr.x;
  const float* __restrict__ d = pr.d;
  for (int v = ch.begin + threadIdx.x; v < ch.end; v += NT) {
    float xv[6], dv[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) { xv[c] = x[c * pl + v]; dv[c] = __ldg(d + c * pl + v); }
#pragma unroll
    for (int c = 0; c < 6; ++c) x[c * pl + v] = xv[c] + dv[c];
  }
}

}  // namespace

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
void launch_mesh_init(const MeshLaunch& L, int k_outer, float dmin, float dmax) {
  if (L.dim == 2) return launch_wg_init(L, k_outer, dmin, dmax);
  if (L.dim == 12) return launch_ed_init(L, k_outer, dmin, dmax);
  launch_pdl(k_mesh_init_v, L.nvchunks, NT, 0, L.stream, L.probs, L.vchunks);
  if (L.grid3)
    launch_pdl(k_mesh_init_pull<true>, L.nvchunks, NT, 0, L.stream, L.probs, L.vchunks, L.part, k_outer, dmin, dmax);
  else
    launch_pdl(k_mesh_init_pull<false>, L.nvchunks, NT, 0, L.stream, L.probs, L.vchunks, L.part, k_outer, dmin,
               dmax);
}

void launch_mesh_apply(const MeshLaunch& L, const float* p_override, int par, int update) {
  if (L.dim == 2) return launch_wg_apply(L, p_override, par, update);
  if (L.dim == 12) return launch_ed_apply(L, p_override, par, update);
  if (!L.grid3 && L.tchunks) {
    launch_pdl(k_mesh_apply_tiled, L.ntchunks, NT, 0, L.stream, L.probs, L.tchunks, L.part, p_override, par, update);
    return;
  }
  launch_pdl(k_mesh_apply_v, L.nvchunks, NT, 0, L.stream, L.probs, L.vchunks, p_override, par, update);
  const int pcur = update ? par + 1 : par;
  if (L.grid3)
    launch_pdl(k_mesh_apply_pull<true>, L.nvchunks, NT, 0, L.stream, L.probs, L.vchunks, L.part, p_override, pcur);
  else
    launch_pdl(k_mesh_apply_pull<false>, L.nvchunks, NT, 0, L.stream, L.probs, L.vchunks, L.part, p_override, pcur);
}

void launch_mesh_update(const MeshLaunch& L, int par) {
  if (L.dim == 2) return launch_wg_update(L, par);
  if (L.dim == 12) return launch_ed_update(L, par);
  launch_pdl(k_mesh_update, L.nvchunks, NT, 0, L.stream, L.probs, L.vchunks, L.part, par);
}

void launch_mesh_energy(const MeshLaunch& L, int mode, int hist_idx) {
  if (L.dim == 2) return launch_wg_energy(L, mode, hist_idx);
  if (L.dim == 12) return launch_ed_energy(L, mode, hist_idx);
  if (!L.grid3) launch_pdl(k_mesh_energy_v, L.nvchunks, NT, 0, L.stream, L.probs, L.vchunks, mode);
  if (L.grid3)
    launch_pdl(k_mesh_energy<true>, L.nvchunks, NT, 0, L.stream, L.probs, L.vchunks, L.part, mode, hist_idx);
  else
    launch_pdl(k_mesh_energy<false>, L.nvchunks, NT, 0, L.stream, L.probs, L.vchunks, L.part, mode, hist_idx);
}

void launch_mesh_step(const MeshLaunch& L, int cond) {
  if (L.dim == 2) return launch_wg_step(L, cond);
  if (L.dim == 12) return launch_ed_step(L, cond);
  launch_pdl(k_mesh_step, L.nvchunks, NT, 0, L.stream, L.probs, L.vchunks, cond);
}

}  // namespace optgb
