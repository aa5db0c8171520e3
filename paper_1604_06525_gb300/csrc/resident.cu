// The resident PCG loop: all PCG iterations of one outer iteration in ONE
// launch, with the whole PCG state on chip.
//
// A problem whose vectors fit in the shared memory of the device (227 KB on
// each of 152 SMs) does not need to stream them between launches: every block
// owns a fixed run of pixels / vertices and keeps their r, p, q, delta, M^-1
// (and, where they fit, the damping diagonal and the edge lists) in its own
// shared memory for the whole loop.  What leaves the SM in a PCG iteration is
// the direction record of every pixel / vertex (16 .. 48 bytes, gathered by its
// neighbours through L2) and one pair per block and sum.
//
// The launch chain it replaces (two or three launches per PCG iteration) is
// bound by latency, not by work: each launch waits for the whole previous
// grid, loads its scalars and vectors, and ends in a fence, an atomic and a
// last block that sums the partials -- 6 us each however small the problem.
// Here a phase ends in an exchange: every block hands its partial sum to all
// others, and each sums them in the same order, so all hold the same total and
// take the same decisions; the exchange is the barrier too.  Two forms:
//  * one cluster of up to 16 blocks (small problems): sums through distributed
//    shared memory, one hardware cluster barrier, about 500 cycles (1,100 with a
//    sum);
//  * the whole device, one block per SM (cooperative launch): every block stores
//    its sum in a slot of its own cache line and polls the slots of all others
//    (2,500 cycles, 4,200 with the fences that order records).  Slots packed in
//    shared lines cost 9,000: a line that blocks of both dies write is slow to read
//    from the far die (4,500-6,400 cycles against 1,100).  Meetings without a
//    sum poll one counter (1,500; 2,400 with fences).
//
// The arithmetic is that of the per-launch kernels, in the same roundings and
// the same order (grid_algebra.cuh, mesh_algebra.cuh, ...); the dot products are
// the same compensated sums, grouped by block instead of by chunk, so the float32
// alpha and beta are the same and with them every iterate.  (Only the mesh
// energies' records with RES_Z carry w = w(z) + beta w(p_old) in place of w(p).)
//
// Slots: two sets, used in turn; both words of a stored pair carry the sum's number, so
// a slot needs no emptying and a stale one is never taken for the next: a block stores
// sum k + 2 only after sum k
// + 1, which every block reaches after reading those of k.  The counts go on from
// launch to launch (sync->sums, sync->meetings).  Every wait of the device-wide form is
// bounded (ResidentSync); a block that gives up flags s->timeout and returns, the others
// run into their own limit, the later launches of the solve return at once, and the host
// resets the slots.  The cluster form waits at the hardware's barrier, which has no limit
// and needs none: its blocks start together and all take the same path.
#include <algorithm>
#include <cmath>
#include <mutex>

#include "embedded_algebra.cuh"
#include "graph2d_algebra.cuh"
#include "grid_algebra.cuh"
#include "mesh_algebra.cuh"
#include "meet.cuh"
#include "opt_launch.h"

namespace optgb {

namespace {

// Grids: 32 x 8 pixels.  The loop runs over the cells that hold an unknown, not over
// the tiles of the launches: of the 128-pixel tiles that a region to edit touches up to
// half the pixels are fixed, which took shared memory and passes, and now and then the
// loop did not fit (1024^2 Poisson, 30 % free, GN 2 x 20: 0.50 ms, or 0.80 ms in
// launches, by where the region lies; 0.47 ms over the cells).
constexpr int CELL = 256;

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_meet() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// 64-bit store to the same shared variable of another block of the cluster
__device__ __forceinline__ void st_cluster(unsigned long long* local, unsigned rank, unsigned long long v) {
  unsigned a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
               : "=r"(a)
               : "r"((unsigned)__cvta_generic_to_shared(local)), "r"(rank));
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long pack(F2 a) {
  return (unsigned long long)__float_as_uint(a.hi) | ((unsigned long long)__float_as_uint(a.lo) << 32);
}
__device__ __forceinline__ F2 unpack(unsigned long long b) {
  return F2{__uint_as_float((unsigned)b), __uint_as_float((unsigned)(b >> 32))};
}
// A block's sum in its slot: two words that each carry the sum's number, so that each
// says by itself whether it is there.
__device__ __forceinline__ void st_slot(unsigned long long* p, F2 s, unsigned k) {
  const unsigned long long tag = (unsigned long long)k << 32;
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(tag | __float_as_uint(s.hi)),
               "l"(tag | __float_as_uint(s.lo))
               : "memory");
}
__device__ __forceinline__ bool ld_slot(const unsigned long long* p, unsigned k, F2& s) {
  unsigned long long a, b;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
  s = F2{__uint_as_float((unsigned)a), __uint_as_float((unsigned)b)};
  return (unsigned)(a >> 32) == k && (unsigned)(b >> 32) == k;
}
// 2^-64 of a block's sum that float32 cannot hold, by a whole warp (sw: its warps' pairs)
static __device__ __noinline__ F2 block_total64(const F2* sw) {
  const int l = threadIdx.x & 31;
  const double d = [&] {
    double v = l < RW ? f2_to_double(sw[l]) : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v * 0x1p-64;
  }();
  return F2{(float)d, (float)(d - (double)(float)d)};
}
__device__ __forceinline__ double over_double(F2 v, F2 over) {
  return v.hi == kOver ? f2_to_double(over) * 0x1p64 : f2_to_double(v);
}

// Meeting of all blocks: what any thread wrote to global memory before is
// visible to every thread of every block after.  Returns false if a block did
// not arrive in time.
template <bool CL>
__device__ __forceinline__ bool meet(Meet& M) {
  if (CL) {
    cluster_meet();
    return true;
  }
  return meet_device(M);
}

// The same with the total of every thread's pair, equal in every thread of
// every block.  FENCE: global writes are ordered too (a cluster's barrier always
// does).
template <bool CL, bool FENCE>
__device__ __forceinline__ bool meet_sum(Meet& M, F2 acc, Sum& total) {
  __shared__ F2 sw[RW];
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  acc = warp_sum_f2(acc);
  if (l == 0) sw[w] = acc;
  __syncthreads();
  auto block_total = [&] {
    F2 v = sw[l % RW];
#pragma unroll
    for (int o = RW / 2; o > 0; o >>= 1) v = f2_shfl_xor_add(v, o);
    return v;
  };
  M.sums += 1;
  const unsigned k = M.sums, n = gridDim.x;
  if (CL) {
    __shared__ unsigned long long part[2][RES_CLUSTER], over[2][RES_CLUSTER];
    if (w == 0) {
      F2 v = block_total();
      if (!isfinite(v.hi)) {
        const F2 o = block_total64(sw);
        if (l < n) st_cluster(&over[k & 1][cluster_rank()], l, pack(o));
        v = F2{kOver, 0.f};
      }
      if (l < n) st_cluster(&part[k & 1][cluster_rank()], l, pack(v));
      __syncwarp();
    }
    cluster_meet();
    const int j = l % RES_CLUSTER;
    F2 t = j < n ? unpack(part[k & 1][j]) : f2_zero();
#pragma unroll
    for (int o = RES_CLUSTER / 2; o > 0; o >>= 1) t = f2_shfl_xor_add(t, o);
    total = Sum{t.hi, t.lo, 0};
    if (!sum_finite(total))
      total = lanes_total64(l < n ? over_double(unpack(part[k & 1][l]), unpack(over[k & 1][l])) : 0.0, 32, 1);
    return true;
  } else {
    constexpr int NP = RES_MAX_BLOCKS / 32;       // polling warps, one slot a thread
    __shared__ F2 sg[NP], so[NP];
    __shared__ int s_ok[NP];
    unsigned long long (*const slot)[16] = M.sy->slot[k & 1];
    if (w == 0) {
      F2 v = block_total();
      if (!isfinite(v.hi)) {
        const F2 o = block_total64(sw);
        if (l == 0) st_slot(&slot[blockIdx.x][2], o, k);
        v = F2{kOver, 0.f};
      }
      if (FENCE) __threadfence();
      if (l == 0) st_slot(slot[blockIdx.x], v, k);
    }
    if (w < NP) {
      const bool on = threadIdx.x < n;
      const unsigned long long* p = slot[on ? threadIdx.x : 0];
      F2 v;
      unsigned long long t0 = 0;
      int ok = 1;
      for (int spin = 0; !ld_slot(p, k, v) && ok; ++spin) ok = !waited_too_long(spin, t0, M.limit);
      if (FENCE) __threadfence();
      ok = __all_sync(0xffffffffu, ok);
      F2 t = warp_sum_f2(on ? v : f2_zero());
      if (!isfinite(__shfl_sync(0xffffffffu, t.hi, 0))) {
        // a kOver among them, or too much in all: 2^-64 of the float64 sum beside kOver
        F2 o = f2_zero();
        t0 = 0;
        int there = 1;
        if (on && v.hi == kOver)
          for (int spin = 0; !ld_slot(p + 2, k, o) && there; ++spin) there = !waited_too_long(spin, t0, M.limit);
        ok = __all_sync(0xffffffffu, there) && ok;
        double d = on ? over_double(v, o) : 0.0;
        for (int b = 16; b > 0; b >>= 1) d += __shfl_xor_sync(0xffffffffu, d, b);
        d *= 0x1p-64;
        if (l == 0) so[w] = F2{(float)d, (float)(d - (double)(float)d)};
        t = F2{kOver, 0.f};
      }
      if (l == 0) {
        sg[w] = t;
        s_ok[w] = ok;
      }
    }
    __syncthreads();
    M.limit = M.later;
    F2 t = sg[0];
    int ok = s_ok[0];
#pragma unroll
    for (int j = 1; j < NP; ++j) {
      f2_add_f2(t, sg[j]);
      ok &= s_ok[j];
    }
    total = Sum{t.hi, t.lo, 0};
    if (!sum_finite(total)) total = lanes_total64(l < NP ? over_double(sg[l], so[l]) : 0.0, 32, 1);
    return ok != 0;
  }
}

// ---------------------------------------------------------------------------
// direction records
// ---------------------------------------------------------------------------
// NR float4 per pixel / vertex, in rec: two buffers of p and one of z = M^-1 r.  Grids keep
// them for the listed cells only, so that they take what the free pixels need and not what
// the image does (a 4000^2 image would hold 770 MB): row by row of cells, and within one
// the pixels row by row, as in the image without its other cells.
// With RES_Z a neighbour forms the new direction itself, p = z + beta p_old, from
// the z published before the exchange that yields beta: one exchange fewer per
// iteration for twice the records read.  Without, p is published in a phase of
// its own.
struct Records {
  const float4* p;      // p (use_z: p_old)
  const float4* z;
  float beta;
  bool use_z;
};
__device__ __forceinline__ float4 load_rec(const Records& R, long long k) {
  float4 v;
  if (!R.use_z) return R.p[k];
  v = R.z[k];
  if (R.beta != 0.f) {
    const float4 o = R.p[k];
    v.x = __fmaf_rn(R.beta, o.x, v.x);
    v.y = __fmaf_rn(R.beta, o.y, v.y);
    v.z = __fmaf_rn(R.beta, o.z, v.z);
    v.w = __fmaf_rn(R.beta, o.w, v.w);
  }
  return v;
}

// ---------------------------------------------------------------------------
// the energies
// ---------------------------------------------------------------------------
// A kind K gives, for local unit j of the block (global unit u):
//   init(c, u, j)          whether u is a pixel / vertex; prepares what K keeps
//   index(c, j)            its index in the planes
//   publish(c, j, v, dst)  a vector's record (p or z)
// and the rows of (J^T J) p without damping: grids by fetch (a pixel's
// neighbours) and rows; graphs see below.

// --- grids -----------------------------------------------------------------
struct GridCtx {
  const GridProb& pr;
  const int* cells;
  int u0;
  float4* geo;          // warp: cos / sin of theta and UrShape, by record
  int* idx;             // shared: record of each unit
  int* flg;             // shared: neighbour flags of each unit
  // shared, of each of the block's cells: the record of its first pixel, the records of a
  // row of pixels, the first pixel's of the last row of the cell above and of the cell below
  const int4* cell;
};

struct GridUnits {
  using Prob = GridProb;
  using Ctx = GridCtx;
  static constexpr bool GRAPH = false;
  static constexpr int NR = 1;
  static __device__ __forceinline__ bool locate(const GridCtx& c, int u, int& x, int& y) {
    const GridProb& pr = c.pr;
    const int cc = c.cells[u / CELL], t = u % CELL;
    x = (cc & 0xffff) * TW + (t & 31);
    y = (cc >> 16) * TH + (t >> 5);
    return x < pr.W && y < pr.H;
  }
  static __device__ __forceinline__ int record(const GridCtx& c, int j) {
    const int4 ci = c.cell[j / CELL];
    return ci.x + (j % CELL) / TW * ci.y + j % TW;
  }
  static __device__ __forceinline__ int index(const GridCtx& c, int j) {
    int x, y;
    locate(c, c.u0 + j, x, y);
    return y * c.pr.P + x;
  }
  // the records left, right, above and below of unit j's
  static __device__ __forceinline__ void near_records(const GridCtx& c, int j, int (&n)[4]) {
    const int4 ci = c.cell[j / CELL];
    const int i = c.idx[j], t = j % CELL;
    n[0] = i - 1;
    n[1] = i + 1;
    n[2] = t >= TW ? i - ci.y : ci.z + t;
    n[3] = t < CELL - TW ? i + ci.y : ci.w + t % TW;
  }
};

struct WarpKind : GridUnits {
  static constexpr int NX = 3, NM = 2;
  static __device__ __forceinline__ constexpr int mp(int k) { return k == 2 ? 1 : 0; }
  // flags: neighbours left, right, above, below (bits 0-3), own pixel (4)
  // unmasked, handle (5)
  static __device__ __forceinline__ bool init(const GridCtx& c, int u, int j) {
    const GridProb& pr = c.pr;
    int x, y;
    if (!locate(c, u, x, y)) {
      c.idx[j] = -1;
      return false;
    }
    const int i = y * pr.P + x;
    const uint8_t* mk = pr.mask;
    int f = 0;
    if (x > 0 && !(mk && mk[i - 1])) f |= 1;
    if (x + 1 < pr.W && !(mk && mk[i + 1])) f |= 2;
    if (y > 0 && !(mk && mk[i - pr.P])) f |= 4;
    if (y + 1 < pr.H && !(mk && mk[i + pr.P])) f |= 8;
    if (!(mk && mk[i])) f |= 16;
    const int t = (y / TH) * pr.ntx + x / pr.tw;
    for (int h = pr.hbeg[t]; h < pr.hbeg[t + 1]; ++h)
      if (pr.hpix[h] == i) f |= 32;
    c.idx[j] = record(c, j);
    c.flg[j] = f;
    float cs, sn;
    if (pr.csn) {
      cs = pr.csn[i];
      sn = pr.csn[pr.plane + i];
    } else {
      sincosf(pr.x[2 * pr.plane + i], &sn, &cs);
    }
    c.geo[c.idx[j]] = make_float4(cs, sn, __ldg(pr.c + i), __ldg(pr.c + pr.plane + i));
    return true;
  }
  static __device__ __forceinline__ void publish(const GridCtx& c, int j, const float (&p)[NX], float4* dst) {
    dst[c.idx[j]] = make_float4(p[0], p[1], p[2], 0.f);
  }
  static __device__ __forceinline__ WarpPix pix(const GridCtx& c, const float4& p, int i) {
    const float4 g = c.geo[i];
    return WarpPix{p.x, p.y, p.z, g.x, g.y, g.z, g.w};
  }
  struct Near {
    WarpPix o, n[4];
  };
  static __device__ __forceinline__ void fetch(const GridCtx& c, int j, const Records& R, Near& N) {
    const int i = c.idx[j], f = c.flg[j];
    int in[4];
    near_records(c, j, in);
    N.o = pix(c, make_float4(0.f, 0.f, 0.f, 0.f), i);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int n = (f >> k) & 1 ? in[k] : i;
      N.n[k] = pix(c, load_rec(R, n), n);
    }
  }
  static __device__ __forceinline__ void rows(const GridCtx& c, int j, const float (&p)[NX], Near& N, float (&q)[NX]) {
    const GridProb& pr = c.pr;
    const int f = c.flg[j];
    q[0] = q[1] = q[2] = 0.f;
    if (!(f & 16)) return;
    N.o.px = p[0]; N.o.py = p[1]; N.o.pt = p[2];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if ((f >> k) & 1) warp_pair(N.o, N.n[k], q[0], q[1], q[2]);
#pragma unroll
    for (int k = 0; k < 3; ++k) q[k] = __fmul_rn(pr.w_reg, q[k]);
    if (f & 32) {
      q[0] = __fmaf_rn(pr.w_fit, p[0], q[0]);
      q[1] = __fmaf_rn(pr.w_fit, p[1], q[1]);
    }
  }
};

struct PoissonKind : GridUnits {
  static constexpr int NX = 4, NM = 1;
  static __device__ __forceinline__ constexpr int mp(int) { return 0; }
  // flags: neighbours left, right, above, below free (bits 0-3), own pixel free
  // (4), S = diag(J^T J) (from bit 8)
  static __device__ __forceinline__ bool init(const GridCtx& c, int u, int j) {
    const GridProb& pr = c.pr;
    int x, y;
    c.idx[j] = -1;
    if (!locate(c, u, x, y)) return false;
    const int i = y * pr.P + x;
    const uint8_t* mk = pr.mask;
    if (mk && mk[i]) return false;        // fixed: no unknown
    int f = 0, S = 0;
    auto nb = [&](bool in, int o, int bit) {
      if (!in) return;
      const bool free = !(mk && mk[i + o]);
      S += free ? 2 : 1;
      if (free) f |= bit;
    };
    nb(x > 0, -1, 1);
    nb(x + 1 < pr.W, 1, 2);
    nb(y > 0, -pr.P, 4);
    nb(y + 1 < pr.H, pr.P, 8);
    c.idx[j] = record(c, j);
    c.flg[j] = f | (S << 8);
    return true;
  }
  static __device__ __forceinline__ void publish(const GridCtx& c, int j, const float (&p)[NX], float4* dst) {
    dst[c.idx[j]] = make_float4(p[0], p[1], p[2], p[3]);
  }
  struct Near {
    float4 n[4];
  };
  static __device__ __forceinline__ void fetch(const GridCtx& c, int j, const Records& R, Near& N) {
    const int f = c.flg[j];
    int in[4];
    near_records(c, j, in);
#pragma unroll
    for (int k = 0; k < 4; ++k) N.n[k] = (f >> k) & 1 ? load_rec(R, in[k]) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  static __device__ __forceinline__ void rows(const GridCtx& c, int j, const float (&p)[NX], Near& N, float (&q)[NX]) {
    const float S = (float)(c.flg[j] >> 8);
    const float4(&n)[4] = N.n;
    q[0] = pois_row(S, p[0], n[0].x, n[1].x, n[2].x, n[3].x);
    q[1] = pois_row(S, p[1], n[0].y, n[1].y, n[2].y, n[3].y);
    q[2] = pois_row(S, p[2], n[0].z, n[1].z, n[2].z, n[3].z);
    q[3] = pois_row(S, p[3], n[0].w, n[1].w, n[2].w, n[3].w);
  }
};

// --- graphs ----------------------------------------------------------------
// A block keeps a table of everything its vertices see: its own units (entries
// 0 .. cap - 1) and, behind them, one entry per edge that leaves the block
// (staged with one load of all their records at once, before the gather): ND
// floats that change (the direction) and NS that do not (the geometry), each a
// plane of `tab` floats.  Edge lists hold table entries.  Without the table
// (voxel grids, one-way edges, too many edges leave) neighbours are read from
// their records, and lists hold vertices.
//
// A voxel is gathered by RES_LANES threads where a block has few of them (see
// resident_plan): each evaluates every RES_LANES-th neighbour, and the terms are added in
// list order all the same.
struct GraphCtx {
  const MeshProb& pr;
  int u0, cap, tab;
  bool staged;
  const int* lst;       // neighbours (staged: table entries)
  const int* row;       // the block's run of the rows of lst
  int* flg;             // shared: handle flag of each unit
  float* dyn;           // ND planes; the first PT hold the direction's first PT components
  float* ext;           // the other components of the direction, NX - PT planes of cap
  float* geo;           // NS planes (staged)
};

struct GraphUnits {
  using Prob = MeshProb;
  using Ctx = GraphCtx;
  static constexpr bool GRAPH = true;
  static __device__ __forceinline__ int index(const GraphCtx& c, int j) { return c.u0 + j; }
  static __device__ __forceinline__ bool init(const GraphCtx& c, int u, int j) {
    c.flg[j] = handle_of(c.pr, u) >= 0;
    return true;
  }
};

template <bool G3_>
struct MeshKind : GraphUnits {
  static constexpr bool G3 = G3_;
  static constexpr int NX = 6, NM = 4, NR = 2, PT = 3, ND = 6, NS = 7, NT_ = 6;
  static __device__ __forceinline__ constexpr int mp(int k) { return k < 3 ? 0 : k - 2; }
  static __device__ __forceinline__ void geometry(const MeshProb& pr, int v, float (&g)[NS]) {
    const GeoRec r = load_geo(pr.grec, v);
#pragma unroll
    for (int k = 0; k < 3; ++k) g[k] = r.U[k];
#pragma unroll
    for (int k = 0; k < 4; ++k) g[3 + k] = r.q[k];
  }
  // the components of the record behind the PT planes: the angular velocity
  static __device__ __forceinline__ void derive(const GraphCtx& c, int j, const float (&p)[NX], float (&d)[ND]) {
    float w[3];
    angular_velocity(load_axes(c.pr, c.u0 + j), p[3], p[4], p[5], w);
#pragma unroll
    for (int k = 0; k < 3; ++k) { d[k] = p[k]; d[3 + k] = w[k]; }
  }
  static __device__ __forceinline__ void pack_rec(const float (&d)[ND], int v, float4* dst) {
    dst[2 * (size_t)v] = make_float4(d[0], d[1], d[2], d[3]);
    dst[2 * (size_t)v + 1] = make_float4(d[4], d[5], 0.f, 0.f);
  }
  static __device__ __forceinline__ void unpack_rec(const Records& R, int v, float (&d)[ND]) {
    const float4 a = load_rec(R, 2 * (long long)v), b = load_rec(R, 2 * (long long)v + 1);
    d[0] = a.x; d[1] = a.y; d[2] = a.z; d[3] = a.w; d[4] = b.x; d[5] = b.y;
  }
  struct Own {
    float pd[3], w[3], U[3], D[3][3];
  };
  static __device__ __forceinline__ void own(const float (&)[NX], const float (&d)[ND], const float (&g)[NS], Own& o) {
    const float q[4] = {g[3], g[4], g[5], g[6]};
#pragma unroll
    for (int k = 0; k < 3; ++k) { o.pd[k] = d[k]; o.w[k] = d[3 + k]; o.U[k] = g[k]; }
    quat_delta_matrix(q, o.D);
  }
  static __device__ __forceinline__ void terms(const MeshProb&, const Own& o, const float (&d)[ND],
                                               const float (&g)[NS], bool out, bool in, float (&t)[NT_]) {
    const float pj[3] = {d[0], d[1], d[2]}, wj[3] = {d[3], d[4], d[5]};
    GeoRec gj;
#pragma unroll
    for (int k = 0; k < 3; ++k) gj.U[k] = g[k];
#pragma unroll
    for (int k = 0; k < 4; ++k) gj.q[k] = g[3 + k];
    float f[3], tq[3];
    mesh_terms(o.pd, o.w, o.U, o.D, pj, wj, gj, out, in, f, tq);
#pragma unroll
    for (int k = 0; k < 3; ++k) { t[k] = f[k]; t[3 + k] = tq[k]; }
  }
  static __device__ __forceinline__ void rows(const GraphCtx& c, int j, const float (&p)[NX], const float (&t)[NT_],
                                              float (&q)[NX]) {
    const MeshProb& pr = c.pr;
    const float tq[3] = {t[3], t[4], t[5]};
    float ga[3];
    axis_rows(load_axes(pr, c.u0 + j), tq, ga);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      q[k] = pr.w_reg * t[k];
      if (c.flg[j]) q[k] = fmaf(pr.w_fit, p[k], q[k]);
      q[3 + k] = -pr.w_reg * ga[k];
    }
  }
};

struct WarpGraphKind : GraphUnits {
  static constexpr bool G3 = false;
  static constexpr int NX = 3, NM = 2, NR = 1, PT = 3, ND = 3, NS = 4, NT_ = 3;
  static __device__ __forceinline__ constexpr int mp(int k) { return k == 2 ? 1 : 0; }
  static __device__ __forceinline__ void geometry(const MeshProb& pr, int v, float (&g)[NS]) {
    const float4 a = __ldg(pr.grec + v);
    g[0] = a.x; g[1] = a.y; g[2] = a.z; g[3] = a.w;
  }
  static __device__ __forceinline__ void derive(const GraphCtx&, int, const float (&p)[NX], float (&d)[ND]) {
#pragma unroll
    for (int k = 0; k < 3; ++k) d[k] = p[k];
  }
  static __device__ __forceinline__ void pack_rec(const float (&d)[ND], int v, float4* dst) {
    dst[v] = make_float4(d[0], d[1], d[2], 0.f);
  }
  static __device__ __forceinline__ void unpack_rec(const Records& R, int v, float (&d)[ND]) {
    const float4 a = load_rec(R, v);
    d[0] = a.x; d[1] = a.y; d[2] = a.z;
  }
  struct Own {
    float4 p, g;
  };
  static __device__ __forceinline__ void own(const float (&p)[NX], const float (&)[ND], const float (&g)[NS], Own& o) {
    o.p = make_float4(p[0], p[1], p[2], 0.f);
    o.g = make_float4(g[0], g[1], g[2], g[3]);
  }
  static __device__ __forceinline__ void terms(const MeshProb&, const Own& o, const float (&d)[ND],
                                               const float (&g)[NS], bool out, bool in, float (&t)[NT_]) {
    wg_terms(o.p, o.g, make_float4(d[0], d[1], d[2], 0.f), make_float4(g[0], g[1], g[2], g[3]), out, in, t);
  }
  static __device__ __forceinline__ void rows(const GraphCtx& c, int j, const float (&p)[NX], const float (&t)[NT_],
                                              float (&q)[NX]) {
    wg_rows(c.pr, t, p, c.flg[j] != 0, q);
  }
};

struct EmbeddedKind : GraphUnits {
  static constexpr bool G3 = false;
  static constexpr int NX = NXE, NM = NME, NR = 3, PT = NXE, ND = NXE, NS = 3, NT_ = 12;
  static __device__ __forceinline__ constexpr int mp(int k) { return k < 3 ? 0 : k - 2; }
  static __device__ __forceinline__ void geometry(const MeshProb& pr, int v, float (&g)[NS]) {
    const float4 a = __ldg(pr.grec + v);
    g[0] = a.x; g[1] = a.y; g[2] = a.z;
  }
  static __device__ __forceinline__ void derive(const GraphCtx&, int, const float (&p)[NX], float (&d)[ND]) {
#pragma unroll
    for (int k = 0; k < ND; ++k) d[k] = p[k];
  }
  static __device__ __forceinline__ void pack_rec(const float (&d)[ND], int v, float4* dst) { store12(dst, v, d); }
  static __device__ __forceinline__ void unpack_rec(const Records& R, int v, float (&d)[ND]) {
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      const float4 a = load_rec(R, 3 * (long long)v + t);
      d[4 * t] = a.x; d[4 * t + 1] = a.y; d[4 * t + 2] = a.z; d[4 * t + 3] = a.w;
    }
  }
  struct Own {
    float p[NX];
    float4 u;
  };
  static __device__ __forceinline__ void own(const float (&p)[NX], const float (&)[ND], const float (&g)[NS], Own& o) {
#pragma unroll
    for (int k = 0; k < NX; ++k) o.p[k] = p[k];
    o.u = make_float4(g[0], g[1], g[2], 0.f);
  }
  static __device__ __forceinline__ void terms(const MeshProb& pr, const Own& o, const float (&d)[ND],
                                               const float (&g)[NS], bool out, bool in, float (&t)[NT_]) {
    float f[3], m[9];
    ed_terms(pr.w_reg, o.p, o.u, d, make_float4(g[0], g[1], g[2], 0.f), out, in, f, m);
#pragma unroll
    for (int k = 0; k < 3; ++k) t[k] = f[k];
#pragma unroll
    for (int k = 0; k < 9; ++k) t[3 + k] = m[k];
  }
  static __device__ __forceinline__ void rows(const GraphCtx& c, int j, const float (&p)[NX], const float (&t)[NT_],
                                              float (&q)[NX]) {
    const float f[3] = {t[0], t[1], t[2]};
    float g[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) g[k] = t[3 + k];
    ed_rows(c.pr, c.u0 + j, p, f, g, c.flg[j] != 0, q);
  }
};

// The edge sums t of unit j (ok: there is one), on voxel grids by LANES consecutive
// threads of a warp; all of them get the result.  Called by whole warps.
template <class K, int LANES>
__device__ __forceinline__ void graph_sums(const GraphCtx& c, int j, bool ok, const typename K::Own& o,
                                           const Records& R, float (&t)[K::NT_]) {
  constexpr int NT_ = K::NT_;
  const MeshProb& pr = c.pr;
#pragma unroll
  for (int k = 0; k < NT_; ++k) t[k] = 0.f;
  const int lane = threadIdx.x % LANES;
  auto fetch = [&](int e, float (&d)[K::ND], float (&g)[K::NS]) {
    if (c.staged) {
#pragma unroll
      for (int k = 0; k < K::ND; ++k) d[k] = c.dyn[k * c.tab + e];
#pragma unroll
      for (int k = 0; k < K::NS; ++k) g[k] = c.geo[k * c.tab + e];
    } else {
      K::unpack_rec(R, e, d);
      K::geometry(pr, e, g);
    }
  };
  auto nbr = [&](int e, bool out, bool in, float (&v)[NT_]) {
    float d[K::ND], g[K::NS];
    fetch(e, d, g);
    K::terms(pr, o, d, g, out, in, v);
  };
  if (K::G3) {
    const Stencil3 st = stencil3(pr, c.u0 + (ok ? j : 0));
    if (LANES == 1) {
      const int i = c.u0 + j;
#pragma unroll
      for (int r = 0; r < 6; r += 2) {
        float d1[K::ND], g1[K::NS], d2[K::ND], g2[K::NS], v[NT_];
        const bool on1 = ok && st.ok[r], on2 = ok && st.ok[r + 1];
        if (on1) fetch(i + st.off[r], d1, g1);
        if (on2) fetch(i + st.off[r + 1], d2, g2);
        if (on1) {
          K::terms(pr, o, d1, g1, true, true, v);
#pragma unroll
          for (int n = 0; n < NT_; ++n) t[n] += v[n];
        }
        if (on2) {
          K::terms(pr, o, d2, g2, true, true, v);
#pragma unroll
          for (int n = 0; n < NT_; ++n) t[n] += v[n];
        }
      }
      return;
    }
#pragma unroll
    for (int r = 0; r < 6; r += LANES) {
      float v[NT_];
      // the thread's neighbour of this round
      int off = 0;
      bool has = false;
#pragma unroll
      for (int s = 0; s < LANES; ++s)
        if (r + s < 6 && lane == s) { off = st.off[r + s < 6 ? r + s : 0]; has = ok && st.ok[r + s < 6 ? r + s : 0]; }
      if (has) nbr(c.u0 + j + off, true, true, v);
#pragma unroll
      for (int s = 0; s < LANES; ++s) {
        const bool from = __shfl_sync(0xffffffffu, (int)has, s, LANES) != 0;
#pragma unroll
        for (int k = 0; k < NT_; ++k) {
          const float a = __shfl_sync(0xffffffffu, has ? v[k] : 0.f, s, LANES);
          if (from) t[k] += a;
        }
      }
    }
    return;
  }
  const int o0 = ok ? c.row[j] : 0, deg = ok ? c.row[j + 1] - o0 : 0;
  const bool sym = pr.sym != 0;
  // two neighbours at a time: their records are in flight together
  for (int k = 0; k < deg; k += 2) {
    float d1[K::ND], g1[K::NS], d2[K::ND], g2[K::NS], v[NT_];
    const bool two = k + 1 < deg;
    const int e1 = c.lst[o0 + k], e2 = two ? c.lst[o0 + k + 1] : e1;
    fetch(e1, d1, g1);
    if (two) fetch(e2, d2, g2);
    K::terms(pr, o, d1, g1, true, sym, v);
#pragma unroll
    for (int n = 0; n < NT_; ++n) t[n] += v[n];
    if (two) {
      K::terms(pr, o, d2, g2, true, sym, v);
#pragma unroll
      for (int n = 0; n < NT_; ++n) t[n] += v[n];
    }
  }
  if (!sym && ok) {
    for (int k = pr.irow[c.u0 + j]; k < pr.irow[c.u0 + j + 1]; ++k) {
      float v[NT_];
      nbr(pr.isrc[k], false, true, v);
#pragma unroll
      for (int n = 0; n < NT_; ++n) t[n] += v[n];
    }
  }
}

// ---------------------------------------------------------------------------
// the loop
// ---------------------------------------------------------------------------
template <int N>
struct Lanes {
  static constexpr int value = N;
};

template <class K, bool CL>
__global__ void __launch_bounds__(RT, 1) k_pcg_resident(const typename K::Prob* __restrict__ probs,
                                                        const int* __restrict__ cells,
                                                        const int4* __restrict__ places, ResidentSync* sync,
                                                        const ResidentPlan rp, float4* rec, int inner, int step,
                                                        int csn_out) {
  constexpr int NX = K::NX, NM = K::NM;
  extern __shared__ float sh[];
  const typename K::Prob pr = probs[0];
  if (CL) pdl_begin();
  Scalars* s = pr.s;
  // (the same for every block: none has passed an exchange; after a launch whose exchanges
  // failed the counts no longer match, and the rest of the solve does not wait on them)
  if (s->done || !s->pcg_active || s->timeout) return;
  if (!CL && sync->absent && blockIdx.x + 1 == gridDim.x) return;
  Meet M = CL ? Meet{} : meet_begin(sync);
  const int tid = threadIdx.x;
  const int u0 = blockIdx.x * rp.per, cnt = min(rp.per, rp.n - u0), cap = rp.per;
  const long long pl = rp.plane;
  const bool zrec = (rp.flags & RES_Z) != 0, lm = pr.lm != 0;
  const float lam = lm ? s->lambda_f : 0.0f;
  float4* const recp[2] = {rec, rec + (zrec ? K::NR * rp.recs : 0)};
  float4* const recz = rec + 2 * K::NR * rp.recs;
  float* cur = sh;
  auto take = [&](int words) { float* r = cur; cur += words; return r; };
  float* const sr = take(NX * cap);
  float* const sq = take(NX * cap);
  float* const sm = take(NM * cap);
  int* const flg = reinterpret_cast<int*>(take(cap));
  // delta and the damping diagonal in shared memory where they fit (grids:
  // always), else in their planes
  float* sd = pr.d + u0;
  long long ds = pl;
  if (rp.flags & RES_D) { sd = take(NX * cap); ds = cap; }
  const float* sc = pr.dc + u0;
  long long cs = pl;
  float* sc_w = nullptr;
  if (lm && (rp.flags & RES_DC)) { sc = sc_w = take(NM * cap); cs = cap; }
  // the direction: grids NX planes, graphs the table's first PT and NX - PT more
  int* idx = nullptr;
  float *sp = nullptr, *sx = nullptr;
  int tab = cap;
  typename K::Ctx ctx = [&] {
    if constexpr (K::GRAPH) {
      tab = cap + rp.slots;
      sx = take((NX - K::PT) * cap);
      sp = take(K::ND * tab);
      const int* row = pr.orow + u0;
      const int* lst = pr.e1;
      GraphCtx c{pr, u0, cap, tab, false, lst, row, flg, sp, sx, nullptr};
      if (rp.flags & RES_LIST) {
        int* srow = reinterpret_cast<int*>(take(cap + 1));
        const int e0 = pr.orow[u0], e1 = pr.orow[u0 + cnt];
        for (int j = tid; j <= cnt; j += RT) srow[j] = pr.orow[u0 + j] - e0;
        c.row = srow;
        int far = 0;
        if (rp.slots > 0) {
          c.geo = take(K::NS * tab);
          for (int e = e0 + tid; e < e1; e += RT) far += (unsigned)(pr.e1[e] - u0) >= (unsigned)cnt;
        }
        int* sl = reinterpret_cast<int*>(cur);
        // how many edges leave the block, and whether their entries fit
        __shared__ int s_far, s_next;
        if (tid == 0) s_far = s_next = 0;
        __syncthreads();
        if (far) atomicAdd(&s_far, far);
        __syncthreads();
        c.staged = pr.sym && rp.slots > 0 && s_far <= rp.slots;
        for (int e = e0 + tid; e < e1; e += RT) {
          int t = pr.e1[e];
          if (c.staged) {
            if ((unsigned)(t - u0) < (unsigned)cnt) {
              t -= u0;
            } else {
              // (which entry an edge gets does not matter: sums follow the list)
              const int k = atomicAdd(&s_next, 1);
              float g[K::NS];
              K::geometry(pr, t, g);
#pragma unroll
              for (int n = 0; n < K::NS; ++n) c.geo[n * tab + cap + k] = g[n];
              sl[e1 - e0 + k] = t;
              t = cap + k;
            }
          }
          sl[e - e0] = t;
        }
        c.lst = sl;
        __syncthreads();
      }
      return c;
    } else {
      sp = take(NX * cap);
      idx = reinterpret_cast<int*>(take(cap));
      int4* const cell = reinterpret_cast<int4*>(take(cap / CELL * 4));     // (16-byte aligned: cap is 256 k)
      for (int k = tid; k < cnt / CELL; k += RT) cell[k] = places[u0 / CELL + k];
      __syncthreads();
      return GridCtx{pr, cells, u0, rec + 3 * rp.recs, idx, flg, cell};
    }
  }();
  // the vertices behind the entries of edges that leave the block
  const int* far_id = nullptr;
  int nfar = 0;
  if constexpr (K::GRAPH) {
    if (ctx.staged) {
      const int ne = ctx.row[cnt];
      far_id = ctx.lst + ne;
      // count: entries were handed out from 0
      __shared__ int s_n;
      if (tid == 0) s_n = 0;
      __syncthreads();
      int n = 0;
      for (int e = tid; e < ne; e += RT) n += ctx.lst[e] >= cap;
      if (n) atomicAdd(&s_n, n);
      __syncthreads();
      nfar = s_n;
    }
  }
  auto skip = [&](int j) { return !K::GRAPH && idx[j] < 0; };
  auto p_at = [&](int k, int j) -> float& {
    if constexpr (K::GRAPH) return k < K::PT ? sp[k * tab + j] : sx[(k - K::PT) * cap + j];
    else return sp[k * cap + j];
  };
  // keeps p of unit j and publishes its record
  auto put_p = [&](int j, const float (&p)[NX], float4* dst) {
#pragma unroll
    for (int k = 0; k < NX; ++k) p_at(k, j) = p[k];
    if constexpr (K::GRAPH) {
      float d[K::ND];
      K::derive(ctx, j, p, d);
#pragma unroll
      for (int k = K::PT; k < K::ND; ++k) sp[k * tab + j] = d[k];
      K::pack_rec(d, u0 + j, dst);
    } else {
      K::publish(ctx, j, p, dst);
    }
  };
  auto put_z = [&](int j, const float (&z)[NX]) {
    if constexpr (K::GRAPH) {
      float d[K::ND];
      K::derive(ctx, j, z, d);
      K::pack_rec(d, u0 + j, recz);
    } else {
      K::publish(ctx, j, z, recz);
    }
  };

  // state of the block's units; the first direction is z = M^-1 r
  for (int j = tid; j < cnt; j += RT) {
    if (!K::init(ctx, u0 + j, j)) continue;
    const long long i = K::index(ctx, j);
    float p[NX], m[NM];
#pragma unroll
    for (int k = 0; k < NM; ++k) {
      m[k] = pr.m[k * pl + i];
      sm[k * cap + j] = m[k];
      if (sc_w) sc_w[k * cap + j] = pr.dc[k * pl + i];
    }
#pragma unroll
    for (int k = 0; k < NX; ++k) {
      const float r = pr.r[k * pl + i];
      p[k] = __fmul_rn(m[K::mp(k)], r);
      sr[k * cap + j] = r;
      sd[k * ds + j] = 0.f;
    }
    put_p(j, p, recp[0]);
    if constexpr (K::GRAPH) {
      if (ctx.staged) {
        float g[K::NS];
        K::geometry(pr, u0 + j, g);
#pragma unroll
        for (int n = 0; n < K::NS; ++n) ctx.geo[n * tab + j] = g[n];
      }
    }
  }
  Sum rz = s->rz_sum, pq = sum_zero();        // the same values in every thread
  int iters = 0, nonfinite = 0, active = 1;
  float alpha = 0.f, beta = 0.f;
  bool met = meet<CL>(M);
  for (int it = 0; met && it < inner; ++it) {
    const Records R = {recp[zrec && it > 0 ? (it - 1) & 1 : 0], recz, beta, zrec && it > 0};
    if (it > 0) {
      // p = z + beta p, for the neighbours
      for (int j = tid; j < cnt; j += RT) {
        if (skip(j)) continue;
        float p[NX];
#pragma unroll
        for (int k = 0; k < NX; ++k) {
          const float z = __fmul_rn(sm[K::mp(k) * cap + j], sr[k * cap + j]);
          p[k] = beta != 0.f ? __fmaf_rn(beta, p_at(k, j), z) : z;
        }
        put_p(j, p, recp[zrec ? it & 1 : 0]);
      }
      if (!zrec && !(met = meet<CL>(M))) break;
    }
    // q = (J^T J + lambda D) p, p.q -> alpha
    F2 acc = f2_zero();
    auto finish_rows = [&](int j, const float (&p)[NX], float (&q)[NX]) {
      if (lm) {
        float c[NM];                          // (all loads before the stores)
#pragma unroll
        for (int k = 0; k < NM; ++k) c[k] = __fmul_rn(lam, sc[k * cs + j]);
#pragma unroll
        for (int k = 0; k < NX; ++k) q[k] = __fmaf_rn(c[K::mp(k)], p[k], q[k]);
      }
#pragma unroll
      for (int k = 0; k < NX; ++k) {
        sq[k * cap + j] = q[k];
        f2_add_prod(acc, p[k], q[k]);
      }
    };
    if constexpr (K::GRAPH) {
      if (ctx.staged) {
        for (int k = tid; k < nfar; k += RT) {
          float d[K::ND];
          K::unpack_rec(R, far_id[k], d);
#pragma unroll
          for (int n = 0; n < K::ND; ++n) sp[n * tab + cap + k] = d[n];
        }
      }
      __syncthreads();
      auto gather = [&](auto lanes) {
        constexpr int LANES = decltype(lanes)::value;
        for (int j0 = 0; j0 < cnt; j0 += RT / LANES) {
          const int j = j0 + tid / LANES;
          const bool ok = j < cnt;
          float p[NX], d[K::ND], g[K::NS], t[K::NT_], q[NX];
          typename K::Own o;
          if (ok) {
#pragma unroll
            for (int k = 0; k < NX; ++k) p[k] = p_at(k, j);
#pragma unroll
            for (int k = 0; k < K::ND; ++k) d[k] = sp[k * tab + j];
            if (ctx.staged) {
#pragma unroll
              for (int k = 0; k < K::NS; ++k) g[k] = ctx.geo[k * tab + j];
            } else {
              K::geometry(pr, u0 + j, g);
            }
            K::own(p, d, g, o);
          }
          graph_sums<K, LANES>(ctx, j, ok, o, R, t);
          if (ok && tid % LANES == 0) {
            K::rows(ctx, j, p, t, q);
            finish_rows(j, p, q);
          }
        }
      };
      bool one = true;
      if constexpr (K::G3) {
        one = rp.lanes == 1;
        if (!one) gather(Lanes<RES_LANES>{});
      }
      if (one) gather(Lanes<1>{});
    } else {
      // two pixels at a time: their neighbours' records are in flight together
      for (int j = tid; j < cnt; j += 2 * RT) {
        const int j2 = j + RT;
        const bool on1 = !skip(j), on2 = j2 < cnt && !skip(j2);
        typename K::Near n1, n2;
        if (on1) K::fetch(ctx, j, R, n1);
        if (on2) K::fetch(ctx, j2, R, n2);
        float p[NX], q[NX];
        if (on1) {
#pragma unroll
          for (int k = 0; k < NX; ++k) p[k] = p_at(k, j);
          K::rows(ctx, j, p, n1, q);
          finish_rows(j, p, q);
        }
        if (on2) {
#pragma unroll
          for (int k = 0; k < NX; ++k) p[k] = p_at(k, j2);
          K::rows(ctx, j2, p, n2, q);
          finish_rows(j2, p, q);
        }
      }
    }
    if (!(met = meet_sum<CL, false>(M, acc, pq))) break;
    if (!(pq.hi > 0.f && sum_finite(pq))) {   // breakdown
      alpha = 0.f;
      active = 0;
      nonfinite = !sum_finite(pq);
      break;
    }
    alpha = sum_quot(rz, pq);
    // delta += alpha p, r -= alpha q, r.z -> beta
    acc = f2_zero();
    for (int j = tid; j < cnt; j += RT) {
      if (skip(j)) continue;
      float z[NX], d[NX];                     // (all loads of delta before its stores)
#pragma unroll
      for (int k = 0; k < NX; ++k) d[k] = sd[k * ds + j];
#pragma unroll
      for (int k = 0; k < NX; ++k) sd[k * ds + j] = __fmaf_rn(alpha, p_at(k, j), d[k]);
#pragma unroll
      for (int k = 0; k < NX; ++k) {
        const float r = __fmaf_rn(-alpha, sq[k * cap + j], sr[k * cap + j]);
        sr[k * cap + j] = r;
        z[k] = __fmul_rn(sm[K::mp(k) * cap + j], r);
        f2_add_prod(acc, r, z[k]);
      }
      if (zrec) put_z(j, z);
    }
    Sum rz2 = sum_zero();
    met = zrec ? meet_sum<CL, true>(M, acc, rz2) : meet_sum<CL, false>(M, acc, rz2);
    if (!met) break;
    iters += 1;
    beta = sum_quot(rz2, rz);
    rz = rz2;
    if (rz.hi == 0.f || !sum_finite(rz)) {
      active = 0;
      nonfinite = !sum_finite(rz);
      break;
    }
  }
  if (!met) {
    if (tid == 0) s->timeout = 1;
    return;
  }
  if ((rp.flags & RES_D) || step) {
    for (int j = tid; j < cnt; j += RT) {
      if (skip(j)) continue;
      const long long i = K::index(ctx, j);
      float d[NX], x[NX];
#pragma unroll
      for (int k = 0; k < NX; ++k) {
        d[k] = sd[k * ds + j];
        if (step) x[k] = pr.x[k * pl + i];
      }
#pragma unroll
      for (int k = 0; k < NX; ++k) {
        if (rp.flags & RES_D) pr.d[k * pl + i] = d[k];
        if (step) pr.x[k * pl + i] = x[k] = __fadd_rn(x[k], d[k]);
      }
      if constexpr (!K::GRAPH) {
        if (NX == 3 && step && csn_out && pr.csn) {
          float sn, cn;
          sincosf(x[2], &sn, &cn);
          pr.csn[i] = cn;
          pr.csn[pl + i] = sn;
        }
      }
    }
  }
  if (blockIdx.x == 0 && tid == 0) {
    s->rz = sum_double(rz);
    s->rz_sum = rz;
    s->pq = sum_double(pq);
    s->alpha_f = alpha;
    s->beta_f = beta;
    s->pcg_iters += iters;
    if (!active) s->pcg_active = 0;
    if (nonfinite) s->nonfinite = 1;
    if (!CL) {
      sync->meetings = M.base + M.meetings * gridDim.x;
      sync->sums = M.sums & 3u;
    }
  }
}

// Self-test: `rounds` meetings (kind 0) or sums, with and without ordered writes (kind 1).
__global__ void __launch_bounds__(RT, 1) k_exchange_selftest(ResidentSync* sync, int kind, int rounds, int* out) {
  if (sync->absent && blockIdx.x + 1 == gridDim.x) return;
  Meet M = meet_begin(sync);
  bool met = true;
  for (int r = 1; r <= rounds && met; ++r) {
    if (kind == 0) {
      met = meet_device(M);
      continue;
    }
    const F2 mine = {(float)r, 0.f};
    Sum total = sum_zero();
    met = r & 1 ? meet_sum<false, true>(M, mine, total) : meet_sum<false, false>(M, mine, total);
    if (met && sum_double(total) != (double)r * RT * gridDim.x) out[1] = 1;
  }
  if (threadIdx.x != 0) return;
  if (!met) out[0] = 1;
  if (met && blockIdx.x == 0) {
    sync->meetings = M.base + M.meetings * gridDim.x;
    sync->sums = M.sums;
  }
}

template <class K, bool CL>
cudaError_t launch(const typename K::Prob* probs, const int* cells, const int4* places, ResidentSync* sync, const ResidentPlan& rp,
                   float4* rec, int inner, int step, int csn_out, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(rp.blocks);
  cfg.blockDim = dim3(RT);
  cfg.dynamicSmemBytes = rp.smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  if (CL) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = rp.blocks;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
  } else {
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = CL ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, k_pcg_resident<K, CL>, probs, cells, places, sync, rp, rec, inner, step, csn_out);
}
template <class K>
cudaError_t launch(const typename K::Prob* probs, const int* cells, const int4* places, ResidentSync* sync, const ResidentPlan& rp,
                   float4* rec, int inner, int step, int csn_out, cudaStream_t st) {
  return rp.cluster ? launch<K, true>(probs, cells, places, sync, rp, rec, inner, step, csn_out, st)
                    : launch<K, false>(probs, cells, places, sync, rp, rec, inner, step, csn_out, st);
}

struct DeviceLimits {
  int sms = 0, smem = 0;        // 0: the resident loop is not available
  int cluster = 0;              // blocks of a cluster (0: none)
};

template <class K>
bool raise_limits(DeviceLimits& d, int optin) {
  cudaFuncAttributes fa;
  for (const void* k : {(const void*)k_pcg_resident<K, false>, (const void*)k_pcg_resident<K, true>}) {
    if (cudaFuncGetAttributes(&fa, k) != cudaSuccess) return false;
    const int room = optin - (int)fa.sharedSizeBytes;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, room) != cudaSuccess) return false;
    d.smem = std::min(d.smem, room);
  }
  int per = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_pcg_resident<K, false>, RT, d.smem) != cudaSuccess ||
      per < 1)
    return false;
  // the largest cluster that fits with full shared memory
  if (cudaFuncSetAttribute(k_pcg_resident<K, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
    (void)cudaGetLastError();
  int best = 0;
  for (int c = RES_CLUSTER; c >= 2 && !best; c /= 2) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(c);
    cfg.blockDim = dim3(RT);
    cfg.dynamicSmemBytes = d.smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = c;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_pcg_resident<K, true>, &cfg) == cudaSuccess && n >= 1) best = c;
    else (void)cudaGetLastError();
  }
  d.cluster = std::min(d.cluster, best);
  return true;
}

// SMs, dynamic shared memory and cluster size of the current device, with
// the kernels' limits raised (once per device).
DeviceLimits device_limits() {
  static std::mutex mu;
  static DeviceLimits lim[128];
  static bool known[128] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 128) return DeviceLimits{};
  std::lock_guard<std::mutex> lk(mu);
  if (known[dev]) return lim[dev];
  DeviceLimits d;
  int coop = 0, optin = 0;
  bool ok = cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && coop &&
            cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess;
  d.smem = optin;
  d.cluster = RES_CLUSTER;
  ok = ok && raise_limits<WarpKind>(d, optin) && raise_limits<PoissonKind>(d, optin) &&
       raise_limits<MeshKind<false>>(d, optin) && raise_limits<MeshKind<true>>(d, optin) &&
       raise_limits<WarpGraphKind>(d, optin) && raise_limits<EmbeddedKind>(d, optin);
  if (!ok) {
    (void)cudaGetLastError();
    d = DeviceLimits{};
  }
  d.sms = std::min(d.sms, RES_MAX_BLOCKS);
  known[dev] = true;
  lim[dev] = d;
  return d;
}

struct Shape {
  int NX, NM, NR;
  int PT, ND, NS;       // graphs: table planes
};
template <class K>
Shape graph_shape() {
  return {K::NX, K::NM, K::NR, K::PT, K::ND, K::NS};
}
Shape shape_of(int kind) {
  switch (kind) {
    case K_WARP: return {WarpKind::NX, WarpKind::NM, WarpKind::NR, WarpKind::NX, WarpKind::NX, 0};
    case K_POISSON: return {PoissonKind::NX, PoissonKind::NM, PoissonKind::NR, PoissonKind::NX, PoissonKind::NX, 0};
    case K_WARPG: return graph_shape<WarpGraphKind>();
    case K_EMBED: return graph_shape<EmbeddedKind>();
    default: return graph_shape<MeshKind<false>>();
  }
}

}  // namespace

// float4 the loop needs for `recs` records in each buffer
size_t resident_records(int kind, long long recs) {
  const Shape s = shape_of(kind);
  return (size_t)(3 * s.NR + (kind == K_WARP ? 1 : 0)) * recs;
}

// Times below: LM 2 x 15, us.
// Up to so many units one cluster takes the problem: it is as fast or faster for every
// kind below (warp of 4,800 pixels 245 against 307 over the device, mesh of 642 vertices 293
// / 315, of 2,562 310 / 331, sheet of 7,920 354 / 346, embedded 2,562 358 / 364, graph 7,650 288
// / 324), and slower above where a unit is much work (mesh of 10,242 431 / 337, embedded
// 527 / 388, volume 24^3 476 / 361; 15,360 pixels 318 / 311).
#ifndef RES_CLUSTER_UNITS
#define RES_CLUSTER_UNITS 8192
#endif
// Over the device, up to so many voxels a block RES_LANES threads share one: 26^3 373 against
// 405 with one thread, 40^3 563 against 424.  (Edge lists lose: mesh of 2,562 350 / 310.)
#ifndef RES_LANE_UNITS
#define RES_LANE_UNITS 256
#endif
// Over the device, up to so many units z goes through records (RES_Z): one meeting an
// iteration less for twice the records read.  Sheet of 32,040 366 against 375 without, mesh
// of 10,242 346 / 365, graph 328 / 338, pixels equal; still 1 to 4 % at 62,500; far above the
// reads cost more (LM / GN 2 x 30: embedded 163,842 3.02 / 1.97 ms, Poisson of 315,000 pixels 699 /
// 614).
#ifndef RES_Z_UNITS
#define RES_Z_UNITS 32768
#endif
// Blocks, shared memory and what it holds for a problem of n units (pixels of
// the listed cells, or vertices); blocks = 0 if the state does
// not fit.  orow: the CSR rows of a graph whose edges are given both ways (else
// NULL).
ResidentPlan resident_plan(int kind, int n, long long plane, int lm, const int* orow) {
  ResidentPlan rp = {};
  const DeviceLimits d = device_limits();
  if (d.smem <= 0 || n <= 0) return rp;
  const bool grid = kind == K_WARP || kind == K_POISSON;
  const Shape s = shape_of(kind);
  const int quantum = grid ? CELL : 32;
  const long long room = d.smem / 4;
  auto fill = [&](int blocks, int least) {
    rp = ResidentPlan{};
    rp.n = n;
    rp.plane = plane;
    const long long want = std::max<long long>(least, (n + (long long)blocks - 1) / blocks);
    rp.per = (int)((want + quantum - 1) / quantum * quantum);
    rp.blocks = (n + rp.per - 1) / rp.per;
    rp.recs = grid ? n : plane;
    const long long per = rp.per;
    // r, q, M^-1, flags; the direction and what is derived from it; records and cells
    long long words = per * (2 * s.NX + s.NM + 1 + (s.NX - s.PT) + s.ND + (grid ? 1 : 0)) + (grid ? per / CELL * 4 : 0);
    auto take = [&](long long w, int flag) {
      if (words + w > room) return false;
      words += w;
      rp.flags |= flag;
      return true;
    };
    if (words > room) return false;
    rp.lanes = 1;
    if (orow) {
      int most = 0;
      for (int b = 0; b < rp.blocks; ++b)
        most = std::max(most, orow[std::min(n, (b + 1) * rp.per)] - orow[b * rp.per]);
      // the lists, and the table: entries for as many edges as leave a run of
      // that many vertices in locality order (measured at most 14 sqrt(per) on
      // sheets and 22 on icospheres; a block where more leave reads records)
      const long long slots = std::min<long long>(most, (long long)(24.0 * std::sqrt((double)per)) + 32);
      if (take(per + 1 + most + slots * (s.ND + 1) + s.NS * (per + slots), RES_LIST)) rp.slots = (int)slots;
      else take(per + 1 + most, RES_LIST);
    }
    const bool dfit = take(per * s.NX, RES_D);
    const bool cfit = !lm || take(per * s.NM, RES_DC);
    if (grid && !(dfit && cfit)) return false;
    rp.smem = (int)(words * 4);
    return true;
  };
  if (n <= RES_CLUSTER_UNITS && d.cluster >= 8 && fill(d.cluster, 256) && (rp.flags & RES_D)) {
    rp.cluster = 1;
    return rp;
  }
  if (!fill(d.sms, grid ? CELL : 64)) return ResidentPlan{};
  if (n <= RES_Z_UNITS) rp.flags |= RES_Z;
  if (kind == K_VOLUME && rp.per <= RES_LANE_UNITS) rp.lanes = RES_LANES;
  return rp;
}

cudaError_t launch_exchange_selftest(ResidentSync* sync, int kind, int rounds, int* out, cudaStream_t st) {
  void* args[] = {&sync, &kind, &rounds, &out};
  return cudaLaunchCooperativeKernel((const void*)k_exchange_selftest, dim3(5), dim3(RT), args, 0, st);
}

cudaError_t launch_resident_grid(int kind, const GridProb* probs, const int* cells, const int4* places, ResidentSync* sync,
                                 const ResidentPlan& rp, float4* rec, int inner, int step, int csn_out,
                                 cudaStream_t st) {
  return kind == K_WARP ? launch<WarpKind>(probs, cells, places, sync, rp, rec, inner, step, csn_out, st)
                        : launch<PoissonKind>(probs, cells, places, sync, rp, rec, inner, step, 0, st);
}

cudaError_t launch_resident_graph(int kind, const MeshProb* probs, ResidentSync* sync, const ResidentPlan& rp,
                                  float4* rec, int inner, int step, cudaStream_t st) {
  switch (kind) {
    case K_VOLUME: return launch<MeshKind<true>>(probs, nullptr, nullptr, sync, rp, rec, inner, step, 0, st);
    case K_WARPG: return launch<WarpGraphKind>(probs, nullptr, nullptr, sync, rp, rec, inner, step, 0, st);
    case K_EMBED: return launch<EmbeddedKind>(probs, nullptr, nullptr, sync, rp, rec, inner, step, 0, st);
    default: return launch<MeshKind<false>>(probs, nullptr, nullptr, sync, rp, rec, inner, step, 0, st);
  }
}

}  // namespace optgb
