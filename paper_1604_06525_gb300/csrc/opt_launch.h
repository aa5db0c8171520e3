// Host-side launch descriptors and launchers of the solver kernels.
#pragma once

#include "opt_internal.cuh"

namespace optgb {

struct GridLaunch {
  const GridProb* probs;
  const Chunk* chunks;
  const int* tiles;
  double* part;
  int nchunks;
  cudaStream_t stream;
  int tw;        // tile width of every problem in the launch (32 or 128)
  int masked;    // every problem in the launch has a mask (wide warp kernel variant)
  int lattice;   // every problem in the launch has GridProb::lattice (wide warp kernel variant)
};

struct MeshLaunch {
  const MeshProb* probs;
  const Chunk* vchunks;
  const Chunk* echunks;
  double* part;
  int nvchunks, nechunks;
  cudaStream_t stream;
  int dim;       // 3: ARAP mesh (6 unknowns per vertex); 2: warp on a graph (3 unknowns);
                 // 12: embedded deformation (12 unknowns)
  int grid3;     // dim 3 on a W x H x D voxel grid: neighbours from the 7-point stencil, not the lists
  const Chunk* tchunks;   // one chunk per vertex tile (tiled ARAP-mesh apply), NULL if not every problem is tiled
  int ntchunks;
};

// Launches kernel k with programmatic stream serialization (the kernel must
// begin with pdl_begin()).  Works inside stream capture as well.
template <typename... KArgs, typename... Args>
inline void launch_pdl(void (*k)(KArgs...), unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                       Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k, static_cast<KArgs>(args)...);
}

// grid_kernels.cu
cudaError_t grid_kernels_prepare();   // one-time kernel attributes (call outside capture)
// csn_in (wide warps): PCGInit reads cos / sin of theta from the planes an
// outer update (csn_out) or launch_grid_csn wrote instead of evaluating them
void launch_grid_init(int kind, const GridLaunch& L, int k_outer, float dmin, float dmax, int csn_in);
void launch_grid_apply(int kind, const GridLaunch& L, const float* p_override, int par, int update);
void launch_grid_update(int kind, const GridLaunch& L, int par);
void launch_grid_energy(int kind, const GridLaunch& L, int mode, int hist_idx);
// Single-reduction PCG (warp or Poisson on 128-pixel tiles; problems planned
// with z / w buffers): iteration `it` (0 starts from r_0, M^-1), and the
// pending step of the last iteration (p of parity par = the iteration count);
// step = 1 also applies the Gauss-Newton update x += delta (csn_out, warp:
// and cos / sin of theta)
void launch_grid_fused(int kind, const GridLaunch& L, int it);
void launch_grid_fused_fin(int kind, const GridLaunch& L, int par, int step, int csn_out);
void launch_grid_step(int kind, const GridLaunch& L, int cond, int csn_out);
// cos / sin of theta at the current unknowns into the cos / sin planes (wide warps)
void launch_grid_csn(const GridLaunch& L);
// Poisson, tile width 128: the degree plane the wide kernels read (S_i + 1 on
// free pixels, 0 elsewhere; pitched like the mask, P x H bytes)
void launch_pois_sdeg(int W, int H, int P, const uint8_t* mask, uint8_t* out, cudaStream_t st);
// found (device, two zeros before): [0] a constant is not finite, [1] (lattice != 0) the
// first two planes are not the pixel lattice up to an offset
void launch_grid_check(int W, int H, int P, const float* c, long long plane, int nc, int lattice, int* found,
                       cudaStream_t st);
// Persistent PCG loop (wide warp tiles only): the largest chunk count whose
// blocks are all resident at once (0 if unknown), and the cooperative launch
// of n_inner PCG iterations (applyJTJ + update) starting at parity par0.
int grid_coop_capacity(int masked);
cudaError_t launch_grid_pcg_coop(const GridLaunch& L, GridBarrier* gb, int par0, int n_inner);
// bounded staging-wait self-test (complete = 0: the wait runs out)
cudaError_t launch_staging_selftest(int complete, unsigned long long limit_ns, int* out, cudaStream_t st);
cudaError_t launch_barrier_selftest(GridBarrier* gb, int nblocks, unsigned int expected, int rounds,
                                    unsigned long long limit_ns, cudaStream_t st);

// resident.cu: the PCG loop of one outer iteration in one launch with the state
// on chip.  orow (graphs; NULL for voxel grids): host copy of the CSR rows.
// cells (grids): the 32 x 8 pixel cells with an unknown, (row << 16) | column, ascending;
// places: of each cell, GridCtx::cell (resident.cu).
// rec: resident_records() float4.  step: x += delta at the end (Gauss-Newton);
// csn_out (wide warps): also cos / sin of the new theta.
ResidentPlan resident_plan(int kind, int n, long long plane, int lm, const int* orow);
size_t resident_records(int kind, long long recs);
cudaError_t launch_resident_grid(int kind, const GridProb* probs, const int* cells, const int4* places, ResidentSync* sync,
                                 const ResidentPlan& rp, float4* rec, int inner, int step, int csn_out,
                                 cudaStream_t st);
cudaError_t launch_resident_graph(int kind, const MeshProb* probs, ResidentSync* sync, const ResidentPlan& rp,
                                  float4* rec, int inner, int step, cudaStream_t st);

// Self-tests: `rounds` exchanges of 5 blocks (kind 0: meetings, 1: float32 sums; fp64.cu:
// sums and meetings of the float64 loop).  out: [0] a wait ran out, [1] a total was wrong
cudaError_t launch_exchange_selftest(ResidentSync* sync, int kind, int rounds, int* out, cudaStream_t st);
cudaError_t launch_exchange_selftest64(ResidentSync* sync, int rounds, int* out, cudaStream_t st);

// edge_plan.cu: the edges of a graph in the internal vertex order.  v0, v1: the
// caller's; iperm: internal number of every caller vertex; e0, e1, isrc: E entries; orow,
// irow: V + 1 zeros before the call; cursor: 2 (V + 1); degw: w_fit at handles, else 0,
// before the call; flags (zeros): [0] an edge is no edge, [1] some edge is given one way, [2]
// how many long rows there are; long_rows: the first EDGE_LONG_ROWS of them (a vertex, or V +
// it for its in-edges), which the caller sorts, then asks for flags[1] again.
constexpr int EDGE_LONG_ROWS = 64;
struct EdgePlan {
  const int *v0, *v1, *iperm;
  int V, E;
  int *e0, *e1, *orow, *irow, *isrc, *cursor;
  float* degw;
  float w_reg;
  int *flags, *long_rows;
};
cudaError_t launch_edge_plan(const EdgePlan& p, cudaStream_t st);
cudaError_t launch_edge_sym(const EdgePlan& p, cudaStream_t st);

// graph_kernels.cu
void launch_mesh_init(const MeshLaunch& L, int k_outer, float dmin, float dmax);
void launch_mesh_apply(const MeshLaunch& L, const float* p_override, int par, int update);
void launch_mesh_update(const MeshLaunch& L, int par);
void launch_mesh_energy(const MeshLaunch& L, int mode, int hist_idx);
void launch_mesh_step(const MeshLaunch& L, int cond);

// graph2d_kernels.cu (dim == 2; reached through the launch_mesh_* functions)
void launch_wg_init(const MeshLaunch& L, int k_outer, float dmin, float dmax);
void launch_wg_apply(const MeshLaunch& L, const float* p_override, int par, int update);
void launch_wg_update(const MeshLaunch& L, int par);
void launch_wg_energy(const MeshLaunch& L, int mode, int hist_idx);
void launch_wg_step(const MeshLaunch& L, int cond);

// embedded_kernels.cu (dim == 12; reached through the launch_mesh_* functions)
void launch_ed_init(const MeshLaunch& L, int k_outer, float dmin, float dmax);
void launch_ed_apply(const MeshLaunch& L, const float* p_override, int par, int update);
void launch_ed_update(const MeshLaunch& L, int par);
void launch_ed_energy(const MeshLaunch& L, int mode, int hist_idx);
void launch_ed_step(const MeshLaunch& L, int cond);

}  // namespace optgb
