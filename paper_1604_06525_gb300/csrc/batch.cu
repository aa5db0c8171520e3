// Batched solves: many uneven problems advanced together, one launch per
// phase for the whole batch (the batched precision form of the solver).
//
// The solver kernels already read their problem from a table (probs[chunk.prob])
// and reduce per problem, so a batch is a combined table: every member's
// descriptor (with its own device scalars, vectors and energy history), a
// combined list of tiles (grid) or vertex / edge ranges (graph), and chunks that
// never straddle two problems.  Each phase (PCGInit, applyJTJ, vector update,
// outer update, energies) is one launch per energy kind covering all members;
// members advance in lock-step through the same outer / inner counts, and every
// scalar (alpha, beta, energies, LM damping) stays per problem on the
// device.  The whole batched solve is captured once as a CUDA graph.
//
// The chunk granularity (tiles per chunk) is picked by a small autotuner that
// times one outer iteration of the batch for each candidate.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <memory>
#include <vector>

#include "opt_gb300.h"
#include "opt_internal.cuh"
#include "opt_launch.h"
#include "opt_problem.h"

using namespace optgb;

namespace {

#define BCK(call)                                              \
  do {                                                         \
    cudaError_t e_ = (call);                                   \
    if (e_ != cudaSuccess) {                                   \
      (void)cudaGetLastError();                                \
      return e_ == cudaErrorMemoryAllocation ? OPT_ERR_OOM : OPT_ERR_CUDA; \
    }                                                          \
  } while (0)

struct PlaneCopy {
  const float* src;
  float* dst;
  int rows, cols;
  int src_pitch, dst_pitch;   // in floats
  const int* perm;            // graphs (one row): internal vertex k = caller vertex perm[k]
  int to_caller;              // with perm: 1 = internal -> caller order, 0 = caller -> internal
  int pad;
};

__global__ void k_copy_planes(const PlaneCopy* __restrict__ tab, int n) {
  const PlaneCopy c = tab[blockIdx.y];
  const long long total = (long long)c.rows * c.cols;
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < total;
       k += (long long)gridDim.x * blockDim.x) {
    if (c.perm) {
      const int v = c.perm[k];
      if (c.to_caller) c.dst[v] = c.src[k];
      else c.dst[k] = c.src[v];
      continue;
    }
    const int r = (int)(k / c.cols), col = (int)(k - (long long)r * c.cols);
    c.dst[(long long)r * c.dst_pitch + col] = c.src[(long long)r * c.src_pitch + col];
  }
}

__global__ void k_reset_tab(Scalars* const* __restrict__ tab, int n, double lambda0) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) scalars_reset(tab[i], lambda0);
}

__global__ void k_lm_decide_tab(Scalars* const* __restrict__ tab, int n, double eta, double lmin, double lmax,
                                double rel_tol) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) lm_decide(tab[i], eta, lmin, lmax, rel_tol);
}

// Each member's round record (server rounds).
__global__ void k_record_round(Scalars* const* __restrict__ tab, int n, RoundRec* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const Scalars* t = tab[i];
  out[i] = RoundRec{t->E, t->E_trial, t->accept, t->outer_done};
}

// Copies every member's scalars and energy history into contiguous buffers.
__global__ void k_gather_results(Scalars* const* __restrict__ tab, double* const* __restrict__ hist, int n,
                                 int hlen, Scalars* __restrict__ s_out, double* __restrict__ h_out) {
  const int i = blockIdx.x;
  if (i >= n) return;
  if (threadIdx.x == 0) s_out[i] = *tab[i];
  for (int k = threadIdx.x; k < hlen; k += blockDim.x) h_out[(long long)i * hlen + k] = hist[i][k];
}

template <class T>
opt_status balloc(std::vector<void*>& allocs, T** ptr, size_t n) {
  void* p = nullptr;
  BCK(cudaMalloc(&p, std::max<size_t>(n, 1) * sizeof(T)));
  allocs.push_back(p);
  *ptr = static_cast<T*>(p);
  return OPT_OK;
}

template <class T>
opt_status bupload(std::vector<void*>& allocs, T** ptr, const std::vector<T>& v) {
  opt_status s = balloc(allocs, ptr, v.size());
  if (s != OPT_OK) return s;
  if (!v.empty()) BCK(cudaMemcpy(*ptr, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice));
  return OPT_OK;
}

struct GridGroup {
  int kind = 0;
  int tw = 32;
  int masked = 0;
  int lattice = 0;                     // every member has GridProb::lattice
  std::vector<int> members;            // indices into opt_batch::probs
  GridProb* d_probs = nullptr;
  std::vector<GridProb> h_probs;       // as on the device
  Chunk* d_chunks = nullptr;
  int* d_tiles = nullptr;
  double* d_part = nullptr;
  int nchunks = 0;
};

struct MeshGroup {
  int dim = 3;                         // 3: ARAP mesh, 2: warp on a graph, 12: embedded deformation
  int grid3 = 0;                       // volumetric problems (7-point stencil)
  std::vector<int> members;
  MeshProb* d_probs = nullptr;
  std::vector<MeshProb> h_probs;       // as on the device
  Chunk* d_vch = nullptr;
  Chunk* d_ech = nullptr;
  Chunk* d_tch = nullptr;              // tile chunks of the tiled ARAP-mesh apply (NULL: some member untiled)
  double* d_part = nullptr;
  int nv = 0, ne = 0, nt = 0;
};

}  // namespace

struct opt_batch {
  std::vector<opt_problem*> probs;
  std::vector<GridGroup> grids;
  MeshGroup graphs[4];               // [0]: ARAP meshes, [1]: warps on graphs, [2]: volumes,
                                     // [3]: embedded deformation
  int tiles_per_chunk = 0;          // 0 = default
  std::vector<void*> table_allocs;  // rebuilt with the chunking
  std::vector<void*> allocs;        // fixed for the batch's life
  Scalars** d_stab = nullptr;
  double** d_htab = nullptr;
  std::vector<double*> h_htab;      // as on the device (none yet: nullptr)
  PlaneCopy* d_copy_in = nullptr;
  PlaneCopy* d_copy_out = nullptr;
  int ncopy = 0, max_plane = 0;
  Scalars* d_sout = nullptr;
  double* d_hout = nullptr;
  int hcap = 0;
  RoundRec* d_rounds = nullptr;     // server rounds: records, round-major
  int rounds_cap = 0;
  cudaStream_t cap_stream = nullptr;
  cudaGraphExec_t gexec = nullptr;
  std::vector<double> gkey;
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
  // a stream for each group after the first, with the event that ends its work;
  // the event that begins it
  std::vector<cudaStream_t> side;
  std::vector<cudaEvent_t> side_done;
  cudaEvent_t fork = nullptr;

  ~opt_batch() {
    for (cudaStream_t t : side) cudaStreamDestroy(t);
    for (cudaEvent_t e : side_done) cudaEventDestroy(e);
    if (fork) cudaEventDestroy(fork);
    if (gexec) cudaGraphExecDestroy(gexec);
    if (cap_stream) cudaStreamDestroy(cap_stream);
    if (ev0) cudaEventDestroy(ev0);
    if (ev1) cudaEventDestroy(ev1);
    for (void* p : table_allocs) cudaFree(p);
    for (void* p : allocs) cudaFree(p);
  }
};

namespace {

bool is_grid_kind(int k) { return k == K_WARP || k == K_POISSON; }

// Tiles per chunk of a group of grids: the fewest for which all chunks of the
// group are on the device at once, two blocks per SM (the residency of the
// wide-tile kernels).  A member's own split is for the device to itself -- one
// tile per block up to 304 tiles -- and in a group every such block pays the
// descriptor, the partial sums and its share of another wave: 96 warps of 32^2 to
// 512^2, GN 3 x 10: 9.1 ms with the members' own splits, 6.5 ms so; at most 4 or 6
// tiles per chunk 6.8 and 6.7 ms, two or four waves of smaller chunks 7.0 and 6.9 ms.
// With so many members that one wave would take chunks half as large again as a
// block's even share, a quarter of that share: the device then evens itself out.
int one_wave_tiles(const std::vector<int>& ntiles, int blocks) {
  const auto chunks = [&](int per) {
    long long c = 0;
    for (int t : ntiles) c += (t + per - 1) / per;
    return c;
  };
  int lo = 1, hi = 1;
  for (int t : ntiles) hi = std::max(hi, t);
  while (lo < hi) {
    const int mid = (lo + hi) / 2;
    if (chunks(mid) <= blocks) hi = mid;
    else lo = mid + 1;
  }
  long long total = 0;
  for (int t : ntiles) total += t;
  return 2ll * lo * blocks <= 3 * total || lo == 1 ? lo : std::max<int>(1, (int)(total / (4ll * blocks)));
}

// (Re)builds the combined work tables with `tpc` tiles per chunk (0 = each
// member's own chunking, or one_wave_tiles() of its group where that is coarser).
opt_status build_tables(opt_batch* b, int tpc) {
  cudaDeviceSynchronize();
  for (void* p : b->table_allocs) cudaFree(p);
  b->table_allocs.clear();
  if (b->gexec) {
    cudaGraphExecDestroy(b->gexec);
    b->gexec = nullptr;
    b->gkey.clear();
  }
  for (GridGroup& g : b->grids) {
    std::vector<GridProb> gp;
    std::vector<Chunk> chunks;
    std::vector<int> tiles, nt;
    for (int i : g.members) nt.push_back(b->probs[i]->ntiles);
    g.lattice = 1;
    for (int i : g.members) g.lattice = g.lattice && b->probs[i]->hg.lattice;
    const int wave = one_wave_tiles(nt, 2 * b->probs[0]->sms);
    for (size_t mi = 0; mi < g.members.size(); ++mi) {
      opt_problem* pb = b->probs[g.members[mi]];
      const std::vector<int>& t = pb->h_tiles;
      GridProb d = pb->hg;
      d.chunk_begin = (int)chunks.size();
      const int base = (int)tiles.size();
      if (tpc > 0) {
        for (int s = 0; s < pb->ntiles; s += tpc)
          chunks.push_back(Chunk{(int)mi, base + s, base + std::min(s + tpc, pb->ntiles), 0});
      } else if ((pb->ntiles + wave - 1) / wave < (int)pb->h_chunks.size()) {
        const int n = (pb->ntiles + wave - 1) / wave;   // sizes differ by at most one tile
        for (int k = 0; k < n; ++k)
          chunks.push_back(Chunk{(int)mi, base + (int)((long long)pb->ntiles * k / n),
                                 base + (int)((long long)pb->ntiles * (k + 1) / n), 0});
      } else {
        // the member's own split: identical reductions to its solo solve
        for (Chunk c : pb->h_chunks) chunks.push_back(Chunk{(int)mi, base + c.begin, base + c.end, 0});
      }
      d.chunk_end = (int)chunks.size();
      tiles.insert(tiles.end(), t.begin(), t.end());
      gp.push_back(d);
    }
    opt_status s;
    if ((s = bupload(b->table_allocs, &g.d_probs, gp)) != OPT_OK) return s;
    if ((s = bupload(b->table_allocs, &g.d_chunks, chunks)) != OPT_OK) return s;
    if ((s = bupload(b->table_allocs, &g.d_tiles, tiles)) != OPT_OK) return s;
    if ((s = balloc(b->table_allocs, &g.d_part, 8 * chunks.size())) != OPT_OK) return s;   // up to 4 Sums
    g.nchunks = (int)chunks.size();
    g.h_probs = gp;
  }
  for (MeshGroup& g : b->graphs) {
    if (g.members.empty()) continue;
    std::vector<MeshProb> mp;
    std::vector<Chunk> vch, ech, tch;
    bool tiled = true;
    for (size_t mi = 0; mi < g.members.size(); ++mi) {
      const opt_problem* pm = b->probs[g.members[mi]];
      tiled = tiled && pm->d_tchunks && pm->apply_form;
    }
    for (size_t mi = 0; mi < g.members.size(); ++mi) {
      opt_problem* pb = b->probs[g.members[mi]];
      const std::vector<Chunk>& v = pb->h_vch;
      const std::vector<Chunk>& e = pb->h_ech;
      MeshProb d = pb->hm;
      d.vchunk_begin = (int)vch.size();
      for (Chunk c : v) { c.prob = (int)mi; vch.push_back(c); }
      d.vchunk_end = (int)vch.size();
      d.echunk_begin = (int)ech.size();
      for (Chunk c : e) { c.prob = (int)mi; ech.push_back(c); }
      d.echunk_end = (int)ech.size();
      d.tchunk_begin = (int)tch.size();
      if (tiled) {
        for (Chunk c : pb->h_tch) { c.prob = (int)mi; tch.push_back(c); }
      }
      d.tchunk_end = (int)tch.size();
      mp.push_back(d);
    }
    opt_status s;
    if ((s = bupload(b->table_allocs, &g.d_probs, mp)) != OPT_OK) return s;
    if ((s = bupload(b->table_allocs, &g.d_vch, vch)) != OPT_OK) return s;
    if ((s = bupload(b->table_allocs, &g.d_ech, ech)) != OPT_OK) return s;
    g.d_tch = nullptr;
    if (tiled && (s = bupload(b->table_allocs, &g.d_tch, tch)) != OPT_OK) return s;
    if ((s = balloc(b->table_allocs, &g.d_part, 2 * std::max({vch.size(), ech.size(), tch.size()}))) != OPT_OK)
      return s;
    g.nv = (int)vch.size();
    g.ne = (int)ech.size();
    g.nt = tiled ? (int)tch.size() : 0;
    g.h_probs = mp;
  }
  b->tiles_per_chunk = tpc;
  return OPT_OK;
}

GridLaunch gl(const GridGroup& g, cudaStream_t st) {
  return GridLaunch{g.d_probs, g.d_chunks, g.d_tiles, g.d_part, g.nchunks, st, g.tw, g.masked, g.lattice};
}
MeshLaunch ml(const MeshGroup& g, cudaStream_t st) {
  return MeshLaunch{g.d_probs, g.d_vch, g.d_ech, g.d_part, g.nv, g.ne, st, g.dim, g.grid3, g.d_tch, g.nt};
}

// Uploads the members' descriptors with the solve's flags (outside any capture).
opt_status refresh_descriptors(opt_batch* b, int lm, int use_precond, int outer, cudaStream_t st) {
  for (opt_problem* pb : b->probs) {
    if (pb->Ehist_cap < outer + 1) {
      double* e = nullptr;
      void* p = nullptr;
      BCK(cudaMalloc(&p, sizeof(double) * (outer + 1)));
      pb->allocs.push_back(p);
      pb->pooled.push_back(false);
      e = static_cast<double*>(p);
      pb->d_Ehist = e;
      pb->Ehist_cap = outer + 1;
      if (pb->gexec) {
        cudaGraphExecDestroy(pb->gexec);
        pb->gexec = nullptr;
        pb->gkey.clear();
      }
    }
  }
  bool waited = false;
  // copies host -> device only what differs from what is there, after the stream's work
  const auto put = [&](void* dev, void* there, const void* want, size_t bytes) -> opt_status {
    if (!std::memcmp(there, want, bytes)) return OPT_OK;
    if (!waited) BCK(cudaStreamSynchronize(st));
    waited = true;
    BCK(cudaMemcpy(dev, want, bytes, cudaMemcpyHostToDevice));
    std::memcpy(there, want, bytes);
    return OPT_OK;
  };
  const auto refresh = [&](auto& g) -> opt_status {
    auto want = g.h_probs;
    for (size_t i = 0; i < want.size(); ++i) {
      want[i].lm = lm;
      want[i].use_precond = use_precond;
      want[i].Ehist = b->probs[g.members[i]]->d_Ehist;
      want[i].jtf_out = nullptr;
      want[i].diag_out = nullptr;
    }
    return put(g.d_probs, g.h_probs.data(), want.data(), want.size() * sizeof(want[0]));
  };
  opt_status s;
  for (GridGroup& g : b->grids)
    if ((s = refresh(g)) != OPT_OK) return s;
  for (MeshGroup& g : b->graphs)
    if (!g.members.empty() && (s = refresh(g)) != OPT_OK) return s;
  std::vector<double*> ht;
  for (opt_problem* pb : b->probs) ht.push_back(pb->d_Ehist);
  b->h_htab.resize(ht.size(), nullptr);
  return put(b->d_htab, b->h_htab.data(), ht.data(), ht.size() * sizeof(double*));
}

void enqueue_copies(opt_batch* b, const PlaneCopy* tab, cudaStream_t st) {
  if (b->ncopy == 0) return;
  const int bx = std::max(1, std::min(64, (b->max_plane + 255) / 256));
  k_copy_planes<<<dim3(bx, b->ncopy), 256, 0, st>>>(tab, b->ncopy);
}

// The groups of a batch touch nothing of one another's between two LM decisions, so
// each takes its launches on a stream of its own, from fork_groups() to
// join_groups(): a small group's kernels, which leave most of the device idle, run
// beside a large group's instead of before and after them (96 warps of 32^2 to 512^2,
// GN 3 x 10, narrow and wide tiles: 6.5 -> 5.9 ms; 22 warps up to 251^2: 1.62 ->
// 1.31 ms; a served mix of warps and meshes, LM 4 x 10: 14.0 -> 12.2 ms).
template <class Grid, class Graph>
void for_groups(opt_batch* b, cudaStream_t st, Grid&& grid, Graph&& graph) {
  size_t lane = 0;
  const auto next = [&] { return lane++ == 0 ? st : b->side[lane - 2]; };
  for (GridGroup& g : b->grids) grid(g, gl(g, next()));
  for (const MeshGroup& g : b->graphs)
    if (!g.members.empty()) graph(ml(g, next()));
}
void fork_groups(opt_batch* b, cudaStream_t st) {
  if (b->side.empty()) return;
  cudaEventRecord(b->fork, st);
  for (cudaStream_t t : b->side) cudaStreamWaitEvent(t, b->fork, 0);
}
void join_groups(opt_batch* b, cudaStream_t st) {
  for (size_t k = 0; k < b->side.size(); ++k) {
    cudaEventRecord(b->side_done[k], b->side[k]);
    cudaStreamWaitEvent(st, b->side_done[k], 0);
  }
}

// wide-tile warp and Poisson groups take the single-reduction PCG iteration when
// asked for (as a solo solve of each member would), the others the two-pass one
bool group_fused(const GridGroup& g, const opt_solve_params& p) {
  return p.pcg_form == 1 && p.inner > 0 && (g.kind == K_WARP || g.kind == K_POISSON) && g.tw == 128;
}

// PCGInit and `inner` PCG iterations of every group.  k: outer iteration; csn_in:
// the wide warps' cos / sin of theta come from the previous outer update; fin_step,
// csn_out: the single-reduction groups' last step also does x += delta.
void enqueue_pcg(opt_batch* b, const opt_solve_params& p, cudaStream_t st, int k, int csn_in, int fin_step,
                 int csn_out) {
  const float dmin = (float)p.diag_min, dmax = (float)p.diag_max;
  for_groups(
      b, st,
      [&](const GridGroup& g, const GridLaunch& L) {
        const bool fused = group_fused(g, p);
        launch_grid_init(g.kind, L, k, dmin, dmax, csn_in);
        for (int i = 0; i < p.inner; ++i) {
          if (fused) {
            launch_grid_fused(g.kind, L, i);
          } else {
            launch_grid_apply(g.kind, L, nullptr, i, 1);
            launch_grid_update(g.kind, L, i);
          }
        }
        if (fused) launch_grid_fused_fin(g.kind, L, p.inner, fin_step, csn_out);
      },
      [&](const MeshLaunch& L) {
        launch_mesh_init(L, k, dmin, dmax);
        for (int i = 0; i < p.inner; ++i) {
          launch_mesh_apply(L, nullptr, i, 1);
          launch_mesh_update(L, i);
        }
      });
}
void enqueue_energy(opt_batch* b, cudaStream_t st, int mode, int hist) {
  for_groups(
      b, st, [&](const GridGroup& g, const GridLaunch& L) { launch_grid_energy(g.kind, L, mode, hist); },
      [&](const MeshLaunch& L) { launch_mesh_energy(L, mode, hist); });
}
// `fused_too`: the single-reduction groups have not stepped yet
void enqueue_step(opt_batch* b, const opt_solve_params& p, cudaStream_t st, int conditional, int csn_out,
                  bool fused_too) {
  for_groups(
      b, st,
      [&](const GridGroup& g, const GridLaunch& L) {
        if (fused_too || !group_fused(g, p)) launch_grid_step(g.kind, L, conditional, csn_out);
      },
      [&](const MeshLaunch& L) { launch_mesh_step(L, conditional); });
}

// The whole solve as stream work.
void enqueue_batch(opt_batch* b, const opt_solve_params& p, bool lm, cudaStream_t st, int outer, bool write_back) {
  const int n = (int)b->probs.size();
  enqueue_copies(b, b->d_copy_in, st);
  k_reset_tab<<<(n + 127) / 128, 128, 0, st>>>(b->d_stab, n, lm ? p.lambda0 : 0.0);
  fork_groups(b, st);
  for (int k = 0; k < outer; ++k) {
    // from the second outer iteration on, the wide warps' cos / sin of theta
    // come from the previous outer update
    const int csn_next = k + 1 < outer;
    enqueue_pcg(b, p, st, k, k > 0, lm ? 0 : 1, lm ? 0 : csn_next);
    if (!lm) {
      enqueue_step(b, p, st, 0, csn_next, false);
    } else {
      enqueue_energy(b, st, 1, -2);
      join_groups(b, st);
      k_lm_decide_tab<<<(n + 127) / 128, 128, 0, st>>>(b->d_stab, n, p.eta, p.lambda_min, p.lambda_max, p.rel_tol);
      fork_groups(b, st);
      enqueue_step(b, p, st, 1, csn_next, true);
    }
  }
  enqueue_energy(b, st, 0, lm ? -1 : outer);
  join_groups(b, st);
  if (write_back) enqueue_copies(b, b->d_copy_out, st);
}

opt_status batch_solve(opt_batch* b, const opt_solve_params* prm_in, opt_report* reports, float* ms_out, bool lm,
                       bool write_back = true) {
  if (!b) return OPT_ERR_INVALID_ARG;
  opt_solve_params p;
  if (prm_in) p = *prm_in;
  else opt_solve_params_default(&p);
  if (p.outer < 1 || p.inner < 0 || p.materialized || p.pcg_form < 0 || p.pcg_form > 1) return OPT_ERR_INVALID_ARG;
  if (lm && (!(p.lambda0 >= 0.0) || !(p.lambda_min <= p.lambda_max) || !(p.diag_min <= p.diag_max)))
    return OPT_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)p.stream;
  opt_status s = refresh_descriptors(b, lm ? 1 : 0, p.use_precond, p.outer, st);
  if (s != OPT_OK) return s;
  const int n = (int)b->probs.size();
  const int hlen = p.outer + 1;
  if (b->hcap < hlen) {
    // the members' scalars and histories next to each other: one copy fetches them
    BCK(cudaStreamSynchronize(st));
    char* r = nullptr;
    if ((s = balloc(b->allocs, &r, n * (sizeof(Scalars) + hlen * sizeof(double)))) != OPT_OK) return s;
    b->d_sout = reinterpret_cast<Scalars*>(r);
    b->d_hout = reinterpret_cast<double*>(b->d_sout + n);
    b->hcap = hlen;
  }
  const std::vector<double> key = {double(p.outer), double(p.inner), double(lm), double(p.use_precond), p.lambda0,
                                   p.lambda_min, p.lambda_max, p.diag_min, p.diag_max, p.eta, p.rel_tol,
                                   double(write_back), double(p.pcg_form)};
  if (p.use_graph) {
    if (!b->gexec || key != b->gkey) {
      if (b->gexec) {
        cudaGraphExecDestroy(b->gexec);
        b->gexec = nullptr;
      }
      cudaGraph_t g = nullptr;
      BCK(cudaStreamBeginCapture(b->cap_stream, cudaStreamCaptureModeThreadLocal));
      enqueue_batch(b, p, lm, b->cap_stream, p.outer, write_back);
      const cudaError_t e = cudaStreamEndCapture(b->cap_stream, &g);
      if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return OPT_ERR_CUDA;
      }
      const cudaError_t e2 = cudaGraphInstantiate(&b->gexec, g, 0);
      cudaGraphDestroy(g);
      if (e2 != cudaSuccess) {
        (void)cudaGetLastError();
        return OPT_ERR_CUDA;
      }
      b->gkey = key;
    }
    BCK(cudaEventRecord(b->ev0, st));
    BCK(cudaGraphLaunch(b->gexec, st));
    BCK(cudaEventRecord(b->ev1, st));
  } else {
    BCK(cudaEventRecord(b->ev0, st));
    enqueue_batch(b, p, lm, st, p.outer, write_back);
    BCK(cudaEventRecord(b->ev1, st));
  }
  k_gather_results<<<n, 128, 0, st>>>(b->d_stab, b->d_htab, n, hlen, b->d_sout, b->d_hout);
  BCK(cudaGetLastError());
  std::vector<char> res(n * (sizeof(Scalars) + hlen * sizeof(double)));
  BCK(cudaMemcpyAsync(res.data(), b->d_sout, res.size(), cudaMemcpyDeviceToHost, st));
  BCK(cudaStreamSynchronize(st));
  float ms = 0.f;
  BCK(cudaEventElapsedTime(&ms, b->ev0, b->ev1));
  if (ms_out) *ms_out = ms;
  std::vector<Scalars> sv(n);
  std::vector<double> hv((size_t)n * hlen);
  std::memcpy(sv.data(), res.data(), n * sizeof(Scalars));
  std::memcpy(hv.data(), res.data() + n * sizeof(Scalars), hv.size() * sizeof(double));
  bool nonfinite = false, timeout = false, misaligned = false;
  for (int i = 0; i < n; ++i) {
    const Scalars& t = sv[i];
    nonfinite |= t.nonfinite != 0;
    timeout |= t.timeout != 0;
    misaligned |= t.misaligned != 0;
    if (!reports) continue;
    opt_report& r = reports[i];
    const int od = lm ? t.outer_done : p.outer;
    r.outer_done = od;
    r.pcg_done = t.pcg_iters;
    r.accepted = lm ? t.accepted_total : p.outer;
    r.converged = t.converged;
    r.E0 = hv[(size_t)i * hlen];
    r.E_final = hv[(size_t)i * hlen + od];
    r.lambda_final = lm ? t.lambda : 0.0;
    if (r.E_history) std::memcpy(r.E_history, &hv[(size_t)i * hlen], sizeof(double) * (od + 1));
    r.ms = ms;
  }
  if (timeout) return OPT_ERR_TIMEOUT;
  if (misaligned) return OPT_ERR_CUDA;
  return nonfinite ? OPT_ERR_NUMERIC : OPT_OK;
}

}  // namespace

extern "C" {

opt_status opt_batch_create(opt_problem* const* probs, int32_t n, opt_batch** out) {
  if (!out) return OPT_ERR_INVALID_ARG;
  *out = nullptr;
  if (!probs || n < 1) return OPT_ERR_INVALID_ARG;
  for (int i = 0; i < n; ++i)
    if (!probs[i]) return OPT_ERR_INVALID_ARG;
  for (int i = 0; i < n; ++i)
    for (int j = i + 1; j < n && n <= 4096; ++j)
      if (probs[i] == probs[j]) return OPT_ERR_INVALID_ARG;
  std::unique_ptr<opt_batch> b(new opt_batch());
  b->probs.assign(probs, probs + n);
  // one launch group per (kind, tile width, mask presence): each group runs
  // one kernel variant
  for (int kind : {(int)K_WARP, (int)K_POISSON})
    for (int tw : {32, 128})
      for (int masked : {0, 1}) {
        GridGroup g;
        g.kind = kind;
        g.tw = tw;
        g.masked = masked;
        for (int i = 0; i < n; ++i)
          if (probs[i]->kind == kind && probs[i]->hg.tw == tw && (probs[i]->hg.mask != nullptr) == (masked != 0))
            g.members.push_back(i);
        if (!g.members.empty()) b->grids.push_back(g);
      }
  b->graphs[1].dim = 2;
  b->graphs[2].grid3 = 1;
  b->graphs[3].dim = 12;
  for (int i = 0; i < n; ++i) {
    if (probs[i]->kind == K_MESH) b->graphs[0].members.push_back(i);
    if (probs[i]->kind == K_WARPG) b->graphs[1].members.push_back(i);
    if (probs[i]->kind == K_VOLUME) b->graphs[2].members.push_back(i);
    if (probs[i]->kind == K_EMBED) b->graphs[3].members.push_back(i);
  }
  BCK(cudaStreamCreateWithFlags(&b->cap_stream, cudaStreamNonBlocking));
  BCK(cudaEventCreate(&b->ev0));
  BCK(cudaEventCreate(&b->ev1));
  size_t ngroups = b->grids.size();
  for (const MeshGroup& g : b->graphs) ngroups += !g.members.empty();
  if (ngroups > 1) BCK(cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming));
  for (size_t k = 1; k < ngroups; ++k) {
    cudaStream_t t = nullptr;
    cudaEvent_t e = nullptr;
    BCK(cudaStreamCreateWithFlags(&t, cudaStreamNonBlocking));
    b->side.push_back(t);
    BCK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    b->side_done.push_back(e);
  }
  // scalar and history tables, plane copies
  std::vector<Scalars*> stab;
  std::vector<PlaneCopy> cin, cout_;
  int maxp = 0;
  for (opt_problem* pb : b->probs) {
    stab.push_back(pb->d_s);
    for (int c = 0; c < pb->nx; ++c) {
      if (is_grid_kind(pb->kind)) {
        cin.push_back(PlaneCopy{pb->user_x[c], pb->x + c * pb->plane, pb->H, pb->W, pb->W, pb->P, nullptr, 0, 0});
        cout_.push_back(PlaneCopy{pb->x + c * pb->plane, pb->user_x[c], pb->H, pb->W, pb->P, pb->W, nullptr, 0, 0});
      } else {
        cin.push_back(PlaneCopy{pb->user_x[c], pb->x + c * pb->plane, 1, pb->V, pb->V, pb->V, pb->d_perm, 0, 0});
        cout_.push_back(PlaneCopy{pb->x + c * pb->plane, pb->user_x[c], 1, pb->V, pb->V, pb->V, pb->d_perm, 1, 0});
      }
      maxp = std::max<int>(maxp, (int)pb->ulen);
    }
  }
  opt_status s;
  if ((s = bupload(b->allocs, &b->d_stab, stab)) != OPT_OK) return s;
  if ((s = balloc(b->allocs, &b->d_htab, (size_t)n)) != OPT_OK) return s;
  if ((s = bupload(b->allocs, &b->d_copy_in, cin)) != OPT_OK) return s;
  if ((s = bupload(b->allocs, &b->d_copy_out, cout_)) != OPT_OK) return s;
  if ((s = balloc(b->allocs, &b->d_sout, (size_t)n)) != OPT_OK) return s;
  b->ncopy = (int)cin.size();
  b->max_plane = maxp;
  if ((s = build_tables(b.get(), 0)) != OPT_OK) return s;
  *out = b.release();
  return OPT_OK;
}

opt_status opt_batch_destroy(opt_batch* b) {
  if (!b) return OPT_OK;
  cudaDeviceSynchronize();
  delete b;
  return OPT_OK;
}

opt_status opt_batch_set_chunking(opt_batch* b, int32_t tiles_per_chunk) {
  if (!b || tiles_per_chunk < 0 || tiles_per_chunk > 4096) return OPT_ERR_INVALID_ARG;
  return build_tables(b, tiles_per_chunk);
}

opt_status opt_batch_solve_gn(opt_batch* b, const opt_solve_params* params, opt_report* reports, float* ms) {
  return batch_solve(b, params, reports, ms, false);
}

opt_status opt_batch_solve_lm(opt_batch* b, const opt_solve_params* params, opt_report* reports, float* ms) {
  return batch_solve(b, params, reports, ms, true);
}

opt_status opt_batch_autotune(opt_batch* b, const opt_solve_params* params, int32_t* chosen, float* best_ms) {
  if (!b) return OPT_ERR_INVALID_ARG;
  opt_solve_params p;
  if (params) p = *params;
  else opt_solve_params_default(&p);
  p.outer = 1;
  p.inner = std::max(1, std::min(p.inner, 4));
  p.use_graph = 1;
  const int cand[] = {0, 1, 2, 4, 8, 16};
  int best = 0;
  float bms = 1e30f;
  for (int c : cand) {
    opt_status s = build_tables(b, c);
    if (s != OPT_OK) return s;
    float t = 0.f, tmin = 1e30f;
    for (int rep = 0; rep < 3; ++rep) {
      s = batch_solve(b, &p, nullptr, &t, false, false);
      if (s != OPT_OK && s != OPT_ERR_NUMERIC) return s;
      if (rep > 0) tmin = std::min(tmin, t);
    }
    if (tmin < bms) {
      bms = tmin;
      best = c;
    }
  }
  opt_status s = build_tables(b, best);
  if (s != OPT_OK) return s;
  if (chosen) *chosen = best;
  if (best_ms) *best_ms = bms;
  return OPT_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Internal interface used by the serving engine (serve.cu): one LM outer
// iteration of every member, without energy-history writes, and a gather of
// the members' scalars.
// ---------------------------------------------------------------------------
namespace optgb {

opt_status batch_prepare_round(opt_batch* b, const opt_solve_params& p, cudaStream_t st) {
  return refresh_descriptors(b, 1, p.use_precond, 1, st);
}

opt_status batch_reserve_rounds(opt_batch* b, int rounds) {
  if (rounds <= b->rounds_cap) return OPT_OK;
  opt_status s = balloc(b->allocs, &b->d_rounds, (size_t)rounds * b->probs.size());
  if (s == OPT_OK) b->rounds_cap = rounds;
  return s;
}

void batch_enqueue_lm_round(opt_batch* b, const opt_solve_params& p, cudaStream_t st, int round) {
  const int n = (int)b->probs.size();
  fork_groups(b, st);
  enqueue_pcg(b, p, st, -2, 0, 0, 0);
  enqueue_energy(b, st, 1, -2);
  join_groups(b, st);
  k_lm_decide_tab<<<(n + 127) / 128, 128, 0, st>>>(b->d_stab, n, p.eta, p.lambda_min, p.lambda_max, p.rel_tol);
  fork_groups(b, st);
  enqueue_step(b, p, st, 1, 0, true);
  join_groups(b, st);
  if (round < b->rounds_cap)
    k_record_round<<<(n + 127) / 128, 128, 0, st>>>(b->d_stab, n, b->d_rounds + (size_t)round * n);
  k_gather_results<<<n, 128, 0, st>>>(b->d_stab, b->d_htab, n, 0, b->d_sout, b->d_hout);
}

opt_status batch_read_scalars(opt_batch* b, Scalars* host_out, RoundRec* rounds_out, int rounds, cudaStream_t st) {
  const size_t n = b->probs.size();
  BCK(cudaMemcpyAsync(host_out, b->d_sout, n * sizeof(Scalars), cudaMemcpyDeviceToHost, st));
  if (rounds_out && rounds > 0 && rounds <= b->rounds_cap)
    BCK(cudaMemcpyAsync(rounds_out, b->d_rounds, (size_t)rounds * n * sizeof(RoundRec), cudaMemcpyDeviceToHost, st));
  BCK(cudaStreamSynchronize(st));
  return OPT_OK;
}

}  // namespace optgb
