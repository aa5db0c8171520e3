// Planning of a graph's edges on the device: renumbered into the internal vertex
// order and sorted by (v0, v1), with the rows of the list, the in-edges of every
// vertex (sources ascending) and its summed edge weights.
//
// Counting sort by vertex, then every row by value: the order of the scatter's
// atomics leaves no trace.  Bound by scattered 4-byte accesses; on a host core the
// same passes took most of a mesh's planning (level-6 icosphere, 245,760 edges: 4.7 ms of
// planning, 1.5 ms so).  One thread sorts a row, so rows of hub vertices (more than
// LONG_ROW) are left to the host, up to EDGE_LONG_ROWS of them: a star of 8,000 leaves is planned
// in 1.3 ms instead of 9.8, one of 200,000 in 25 instead of 420.
#include <algorithm>

#include "opt_internal.cuh"
#include "opt_launch.h"

namespace optgb {

namespace {

__global__ void __launch_bounds__(NT) k_edge_count(const EdgePlan p) {
  for (long long e = blockIdx.x * NT + threadIdx.x; e < p.E; e += gridDim.x * NT) {
    const int a = p.v0[e], b = p.v1[e];
    if (a < 0 || a >= p.V || b < 0 || b >= p.V || a == b) {
      p.flags[0] = 1;
      continue;
    }
    atomicAdd(&p.orow[p.iperm[a] + 1], 1);
    atomicAdd(&p.irow[p.iperm[b] + 1], 1);
  }
}

// Running sums of one list's counts (block 0: out-edges, 1: in-edges), eight a thread
// at a time, and a copy for the scatter to advance.
constexpr int SCAN_T = 1024, SCAN_K = 8;
__global__ void __launch_bounds__(SCAN_T) k_edge_rows(const EdgePlan p) {
  __shared__ int warp_sum[32];
  int* row = blockIdx.x ? p.irow : p.orow;
  int* cur = p.cursor + (blockIdx.x ? p.V + 1 : 0);
  const int n = p.V + 1, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  int carry = 0;
  for (int base = 0; base < n; base += SCAN_T * SCAN_K) {
    int v[SCAN_K], sum = 0;
#pragma unroll
    for (int k = 0; k < SCAN_K; ++k) {
      const int i = base + tid * SCAN_K + k;
      v[k] = sum += i < n ? row[i] : 0;
    }
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o *= 2) {
      const int t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) warp_sum[w] = incl;
    __syncthreads();
    if (w == 0) {
      int t = warp_sum[lane];
#pragma unroll
      for (int o = 1; o < 32; o *= 2) {
        const int u = __shfl_up_sync(0xffffffffu, t, o);
        if (lane >= o) t += u;
      }
      warp_sum[lane] = t;
    }
    __syncthreads();
    const int before = carry + (w ? warp_sum[w - 1] : 0) + incl - sum;
#pragma unroll
    for (int k = 0; k < SCAN_K; ++k) {
      const int i = base + tid * SCAN_K + k;
      if (i < n) row[i] = cur[i] = before + v[k];
    }
    carry += warp_sum[31];
    __syncthreads();
  }
}

__global__ void __launch_bounds__(NT) k_edge_scatter(const EdgePlan p) {
  if (p.flags[0]) return;
  for (long long e = blockIdx.x * NT + threadIdx.x; e < p.E; e += gridDim.x * NT) {
    const int a = p.iperm[p.v0[e]], b = p.iperm[p.v1[e]];
    p.e1[atomicAdd(&p.cursor[a], 1)] = b;
    p.isrc[atomicAdd(&p.cursor[p.V + 1 + b], 1)] = a;
  }
}

// Ascending order of x[0, n): by insertion, long rows (hub vertices) by heap.
__device__ void sort_row(int* x, int n) {
  if (n <= 48) {
    for (int k = 1; k < n; ++k) {
      const int v = x[k];
      int m = k;
      for (; m > 0 && x[m - 1] > v; --m) x[m] = x[m - 1];
      x[m] = v;
    }
    return;
  }
  const auto sift = [&](int root, int end) {
    const int v = x[root];
    for (int c; (c = 2 * root + 1) < end; root = c) {
      if (c + 1 < end && x[c + 1] > x[c]) ++c;
      if (x[c] <= v) break;
      x[root] = x[c];
    }
    x[root] = v;
  };
  for (int k = n / 2 - 1; k >= 0; --k) sift(k, n);
  for (int end = n - 1; end > 0; --end) {
    const int v = x[0];
    x[0] = x[end];
    x[end] = v;
    sift(0, end);
  }
}

// Whether the host sorts row t (a vertex, or V + it for its in-edges) of n entries.
constexpr int LONG_ROW = 512;
__device__ bool left_to_host(const EdgePlan& p, int t, int n) {
  if (n <= LONG_ROW) return false;
  const int k = atomicAdd(&p.flags[2], 1);
  if (k >= EDGE_LONG_ROWS) return false;
  p.long_rows[k] = t;
  return true;
}

// One thread per vertex and list: its row in order; for out-edges also the row's
// sources and the vertex' weight (w_reg added once for each edge it is an end of).
__global__ void __launch_bounds__(NT) k_edge_sort(const EdgePlan p) {
  if (p.flags[0]) return;
  const long long t = blockIdx.x * (long long)NT + threadIdx.x;
  if (t >= 2ll * p.V) return;
  if (t >= p.V) {
    const int v = (int)(t - p.V), n = p.irow[v + 1] - p.irow[v];
    if (!left_to_host(p, (int)t, n)) sort_row(p.isrc + p.irow[v], n);
    return;
  }
  const int v = (int)t, b = p.orow[v], e = p.orow[v + 1];
  if (!left_to_host(p, v, e - b)) sort_row(p.e1 + b, e - b);
  for (int k = b; k < e; ++k) p.e0[k] = v;
  float w = p.degw[v];
  for (int k = (e - b) + (p.irow[v + 1] - p.irow[v]); k > 0; --k) w += p.w_reg;
  p.degw[v] = w;
}

// flags[1] = 1 unless every edge is given both ways.
__global__ void __launch_bounds__(NT) k_edge_sym(const EdgePlan p) {
  if (p.flags[0]) return;
  bool same = true;
  const long long n = max((long long)p.E, p.V + 1ll);
  for (long long k = blockIdx.x * (long long)NT + threadIdx.x; k < n; k += (long long)gridDim.x * NT) {
    if (k < p.E) same = same && p.e1[k] == p.isrc[k];
    if (k <= p.V) same = same && p.orow[k] == p.irow[k];
  }
  if (!same) p.flags[1] = 1;
}

}  // namespace

cudaError_t launch_edge_plan(const EdgePlan& p, cudaStream_t st) {
  const auto blocks = [](long long n) { return (unsigned)std::max(1ll, std::min((n + NT - 1) / NT, 4096ll)); };
  k_edge_count<<<blocks(p.E), NT, 0, st>>>(p);
  k_edge_rows<<<2, SCAN_T, 0, st>>>(p);
  k_edge_scatter<<<blocks(p.E), NT, 0, st>>>(p);
  k_edge_sort<<<(unsigned)((2ll * p.V + NT - 1) / NT), NT, 0, st>>>(p);
  return launch_edge_sym(p, st);
}

cudaError_t launch_edge_sym(const EdgePlan& p, cudaStream_t st) {
  k_edge_sym<<<(unsigned)std::min((std::max<long long>(p.E, p.V + 1ll) + NT - 1) / NT, 4096ll), NT, 0, st>>>(p);
  return cudaGetLastError();
}

}  // namespace optgb
