// Meetings of all blocks of a cooperative launch (one block per SM) through
// global memory, for the resident PCG loops (resident.cu says what they cost and
// why the slots lie as they do; fp64.cu).
#pragma once

#include "opt_internal.cuh"

namespace optgb {

constexpr int RT = 512;               // threads per block of a resident loop
constexpr int RW = RT / 32;

__device__ __forceinline__ unsigned ld_relaxed(const unsigned* p) {
  unsigned v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long ld_relaxed(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void red_add(unsigned* p, unsigned v) {
  asm volatile("red.relaxed.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// A wait's time limit: called now and then while waiting.
__device__ __forceinline__ bool waited_too_long(int spin, unsigned long long& t0, unsigned long long limit) {
  if ((spin & 255) != 255) return false;
  const unsigned long long now = global_ns();
  if (t0 == 0) t0 = now;
  return now - t0 > limit;
}

// What a launch knows of the device-wide exchanges: those done so far, by kind, and how
// long the next wait and the later ones may take.
struct Meet {
  ResidentSync* sy;
  unsigned base, meetings, sums;
  unsigned long long limit, later;
};
__device__ __forceinline__ Meet meet_begin(ResidentSync* sy) {
  return Meet{sy, sy->meetings, 0u, sy->sums, sy->first_ns, sy->wait_ns};
}

// Meeting of all blocks: what any thread wrote to global memory before is
// visible to every thread of every block after.  Returns false if a block did
// not arrive in time.
__device__ __forceinline__ bool meet_device(Meet& M) {
  __shared__ int s_ok;
  __syncthreads();
  M.meetings += 1;
  if (threadIdx.x == 0) {
    __threadfence();
    red_add(&M.sy->counter, 1u);
    const unsigned want = M.base + M.meetings * gridDim.x;
    unsigned long long t0 = 0;
    int ok = 1;
    for (int spin = 0; ok && (int)(ld_relaxed(&M.sy->counter) - want) < 0; ++spin) ok = !waited_too_long(spin, t0, M.limit);
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  M.limit = M.later;
  return s_ok != 0;
}

}  // namespace optgb
