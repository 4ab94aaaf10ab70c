// Pieces the stack-march kernels share.
#pragma once

#include <algorithm>
#include <cmath>

#include "internal.cuh"

namespace fitrig {

// Approximate reciprocal (rcp.approx.ftz: relative error below 2^-23).
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Maxima of a march.  Every warp of every CTA has one for the stack and, with
// the running M, one per snapshot, and all CTAs are at about the same
// snapshot, so that an atomic each would queue up at one address (64 x 4096^2,
// w = 5, running M: 1.4 M of them, march 2.12 ms).  The words only grow during a
// launch, so a warp looks first (past the L1 cache) and leaves a maximum that is
// no larger than what is there: 0.71 ms, the march without running M 0.69.  (The
// sliding march spends far longer between snapshots and keeps its atomics.)
__device__ __forceinline__ void raise_max(unsigned* word, unsigned key) {
  if (key > __ldcg(word)) atomicMax(word, key);
}

// This warp's maximum of v into *key (every lane calls it; -inf is skipped).
__device__ __forceinline__ void warp_raise_max(float v, unsigned* key) {
  const unsigned k = __reduce_max_sync(0xffffffffu, v > -INFINITY ? f32_key(v) : 0u);
  if ((threadIdx.x & 31) == 0 && k) raise_max(key, k);
}

// The snapshots' maxima: lane 0 notes each in shared memory, and the warp looks
// at sixteen words together.  put() is called by every lane of a full warp for
// j = 0 .. L - 1 in order.
constexpr int kSnapChunk = 16;
__device__ __forceinline__ void snap_max(unsigned (*hold)[kSnapChunk], unsigned* smax, float v, int j,
                                         int L) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned k = __reduce_max_sync(0xffffffffu, v > -INFINITY ? f32_key(v) : 0u);
  if (lane == 0) hold[warp][j % kSnapChunk] = k;
  if (j % kSnapChunk != kSnapChunk - 1 && j != L - 1) return;
  __syncwarp();
  if (lane <= j % kSnapChunk) {
    const unsigned h = hold[warp][lane];
    if (h) raise_max(smax + (j - j % kSnapChunk) + lane, h);
  }
  __syncwarp();
}

// Maximum of v over the calling threads into *key.  Full warps reduce first;
// the threads of a trailing partial warp (a block size that is not a multiple
// of 32) look for themselves.
__device__ __forceinline__ void max_to(float v, unsigned* key, bool full_warp) {
  if (full_warp) {
    warp_raise_max(v, key);
    return;
  }
  if (v > -INFINITY) raise_max(key, f32_key(v));
}

// The sums and maximum of one tile's PER column partials, added in the order
// of a warp that holds one per lane and adds across the lanes by halves (16, 8,
// 4, 2, 1): node<PER, O, l> is lane l after the step of distance O.  One thread does it, because a warp per
// tile with its fifteen shuffles costs more instructions than a small tile's
// pixels.
template <int PER, int O, int LANE>
__device__ __forceinline__ float3 partials_node(const float4* p) {
  static_assert(PER <= 32, "one partial per lane");
  if constexpr (O == 32) {
    const float4 q = p[LANE];
    return make_float3(q.x, q.y, q.z);
  } else {
    float3 r = partials_node<PER, 2 * O, LANE>(p);
    if constexpr (LANE + O < PER) {   // the absent lanes' zeros change nothing
      const float3 h = partials_node<PER, 2 * O, LANE + O>(p);
      r.x += h.x;
      r.y = fmaxf(r.y, h.y);
      r.z += h.z;
    }
    return r;
  }
}

// Launches a march kernel over its boxes and time segments.  A difference-coded
// stack is decoded from its first snapshot on, so it has one segment.
template <typename K>
cudaError_t launch_segments(K kern, const CUtensorMap* tmap, StackArgs a, cudaStream_t st) {
  const int units = a.nsnap - 2;
  a.seg_units = units;
  if (!a.key) {
    int per_sm = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, a.g.threads,
                                                                        a.g.smem_bytes);
    if (e != cudaSuccess) return e;
    a.seg_units = march_seg_units((int64_t)a.g.gridX * a.g.gridY, per_sm, units);
  }
  const dim3 grid(a.g.gridX, a.g.gridY, (units + a.seg_units - 1) / a.seg_units);
  kern<<<grid, a.g.threads, a.g.smem_bytes, st>>>(*tmap, a);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace fitrig
