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

// Maximum of v over the calling threads into *key.  Full warps reduce with
// shuffles first; the threads of a trailing partial warp (a block size that is
// not a multiple of 32) go straight to the atomic.
__device__ __forceinline__ void max_to(float v, unsigned* key, bool full_warp) {
  if (full_warp) {
    warp_max_to(v, key);
    return;
  }
  if (v > -INFINITY) atomicMax(key, f32_key(v));
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
