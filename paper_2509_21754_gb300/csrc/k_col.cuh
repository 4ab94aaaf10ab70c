// The column march: windows 7 and 9 to 15 (no power of two, too large for a
// thread to own a tile).
//
// One thread per pixel column carries x^(s+1) and D^(s) of V tiles' rows of that
// column in registers; a tile's columns leave one partial (sum Delta, max Delta,
// sum r) per segment of R rows in shared memory, and after the snapshot's
// barrier one thread per tile adds them.  Everything that depends on the window
// is a template value, so a thread's rows are straight-line code with all their
// loads in flight; with the row count a variable (k_stack_tile) each row was a
// branch of its own, its load's and reciprocal's latency exposed, and a warp per
// tile with fifteen shuffles did the sums, as many instructions as a 7 x 7
// tile's pixels.  The segments, their row order and the order of the partials
// are k_stack_tile's, so every tile has the bits it had there.
// Bound by instruction issue (w = 12, FP16, signed: 23 per pixel, 77% of the
// issue slots).  64 x 2048^2, k_stack_tile -> this: w = 7 FP32 1585 -> 192 us
// (84% of the copy bandwidth), 9 1195 -> 286, 10 975 -> 235, 11 1021 -> 286,
// 12 882 -> 220, 12 FP16 signed 847 -> 208, 13 866 -> 243, 14 FP16 766 -> 228,
// 15 765 -> 274.
#pragma once

#include "march.cuh"

namespace fitrig {

// Window-dependent constants of the column march.
template <int W>
struct ColShape {
  static constexpr int kSeg = W <= 8 ? 1 : 2;               // segments of a tile's column
  static constexpr int kR = (W + kSeg - 1) / kSeg;          // rows of the first segment(s)
  static constexpr int kV = W <= 11 ? 2 : 1;                // tiles a thread holds one above another
  static constexpr int kPer = kSeg * W;                     // partials of a tile
  static constexpr int kStride = kPer | 1;                  // odd, in 16-byte entries: no bank conflicts
  // tiles across: an x origin that is a multiple of 8 elements (16 bytes in
  // half precision) and at most 256 columns; the last warp's spare lanes
  // repeat a column and write nothing (15 of 16 threads work at the least)
  static constexpr int kTBX = W == 7 ? 32 : 16;
  static constexpr int kBW = kTBX * W;
  static constexpr int kThreads = (kBW + 31) / 32 * 32;
  static constexpr int kTBY = kV;
  static_assert(kBW % 8 == 0 && kBW <= 256 && kTBX * kTBY <= kThreads, "column march shape");
};

template <typename T, int W, bool SIGNED>
__global__ void __launch_bounds__(ColShape<W>::kThreads) k_stack_col(const __grid_constant__ CUtensorMap tmap,
                                                                     const StackArgs a) {
  using S = ColShape<W>;
  constexpr int BW = S::kBW, NT = S::kTBX * S::kTBY, RV = W * S::kV;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ unsigned hold[S::kThreads / 32][kSnapChunk];
  const int NS = a.g.stages;
  float4* part = reinterpret_cast<float4*>(smem + (size_t)NS * a.g.stage_bytes);
  const uint32_t bar0 = smem_u32(part + 2 * NT * S::kStride);
  const uint32_t stage0 = smem_u32(smem);
  constexpr uint32_t box_bytes = (uint32_t)(BW * S::kTBY * W * (int)sizeof(T));
  const int tid = threadIdx.x;
  const int c = min(tid, BW - 1);
  const int x0 = blockIdx.x * BW, y0 = blockIdx.y * S::kTBY * W;
  const int s0 = blockIdx.z * a.seg_units;                    // first unit of the segment
  const int L = min(a.seg_units, a.nsnap - 2 - s0) + 2;       // its snapshots
  const int z0 = a.zrot + s0;
  if (tid == 0) {
    prefetch_tmap(&tmap);
    for (int i = 0; i < NS; ++i) mbar_init(bar0 + 8 * i, 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (tid == 0) {
    for (int j = 0; j < NS && j < L; ++j) {
      mbar_expect_tx(bar0 + 8 * j, box_bytes);
      tma_load_3d(stage0 + j * (uint32_t)a.g.stage_bytes, &tmap, x0, y0, (z0 + j) % a.nsnap, bar0 + 8 * j);
    }
  }
  // this thread's pixels in a stage, and where its partials go
  float4* const mine = part + (c / W) * S::kStride + c % W;
  float x[RV], d[RV];
#pragma unroll
  for (int i = 0; i < RV; ++i) x[i] = d[i] = 0.f;
  float mx = -INFINITY;
  const uint64_t deadline = globaltimer_ns() + a.timeout_ns;
  int stg = 0, turn = 0;      // turn: first thread of the tiles' threads
  uint32_t phase = 0;
  for (int j = 0; j < L; ++j) {
    const bool ok = mbar_wait_bounded(bar0 + 8 * stg, phase, deadline);
    const T* st = reinterpret_cast<const T*>(smem + (size_t)stg * a.g.stage_bytes) + c;
    float sm = -INFINITY;
    if (ok && j >= 2) {
      // the column's zero test: the smallest |x^(s+1)| (Eq. 5's guard is
      // needed for x = 0 only; the signed quotient also keeps to normal x)
      float mn = INFINITY;
#pragma unroll
      for (int i = 0; i < RV; ++i) mn = fminf(mn, fabsf(x[i]));
      const bool fast = SIGNED ? mn >= 1.17549435e-38f : mn != 0.f;
#pragma unroll
      for (int v = 0; v < S::kV; ++v) {
#pragma unroll
        for (int sg = 0; sg < S::kSeg; ++sg) {
          float s1 = 0.f, s2 = 0.f, s3 = 0.f;
          float dl[S::kR], xr[S::kR];
#pragma unroll
          for (int r = 0; r < S::kR; ++r) {
            if (sg * S::kR + r < W) {
              const int i = v * W + sg * S::kR + r;
              const float xn = to_f32(st[i * BW]);
              sm = fmaxf(sm, xn);
              const float dn = fabsf(xn - x[i]);   // D^(s+1)
              dl[r] = fabsf(dn - d[i]);            // Delta
              xr[r] = x[i];
              s1 += dl[r];
              s2 = fmaxf(s2, dl[r]);
              d[i] = dn;
              x[i] = xn;
            }
          }
          if (fast) {
#pragma unroll
            for (int r = 0; r < S::kR; ++r) {
              if (sg * S::kR + r < W) {
                if (SIGNED) s3 += fminf(dl[r] * rcp_approx(xr[r]), 1.f);
                else s3 += __saturatef(dl[r] * fabsf(rcp_approx(xr[r])));
              }
            }
          } else {
#pragma unroll
            for (int r = 0; r < S::kR; ++r) {
              if (sg * S::kR + r < W) {
                const float ref = SIGNED ? xr[r] : fabsf(xr[r]);
                const float xh = (xr[r] == 0.f) ? kGuardC : ref;   // Eq. 5
                s3 += fminf(__fdividef(dl[r], xh), 1.f);           // Eq. 4
              }
            }
          }
          if (tid < BW)
            mine[(j & 1) * NT * S::kStride + v * S::kTBX * S::kStride + sg * W] =
                make_float4(s1, s2, s3, 0.f);
        }
      }
    } else if (ok) {
#pragma unroll
      for (int i = 0; i < RV; ++i) {
        const float xn = to_f32(st[i * BW]);
        sm = fmaxf(sm, xn);
        d[i] = fabsf(xn - x[i]);   // D^(0) once j == 1
        x[i] = xn;
      }
    }
    if (__syncthreads_or(!ok)) {
      // A stage never completed: flag it, let in-flight copies land (bounded),
      // and leave.  No thread touches the ring after this point.
      if (tid == 0) {
        atomicOr(a.status, kErrTimeout);
        const uint64_t d2 = globaltimer_ns() + 1000000ull;
        for (int jj = j; jj < L && jj < j + NS; ++jj)
          mbar_wait_bounded(bar0 + 8 * (jj % NS), (uint32_t)((jj / NS) & 1), d2);
      }
      return;
    }
    mx = fmaxf(mx, sm);
    if (a.smax) snap_max(hold, a.smax + s0, sm, j, L);
    if (tid == 0 && j + NS < L) {
      fence_proxy_async_smem();
      mbar_expect_tx(bar0 + 8 * stg, box_bytes);
      tma_load_3d(stage0 + stg * (uint32_t)a.g.stage_bytes, &tmap, x0, y0, (z0 + j + NS) % a.nsnap,
                  bar0 + 8 * stg);
    }
    if (++stg == NS) {
      stg = 0;
      phase ^= 1u;
    }
    if (j >= 2) {
      // one thread per tile; the warps that do it change from unit to unit
      int tt = tid - turn;
      if (tt < 0) tt += S::kThreads;
      turn = turn + 32 == S::kThreads ? 0 : turn + 32;
      const int tx = blockIdx.x * S::kTBX + tt % S::kTBX, ty = blockIdx.y * S::kTBY + tt / S::kTBX;
      if (tt < NT && tx < a.Tx && ty < a.Ty) {
        const float3 s = partials_node<S::kPer, 1, 0>(part + ((j & 1) * NT + tt) * S::kStride);
        const float n = (float)(min(W, a.ny - ty * W) * min(W, a.nx - tx * W));
        float v = (s.x / n) * s.y * (s.z / n);
        if (!isfinite(s.x) || !isfinite(v)) v = NAN;
        a.vp[(size_t)(s0 + j - 2) * (size_t)a.vstride + (size_t)ty * a.Tx + tx] = v;
      }
    }
  }
  warp_raise_max(mx, a.gmax);   // (whole warps: kThreads is a multiple of 32)
}

template <typename T, int W, bool SIGNED>
static cudaError_t launch_col_w(const CUtensorMap* tmap, const StackArgs& a, cudaStream_t st) {
  auto kern = k_stack_col<T, W, SIGNED>;
  const cudaError_t lim = allow_smem(kern, a.g.smem_bytes);
  if (lim != cudaSuccess) return lim;
  return launch_segments(kern, tmap, a, st);
}

template <typename T, bool SIGNED>
cudaError_t launch_col(const CUtensorMap* tmap, const StackArgs& a, cudaStream_t st) {
  switch (a.g.w) {
    case 7: return launch_col_w<T, 7, SIGNED>(tmap, a, st);
    case 9: return launch_col_w<T, 9, SIGNED>(tmap, a, st);
    case 10: return launch_col_w<T, 10, SIGNED>(tmap, a, st);
    case 11: return launch_col_w<T, 11, SIGNED>(tmap, a, st);
    case 12: return launch_col_w<T, 12, SIGNED>(tmap, a, st);
    case 13: return launch_col_w<T, 13, SIGNED>(tmap, a, st);
    case 14: return launch_col_w<T, 14, SIGNED>(tmap, a, st);
    case 15: return launch_col_w<T, 15, SIGNED>(tmap, a, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace fitrig
