// Threshold, compaction, components, candidates and their sort.
//
// Selection follows the set {t | z_t > tau} of Sec. 2.4.1 (image branch) and
// Sec. 2.4.2 (eta): z = (v - centre) / scale in FP64.  The comparison is made
// in FP32 against thr = the largest float <= centre + tau * scale, which picks
// exactly the floats v with (double)v > centre + tau * scale.
//
// Compaction is order-preserving (per-block counts, an exclusive scan, and a
// warp-ballot write), so the list of selected tiles is sorted by (unit, t).
// Tiles are merged into 8-connected components per unit (a pulsar spreads over
// one, two or four tiles, Sec. 2.4.2) by a lock-free union-find whose roots
// are always the smallest list index; each component yields one candidate at
// its maximum-z tile (ties: smallest tile index).  The image-branch pixel is
// the tile's arg-max of Delta recomputed from the three snapshots; the
// frequency-branch pixel is the tile centre refined by a parabola through the
// eta of the neighbouring tiles.  Candidates are finally radix-sorted by
// (snapshot, y, x), a unique key, so the output is deterministic.
#include <cfloat>
#include <climits>
#include <cmath>

#include "internal.cuh"

namespace fitrig {

constexpr int kSelThreads = 256;

__device__ __forceinline__ void chunk_range(int64_t N, int nblk, int b, int64_t* lo,
                                            int64_t* hi) {
  const int64_t chunk = (N + nblk - 1) / nblk;
  *lo = (int64_t)b * chunk;
  *hi = *lo + chunk < N ? *lo + chunk : N;
}

// Ordered compaction over the element space [0, groups * stride): each warp
// owns a contiguous chunk of `chunk` elements (a multiple of 128), counts its
// selected entries, and after an exclusive scan of the warp counts writes them
// in order with a warp-level prefix -- no block-wide barriers.  VEC reads four
// entries per lane (16-byte aligned base, stride % 4 == 0).
__device__ __forceinline__ void warp_range(int64_t N, int64_t chunk, int64_t* lo, int64_t* hi) {
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  *lo = w * chunk;
  *hi = *lo + chunk < N ? *lo + chunk : N;
}

template <bool VEC>
__global__ void __launch_bounds__(kSelThreads) k_sel_count(const float* __restrict__ vals,
                                                           int groups, int64_t stride,
                                                           const float* __restrict__ thr,
                                                           int64_t chunk, int* wcnt) {
  const int64_t N = (int64_t)groups * stride;
  int64_t lo, hi;
  warp_range(N, chunk, &lo, &hi);
  const int lane = threadIdx.x & 31;
  int cnt = 0;
  const int step = VEC ? 4 : 1;
  int64_t i = lo + lane * step;
  int g = lo < N ? (int)(lo / stride) : 0;
  int64_t gend = (int64_t)(g + 1) * stride;
  float th = lo < N ? thr[g] : INFINITY;
  for (; i < hi; i += 32 * step) {
    while (i >= gend) {
      ++g;
      gend += stride;
      th = thr[g];
    }
    if (VEC) {
      const float4 q = *reinterpret_cast<const float4*>(vals + i);
      cnt += (q.x > th) + (q.y > th) + (q.z > th) + (q.w > th);
    } else {
      cnt += vals[i] > th;
    }
  }
  for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
  if (lane == 0) wcnt[((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5] = cnt;
}

// Exclusive scan of per-warp (or per-block) counts (one block of 1024 threads;
// sh: its shared memory).
__device__ __forceinline__ void scan_counts(int nblk, const int* blkcnt, int* blkoff, int* total,
                                            int64_t cap, unsigned* status, unsigned* want,
                                            long long* sh) {
  const int per = (nblk + 1023) / 1024;
  const int b0 = threadIdx.x * per;
  long long local = 0;
  for (int b = b0; b < b0 + per && b < nblk; ++b) local += blkcnt[b];
  sh[threadIdx.x] = local;
  __syncthreads();
  for (int d = 1; d < 1024; d <<= 1) {
    const long long add = threadIdx.x >= d ? sh[threadIdx.x - d] : 0;
    __syncthreads();
    sh[threadIdx.x] += add;
    __syncthreads();
  }
  long long run = sh[threadIdx.x] - local;
  for (int b = b0; b < b0 + per && b < nblk; ++b) {
    blkoff[b] = (int)(run < cap ? run : cap);
    run += blkcnt[b];
  }
  if (threadIdx.x == 1023) {
    const long long tot = sh[1023];
    *total = (int)(tot < cap ? tot : cap);
    if (tot > cap) {
      atomicOr(status, kErrCapacity);
      if (want) atomicMax(want, (unsigned)(tot < 0xffffffffll ? tot : 0xffffffffll));
    }
  }
}

__global__ void __launch_bounds__(1024) k_scan_blocks(int nblk, const int* blkcnt, int* blkoff,
                                                      int* total, int64_t cap,
                                                      unsigned* status, unsigned* want) {
  __shared__ long long sh[1024];
  scan_counts(nblk, blkcnt, blkoff, total, cap, status, want, sh);
}

template <bool VEC>
__global__ void __launch_bounds__(kSelThreads) k_sel_write(const float* __restrict__ vals,
                                                           int groups, int64_t stride,
                                                           const float* __restrict__ thr,
                                                           int64_t chunk, const int* woff,
                                                           SelItem* items, uint32_t* sbits,
                                                           int* wbase, int64_t cap,
                                                           unsigned* compmax, int* peak) {
  const int64_t N = (int64_t)groups * stride;
  int64_t lo, hi;
  warp_range(N, chunk, &lo, &hi);
  if (lo >= hi) return;   // warp-uniform
  const int lane = threadIdx.x & 31;
  const int step = VEC ? 4 : 1;
  int64_t run = woff[((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5];
  int g = (int)(lo / stride);
  int64_t gend = (int64_t)(g + 1) * stride;
  for (int64_t base = lo; base < hi; base += 32 * step) {
    const int64_t i = base + lane * step;
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    unsigned bits = 0;
    if (i < hi) {
      while (i >= gend) {
        ++g;
        gend += stride;
      }
      const float th = thr[g];
      if (VEC) {
        const float4 q = *reinterpret_cast<const float4*>(vals + i);
        v[0] = q.x;
        v[1] = q.y;
        v[2] = q.z;
        v[3] = q.w;
        bits = (q.x > th) | ((q.y > th) << 1) | ((q.z > th) << 2) | ((q.w > th) << 3);
      } else {
        v[0] = vals[i];
        bits = v[0] > th;
      }
    }
    const int c = __popc(bits);
    int incl = c;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    int64_t pos = run + incl - c;
    // bitmap words of this iteration (base is a multiple of 32 elements, of
    // 128 with VEC) and the list index of each word's first selected element
    if (VEC) {
      uint32_t word = bits << (4 * (lane & 7));   // lanes 8w..8w+7 hold word w
      word |= __shfl_xor_sync(0xffffffffu, word, 1);
      word |= __shfl_xor_sync(0xffffffffu, word, 2);
      word |= __shfl_xor_sync(0xffffffffu, word, 4);
      if ((lane & 7) == 0) {
        const int64_t wi = (base >> 5) + (lane >> 3);
        sbits[wi] = word;
        wbase[wi] = (int)min(pos, (int64_t)INT_MAX);
      }
    } else {
      const uint32_t word = __ballot_sync(0xffffffffu, bits != 0);
      if (lane == 0) {
        sbits[base >> 5] = word;
        wbase[base >> 5] = (int)min(pos, (int64_t)INT_MAX);
      }
    }
    if (bits) {
      for (int k = 0; k < step; ++k) {
        if (!(bits >> k & 1u)) continue;
        if (pos < cap) {
          const int64_t e = i + k;
          SelItem it;
          it.group = g;
          it.t = (int32_t)(e - (int64_t)g * stride);
          it.v = v[k];
          items[pos] = it;
          compmax[pos] = 0u;   // component state for launch_components
          peak[pos] = INT_MAX;
        }
        ++pos;
      }
    }
    run += total;
  }
}

static int64_t sel_chunk(int64_t N, int nwarps) {
  int64_t c = (N + nwarps - 1) / nwarps;
  return (c + 127) / 128 * 128;
}

static bool sel_vec(const float* vals, int64_t stride) {
  return (reinterpret_cast<uintptr_t>(vals) % 16 == 0) && (stride % 4 == 0);
}

cudaError_t launch_select(const float* vals, int groups, int64_t stride, const float* thr,
                          const SelectScratch& s, unsigned* status, cudaStream_t st) {
  const int nw = s.nblk * (kSelThreads / 32);
  const int64_t chunk = sel_chunk((int64_t)groups * stride, nw);
  if (sel_vec(vals, stride)) {
    k_sel_count<true><<<s.nblk, kSelThreads, 0, st>>>(vals, groups, stride, thr, chunk, s.blkcnt);
    k_scan_blocks<<<1, 1024, 0, st>>>(nw, s.blkcnt, s.blkoff, s.nsel, s.capacity, status,
                                      s.want);
    k_sel_write<true><<<s.nblk, kSelThreads, 0, st>>>(vals, groups, stride, thr, chunk,
                                                      s.blkoff, s.items, s.bits, s.wbase,
                                                      s.capacity, s.compmax, s.peak);
  } else {
    k_sel_count<false><<<s.nblk, kSelThreads, 0, st>>>(vals, groups, stride, thr, chunk, s.blkcnt);
    k_scan_blocks<<<1, 1024, 0, st>>>(nw, s.blkcnt, s.blkoff, s.nsel, s.capacity, status,
                                      s.want);
    k_sel_write<false><<<s.nblk, kSelThreads, 0, st>>>(vals, groups, stride, thr, chunk,
                                                       s.blkoff, s.items, s.bits, s.wbase,
                                                       s.capacity, s.compmax, s.peak);
  }
  count_launches(3);
  return cudaGetLastError();
}

__global__ void k_sum_counts(int nblk, const int* blkcnt, long long* total) {
  __shared__ long long sh[256];
  long long s = 0;
  for (int b = threadIdx.x; b < nblk; b += blockDim.x) s += blkcnt[b];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int d = 128; d > 0; d >>= 1) {
    if (threadIdx.x < d) sh[threadIdx.x] += sh[threadIdx.x + d];
    __syncthreads();
  }
  if (threadIdx.x == 0) *total = sh[0];
}

cudaError_t launch_count_selected(const float* vals, int groups, int64_t stride, const float* thr,
                                  int nblk, int* wcnt, long long* total, cudaStream_t st) {
  const int nw = nblk * (kSelThreads / 32);
  const int64_t chunk = sel_chunk((int64_t)groups * stride, nw);
  if (sel_vec(vals, stride))
    k_sel_count<true><<<nblk, kSelThreads, 0, st>>>(vals, groups, stride, thr, chunk, wcnt);
  else
    k_sel_count<false><<<nblk, kSelThreads, 0, st>>>(vals, groups, stride, thr, chunk, wcnt);
  k_sum_counts<<<1, 256, 0, st>>>(nw, wcnt, total);
  count_launches(2);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- components
__device__ __forceinline__ int64_t item_key(const SelItem& it, int64_t T) {
  return (int64_t)it.group * T + it.t;
}

__device__ __forceinline__ int find_root(int* parent, int x) {
  volatile int* p = parent;
  int y = p[x];
  while (y != x) {
    const int z = p[y];
    if (z != y) p[x] = z;   // path halving; only non-roots are written
    x = y;
    y = p[x];
  }
  return x;
}

__device__ void unite(int* parent, int a, int b, unsigned* status) {
  for (int it = 0; it < (1 << 20); ++it) {
    a = find_root(parent, a);
    b = find_root(parent, b);
    if (a == b) return;
    const int hi = a > b ? a : b, lo = a > b ? b : a;
    const int old = atomicCAS(&parent[hi], hi, lo);
    if (old == hi) return;
    a = old;
    b = lo;
  }
  atomicOr(status, kErrCcLimit);
}


// Horizontal runs: a selected tile whose left neighbour is selected is the next
// list entry after it.  Each warp takes 32 consecutive entries, finds by
// ballot the nearest run start at or before each lane, and points the entry at
// it; a run that began in an earlier warp points at the entry just before the
// warp, so chains only cross warp boundaries.
__global__ void k_cc_runs(const SelItem* __restrict__ items, const int* nsel, int Tx,
                          int* parent) {
  const int n = *nsel;
  const int lane = threadIdx.x & 31;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  for (int base = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; base < n; base += nw * 32) {
    const int i = base + lane;
    bool left = false;
    if (i < n && i > 0) {
      const SelItem me = items[i], pv = items[i - 1];
      left = pv.group == me.group && pv.t == me.t - 1 && (me.t % Tx) != 0;
    }
    const unsigned lmask = __ballot_sync(0xffffffffu, left);
    const unsigned starts = ~lmask & (lane == 31 ? 0xffffffffu : ((2u << lane) - 1u));
    if (i < n) {
      int head;
      if (starts) head = base + 31 - __clz(starts);
      else head = base - 1;   // the run started in an earlier warp
      parent[i] = head;
    }
  }
}

// List index of element e when it is selected, else -1.
__device__ __forceinline__ int sel_index(const uint32_t* __restrict__ sbits,
                                         const int* __restrict__ wbase, int64_t e) {
  const uint32_t w = sbits[e >> 5];
  const uint32_t b = 1u << (e & 31);
  if (!(w & b)) return -1;
  return wbase[e >> 5] + __popc(w & (b - 1u));
}

__global__ void k_cc_union(const SelItem* __restrict__ items, const int* nsel, int Tx, int Ty,
                           int64_t T, const uint32_t* __restrict__ sbits,
                           const int* __restrict__ wbase, int* parent, unsigned* status) {
  const int n = *nsel;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const SelItem me = items[i];
    const int ty = me.t / Tx, tx = me.t - (me.t / Tx) * Tx;
    if (ty == 0) continue;
    // left neighbours are joined by the runs; of the row above, the tile right
    // above covers both diagonals when it is selected (they would be in its run)
    const int64_t up = (int64_t)me.group * T + (int64_t)(ty - 1) * Tx + tx;
    // (indices at or past n belong to a list that overflowed its capacity)
    const int j = sel_index(sbits, wbase, up);
    if (j >= 0) {
      if (j < n) unite(parent, i, j, status);
    } else {
      if (tx > 0) {
        const int jl = sel_index(sbits, wbase, up - 1);
        if (jl >= 0 && jl < n) unite(parent, i, jl, status);
      }
      if (tx + 1 < Tx) {
        const int jr = sel_index(sbits, wbase, up + 1);
        if (jr >= 0 && jr < n) unite(parent, i, jr, status);
      }
    }
  }
}

// After the unions the roots no longer change, so each thread finds its
// entry's root without writing, then points the entry at it (a final value,
// so other walks through it stay valid) and raises the component's largest
// value key.  (Path halving here could store an intermediate ancestor over
// another thread's root and leave an entry outside its component's root.)
__global__ void k_cc_flatten_max(const SelItem* __restrict__ items, const int* nsel, int* parent,
                                 unsigned* compmax) {
  const int n = *nsel;
  volatile int* p = parent;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    int r = i, y = p[i];
    while (y != r) {
      r = y;
      y = p[r];
    }
    p[i] = r;
    atomicMax(&compmax[r], f32_key(items[i].v));   // a component lies in one group
  }
}

// The peak of each component: its entry of largest value, the smallest list
// index on ties (the list is in tile order).
__global__ void k_cc_peak(const SelItem* __restrict__ items, const int* nsel, const int* parent,
                          const unsigned* compmax, int* peak) {
  const int n = *nsel;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int r = parent[i];
    if (f32_key(items[i].v) == compmax[r]) atomicMin(&peak[r], i);
  }
}

cudaError_t launch_components(int Tx, int Ty, int64_t T, const SelectScratch& s,
                              unsigned* status, cudaStream_t st) {
  // (every entry's compmax / peak were initialised by the compaction)
  const int grid = 152 * 16, thr = 256;
  k_cc_runs<<<grid, thr, 0, st>>>(s.items, s.nsel, Tx, s.parent);
  k_cc_union<<<grid, thr, 0, st>>>(s.items, s.nsel, Tx, Ty, T, s.bits, s.wbase, s.parent,
                                   status);
  k_cc_flatten_max<<<grid, thr, 0, st>>>(s.items, s.nsel, s.parent, s.compmax);
  k_cc_peak<<<grid, thr, 0, st>>>(s.items, s.nsel, s.parent, s.compmax, s.peak);
  count_launches(4);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- block-tiled components
// A streaming kernel first thresholds every tile map into a bitmap (one bit
// per tile).  A CTA then takes one kBlkY x kBlkX block of one group's bitmap
// (with a one-tile halo), labels the block's 8-connected components with a
// shared-memory union-find, and finds each component's peak (largest value,
// smallest tile index on ties) as the largest key (value key << 32) | ~t,
// reading the values of the selected tiles only.  A
// component that reaches a selected tile outside the block is a boundary
// component: it gets a global id, its edge tiles get that id in a dense label
// map, and a second kernel unites the ids of selected neighbours across block
// edges.  Every other component's peak is set in the block's bits of the
// dense peak bitmap directly; the merged boundary components' peaks are
// OR'ed in afterwards, and an ordered compaction of the bitmap gives the peak
// list in (group, t) order.
constexpr int kBlkT = kBlkY * kBlkX;
constexpr int kBlkThreads = 256;
static_assert(kBlkY % 32 == 0 && kBlkY <= 64 && kBlkX == 64, "block geometry");
constexpr int kBlkIds = 2 * kBlkX + 2 * (kBlkY - 2);   // boundary components a block can have
constexpr int kBlkPairs = 4 * kBlkIds;                  // cross-edge pairs a block can record
constexpr int kBlkRing = 2 * kBlkX + 2 * (kBlkY - 2);   // edge tiles of a block

__device__ __forceinline__ int find_s(const int* par, int x) {
  const volatile int* p = par;
  int y = p[x];
  while (y != x) {
    x = y;
    y = p[x];
  }
  return x;
}

// Shared-memory union (roots always link the larger index to the smaller).
__device__ void unite_s(int* par, int a, int b, unsigned* status) {
  for (int it = 0; it < (1 << 16); ++it) {
    a = find_s(par, a);
    b = find_s(par, b);
    if (a == b) return;
    const int hi = a > b ? a : b, lo = a > b ? b : a;
    const int old = atomicCAS(&par[hi], hi, lo);
    if (old == hi) return;
    a = old;
    b = lo;
  }
  atomicOr(status, kErrCcLimit);
}

__device__ __forceinline__ int find_g(const int* par, int x) {
  const volatile int* p = par;
  int y = p[x];
  while (y != x) {
    x = y;
    y = p[x];
  }
  return x;
}

__device__ __forceinline__ unsigned long long peak_key(float v, uint32_t t) {
  return ((unsigned long long)f32_key(v) << 32) | (unsigned long long)(0xffffffffu - t);
}

// The ring position r (0 <= r < kBlkRing) of a block's edge as (ly, lx).
__device__ __forceinline__ void ring_pos(int r, int* ly, int* lx) {
  if (r < kBlkX) {
    *ly = 0;
    *lx = r;
  } else if (r < 2 * kBlkX) {
    *ly = kBlkY - 1;
    *lx = r - kBlkX;
  } else {
    const int q = r - 2 * kBlkX;   // the side columns without the corners
    *ly = 1 + (q >> 1);
    *lx = (q & 1) ? kBlkX - 1 : 0;
  }
}

// Cross-block neighbour pair: group, tile and the direction (0..7) of the
// neighbour, packed as (g << 40) | (t << 3) | dir.
__device__ __forceinline__ void dir_offset(int d, int* dy, int* dx) {
  const int k = d < 4 ? d : d + 1;   // skip the centre of the 3 x 3
  *dy = k / 3 - 1;
  *dx = k % 3 - 1;
}

// Run-based labelling on bit masks.  Row y of the block is a 64-bit mask; a
// run is a maximal sequence of set bits, identified by its first bit, and is a
// node of the shared-memory union-find (node y * 64 + start).  Runs of
// adjacent rows are joined when they touch 8-connectedly (overlap after
// dilating one by a bit on each side).
__device__ __forceinline__ uint64_t run_starts(uint64_t m) { return m & ~(m << 1); }

// First bit of the run of m that contains bit b (b set in m).
__device__ __forceinline__ int run_of(uint64_t m, int b) {
  const uint64_t st = run_starts(m) & (b == 63 ? ~0ull : ((2ull << b) - 1ull));
  return 63 - __clzll((long long)st);
}

// Bits s.. of the run of m starting at s.
__device__ __forceinline__ uint64_t run_bits(uint64_t m, int s) {
  const uint64_t from = m >> s;
  const int len = __ffsll((long long)~from) - 1;   // < 64 unless the run reaches bit 63
  const uint64_t ones = (len <= 0 || len >= 64) ? ~0ull : ((1ull << len) - 1ull);
  return (len == 0 ? 0ull : ones) << s;
}

constexpr int kBlkMaxRuns = kBlkT / 2;   // runs of a block (alternating bits at most)

// Selected-tile bitmap: bit (tx & 31) of word tx / 32 of row (g, ty) is
// v > the group's threshold (never for NaN: an invalid tile); bits past the row's end are 0.
// One warp per row: all of the row's loads (coalesced, up to 32 per lane) are
// issued before its ballots.  The first row of each CTA adds its runs (those of
// neighbouring words counted apart) to *b.runs, from which k_blk_cc sees how dense
// the selection is.
constexpr int kMaskThreads = 256;
__global__ void __launch_bounds__(kMaskThreads) k_blk_mask(const float* __restrict__ vals,
                                                           int64_t stride, int Tx, int Ty,
                                                           int64_t nrows,
                                                           const double* __restrict__ cs,
                                                           double tau, double* inv,
                                                           BlockScratch b) {
  pdl_begin();
  if (blockIdx.x == 0 && threadIdx.x == 0) b.counters[1] = b.counters[3] = 0;
  const int lane = threadIdx.x & 31;
  const int64_t r = ((int64_t)blockIdx.x * kMaskThreads + threadIdx.x) >> 5;
  if (r >= nrows) return;
  const int g = (int)(r / Ty), ty = (int)(r - (int64_t)g * Ty);
  // (a launch of its own for the thresholds was one more step of the chain)
  float th = 0.f;
  if (lane == 0) th = group_threshold(cs, g, tau, ty == 0 ? inv + g : nullptr);
  th = __shfl_sync(0xffffffffu, th, 0);
  const float* row = vals + (size_t)g * stride + (int64_t)ty * Tx;
  uint32_t* out = b.sbits + (size_t)r * b.words;
  unsigned runs = 0;
  for (int w0 = 0; w0 < b.words; w0 += 32) {
    float x[32];
#pragma unroll
    for (int u = 0; u < 32; ++u) {
      const int tx = (w0 + u) * 32 + lane;
      x[u] = tx < Tx ? row[tx] : NAN;
    }
    uint32_t mine = 0;
#pragma unroll
    for (int u = 0; u < 32; ++u) {
      const uint32_t bal = __ballot_sync(0xffffffffu, x[u] > th);
      if (lane == u) mine = bal;
    }
    if (w0 + lane < b.words) out[w0 + lane] = mine;
    runs += __popc(mine & ~(mine << 1));
  }
  if (threadIdx.x < 32) {
    runs = __reduce_add_sync(0xffffffffu, runs);
    if (lane == 0 && runs) atomicAdd(b.runs, runs);
  }
}

// The labelling of one block by NT threads, for blocks of at most MAXR runs.
// Returns false, with nothing written, when the block has more (then every
// thread sees it) or with `skip` (the caller's word from memory, looked at once
// the block's own loads are on their way).
template <int NT, int MAXR>
struct BlkShared {
  unsigned long long mrow[kBlkY];   // the block's rows
  unsigned long long htop, hbot;    // halo rows above / below (block columns)
  unsigned long long hleft, hright;   // halo columns (bit = block row)
  unsigned long long pkey[MAXR];    // peak key of each root; its id once known
  uint32_t rinfo[MAXR];             // run: row << 16 | start << 8 | end
  uint32_t bnd[MAXR / 32];          // boundary flag of each root (bit mask)
  uint32_t pw[kBlkY][2];
  int runbase[kBlkY + 1];           // first run of each row; runbase[kBlkY] = runs
  int wrun[NT / 32];
  __align__(4) short par[MAXR];     // union-find over runs (CAS on aligned words)
  uint32_t hcorner;                 // bits: 0 top-left, 1 top-right, 2 bottom-left, 3 bottom-right
  int nsel, nbnd, npair;
};

template <int NT, int MAXR>
__device__ __forceinline__ bool blk_label(BlkShared<NT, MAXR>& sh, const float* __restrict__ vals,
                                          int64_t stride, int Tx, int Ty, const BlockScratch& b,
                                          int64_t bidx, int g, int bx, int by, bool skip,
                                          unsigned* status) {
  static_assert(NT >= 64 && MAXR <= kBlkMaxRuns, "a thread per row");
  constexpr int kIter = (MAXR + NT - 1) / NT;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // this block's slots: boundary ids bidx * kBlkIds + k, pairs bidx * kBlkPairs + k
  const int tx0 = bx * kBlkX, ty0 = by * kBlkY;
  const int w0 = tx0 / 32;
  if (tid == 0) {
    sh.hleft = sh.hright = 0ull;
    sh.hcorner = 0u;
    sh.nsel = sh.nbnd = sh.npair = 0;
  }
  __syncthreads();
  // 1. the block's rows as 64-bit masks, the halo rows, columns and corners,
  // from the bitmap words of rows ty0-1 .. ty0+kBlkY (the words on either side
  // hold the halo columns' bits); outside the map: 0.  The last threads take
  // the halo rows.
  const uint32_t* sb = b.sbits + (size_t)g * Ty * b.words;
  int rc = 0, rincl = 0;
  unsigned long long mine = 0ull;
  for (int q = tid; q < kBlkY + 2; q += NT) {
    const int r = q < kBlkY ? q : (q == kBlkY ? -1 : kBlkY);   // block row
    const int ty = ty0 + r;
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int wx = w0 - 1 + k;
      w[k] = (ty >= 0 && ty < Ty && wx >= 0 && wx < b.words) ? sb[(size_t)ty * b.words + wx] : 0u;
    }
    const unsigned long long m = ((unsigned long long)w[2] << 32) | w[1];
    const bool left = (w[0] >> 31) != 0u, right = (w[3] & 1u) != 0u;
    if (r < 0) {
      sh.htop = m;
      if (left || right) atomicOr(&sh.hcorner, (left ? 1u : 0u) | (right ? 2u : 0u));
    } else if (r >= kBlkY) {
      sh.hbot = m;
      if (left || right) atomicOr(&sh.hcorner, (left ? 4u : 0u) | (right ? 8u : 0u));
    } else {   // q = tid: this thread's row
      mine = m;
      sh.mrow[r] = m;
      sh.pw[r][0] = sh.pw[r][1] = 0u;
      if (left) atomicOr(&sh.hleft, 1ull << r);
      if (right) atomicOr(&sh.hright, 1ull << r);
    }
  }
  if (skip) return false;
  // 2. the run list: counts per row, their scan (one thread per row, the
  // first kBlkY / 32 warps), then each row's runs
  if (tid < kBlkY) {
    rc = __popcll((long long)run_starts(mine));
    rincl = rc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, rincl, o);
      if (lane >= o) rincl += y;
    }
    if (lane == 31) sh.wrun[warp] = rincl;
    int n = __popcll((long long)mine);
#pragma unroll
    for (int o = 16; o; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
    if (lane == 0) atomicAdd(&sh.nsel, n);
  }
  __syncthreads();
  int nr = 0;
#pragma unroll
  for (int w = 0; w < kBlkY / 32; ++w) nr += sh.wrun[w];
  if (nr > MAXR) return false;
  if (tid < kBlkY) {
    int k = rincl - rc;
    for (int w = 0; w < warp; ++w) k += sh.wrun[w];
    sh.runbase[tid] = k;
    if (tid == 0) sh.runbase[kBlkY] = nr;
    for (unsigned long long st = run_starts(mine); st; st &= st - 1, ++k) {
      const int s0 = __ffsll((long long)st) - 1;
      const int e0 = 63 - __clzll((long long)run_bits(mine, s0));
      sh.rinfo[k] = ((uint32_t)tid << 16) | ((uint32_t)s0 << 8) | (uint32_t)e0;
      sh.par[k] = (short)k;
      sh.pkey[k] = 0ull;
    }
  }
  for (int k = tid; k < MAXR / 32; k += NT) sh.bnd[k] = 0u;
  __syncthreads();
  auto run_index = [&](int row, int s0) {   // run of `row` starting at bit s0
    const unsigned long long st = run_starts(sh.mrow[row]);
    return sh.runbase[row] + __popcll((long long)(st & ((1ull << s0) - 1ull)));
  };
  // 3. unions: each run with the touching runs of the row above
  const volatile short* vpar = sh.par;
  auto unite_r = [&](int a, int c) {
    for (int it = 0; it < (1 << 16); ++it) {
      while (vpar[a] != a) a = vpar[a];
      while (vpar[c] != c) c = vpar[c];
      if (a == c) return;
      const int hi = a > c ? a : c, lo = a > c ? c : a;
      // 16-bit compare-and-swap through the aligned 32-bit word
      unsigned* w = reinterpret_cast<unsigned*>(&sh.par[hi & ~1]);
      const unsigned shf = (hi & 1) ? 16u : 0u;
      const unsigned old = *reinterpret_cast<volatile unsigned*>(w);
      if ((int)(short)(old >> shf) != hi) continue;
      const unsigned nw = (old & ~(0xffffu << shf)) | ((unsigned)(unsigned short)lo << shf);
      if (atomicCAS(w, old, nw) == old) return;
    }
    atomicOr(status, kErrCcLimit);
  };
  for (int k = tid; k < nr; k += NT) {
    const uint32_t ri = sh.rinfo[k];
    const int row = ri >> 16, s0 = (ri >> 8) & 255, e0 = ri & 255;
    if (row == 0) continue;
    const unsigned long long rb = (e0 == 63 ? ~0ull : ((2ull << e0) - 1ull)) & ~((1ull << s0) - 1ull);
    const unsigned long long u = sh.mrow[row - 1];
    unsigned long long nb = (rb | (rb << 1) | (rb >> 1)) & u;
    while (nb) {
      const int ub = __ffsll((long long)nb) - 1;
      const int us = run_of(u, ub);
      unite_r(k, run_index(row - 1, us));
      nb &= ~run_bits(u, us);
    }
  }
  __syncthreads();
  // 4. per run: its root (read-only), boundary flag, peak key
  int rootv[kIter];
#pragma unroll
  for (int j = 0; j < kIter; ++j) {
    const int k = tid + j * NT;
    rootv[j] = -1;
    if (k >= nr) continue;
    int r = k;
    while (sh.par[r] != r) r = sh.par[r];
    rootv[j] = r;
    const uint32_t ri = sh.rinfo[k];
    const int row = ri >> 16, s0 = (ri >> 8) & 255, e0 = ri & 255;
    const unsigned long long rb = (e0 == 63 ? ~0ull : ((2ull << e0) - 1ull)) & ~((1ull << s0) - 1ull);
    const unsigned long long dil = rb | (rb << 1) | (rb >> 1);
    bool out = false;
    if (row == 0)
      out = out || (dil & sh.htop) || (s0 == 0 && (sh.hcorner & 1u)) || (e0 == 63 && (sh.hcorner & 2u));
    if (row == kBlkY - 1)
      out = out || (dil & sh.hbot) || (s0 == 0 && (sh.hcorner & 4u)) || (e0 == 63 && (sh.hcorner & 8u));
    // block rows row-1..row+1 as halo-column bits
    const unsigned long long near = row == 0 ? 3ull : (7ull << (row - 1));
    if (s0 == 0) out = out || (sh.hleft & near);
    if (e0 == 63) out = out || (sh.hright & near);
    if (out) atomicOr(&sh.bnd[r >> 5], 1u << (r & 31));
    unsigned long long key = 0ull;
    const uint32_t t0 = (uint32_t)((ty0 + row) * Tx + tx0);
    const float* vr = vals + (size_t)g * stride + t0;
#pragma unroll 4
    for (int c = s0; c <= e0; ++c) {
      const unsigned long long kc = peak_key(vr[c], t0 + (uint32_t)c);
      key = kc > key ? kc : key;
    }
    atomicMax(&sh.pkey[r], key);
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kIter; ++j)
    if (rootv[j] >= 0) sh.par[tid + j * NT] = (short)rootv[j];   // straight to the root
  // 5. roots: an interior component's peak bit; a boundary component's id
#pragma unroll
  for (int j = 0; j < kIter; ++j) {
    const int k = tid + j * NT;
    if (rootv[j] != k) continue;
    const unsigned long long key = sh.pkey[k];
    if (!((sh.bnd[k >> 5] >> (k & 31)) & 1u)) {
      const uint32_t t = 0xffffffffu - (uint32_t)key;
      const int pty = (int)(t / (uint32_t)Tx), ptx = (int)(t - (uint32_t)pty * (uint32_t)Tx);
      const int ply = pty - ty0, plx = ptx - tx0;
      atomicOr(&sh.pw[ply][plx >> 5], 1u << (plx & 31));
    } else {
      const int slot = atomicAdd(&sh.nbnd, 1);   // < kBlkIds: each owns a ring tile
      const int id = (int)(bidx * kBlkIds + slot);
      b.bpar[id] = id;
      b.bgrp[id] = g;
      b.bkey[id] = key;
      b.rkey[id] = key;
      sh.pkey[k] = (unsigned long long)id;   // only this thread reads or writes a root's slot here
    }
  }
  __syncthreads();
  // 6. edge tiles of boundary components: their label, and each selected
  // neighbour across the block edge with a larger tile index as a pair; the
  // block's peak words; the counts
  auto selected = [&](int ly, int lx) -> bool {   // -1 <= ly <= kBlkY, -1 <= lx <= kBlkX
    if (ly >= 0 && ly < kBlkY) {
      if (lx >= 0 && lx < kBlkX) return (sh.mrow[ly] >> lx) & 1ull;
      return ((lx < 0 ? sh.hleft : sh.hright) >> ly) & 1ull;
    }
    if (lx >= 0 && lx < kBlkX) return ((ly < 0 ? sh.htop : sh.hbot) >> lx) & 1ull;
    return (sh.hcorner >> ((ly < 0 ? 0 : 2) + (lx < 0 ? 0 : 1))) & 1u;
  };
  if (sh.nbnd > 0) {
    for (int q = tid; q < kBlkRing; q += NT) {
      int ly, lx;
      ring_pos(q, &ly, &lx);
      if (!selected(ly, lx)) continue;
      const int r = sh.par[run_index(ly, run_of(sh.mrow[ly], lx))];
      if (!((sh.bnd[r >> 5] >> (r & 31)) & 1u)) continue;
      const int64_t t = (int64_t)(ty0 + ly) * Tx + (tx0 + lx);
      b.glab[(size_t)g * stride + t] = (int)sh.pkey[r];
#pragma unroll
      for (int d = 0; d < 8; ++d) {
        int dy, dx;
        dir_offset(d, &dy, &dx);
        const int ny = ly + dy, nx = lx + dx;
        const bool outside = ny < 0 || ny >= kBlkY || nx < 0 || nx >= kBlkX;
        if (!outside || !selected(ny, nx)) continue;
        if (dy * Tx + dx <= 0) continue;   // the other tile records it
        const int k = atomicAdd(&sh.npair, 1);   // < kBlkPairs: at most 4 per ring tile
        b.pairs[bidx * kBlkPairs + k] =
            ((unsigned long long)g << 40) | ((unsigned long long)t << 3) | (unsigned)d;
      }
    }
  }
  for (int q = tid; q < 2 * kBlkY; q += NT) {
    const int ly = q >> 1, wx = q & 1;
    const int ty = ty0 + ly, w = tx0 / 32 + wx;
    if (ty < Ty && w < b.words) b.pbits[((size_t)g * Ty + ty) * b.words + w] = sh.pw[ly][wx];
  }
  __syncthreads();
  if (tid == 0) b.bstat[bidx] = make_int4(sh.nbnd, sh.npair, sh.nsel, 0);
  return true;
}

// A block holds a hundred or two runs where a few per cent of the tiles are
// selected, and its labelling is a chain of short dependent steps: what counts
// is how many blocks an SM has in hand.  Two warps and shared memory for
// kBlkFewRuns runs let 20 blocks share an SM, where 256 threads and room for
// the most runs a block can have (2048) let six: k_blk_cc, 30 sliding maps of 16.8
// M pixels 1378 -> 688 us, 6 maps of 24.2 M tiles 528 -> 420, 62 maps of 672 k 114
// -> 108.  Bound by issue and the divergence of the loops over runs.
// k_blk_cc_full takes what is left, one block to a CTA at a time over the whole
// chip: the blocks of more runs, which k_blk_cc lists; all blocks where the
// selection is dense (kDenseRuns a block on average by the sample of k_blk_mask,
// 12% of the tiles, 4 sigma on sky: k_blk_cc then returns at once); and all blocks
// of maps that fill no more than one wave of its own CTAs.  Selection of 62 maps
// of 672 k tiles at 2 / 3 / 4 / 6 sigma 452 / 373 / 337 / 262 us; every block in
// full 436 / 370 / 335 / 282; listed without the dense rule 516 / 415 / 337 / 259;
// with the blocks found and labelled in turn by a CTA for each 256 of them 4326 / 460
// / 338 / 262.  14 maps of 42 k tiles (224 blocks) at 2 / 6 sigma 51 / 36 us, listed
// 94 / 47.
constexpr int kBlkFewThreads = 64;
constexpr int kBlkFewRuns = 512;
constexpr int kDenseRuns = 360;
constexpr int kBlkFullPerSm = 6;
enum { kFullListed = 0, kFullAll = 1 };   // k_blk_cc_full's blocks

__global__ void __launch_bounds__(kBlkFewThreads, 20) k_blk_cc(const float* __restrict__ vals,
                                                               int64_t stride, int Tx, int Ty,
                                                               unsigned dense, BlockScratch b,
                                                               unsigned* status) {
  pdl_begin();
  __shared__ BlkShared<kBlkFewThreads, kBlkFewRuns> sh;
  const bool skip = *b.runs >= dense;
  const int64_t bidx = ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
  if (!blk_label(sh, vals, stride, Tx, Ty, b, bidx, (int)blockIdx.z, (int)blockIdx.x,
                 (int)blockIdx.y, skip, status) &&
      !skip && threadIdx.x == 0)
    b.full[atomicAdd(&b.counters[3], 1)] = (int)bidx;
}

__global__ void __launch_bounds__(kBlkThreads, kBlkFullPerSm) k_blk_cc_full(
    const float* __restrict__ vals, int64_t stride, int Tx, int Ty, int nblocks, int blocks,
    unsigned dense, BlockScratch b, unsigned* status) {
  pdl_begin();
  __shared__ BlkShared<kBlkThreads, kBlkMaxRuns> sh;
  const int nbx = (Tx + kBlkX - 1) / kBlkX, nby = (Ty + kBlkY - 1) / kBlkY;
  const bool all = blocks == kFullAll || *b.runs >= dense;
  const int n = all ? nblocks : b.counters[3];
  __shared__ int next[2];
  for (int i = blockIdx.x, k = 0; i < n; i = next[k], k ^= 1) {
    const int bidx = all ? i : b.full[i];
    if (threadIdx.x == 0) next[k] = (int)gridDim.x + atomicAdd(&b.counters[1], 1);
    blk_label(sh, vals, stride, Tx, Ty, b, bidx, bidx / (nbx * nby), bidx % nbx, bidx / nbx % nby,
              false, status);
    __syncthreads();   // the next block's memory
  }
}

// Unions of boundary components across block edges: one warp per block joins
// the component ids of the block's recorded neighbour pairs.
__device__ __forceinline__ bool valid_id(const BlockScratch& b, int64_t nblocks, int id) {
  if (id < 0) return false;
  const int64_t blk = id / kBlkIds;
  return blk < nblocks && (id - blk * kBlkIds) < b.bstat[blk].x;
}

// (the loads of words that other warps change go past the L1 cache, so that
// the steps may also follow each other inside one CTA)
__device__ __forceinline__ void blk_merge(int64_t stride, int Tx, int64_t nblocks,
                                          const BlockScratch& b, unsigned* status, int64_t w0,
                                          int64_t nw) {
  const int lane = threadIdx.x & 31;
  for (int64_t blk = w0; blk < nblocks; blk += nw) {
    const int np = b.bstat[blk].y;
    for (int k = lane; k < np; k += 32) {
      const unsigned long long pk = b.pairs[blk * kBlkPairs + k];
      const int g = (int)(pk >> 40);
      const int64_t t = (int64_t)((pk >> 3) & ((1ull << 37) - 1));
      int dy, dx;
      dir_offset((int)(pk & 7u), &dy, &dx);
      const int64_t tn = t + (int64_t)dy * Tx + dx;
      const int* lab = b.glab + (size_t)g * stride;
      // the label map is never cleared: every label read here was written by
      // k_blk_cc of this detect, and the check keeps a stale one harmless
      const int me = lab[t], other = lab[tn];
      if (valid_id(b, nblocks, me) && valid_id(b, nblocks, other)) unite(b.bpar, me, other, status);
    }
  }
}

// Merged peak keys: every boundary component raises its root's key.
__device__ __forceinline__ void blk_resolve(int64_t nblocks, const BlockScratch& b, int64_t w0,
                                            int64_t nw) {
  const int lane = threadIdx.x & 31;
  for (int64_t blk = w0; blk < nblocks; blk += nw) {
    const int n = b.bstat[blk].x;
    for (int k = lane; k < n; k += 32) {
      const int id = (int)(blk * kBlkIds + k);
      const int r = find_g(b.bpar, id);
      if (r != id) atomicMax(&b.rkey[r], b.bkey[id]);
    }
  }
}

// Each merged component's peak bit.
__device__ __forceinline__ void blk_mark(int Tx, int Ty, int64_t nblocks, const BlockScratch& b,
                                         int64_t w0, int64_t nw) {
  const int lane = threadIdx.x & 31;
  for (int64_t blk = w0; blk < nblocks; blk += nw) {
    const int n = b.bstat[blk].x;
    for (int k = lane; k < n; k += 32) {
      const int id = (int)(blk * kBlkIds + k);
      if (__ldcg(&b.bpar[id]) != id) continue;   // roots never change after the unions
      const uint32_t t = 0xffffffffu - (uint32_t)__ldcg(&b.rkey[id]);
      const int ty = (int)(t / (uint32_t)Tx), tx = (int)(t - (uint32_t)ty * (uint32_t)Tx);
      atomicOr(&b.pbits[((size_t)b.bgrp[id] * Ty + ty) * b.words + (tx >> 5)], 1u << (tx & 31));
    }
  }
}

__device__ __forceinline__ int64_t grid_warp() {
  return ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
}
__device__ __forceinline__ int64_t grid_warps() { return ((int64_t)gridDim.x * blockDim.x) >> 5; }

__global__ void k_blk_merge(int64_t stride, int Tx, int64_t nblocks, BlockScratch b,
                            unsigned* status) {
  pdl_begin();
  blk_merge(stride, Tx, nblocks, b, status, grid_warp(), grid_warps());
}

__global__ void k_blk_resolve(int64_t nblocks, BlockScratch b) {
  pdl_begin();
  blk_resolve(nblocks, b, grid_warp(), grid_warps());
}

__global__ void k_blk_mark(int Tx, int Ty, int64_t nblocks, BlockScratch b) {
  pdl_begin();
  blk_mark(Tx, Ty, nblocks, b, grid_warp(), grid_warps());
}

// Ordered compaction of the peak bitmap, one warp per tile row and
// kRowsPerCta rows per CTA: each row's peak count and each CTA's sum, the
// scan of the CTAs' sums, then each row's peaks in order.  A row's offset is
// its CTA's offset plus the counts of the CTA's rows before it.
constexpr int kPbThreads = 256;
constexpr int kRowsPerCta = kPbThreads / 32;

__device__ __forceinline__ int64_t row_offset(const BlockScratch& b, int64_t r) {
  const int64_t r0 = r & ~(int64_t)(kRowsPerCta - 1);
  int64_t off = b.blkoff[r0 / kRowsPerCta];
#pragma unroll
  for (int k = 0; k < kRowsPerCta - 1; ++k)
    if (r0 + k < r) off += b.rowcnt[r0 + k];
  return off;
}

__global__ void __launch_bounds__(kPbThreads) k_pbits_count(int64_t nrows, BlockScratch b) {
  pdl_begin();
  __shared__ int wc[kRowsPerCta];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t r = (int64_t)blockIdx.x * kRowsPerCta + warp;
  int c = 0;
  if (r < nrows) {
    const uint32_t* row = b.pbits + (size_t)r * b.words;
    for (int w = lane; w < b.words; w += 32) c += __popc(row[w]);
  }
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if (lane == 0) {
    wc[warp] = c;
    if (r < nrows) b.rowcnt[r] = c;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int w = 0; w < kRowsPerCta; ++w) t += wc[w];
    b.blkcnt[blockIdx.x] = t;
  }
}

__global__ void __launch_bounds__(kPbThreads) k_pbits_write(int64_t nrows, int Tx, int Ty,
                                                            const float* __restrict__ vals,
                                                            int64_t stride, BlockScratch b,
                                                            SelItem* peaks, int64_t cap) {
  pdl_begin();
  const int lane = threadIdx.x & 31;
  const int64_t r = ((int64_t)blockIdx.x * kPbThreads + threadIdx.x) >> 5;
  if (r >= nrows) return;
  const int g = (int)(r / Ty), ty = (int)(r - (int64_t)g * Ty);
  const uint32_t* row = b.pbits + (size_t)r * b.words;
  const float* vg = vals + (size_t)g * stride;
  int64_t run = row_offset(b, r);
  for (int w0 = 0; w0 < b.words; w0 += 32) {
    const int wx = w0 + lane;
    const uint32_t w = wx < b.words ? row[wx] : 0u;
    const int c = __popc(w);
    int incl = c;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    int64_t pos = run + incl - c;
    run += __shfl_sync(0xffffffffu, incl, 31);
    // every value load of the word first, then the writes
    constexpr int kMaxBits = 8;
    float val[kMaxBits];
    int tt[kMaxBits];
    uint32_t m = w;
    while (m) {
      int nb = 0;
      for (; m && nb < kMaxBits; ++nb) {
        const int bit = __ffs(m) - 1;
        m &= m - 1;
        tt[nb] = ty * Tx + wx * 32 + bit;
        val[nb] = vg[tt[nb]];
      }
      for (int k = 0; k < nb; ++k, ++pos)
        if (pos < cap) peaks[pos] = SelItem{g, tt[k], val[k]};
    }
  }
}

// The selected count (the blocks' sum) against the selection capacity, by one
// CTA of 1024 threads.
__device__ __forceinline__ void blk_check(int64_t nblocks, const BlockScratch& b, int64_t cap,
                                          unsigned* status, unsigned* want, long long* part) {
  long long n = 0;
  for (int64_t i = threadIdx.x; i < nblocks; i += 1024) n += b.bstat[i].z;
  for (int o = 16; o; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = n;
  __syncthreads();
  if (threadIdx.x == 0) {
    long long tot = 0;
    for (int w = 0; w < 32; ++w) tot += part[w];
    if (tot > cap) {
      atomicOr(status, kErrCapacity);
      if (want) atomicMax(want, (unsigned)(tot < 0xffffffffll ? tot : 0xffffffffll));
    }
  }
}

// One CTA scans the row counts of the CTAs of k_pbits_count, another checks
// the capacity.
__global__ void __launch_bounds__(1024) k_blk_scan(int nblk, int64_t nblocks, BlockScratch b,
                                                   int64_t cap, unsigned* status, unsigned* want) {
  pdl_begin();
  __shared__ long long sh[1024];
  if (blockIdx.x == 0)
    scan_counts(nblk, b.blkcnt, b.blkoff, &b.counters[2], cap, status, (unsigned*)nullptr, sh);
  else
    blk_check(nblocks, b, cap, status, want, sh);
}

// Small maps: everything after the labelling in one CTA, whose barriers cost
// a fraction of the launches they replace (unions, peaks, row counts, their scan
// and the check: six).  Bounded by kTailBlocks blocks, four per warp (256 took 39
// us against about 28 in launches of their own), and by the rows whose counts fit
// in shared memory.
constexpr int kTailThreads = 1024;
constexpr int64_t kTailBlocks = 128;
constexpr int64_t kTailRows = 4096;

__global__ void __launch_bounds__(kTailThreads) k_blk_tail(int64_t stride, int Tx, int Ty,
                                                           int64_t nblocks, int64_t nrows,
                                                           BlockScratch b, int64_t cap,
                                                           unsigned* status, unsigned* want) {
  pdl_begin();
  __shared__ union {
    long long scan[1024];
    int rows[kTailRows];
  } sh;
  const int tid = threadIdx.x, warp = tid >> 5;
  blk_merge(stride, Tx, nblocks, b, status, warp, kTailThreads / 32);
  __syncthreads();
  blk_resolve(nblocks, b, warp, kTailThreads / 32);
  __syncthreads();
  blk_mark(Tx, Ty, nblocks, b, warp, kTailThreads / 32);
  __syncthreads();
  // the peaks of every tile row: a thread per bitmap word (the bits set above
  // are past the L1 cache)
  for (int r = tid; r < nrows; r += kTailThreads) sh.rows[r] = 0;
  __syncthreads();
  const int nwords = (int)nrows * b.words;
  for (int i0 = tid; i0 < nwords; i0 += 8 * kTailThreads) {
    uint32_t w[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int i = i0 + k * kTailThreads;
      w[k] = i < nwords ? __ldcg(b.pbits + i) : 0u;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (w[k]) atomicAdd(&sh.rows[(i0 + k * kTailThreads) / b.words], __popc(w[k]));
  }
  __syncthreads();
  for (int r = tid; r < nrows; r += kTailThreads) b.rowcnt[r] = sh.rows[r];
  const int ncta = (int)((nrows + kRowsPerCta - 1) / kRowsPerCta);
  for (int i = tid; i < ncta; i += kTailThreads) {
    int c = 0;
    for (int64_t r = (int64_t)i * kRowsPerCta; r < nrows && r < (int64_t)(i + 1) * kRowsPerCta; ++r)
      c += sh.rows[r];
    b.blkcnt[i] = c;
  }
  __syncthreads();
  scan_counts(ncta, b.blkcnt, b.blkoff, &b.counters[2], cap, status, (unsigned*)nullptr, sh.scan);
  __syncthreads();
  blk_check(nblocks, b, cap, status, want, sh.scan);
}

static int block_words(int Tx) { return (Tx + 31) / 32; }

static int64_t block_count(int groups, int Tx, int Ty) {
  return (int64_t)groups * ((Ty + kBlkY - 1) / kBlkY) * ((Tx + kBlkX - 1) / kBlkX);
}

size_t block_scratch_bytes(int groups, int Tx, int Ty, int64_t stride) {
  const int64_t cap = block_count(groups, Tx, Ty) * kBlkIds;
  const int64_t nw = (int64_t)groups * Ty * block_words(Tx);
  const int64_t nrows = (int64_t)groups * Ty;
  const int64_t nblk = (nrows + kRowsPerCta - 1) / kRowsPerCta;
  size_t bytes = 0;
  auto add = [&](size_t n) { bytes += (n + 255) / 256 * 256; };
  add(sizeof(int) * (size_t)groups * stride);    // glab
  add(sizeof(int) * cap);                        // bpar
  add(sizeof(int) * cap);                        // bgrp
  add(sizeof(unsigned long long) * cap);         // bkey
  add(sizeof(unsigned long long) * cap);         // rkey
  add(sizeof(uint32_t) * nw);                    // pbits
  add(sizeof(uint32_t) * nw);                    // sbits
  add(sizeof(unsigned long long) * block_count(groups, Tx, Ty) * kBlkPairs);   // pairs
  add(sizeof(int4) * block_count(groups, Tx, Ty));   // bstat
  add(sizeof(int) * block_count(groups, Tx, Ty));    // full
  add(sizeof(int) * 4);                          // counters
  add(sizeof(int) * nblk);                       // blkcnt
  add(sizeof(int) * (nblk + 1));                 // blkoff
  add(sizeof(int) * nrows);                      // rowcnt
  return bytes;
}

void block_scratch_carve(void* base, int groups, int Tx, int Ty, int64_t stride, BlockScratch* b) {
  const int64_t cap = block_count(groups, Tx, Ty) * kBlkIds;
  const int64_t nw = (int64_t)groups * Ty * block_words(Tx);
  char* p = static_cast<char*>(base);
  size_t off = 0;
  auto take = [&](size_t n) {
    char* q = p + off;
    off += (n + 255) / 256 * 256;
    return q;
  };
  b->glab = reinterpret_cast<int*>(take(sizeof(int) * (size_t)groups * stride));
  b->bpar = reinterpret_cast<int*>(take(sizeof(int) * cap));
  b->bgrp = reinterpret_cast<int*>(take(sizeof(int) * cap));
  b->bkey = reinterpret_cast<unsigned long long*>(take(sizeof(unsigned long long) * cap));
  b->rkey = reinterpret_cast<unsigned long long*>(take(sizeof(unsigned long long) * cap));
  b->pbits = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * nw));
  b->sbits = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * nw));
  b->pairs = reinterpret_cast<unsigned long long*>(
      take(sizeof(unsigned long long) * block_count(groups, Tx, Ty) * kBlkPairs));
  b->bstat = reinterpret_cast<int4*>(take(sizeof(int4) * block_count(groups, Tx, Ty)));
  b->full = reinterpret_cast<int*>(take(sizeof(int) * block_count(groups, Tx, Ty)));
  b->pcap = block_count(groups, Tx, Ty) * kBlkPairs;
  b->counters = reinterpret_cast<int*>(take(sizeof(int) * 4));
  const int64_t nrows = (int64_t)groups * Ty;
  b->nblk = (int)((nrows + kRowsPerCta - 1) / kRowsPerCta);
  b->blkcnt = reinterpret_cast<int*>(take(sizeof(int) * b->nblk));
  b->blkoff = reinterpret_cast<int*>(take(sizeof(int) * (b->nblk + 1)));
  b->rowcnt = reinterpret_cast<int*>(take(sizeof(int) * nrows));
  b->cap = cap;
  b->words = block_words(Tx);
}

cudaError_t launch_block_select(const float* vals, int groups, int64_t stride, int Tx, int Ty,
                                const double* cs, double tau, double* inv, const BlockScratch& b,
                                SelItem* peaks, int64_t cap, unsigned* status, unsigned* want,
                                cudaStream_t st) {
  // peaks == nullptr: the caller emits straight from the rows (launch_emit_rows)
  const int64_t nblocks = block_count(groups, Tx, Ty);
  if (groups < 1 || groups > 65535 || (Ty + kBlkY - 1) / kBlkY > 65535 ||
      (int64_t)Tx * Ty > 0xffffffffll || nblocks * kBlkIds > INT_MAX ||
      nblocks * kBlkIds > b.cap)
    return cudaErrorInvalidValue;
  // (counters[2], the peak count, is written by the scan below; nothing else
  // is read, so no clearing launch sits between the noise and this chain)
  const int64_t nrows = (int64_t)groups * Ty;
  const int64_t ncta = (nrows + kRowsPerCta - 1) / kRowsPerCta;
  if (ncta > b.nblk) return cudaErrorInvalidValue;   // sized by block_scratch_carve
  int launches = 2;
  cudaError_t e = launch_pdl(k_blk_mask, dim3((unsigned)((nrows * 32 + kMaskThreads - 1) / kMaskThreads)),
                             dim3(kMaskThreads), 0, st, vals, stride, Tx, Ty, nrows, cs, tau, inv, b);
  // runs in the rows that k_blk_mask samples where a block has kDenseRuns
  const double sampled = (double)((nrows + kMaskThreads / 32 - 1) / (kMaskThreads / 32)) / (double)nrows;
  const unsigned dense = (unsigned)std::min(
      4e9, (double)kDenseRuns * sampled * (double)groups * Tx * Ty / (kBlkX * kBlkY) + 1.0);
  if (nblocks <= 152 * kBlkFullPerSm) {
    if (e == cudaSuccess)
      e = launch_pdl(k_blk_cc_full, dim3((unsigned)nblocks), dim3(kBlkThreads), 0, st, vals, stride,
                     Tx, Ty, (int)nblocks, (int)kFullAll, dense, b, status);
  } else {
    const dim3 grid((Tx + kBlkX - 1) / kBlkX, (Ty + kBlkY - 1) / kBlkY, groups);
    if (e == cudaSuccess)
      e = launch_pdl(k_blk_cc, grid, dim3(kBlkFewThreads), 0, st, vals, stride, Tx, Ty, dense, b, status);
    if (e == cudaSuccess)
      e = launch_pdl(k_blk_cc_full, dim3(152 * kBlkFullPerSm), dim3(kBlkThreads), 0, st, vals, stride,
                     Tx, Ty, (int)nblocks, (int)kFullListed, dense, b, status);
    launches += 1;
  }
  if (nblocks <= kTailBlocks && nrows <= kTailRows) {
    if (e == cudaSuccess)
      e = launch_pdl(k_blk_tail, dim3(1), dim3(kTailThreads), 0, st, stride, Tx, Ty, nblocks, nrows,
                     b, cap, status, want);
    launches += 1;
  } else {
    const unsigned wgrid = (unsigned)std::min<int64_t>((nblocks + 7) / 8, 152 * 64);   // a warp per block
    if (e == cudaSuccess)
      e = launch_pdl(k_blk_merge, dim3(wgrid), dim3(256), 0, st, stride, Tx, nblocks, b, status);
    if (e == cudaSuccess) e = launch_pdl(k_blk_resolve, dim3(wgrid), dim3(256), 0, st, nblocks, b);
    if (e == cudaSuccess)
      e = launch_pdl(k_blk_mark, dim3(wgrid), dim3(256), 0, st, Tx, Ty, nblocks, b);
    if (e == cudaSuccess)
      e = launch_pdl(k_pbits_count, dim3((unsigned)ncta), dim3(kPbThreads), 0, st, nrows, b);
    if (e == cudaSuccess)
      e = launch_pdl(k_blk_scan, dim3(2), dim3(1024), 0, st, (int)ncta, nblocks, b, cap, status, want);
    launches += 5;
  }
  if (e == cudaSuccess && peaks) {
    e = launch_pdl(k_pbits_write, dim3((unsigned)ncta), dim3(kPbThreads), 0, st, nrows, Tx, Ty, vals,
                   stride, b, peaks, cap);
    launches += 1;
  }
  if (e != cudaSuccess) return e;
  count_launches(launches);
  return cudaGetLastError();
}

// ---- ordered list of component peaks (sorted by (group, t) like the items)
__global__ void __launch_bounds__(kSelThreads) k_peak_count(const int* nsel, const int* parent,
                                                            const int* peak, int nblk,
                                                            int* blkcnt) {
  __shared__ int wsum[kSelThreads / 32];
  int64_t lo, hi;
  chunk_range(*nsel, nblk, blockIdx.x, &lo, &hi);
  int cnt = 0;
  for (int64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) cnt += peak[parent[i]] == (int)i;
  for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = cnt;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int w = 0; w < kSelThreads / 32; ++w) t += wsum[w];
    blkcnt[blockIdx.x] = t;
  }
}

__global__ void __launch_bounds__(kSelThreads) k_peak_write(const int* nsel, const int* parent,
                                                            const int* peak, int nblk,
                                                            const int* blkoff, int* plist) {
  __shared__ int wcnt[kSelThreads / 32];
  int64_t lo, hi;
  chunk_range(*nsel, nblk, blockIdx.x, &lo, &hi);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int run = blkoff[blockIdx.x];
  for (int64_t base = lo; base < hi; base += blockDim.x) {
    const int64_t i = base + threadIdx.x;
    const bool is_peak = i < hi && peak[parent[i]] == (int)i;
    const unsigned bal = __ballot_sync(0xffffffffu, is_peak);
    if (lane == 0) wcnt[warp] = __popc(bal);
    __syncthreads();
    int before = 0, tile = 0;
    for (int w = 0; w < kSelThreads / 32; ++w) {
      before += w < warp ? wcnt[w] : 0;
      tile += wcnt[w];
    }
    if (is_peak) plist[run + before + __popc(bal & ((1u << lane) - 1u))] = (int)i;
    run += tile;
    __syncthreads();
  }
}

// ---- candidates
// Peak p of an ordered peak list: items[plist[p]], or items[p] without plist.
__device__ __forceinline__ SelItem peak_item(const SelItem* items, const int* plist, int p) {
  return plist ? items[plist[p]] : items[p];
}

__device__ __forceinline__ float load_px(const void* base, int storage, int64_t idx) {
  switch (storage) {
    case FITRIG_BF16: return to_f32(static_cast<const bf16_t*>(base)[idx]);
    case FITRIG_F16: return to_f32(static_cast<const f16_t*>(base)[idx]);
    default: return static_cast<const float*>(base)[idx];
  }
}

__device__ __forceinline__ float parabola(float l, float c, float r) {
  if (!isfinite(l) || !isfinite(c) || !isfinite(r)) return 0.f;
  const float den = l - 2.f * c + r;
  if (!(den < 0.f)) return 0.f;
  const float d = 0.5f * (l - r) / den;
  return fminf(0.5f, fmaxf(-0.5f, d));
}

// Peak offset within [-0.5, 0.5] of the Catmull-Rom cubic spline through the
// samples at -2..2 (m2, m1, c, p1, p2) along one axis of the eta map.  On the
// segment from a (at 0) to b (at 1) with outer neighbours z (at -1) and d (at
// 2):  f(t) = a + t (k1 + t (k2 + t k3)),  k1 = (b - z)/2,
// k2 = (2z - 5a + 4b - d)/2,  k3 = (-z + 3a - 3b + d)/2.  Candidates in order:
// offset 0; the right segment's interior roots of f' (ascending), then +0.5;
// the left segment's (t in [0.5, 1], offset t - 1) roots, then -0.5; strictly
// larger values win.  A missing neighbour at +-1 leaves its side unsearched;
// a missing outer sample is extended linearly.  Roots of f' come from the
// cancellation-free form of the quadratic formula.
__device__ __forceinline__ float cubic_offset(float m2, float m1, float c, float p1, float p2) {
  if (!isfinite(c)) return 0.f;
  float bx = 0.f, bf = c;
  auto segment = [&](float z, float a, float b, float d, float lo, float hi, float shift) {
    const float k1 = 0.5f * (b - z);
    const float k2 = 0.5f * (2.f * z - 5.f * a + 4.f * b - d);
    const float k3 = 0.5f * (-z + 3.f * a - 3.f * b + d);
    auto f = [&](float t) { return a + t * (k1 + t * (k2 + t * k3)); };
    const float A = 3.f * k3, B = 2.f * k2, C = k1;
    const float disc = B * B - 4.f * A * C;
    float r0 = 0.f, r1 = 0.f;
    int nr = 0;
    if (disc >= 0.f) {
      const float q = -0.5f * (B + copysignf(sqrtf(disc), B));
      if (A != 0.f) r0 = q / A, nr = 1;
      if (q != 0.f) {
        if (nr == 0) r0 = C / q;
        else r1 = C / q;
        ++nr;
      }
      if (nr == 2 && r1 < r0) {
        const float t = r0;
        r0 = r1;
        r1 = t;
      }
    }
    if (nr >= 1 && lo < r0 && r0 < hi) {
      const float v = f(r0);
      if (v > bf) bf = v, bx = r0 + shift;
    }
    if (nr == 2 && lo < r1 && r1 < hi) {
      const float v = f(r1);
      if (v > bf) bf = v, bx = r1 + shift;
    }
    const float e = shift == 0.f ? hi : lo;
    const float v = f(e);
    if (v > bf) bf = v, bx = e + shift;
  };
  if (isfinite(p1)) {
    const float d = isfinite(p2) ? p2 : 2.f * p1 - c;
    segment(isfinite(m1) ? m1 : 2.f * c - p1, c, p1, d, 0.f, 0.5f, 0.f);
  }
  if (isfinite(m1)) {
    const float z = isfinite(m2) ? m2 : 2.f * m1 - c;
    segment(z, m1, c, isfinite(p1) ? p1 : 2.f * c - m1, 0.5f, 1.f, -1.f);
  }
  return bx;
}

// The candidate's significance, z = (v - centre) / scale in FP64 (Sec. 2.4.1,
// 2.4.2), rounded to FP32 for the output.
__device__ __forceinline__ float significance(const CandArgs& a, const SelItem& it) {
  return (float)(((double)it.v - a.cs[2 * it.group]) * a.inv[it.group]);
}

// Candidates so far: those before this branch's and its peaks, at most the
// buffer's (by one thread of the emitting kernel; no other one reads it).
__device__ __forceinline__ void set_count(const CandArgs& a, int64_t total, unsigned* status) {
  if (total > a.cap) {
    total = a.cap;
    atomicOr(status, kErrCapacity);
  }
  *a.nout = (int)total;
}

// Frequency branch: one thread per peak; tile-centre order is (y, x) order,
// so the peaks' list order is already the output order.
__global__ void k_emit_freq(CandArgs a, const SelItem* __restrict__ items, const int* np_,
                            const int* __restrict__ plist, unsigned* status) {
  pdl_begin();
  const int np = *np_;
  if (status && blockIdx.x == 0 && threadIdx.x == 0) set_count(a, np, status);
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < np; p += gridDim.x * blockDim.x) {
    const SelItem it = peak_item(items, plist, p);
    const int ty = it.t / a.Tx, tx = it.t - (it.t / a.Tx) * a.Tx;
    const int hw = min(a.w, a.ny - ty * a.w), ww = min(a.w, a.nx - tx * a.w);
    const float e = a.eta[it.t];
    const float el = tx > 0 ? a.eta[it.t - 1] : NAN;
    const float er = tx + 1 < a.Tx ? a.eta[it.t + 1] : NAN;
    const float eu = ty > 0 ? a.eta[it.t - a.Tx] : NAN;
    const float ed = ty + 1 < a.Ty ? a.eta[it.t + a.Tx] : NAN;
    fitrig_candidate c;
    c.x = tx * a.w + (ww - 1) / 2;
    c.y = ty * a.w + (hw - 1) / 2;
    c.snapshot = -1;
    c.significance = significance(a, it);
    c.branch = FITRIG_BRANCH_FREQ;
    c.freq_bin = a.bin[it.t];
    float dx, dy;
    if (a.refine == FITRIG_REFINE_CUBIC) {
      const float el2 = tx > 1 ? a.eta[it.t - 2] : NAN;
      const float er2 = tx + 2 < a.Tx ? a.eta[it.t + 2] : NAN;
      const float eu2 = ty > 1 ? a.eta[it.t - 2 * a.Tx] : NAN;
      const float ed2 = ty + 2 < a.Ty ? a.eta[it.t + 2 * a.Tx] : NAN;
      dx = cubic_offset(el2, el, e, er, er2);
      dy = cubic_offset(eu2, eu, e, ed, ed2);
    } else {
      dx = parabola(el, e, er);
      dy = parabola(eu, e, ed);
    }
    c.xf = (float)(tx * a.w) + 0.5f * (float)(ww - 1) + dx * (float)a.w;
    c.yf = (float)(ty * a.w) + 0.5f * (float)(hw - 1) + dy * (float)a.w;
    if (p < a.cap) a.out[p] = c;
  }
}

__device__ __forceinline__ fitrig_candidate image_candidate(const CandArgs& a, const SelItem& it,
                                                            int tx, int ty, int w, int dx, int dy) {
  fitrig_candidate c;
  c.x = tx * w + dx;
  c.y = ty * w + dy;
  c.snapshot = it.group;
  c.significance = significance(a, it);
  c.branch = FITRIG_BRANCH_IMAGE;
  c.freq_bin = -1;
  c.xf = (float)c.x;
  c.yf = (float)c.y;
  return c;
}

// Image branch, step 1 (otherwise): one warp per peak computes the tile's
// arg-max of Delta (ties: smallest row-major index, same FP32 arithmetic as the
// stack march) and writes the candidate in peak-list order to `tmp`.
__global__ void k_emit_image(CandArgs a, const SelItem* __restrict__ items, const int* np_,
                             const int* __restrict__ plist, fitrig_candidate* tmp) {
  pdl_begin();
  const int np = *np_;
  const int lane = threadIdx.x & 31;
  const int wid = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  for (int p = wid; p < np; p += nw) {
    const SelItem it = peak_item(items, plist, p);
    const int ty = it.t / a.Tx, tx = it.t - (it.t / a.Tx) * a.Tx;
    const int hw = min(a.w, a.ny - ty * a.w), ww = min(a.w, a.nx - tx * a.w);
    int64_t sl[3];   // the unit's three snapshots in the stack
    for (int k = 0; k < 3; ++k)
      sl[k] = (a.zmod > 0 ? (int64_t)((a.zrot + it.group + k) % a.zmod) : (int64_t)(it.group + k)) * a.slice;
    float best = -1.f;
    int bidx = INT_MAX;
    for (int q = lane; q < hw * ww; q += 32) {
      const int dy = q / ww, dx = q - (q / ww) * ww;
      const int64_t off = (int64_t)(ty * a.w + dy) * a.pitch + (tx * a.w + dx);
      float x0, x1, x2;
      if (a.key) {
        // difference-coded stack (plans only: slot = snapshot): decode the
        // pixel in snapshot order with the march's FP32 sums
        x0 = a.key[(int64_t)(ty * a.w + dy) * a.kpitch + (tx * a.w + dx)];
        for (int k = 1; k <= it.group; ++k)
          x0 = __fadd_rn(x0, load_px(a.stack, a.storage, (int64_t)k * a.slice + off));
        x1 = __fadd_rn(x0, load_px(a.stack, a.storage, sl[1] + off));
        x2 = __fadd_rn(x1, load_px(a.stack, a.storage, sl[2] + off));
      } else {
        x0 = load_px(a.stack, a.storage, sl[0] + off);
        x1 = load_px(a.stack, a.storage, sl[1] + off);
        x2 = load_px(a.stack, a.storage, sl[2] + off);
      }
      const float d = fabsf(fabsf(x2 - x1) - fabsf(x1 - x0));
      if (d > best) {
        best = d;
        bidx = q;
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
      const float ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bidx, o);
      if (ob > best || (ob == best && oi < bidx)) {
        best = ob;
        bidx = oi;
      }
    }
    if (lane == 0) tmp[p] = image_candidate(a, it, tx, ty, a.w, bidx % ww, bidx / ww);
  }
}

// Image branch, step 2: peaks are in (unit, tile row, tile column) order.  Each
// run of peaks sharing (unit, tile row) -- a group -- occupies the same output
// positions once sorted by (y, x); inside a group the order is (dy, tx), so a
// stable counting sort on the in-tile row dy finishes it.  A warp scans 32
// consecutive peaks, finds the group heads among them by ballot, and sorts
// each of those groups (which may run past its 32 entries).  A group's first
// 32 peaks are read once and kept in registers between the count and the
// write (most groups are no longer); later ones are read again.
constexpr int kGroupWarps = 8;
constexpr int kMaxW = 128;

// FROM_ARG: the candidates are formed here from the peak list and the
// march's in-tile arg-max (no intermediate list); otherwise they are read
// from `tmp`, where k_emit_image wrote them.
template <bool FROM_ARG>
__global__ void __launch_bounds__(kGroupWarps * 32) k_group_sort(CandArgs a, const int* np_,
                                                                 const fitrig_candidate* tmp,
                                                                 const SelItem* __restrict__ items,
                                                                 const int* __restrict__ plist,
                                                                 const int* base_,
                                                                 unsigned* status) {
  pdl_begin();
  __shared__ int counts[kGroupWarps][kMaxW];
  // one peak: its group (snapshot, tile row) and, for the count and the
  // write, its candidate
  struct Peak {
    SelItem it;   // FROM_ARG
    fitrig_candidate c;
    int snap, row;
  };
  auto head_of = [&](int p, int* snap, int* row) {
    if (FROM_ARG) {
      const SelItem it = peak_item(items, plist, p);
      *snap = it.group;
      *row = it.t / a.Tx;
    } else {
      const fitrig_candidate c = tmp[p];
      *snap = c.snapshot;
      *row = c.y / a.w;
    }
  };
  auto load = [&](int p) -> Peak {
    Peak k;
    if (FROM_ARG) {
      k.it = peak_item(items, plist, p);
      k.snap = k.it.group;
      k.row = k.it.t / a.Tx;
    } else {
      k.c = tmp[p];
      k.snap = k.c.snapshot;
      k.row = k.c.y / a.w;
    }
    return k;
  };
  // the candidate and its in-tile row (FROM_ARG: from the march's arg-max)
  auto finish = [&](Peak& k) -> int {
    if (FROM_ARG) {
      const int ty = k.row, tx = k.it.t - ty * a.Tx;
      const int idx = a.arg[(int64_t)k.it.group * a.stride + k.it.t];
      k.c = image_candidate(a, k.it, tx, ty, a.w, idx % a.w, idx / a.w);
    }
    return k.c.y - k.row * a.w;
  };
  const int np = *np_;
  const int base = base_ ? *base_ : 0;
  if (status && blockIdx.x == 0 && threadIdx.x == 0) set_count(a, (int64_t)base + np, status);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int* cnt = counts[warp];
  const int wid = blockIdx.x * kGroupWarps + warp;
  const int nw = gridDim.x * kGroupWarps;
  for (int p0 = wid * 32; p0 < np; p0 += nw * 32) {
    const int pl = p0 + lane;
    int sn = -1, rw = -1, psn = -2, prw = -2;
    if (pl < np) head_of(pl, &sn, &rw);
    if (lane == 0 && pl > 0 && pl < np) head_of(pl - 1, &psn, &prw);
    const int usn = __shfl_up_sync(0xffffffffu, sn, 1), urw = __shfl_up_sync(0xffffffffu, rw, 1);
    if (lane > 0) {
      psn = usn;
      prw = urw;
    }
    const bool head = pl < np && (sn != psn || rw != prw);
    unsigned heads = __ballot_sync(0xffffffffu, head);
    while (heads) {
      const int hl = __ffs(heads) - 1;
      heads &= heads - 1;
      const int p = p0 + hl;
      const int snap = __shfl_sync(0xffffffffu, sn, hl), gty = __shfl_sync(0xffffffffu, rw, hl);
      for (int k = lane; k < a.w; k += 32) cnt[k] = 0;
      __syncwarp();
      // the group's extent and its count per in-tile row; the first 32 peaks
      // stay in registers
      Peak first;
      int dy0 = kMaxW;
      int end = p;
      for (int q0 = p;; q0 += 32) {
        const int q = q0 + lane;
        Peak k;
        bool in = false;
        if (q < np) {
          k = load(q);
          in = k.snap == snap && k.row == gty;
        }
        int dy = kMaxW;
        if (in) {
          dy = finish(k);
          atomicAdd(&cnt[dy], 1);
        }
        if (q0 == p) {
          first = k;
          dy0 = dy;
        }
        const unsigned bal = __ballot_sync(0xffffffffu, in);   // a prefix of the lanes
        end = q0 + __popc(bal);
        if (bal != 0xffffffffu) break;
      }
      __syncwarp();
      if (lane == 0) {
        int run = 0;
        for (int k = 0; k < a.w; ++k) {
          const int c = cnt[k];
          cnt[k] = run;
          run += c;
        }
      }
      __syncwarp();
      for (int q0 = p; q0 < end; q0 += 32) {
        const int q = q0 + lane;
        const bool valid = q < end;
        Peak k = first;
        int dy = dy0;
        if (q0 != p) {
          dy = kMaxW;
          if (valid) {
            k = load(q);
            dy = finish(k);
          }
        }
        if (!valid) dy = kMaxW;
        // lanes with the same in-tile row: a ballot per row for small
        // windows (the match instruction's unit is slow), a match otherwise;
        // lanes past the group (dy = kMaxW) use none of it
        unsigned peers = 0;
        if (a.w <= 8) {
          for (int d = 0; d < a.w; ++d) {
            const unsigned b = __ballot_sync(0xffffffffu, dy == d);
            if (dy == d) peers = b;
          }
        } else {
          peers = __match_any_sync(0xffffffffu, dy);
        }
        const int rank = __popc(peers & ((1u << lane) - 1u));
        const int off = valid ? cnt[dy] : 0;
        __syncwarp();
        if (valid) {
          const int pos = base + p + off + rank;
          if (pos < a.cap) a.out[pos] = k.c;
          if (lane == __ffs(peers) - 1) cnt[dy] = off + __popc(peers);
        }
        __syncwarp();
      }
    }
  }
}

// Image branch straight from the peak bitmap, w <= kRowsMaxW: one warp per
// tile row writes the row's candidates in (snapshot, y, x) order, a bitmap
// word per lane, 32 words at a time.  Inside a tile row that order is (dy,
// tx), so a peak's place is the row's offset (from the scan of the rows' peak
// counts), the row's peaks in lower in-tile rows, and the peaks of its own
// in-tile row at smaller tx (earlier words, then warp scans of each lane's
// count per in-tile row).  Rows of more than 32 words (WIDE) are counted once
// over all words first.  The in-tile row and column come from the march's
// arg-max; in sliding mode and at w = 1 a tile is its pixel and there is
// nothing to read.  Each lane reads the arg-max byte and value of its first
// kRowsBatch peaks together and keeps them; a lane with more reads the rest
// again.  No peak list, recomputed arg-max or sort is needed: 30 sliding maps
// of 16.8 M pixels, 1.5 M candidates, 742 -> 160 us (k_pbits_write, k_emit_image
// and k_group_sort before); 6 maps of 24.2 M tiles, 7.3 M candidates, 382 -> 284.
// Of pixels as tiles (MAXW = 1: one count instead of eight) six CTAs fit an SM
// instead of four: sliding 32 x 4096^2 4.12 -> 4.08 ms a detect.
constexpr int kRowsMaxW = 8;
constexpr int kRowsBatch = 4;
template <bool WIDE, int MAXW>
__global__ void __launch_bounds__(kPbThreads, MAXW == 1 ? 6 : 4) k_emit_rows(CandArgs a, const float* __restrict__ vals,
                                                          int64_t nrows, BlockScratch b,
                                                          int64_t cap, const int* base_,
                                                          unsigned* status) {
  pdl_begin();
  const int64_t base = base_ ? *base_ : 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) set_count(a, base + b.counters[2], status);
  const int lane = threadIdx.x & 31;
  const int64_t r = ((int64_t)blockIdx.x * kPbThreads + threadIdx.x) >> 5;
  if (r >= nrows || (WIDE && b.rowcnt[r] == 0)) return;
  const int w = MAXW == 1 ? 1 : a.w;
  const int g = (int)(r / a.Ty), ty = (int)(r - (int64_t)g * a.Ty);
  const int t0 = ty * a.Tx;
  const uint32_t* row = b.pbits + (size_t)r * b.words;
  const uint8_t* ag = a.arg ? a.arg + (size_t)g * a.stride + t0 : nullptr;
  const float* vg = vals + (size_t)g * a.stride + t0;
  const int64_t roff = row_offset(b, r);
  auto arg_of = [&](int t) -> int { return MAXW == 1 ? 0 : ag[t]; };
  // place of the next peak of each in-tile row over the words so far
  int next[MAXW];
#pragma unroll
  for (int d = 0; d < MAXW; ++d) next[d] = 0;
  if (WIDE && MAXW > 1) {
    int cnt[MAXW];
#pragma unroll
    for (int d = 0; d < MAXW; ++d) cnt[d] = 0;
    for (int wx = lane; wx < b.words; wx += 32)
      for (uint32_t q = row[wx]; q; q &= q - 1) {
        const int dy = arg_of(wx * 32 + __ffs(q) - 1) / w;
#pragma unroll
        for (int d = 0; d < MAXW; ++d) cnt[d] += dy == d;
      }
    int run = 0;
#pragma unroll
    for (int d = 0; d < MAXW; ++d) {
      next[d] = run;
      int c = cnt[d];
#pragma unroll
      for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
      run += c;
    }
  }
  for (int w0 = 0; w0 < b.words; w0 += 32) {
    const int wx = w0 + lane;
    const uint32_t word = wx < b.words ? row[wx] : 0u;
    int idx[kRowsBatch], tx[kRowsBatch];
    float v[kRowsBatch];
    uint32_t m = word;
#pragma unroll
    for (int k = 0; k < kRowsBatch; ++k) {
      idx[k] = -1;
      tx[k] = 0;
      v[k] = 0.f;
      if (m) {
        tx[k] = wx * 32 + __ffs(m) - 1;
        m &= m - 1;
        idx[k] = arg_of(tx[k]);
        v[k] = vg[tx[k]];
      }
    }
    const uint32_t rest = m;
    int mine[MAXW];
#pragma unroll
    for (int d = 0; d < MAXW; ++d) mine[d] = 0;
#pragma unroll
    for (int k = 0; k < kRowsBatch; ++k) {
      const int dy = idx[k] >= 0 ? idx[k] / w : -1;
#pragma unroll
      for (int d = 0; d < MAXW; ++d) mine[d] += dy == d;
    }
    for (uint32_t q = rest; q; q &= q - 1) {
      const int dy = arg_of(wx * 32 + __ffs(q) - 1) / w;
#pragma unroll
      for (int d = 0; d < MAXW; ++d) mine[d] += dy == d;
    }
    // place of this lane's first peak of each in-tile row: the row's peaks in
    // lower in-tile rows, the earlier words' and the lower lanes' of that row
    int excl[MAXW];
    int run = 0;
#pragma unroll
    for (int d = 0; d < MAXW; ++d) {
      excl[d] = 0;
      int incl = mine[d];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      const int tot = __shfl_sync(0xffffffffu, incl, 31);
      if (WIDE) {
        excl[d] = next[d] + incl - mine[d];
        next[d] += tot;
      } else {
        excl[d] = run + incl - mine[d];
        run += tot;
      }
    }
    auto put = [&](int t, int i, float val) {
      const int dy = i / w, dx = i - dy * w;
      int j = 0;
#pragma unroll
      for (int d = 0; d < MAXW; ++d)
        if (dy == d) j = excl[d]++;
      const int64_t n = roff + j;   // place among the image candidates
      const int64_t pos = base + n;
      if (n < cap && pos < a.cap)
        a.out[pos] = image_candidate(a, SelItem{g, t0 + t, val}, t, ty, w, dx, dy);
    };
#pragma unroll
    for (int k = 0; k < kRowsBatch; ++k)
      if (idx[k] >= 0) put(tx[k], idx[k], v[k]);
    for (uint32_t q = rest; q; q &= q - 1) {
      const int t = wx * 32 + __ffs(q) - 1;
      put(t, arg_of(t), vg[t]);
    }
    if (!WIDE) break;
  }
}

__global__ void k_add_count(int* total, const int* part) {
  *total += *part;
}

// Copies the first min(*n, cap) candidates to mapped host memory, so only the
// candidates that exist cross the host link.
__global__ void k_export(const fitrig_candidate* __restrict__ src, const int* n,
                         fitrig_candidate* dst, int cap) {
  const int m = min(*n, cap);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x)
    dst[i] = src[i];
}

cudaError_t launch_export_candidates(const fitrig_candidate* src, const int* n,
                                     fitrig_candidate* dst, int cap, cudaStream_t st) {
  k_export<<<64, 256, 0, st>>>(src, n, dst, cap);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_emit_peaks(const CandArgs& a, const SelItem* peaks, const int* npeak,
                              const int* base, fitrig_candidate* tmp, unsigned* status,
                              cudaStream_t st) {
  cudaError_t e;
  int launches = 1;
  if (a.branch == FITRIG_BRANCH_FREQ) {
    e = launch_pdl(k_emit_freq, dim3(152 * 4), dim3(256), 0, st, a, peaks, npeak,
                   (const int*)nullptr, status);
  } else if (a.arg) {
    e = launch_pdl(k_group_sort<true>, dim3(152 * 4), dim3(kGroupWarps * 32), 0, st, a, npeak,
                   (const fitrig_candidate*)tmp, peaks, (const int*)nullptr, base, status);
  } else {
    e = launch_pdl(k_emit_image, dim3(152 * 4), dim3(256), 0, st, a, peaks, npeak,
                   (const int*)nullptr, tmp);
    if (e == cudaSuccess)
      e = launch_pdl(k_group_sort<false>, dim3(152 * 4), dim3(kGroupWarps * 32), 0, st, a, npeak,
                     (const fitrig_candidate*)tmp, peaks, (const int*)nullptr, base, status);
    launches = 2;
  }
  count_launches(launches);
  return e;
}

cudaError_t launch_emit_rows(const CandArgs& a, const float* vals, int groups, const BlockScratch& b,
                             int64_t cap, const int* base, unsigned* status, cudaStream_t st) {
  if ((!a.arg && a.w != 1) || a.w < 1 || a.w > kRowsMaxW ||
      ((int64_t)groups * a.Ty + kRowsPerCta - 1) / kRowsPerCta > b.nblk)
    return cudaErrorInvalidValue;
  const int64_t nrows = (int64_t)groups * a.Ty;
  const dim3 grid((unsigned)((nrows * 32 + kPbThreads - 1) / kPbThreads));
  cudaError_t e;
  if (a.w == 1)
    e = launch_pdl(k_emit_rows<true, 1>, grid, dim3(kPbThreads), 0, st, a, vals, nrows, b, cap, base,
                   status);
  else if (b.words > 32)
    e = launch_pdl(k_emit_rows<true, kRowsMaxW>, grid, dim3(kPbThreads), 0, st, a, vals, nrows, b,
                   cap, base, status);
  else
    e = launch_pdl(k_emit_rows<false, kRowsMaxW>, grid, dim3(kPbThreads), 0, st, a, vals, nrows, b,
                   cap, base, status);
  count_launches(1);
  return e;
}

cudaError_t launch_emit_candidates(const CandArgs& a, const SelectScratch& s, int* base,
                                   fitrig_candidate* tmp, unsigned* status, cudaStream_t st) {
  // ordered list of component peaks
  k_peak_count<<<s.nblk, kSelThreads, 0, st>>>(s.nsel, s.parent, s.peak, s.nblk, s.blkcnt);
  k_scan_blocks<<<1, 1024, 0, st>>>(s.nblk, s.blkcnt, s.blkoff, s.npeak, s.capacity, status,
                                    nullptr);
  k_peak_write<<<s.nblk, kSelThreads, 0, st>>>(s.nsel, s.parent, s.peak, s.nblk, s.blkoff,
                                               s.plist);
  if (a.branch == FITRIG_BRANCH_FREQ) {
    k_emit_freq<<<152 * 4, 256, 0, st>>>(a, s.items, s.npeak, s.plist, nullptr);
    count_launches(4);
  } else {
    if (a.arg) {
      k_group_sort<true><<<152 * 4, kGroupWarps * 32, 0, st>>>(a, s.npeak, tmp, s.items, s.plist,
                                                               base, nullptr);
      count_launches(4);
    } else {
      k_emit_image<<<152 * 4, 256, 0, st>>>(a, s.items, s.npeak, s.plist, tmp);
      k_group_sort<false><<<152 * 4, kGroupWarps * 32, 0, st>>>(a, s.npeak, tmp, s.items,
                                                                s.plist, base, nullptr);
      count_launches(5);
    }
  }
  // running total of candidates
  k_add_count<<<1, 1, 0, st>>>(a.nout, s.npeak);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace fitrig
