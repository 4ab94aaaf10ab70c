// Image-frequency branch (Sec. 2.4.2): per tile, the series of the tile
// statistic over the n = L - 2 units, its mean removed (the DC term of Eq.
// eta), an unnormalised DFT of exact length n, and
//   eta_t = max_{k=1..floor(n/2)} |X_k|   (h = maximum spectral magnitude)
// with the arg-max bin (smallest k on ties), or, with hmax > 1, h = the
// incoherent harmonic sum
//   eta_t = max_{m = 1, 2, 4, .., hmax} max_{k: m k <= floor(n/2)}
//           (|X_k| + |X_2k| + .. + |X_mk|) / sqrt(m)
// with the fundamental k (ties: smaller m, then smaller k).  Sec. 2.4.2 names
// harmonic summing as a choice of h without a formula; this is the classic
// incoherent form.
//
// The series used is v_t(s) = mean(Delta) max(Delta) mean(r), i.e. the tLISI
// complement times M^2 with one M for the stack, so |X_k| of tLISI is |X_k|/M^2
// and the z-score of eta is unchanged.
//
// One thread per tile; the series is staged in shared memory (coalesced over
// tiles).  Real input: pairs y_s, y_{n-s} are folded into e_s = y_s + y_{n-s}
// and o_s = y_s - y_{n-s}, so that Re X_k = y_0 + sum e_s cos + [n even]
// (-1)^k y_{n/2} and Im X_k = -sum o_s sin, halving the multiply-adds.  The
// twiddles cos/sin(2 pi k s / n) come from a table filled on the host in FP64.
#include <algorithm>
#include <cmath>

#include "internal.cuh"

namespace fitrig {

constexpr int kDftThreads = 128;

// The harmonic sum over one tile's magnitudes |X_k| = mag[(k - 1) * stride],
// k = 1..K, in the order (m ascending, k ascending) so that ties keep the
// smaller m, then the smaller k.
__device__ __forceinline__ void harmonic_best(const float* mag, int stride, int K, int hmax,
                                              float& best, int& bk) {
  best = -1.f;
  bk = 1;
  for (int m = 1; m <= hmax && m <= K; m <<= 1) {
    const float inv = 1.f / sqrtf((float)m);
    for (int k = 1; k * m <= K; ++k) {
      float acc = 0.f;
      for (int j = 1; j <= m; ++j) acc += mag[(j * k - 1) * stride];
      acc *= inv;
      if (acc > best) {
        best = acc;
        bk = k;
      }
    }
  }
}

__global__ void __launch_bounds__(kDftThreads) k_dft(const float* __restrict__ vp, int n,
                                                     int64_t T, int64_t vs,
                                                     const float2* __restrict__ tw,
                                                     const float* __restrict__ wts,
                                                     float* eta, int* bin) {
  extern __shared__ float ys[];   // [n][kDftThreads]
  const int tid = threadIdx.x;
  const int64_t t = (int64_t)blockIdx.x * kDftThreads + tid;
  const bool live = t < T;
  bool ok = live;
  float s = 0.f, comp = 0.f;
  for (int q = 0; q < n; ++q) {
    const float v = live ? (wts ? vp[(size_t)q * vs + t] * wts[q] : vp[(size_t)q * vs + t]) : 0.f;
    ok = ok && isfinite(v);
    ys[q * kDftThreads + tid] = v;
    const float y = v - comp;
    const float u = s + y;
    comp = (u - s) - y;
    s = u;
  }
  if (!live) return;
  if (!ok) {
    eta[t] = NAN;
    bin[t] = -1;
    return;
  }
  const float mean = s / (float)n;
  const int H = (n - 1) / 2;        // folded pairs s = 1..H
  const bool even = (n & 1) == 0;
  const float y0 = ys[tid] - mean;
  const float ymid = even ? ys[(n / 2) * kDftThreads + tid] - mean : 0.f;
  for (int q = 1; q <= H; ++q) {
    const float a = ys[q * kDftThreads + tid] - mean;
    const float b = ys[(n - q) * kDftThreads + tid] - mean;
    ys[q * kDftThreads + tid] = a + b;         // e_q
    ys[(n - q) * kDftThreads + tid] = a - b;   // o_q
  }
  const int K = n / 2;
  float best = -1.f;
  int bk = 1;
  for (int k = 1; k <= K; ++k) {
    float re = y0 + ((even && (k & 1)) ? -ymid : ymid);
    float im = 0.f;
    const float2* twk = tw + (size_t)(k - 1) * H;
    for (int q = 1; q <= H; ++q) {
      const float2 cs = twk[q - 1];
      re = fmaf(ys[q * kDftThreads + tid], cs.x, re);
      im = fmaf(ys[(n - q) * kDftThreads + tid], cs.y, im);
    }
    const float m2 = re * re + im * im;
    if (m2 > best) {
      best = m2;
      bk = k;
    }
  }
  eta[t] = sqrtf(best);
  bin[t] = bk;
}

// Short series (n <= 2*KMAX + 1): the pair loop runs outermost and the
// accumulators of every bin stay in registers; each twiddle is a shared-memory
// broadcast, so one load feeds two multiply-adds.
template <int KMAX, bool HARM>
__global__ void __launch_bounds__(kDftThreads) k_dft_short(const float* __restrict__ vp, int n,
                                                           int64_t T, int64_t vs,
                                                           const float2* __restrict__ tw,
                                                           const float* __restrict__ wts,
                                                           int hmax, float* eta, int* bin) {
  extern __shared__ float2 tws[];   // [H][K] twiddles, pair-major, then [n][threads] series
  const int H = (n - 1) / 2, K = n / 2;
  float* ys = reinterpret_cast<float*>(tws + H * K);
  for (int i = threadIdx.x; i < H * K; i += blockDim.x) {
    const int q = i / K, k = i - (i / K) * K;
    tws[i] = tw[(size_t)k * H + q];
  }
  __syncthreads();
  // (a CTA takes many groups of tiles: its twiddle table costs more than a group)
  for (int64_t t = (int64_t)blockIdx.x * kDftThreads + threadIdx.x; t < T;
       t += (int64_t)gridDim.x * kDftThreads) {
    float s = 0.f, comp = 0.f;
    bool ok = true;
    float* my = ys + threadIdx.x;
    for (int q = 0; q < n; ++q) {
      const float v = wts ? vp[(size_t)q * vs + t] * wts[q] : vp[(size_t)q * vs + t];
      ok = ok && isfinite(v);
      my[q * kDftThreads] = v;
      const float y = v - comp;
      const float u = s + y;
      comp = (u - s) - y;
      s = u;
    }
    if (!ok) {
      eta[t] = NAN;
      bin[t] = -1;
      continue;
    }
    const float mean = s / (float)n;
    const bool even = (n & 1) == 0;
    const float y0 = my[0] - mean;
    const float ymid = even ? my[(n / 2) * kDftThreads] - mean : 0.f;
    float re[KMAX], im[KMAX];
#pragma unroll
    for (int k = 0; k < KMAX; ++k) {
      re[k] = y0 + ((even && ((k + 1) & 1)) ? -ymid : ymid);
      im[k] = 0.f;
    }
    for (int q = 1; q <= H; ++q) {
      const float a = my[q * kDftThreads] - mean;
      const float b = my[(n - q) * kDftThreads] - mean;
      const float e = a + b, o = a - b;
      const float2* row = tws + (q - 1) * K;
#pragma unroll
      for (int k = 0; k < KMAX; ++k) {
        if (k < K) {
          const float2 cs = row[k];
          re[k] = fmaf(e, cs.x, re[k]);
          im[k] = fmaf(o, cs.y, im[k]);
        }
      }
    }
    float best = -1.f;
    int bk = 1;
    if constexpr (HARM) {
      // the series is spent: its column holds the magnitudes for the harmonic sum
#pragma unroll
      for (int k = 0; k < KMAX; ++k)
        if (k < K) my[k * kDftThreads] = sqrtf(re[k] * re[k] + im[k] * im[k]);
      harmonic_best(my, kDftThreads, K, hmax, best, bk);
      eta[t] = best;
      bin[t] = bk;
    } else {
#pragma unroll
      for (int k = 0; k < KMAX; ++k) {
        if (k < K) {
          const float m2 = re[k] * re[k] + im[k] * im[k];
          if (m2 > best) {
            best = m2;
            bk = k + 1;
          }
        }
      }
      eta[t] = sqrtf(best);
      bin[t] = bk;
    }
  }
}

// Even n = 2m (n <= 66): the transform splits into the two length-m DFTs of
// the even- and odd-indexed samples, X_k = E_k + W^k O_k with W = e^(-2 pi i/n)
// (a radix-2 decimation in time).  E and O are DFTs of real series, so only
// their bins k = 0..floor(m/2) are formed (the others are complex conjugates,
// E_(m-k) = conj(E_k)), each from folded pairs of samples; one shared-memory
// twiddle then feeds four multiply-adds (both halves, real and imaginary
// parts), half the work of the direct form.  X_m = E_0 - O_0 (Nyquist).
// Twiddles come from the host's FP64 table of 2 pi q / n (its first row) by
// symmetry.
template <int KH, bool HARM>
__global__ void __launch_bounds__(kDftThreads) k_dft_even(const float* __restrict__ vp, int n,
                                                          int64_t T, int64_t vs,
                                                          const float2* __restrict__ tw,
                                                          const float* __restrict__ wts,
                                                          int hmax, float* eta, int* bin) {
  extern __shared__ float2 sm2[];
  const int m = n / 2, Hm = (m - 1) / 2, K = m / 2, H = (n - 1) / 2;
  float2* th = sm2;                                 // [Hm][K]: 2 pi j k / m, j,k >= 1
  float2* tk = th + (Hm > 0 ? Hm * K : 0);          // [m]: 2 pi k / n
  float* ys = reinterpret_cast<float*>(tk + m);     // [n][kDftThreads]
  // (cos, sin) of 2 pi a / n from the table row q = 1..H and symmetry
  auto ang = [&](int a) -> float2 {
    if (a == 0) return make_float2(1.f, 0.f);
    if (2 * a == n) return make_float2(-1.f, 0.f);
    if (a <= H) return tw[a - 1];
    const float2 c = tw[n - a - 1];
    return make_float2(c.x, -c.y);
  };
  for (int i = threadIdx.x; i < Hm * K; i += blockDim.x) {
    const int j = i / K + 1, k = i - (i / K) * K + 1;
    th[i] = ang((2 * j * k) % n);
  }
  for (int k = threadIdx.x; k < m; k += blockDim.x) tk[k] = ang(k);
  __syncthreads();
  float* my = ys + threadIdx.x;
  // (a CTA takes many groups of tiles: its twiddle tables cost more than a group
  // of short series; a thread's column of ys is its own, so no barrier is needed)
  for (int64_t t = (int64_t)blockIdx.x * kDftThreads + threadIdx.x; t < T;
       t += (int64_t)gridDim.x * kDftThreads) {
    // the series arrives by asynchronous global -> shared copies, all n of a
    // thread in flight at once (coalesced over the CTA's tiles)
    for (int q = 0; q < n; ++q) {
      const uint32_t dst = smem_u32(my + q * kDftThreads);
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst),
                   "l"(vp + (size_t)q * vs + t)
                   : "memory");
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    float sum = 0.f;
    bool ok = true;
    for (int q = 0; q < n; ++q) {
      float v = my[q * kDftThreads];
      if (wts) {
        v *= wts[q];
        my[q * kDftThreads] = v;
      }
      ok = ok && isfinite(v);
      sum += v;
    }
    if (!ok) {
      eta[t] = NAN;
      bin[t] = -1;
      continue;
    }
    const float mean = sum / (float)n;
    auto ye = [&](int j) { return my[(2 * j) * kDftThreads] - mean; };       // y_(2j)
    auto yo = [&](int j) { return my[(2 * j + 1) * kDftThreads] - mean; };   // y_(2j+1)
    const float ye0 = ye(0), yo0 = yo(0);
    const bool meven = (m & 1) == 0;
    const float yem = meven ? ye(m / 2) : 0.f, yom = meven ? yo(m / 2) : 0.f;
    float E0 = ye0 + yem, O0 = yo0 + yom;   // bin 0 of each half
    float er[KH], es[KH], orr[KH], os[KH];  // bins 1..K: real parts, and the sums of
                                            // the odd folds times sin (imag = -that)
#pragma unroll
    for (int k = 0; k < KH; ++k) {
      const float sg = ((k + 1) & 1) ? -1.f : 1.f;   // (-1)^(k+1)
      er[k] = ye0 + sg * yem;
      orr[k] = yo0 + sg * yom;
      es[k] = 0.f;
      os[k] = 0.f;
    }
    for (int j = 1; j <= Hm; ++j) {
      const float a = ye(j), b = ye(m - j), c = yo(j), d = yo(m - j);
      const float ee = a + b, eo = a - b, oe = c + d, oo = c - d;
      E0 += ee;
      O0 += oe;
      const float2* row = th + (j - 1) * K;
#pragma unroll
      for (int k = 0; k < KH; ++k) {
        if (k < K) {
          const float2 w = row[k];
          er[k] = fmaf(ee, w.x, er[k]);
          es[k] = fmaf(eo, w.y, es[k]);
          orr[k] = fmaf(oe, w.x, orr[k]);
          os[k] = fmaf(oo, w.y, os[k]);
        }
      }
    }
    // X_k = E_k + W^k O_k, W^k = (c, -s):  Re = Er + c Or + s Oi,  Im = Ei + c Oi - s Or
    float best = -1.f;
    int bk = 1;
    // with harmonic summing the spent series column collects |X_k| at row k - 1
    constexpr bool harm = HARM;
    auto take = [&](int k, float Er, float Ei, float Or, float Oi) {
      const float2 w = tk[k];
      const float re = Er + w.x * Or + w.y * Oi;
      const float im = Ei + w.x * Oi - w.y * Or;
      const float m2 = re * re + im * im;
      if constexpr (harm) my[(k - 1) * kDftThreads] = sqrtf(m2);
      if (m2 > best || (m2 == best && k < bk)) {
        best = m2;
        bk = k;
      }
    };
#pragma unroll
    for (int k = 0; k < KH; ++k) {
      if (k < K) {
        take(k + 1, er[k], -es[k], orr[k], -os[k]);                    // bin k+1
        if (m - (k + 1) > K) take(m - (k + 1), er[k], es[k], orr[k], os[k]);   // its mirror
      }
    }
    {
      const float x = E0 - O0;   // bin m
      const float m2 = x * x;
      if constexpr (HARM) my[(m - 1) * kDftThreads] = fabsf(x);
      if (m2 > best || (m2 == best && m < bk)) {
        best = m2;
        bk = m;
      }
    }
    if constexpr (HARM) {
      harmonic_best(my, kDftThreads, m, hmax, best, bk);
      eta[t] = best;
      bin[t] = bk;
    } else {
      eta[t] = sqrtf(best);
      bin[t] = bk;
    }
  }
}

// Long series (n up to kLongMaxN) and harmonic sums beyond the short kernels:
// one warp per tile, a CTA stages the series of kLongWarps consecutive tiles
// (each cube row a 32-byte segment) and transposes them into shared memory.
// Lane l forms bins k = l + 1 + 32 j, kLongB at a time, over the folded pairs
// (e_q, o_q) read as broadcasts; the phasor (cos, sin)(2 pi k q / n) advances by
// one complex multiply per step and is re-seeded from the host's FP64 table
// every kSeed steps, so its rounding error stays that of a few dozen
// multiplies.  The magnitudes go to shared memory for the maximum or the
// harmonic sum, which the warp then reduces.
constexpr int kLongWarps = 8;
constexpr int kLongMaxN = 4096;
constexpr int kLongB = 4;
constexpr int kSeed = 32;

// Warp reduction of one tile's squared magnitudes mk[k] = |X_k|^2, k = 1..K:
// the maximum magnitude (hmax = 1) or the largest harmonic sum, with its bin
// (ties: smaller m, then smaller k).  Lane 0 writes eta and the bin.
__device__ __forceinline__ void warp_spectrum_best(const float* mk, int K, int hmax, int lane,
                                                   float* eta, int* bin) {
  float best = -1.f;
  int bk = 1, bm = 1;
  if (hmax <= 1) {
    for (int k = 1 + lane; k <= K; k += 32) {
      const float v = mk[k];
      if (v > best) {
        best = v;
        bk = k;
      }
    }
  } else {
    for (int m = 1; m <= hmax && m <= K; m <<= 1) {
      const float inv = 1.f / sqrtf((float)m);
      for (int k = 1 + lane; k * m <= K; k += 32) {
        float acc = 0.f;
        for (int j = 1; j <= m; ++j) acc += sqrtf(mk[j * k]);
        acc *= inv;
        if (acc > best) {
          best = acc;
          bk = k;
          bm = m;
        }
      }
    }
  }
  // warp arg-max: larger value, then smaller m, then smaller k
#pragma unroll
  for (int off = 16; off; off >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, best, off);
    const int okk = __shfl_xor_sync(0xffffffffu, bk, off);
    const int om = __shfl_xor_sync(0xffffffffu, bm, off);
    if (ov > best || (ov == best && (om < bm || (om == bm && okk < bk)))) {
      best = ov;
      bk = okk;
      bm = om;
    }
  }
  if (lane == 0) {
    *eta = hmax <= 1 ? sqrtf(best) : best;
    *bin = bk;
  }
}

__host__ __device__ constexpr int long_ldy(int n) { return (n + 27) / 32 * 32 + 4; }

__global__ void __launch_bounds__(kLongWarps * 32) k_dft_long(const float* __restrict__ vp, int n,
                                                              int64_t T, int64_t vs,
                                                              const float2* __restrict__ tw,
                                                              const float* __restrict__ wts,
                                                              int hmax, float* eta, int* bin) {
  extern __shared__ float lsm[];
  const int K = n / 2, H = (n - 1) / 2, ldy = long_ldy(n);
  float* ys = lsm;                                 // [kLongWarps][ldy]
  float* mg = lsm + kLongWarps * ldy;              // [kLongWarps][K + 1]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t t0 = (int64_t)blockIdx.x * kLongWarps;
  for (int i = threadIdx.x; i < n * kLongWarps; i += blockDim.x) {
    const int q = i / kLongWarps, c = i - q * kLongWarps;
    const int64_t t = t0 + c;
    float v = t < T ? vp[(size_t)q * vs + t] : 0.f;
    if (wts) v *= wts[q];
    ys[c * ldy + q] = v;
  }
  __syncthreads();
  const int64_t t = t0 + warp;
  if (t >= T) return;
  float* y = ys + warp * ldy;
  float sum = 0.f;
  bool ok = true;
  for (int q = lane; q < n; q += 32) {
    const float v = y[q];
    ok = ok && isfinite(v);
    sum += v;
  }
  ok = __all_sync(0xffffffffu, ok);
#pragma unroll
  for (int off = 16; off; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
  if (!ok) {
    if (lane == 0) {
      eta[t] = NAN;
      bin[t] = -1;
    }
    return;
  }
  const float mean = sum / (float)n;
  __syncwarp();
  for (int q = 1 + lane; q <= H; q += 32) {
    const float a = y[q] - mean, b = y[n - q] - mean;
    y[q] = a + b;       // e_q
    y[n - q] = a - b;   // o_q
  }
  __syncwarp();
  const bool even = (n & 1) == 0;
  const float y0 = y[0] - mean;
  const float ymid = even ? y[n / 2] - mean : 0.f;
  // (cos, sin) of 2 pi a / n, 0 <= a < n, from the table's first row and symmetry
  auto ang = [&](int a) -> float2 {
    if (a == 0) return make_float2(1.f, 0.f);
    if (2 * a == n) return make_float2(-1.f, 0.f);
    if (a <= H) return tw[a - 1];
    const float2 c = tw[n - a - 1];
    return make_float2(c.x, -c.y);
  };
  float* mk = mg + warp * (K + 1);   // |X_k|^2 at mk[k]
  for (int kb = 1; kb <= K; kb += 32 * kLongB) {
    int kk[kLongB];
    float re[kLongB], im[kLongB], c[kLongB], sn[kLongB], wc[kLongB], ws[kLongB];
#pragma unroll
    for (int b = 0; b < kLongB; ++b) {
      kk[b] = min(kb + lane + 32 * b, K);
      re[b] = y0 + ((even && (kk[b] & 1)) ? -ymid : ymid);
      im[b] = 0.f;
      const float2 w = ang(kk[b]);
      wc[b] = w.x;
      ws[b] = w.y;
    }
    for (int q0 = 1; q0 <= H; q0 += kSeed) {
#pragma unroll
      for (int b = 0; b < kLongB; ++b) {
        const float2 e = ang((int)(((int64_t)kk[b] * q0) % n));
        c[b] = e.x;
        sn[b] = e.y;
      }
      const int qe = min(H, q0 + kSeed - 1);
      for (int q = q0; q <= qe; ++q) {
        const float e = y[q], o = y[n - q];
#pragma unroll
        for (int b = 0; b < kLongB; ++b) {
          re[b] = fmaf(e, c[b], re[b]);
          im[b] = fmaf(o, sn[b], im[b]);
          const float cn = fmaf(c[b], wc[b], -sn[b] * ws[b]);
          sn[b] = fmaf(sn[b], wc[b], c[b] * ws[b]);
          c[b] = cn;
        }
      }
    }
#pragma unroll
    for (int b = 0; b < kLongB; ++b)
      if (kb + lane + 32 * b <= K) mk[kk[b]] = re[b] * re[b] + im[b] * im[b];
  }
  __syncwarp();
  warp_spectrum_best(mk, K, hmax, lane, eta + t, bin + t);
}

// Composite lengths of the long path: one step of Cooley and Tukey's splitting
// (Math. Comp. 19, 1965) with n = P M, X_q = sum_p W_n^(p q) S_p[q mod M], S_p
// the length-M DFT of y_p, y_(p+P), ..  The sub-series are real, so S_p[M - k]
// is the conjugate of S_p[k] and only k <= M/2 is summed, from folded pairs as
// in the direct kernels; a lane holds two bins of kMixP sub-series, so one
// table entry feeds 4 kMixP multiply-adds and one pair of broadcast loads four.
// n = 1498 = 14 x 107: about 9 k instructions per tile and warp against the
// direct kernel's 116 k; every twiddle is a table entry (the direct kernel
// advances a phasor), so the rounding error is smaller too.  4096 series of
// 1498 points, harmonic sums to 8: 988 -> 138 us; 16,384 of 300 / 1001 / 4095:
// 208 / 1298 / 38383 -> 70 / 218 / 4121 us; 998 = 2 x 499: 1300 -> 1056.  Bound by
// the shared-memory loads of the pairs and table entries.  One warp per tile;
// the table (full circle) and the WARPS tiles' series and sub-spectra are in
// shared memory.
constexpr int kMixP = 8;
constexpr int kMixK = 2;

__host__ __device__ constexpr int mixed_lds(int n, int P) { return P * (n / P / 2 + 1); }

template <int WARPS>
__global__ void __launch_bounds__(WARPS * 32) k_dft_mixed(const float* __restrict__ vp, int n, int P,
                                                          int64_t T, int64_t vs,
                                                          const float2* __restrict__ tw,
                                                          const float* __restrict__ wts, int hmax,
                                                          float* eta, int* bin) {
  extern __shared__ float2 msm[];
  const int K = n / 2, H = (n - 1) / 2, M = n / P, MB = M / 2 + 1, HM = (M - 1) / 2;
  const int ldy = long_ldy(n), lds = mixed_lds(n, P);
  float2* tb = msm;                                           // [n] (cos, sin)(2 pi a / n)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* S = tb + n + warp * lds;                            // [P][MB]
  float* ys = reinterpret_cast<float*>(tb + n + WARPS * lds);   // [WARPS][ldy]
  const int64_t t0 = (int64_t)blockIdx.x * WARPS;
  for (int i = threadIdx.x; i < n * WARPS; i += WARPS * 32) {
    const int q = i / WARPS, c = i - q * WARPS;
    const int64_t t = t0 + c;
    float v = t < T ? vp[(size_t)q * vs + t] : 0.f;
    if (wts) v *= wts[q];
    ys[c * ldy + q] = v;
  }
  for (int a = threadIdx.x; a < n; a += WARPS * 32) {
    float2 e;
    if (a == 0) e = make_float2(1.f, 0.f);
    else if (2 * a == n) e = make_float2(-1.f, 0.f);
    else if (a <= H) e = tw[a - 1];
    else {
      e = tw[n - a - 1];
      e.y = -e.y;
    }
    tb[a] = e;
  }
  __syncthreads();
  const int64_t t = t0 + warp;
  if (t >= T) return;
  float* y = ys + warp * ldy;
  float sum = 0.f;
  bool ok = true;
  for (int q = lane; q < n; q += 32) {
    const float v = y[q];
    ok = ok && isfinite(v);
    sum += v;
  }
  ok = __all_sync(0xffffffffu, ok);
#pragma unroll
  for (int off = 16; off; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
  if (!ok) {
    if (lane == 0) {
      eta[t] = NAN;
      bin[t] = -1;
    }
    return;
  }
  const float mean = sum / (float)n;
  const bool even = (M & 1) == 0;
  __syncwarp();
  // the folded pairs of every sub-series: y_(p + P j), j = 1..HM, lie at i + P
  for (int i = lane; i < P * HM; i += 32) {
    const int p = i % P, hi = p + P * (M - 1 - i / P);
    const float a = y[i + P] - mean, b = y[hi] - mean;
    y[i + P] = a + b;   // e
    y[hi] = a - b;      // o
  }
  for (int p = lane; p < P; p += 32) {
    y[p] -= mean;
    if (even) y[p + P * (M / 2)] -= mean;
  }
  __syncwarp();
  for (int kb = 0; kb < MB; kb += 32 * kMixK) {
    int kk[kMixK];
#pragma unroll
    for (int b = 0; b < kMixK; ++b) kk[b] = min(kb + lane + 32 * b, MB - 1);
    for (int p0 = 0; p0 < P; p0 += kMixP) {
      float re[kMixK][kMixP], im[kMixK][kMixP];
#pragma unroll
      for (int i = 0; i < kMixP; ++i) {
        const int p = min(p0 + i, P - 1);
        const float y0 = y[p], ym = even ? y[p + P * (M / 2)] : 0.f;
#pragma unroll
        for (int b = 0; b < kMixK; ++b) {
          re[b][i] = y0 + ((kk[b] & 1) ? -ym : ym);
          im[b][i] = 0.f;
        }
      }
      int a[kMixK];
#pragma unroll
      for (int b = 0; b < kMixK; ++b) a[b] = 0;
      const float* ye = y + p0;
      const float* yo = y + p0 + P * M;
      for (int j = 1; j <= HM; ++j) {
        ye += P;
        yo -= P;
        float2 c[kMixK];
#pragma unroll
        for (int b = 0; b < kMixK; ++b) {
          a[b] += kk[b];
          if (a[b] >= M) a[b] -= M;
          c[b] = tb[a[b] * P];
        }
#pragma unroll
        for (int i = 0; i < kMixP; ++i) {
          if (p0 + i >= P) break;   // (uniform)
          const float e = ye[i], o = yo[i];
#pragma unroll
          for (int b = 0; b < kMixK; ++b) {
            re[b][i] = fmaf(e, c[b].x, re[b][i]);
            im[b][i] = fmaf(o, c[b].y, im[b][i]);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < kMixP; ++i)
        if (p0 + i < P) {
#pragma unroll
          for (int b = 0; b < kMixK; ++b)
            if (kb + lane + 32 * b < MB) S[(p0 + i) * MB + kk[b]] = make_float2(re[b][i], -im[b][i]);
        }
    }
  }
  __syncwarp();
  float* mk = y;   // the series is spent: |X_q|^2 at mk[q]
  for (int q = 1 + lane; q <= K; q += 32) {
    int k = q % M;
    const bool mirror = k >= MB;
    if (mirror) k = M - k;
    const float sg = mirror ? -1.f : 1.f;   // conjugate of S_p[M - k]
    float2 x = S[k];
    x.y *= sg;
    int a = 0;
    for (int p = 1; p < P; ++p) {
      a += q;
      if (a >= n) a -= n;
      const float2 w = tb[a];
      float2 v = S[p * MB + k];
      v.y *= sg;
      x.x = fmaf(w.x, v.x, fmaf(w.y, v.y, x.x));
      x.y = fmaf(w.x, v.y, fmaf(-w.y, v.x, x.y));
    }
    mk[q] = x.x * x.x + x.y * x.y;
  }
  __syncwarp();
  warp_spectrum_best(mk, K, hmax, lane, eta + t, bin + t);
}

// The divisor P of n whose splitting costs least, in instructions per warp
// and tile, or 0 when the direct kernel (six multiply-adds and two loads per
// pair and four bins) costs less: primes, and twice a prime below about 70.
static int mixed_split(int n) {
  const int K = n / 2, H = (n - 1) / 2;
  int best = 0;
  int64_t cost = (int64_t)((K + 32 * kLongB - 1) / (32 * kLongB)) * H * (6 * kLongB + 2) * 4 / 5;
  for (int P = 2; P <= n / 3; ++P) {
    if (n % P) continue;
    const int M = n / P, MB = M / 2 + 1;
    const int64_t sub = (int64_t)((MB + 32 * kMixK - 1) / (32 * kMixK)) * (M / 2) *
                        ((P + kMixP - 1) / kMixP * 5 * kMixK + P * (2 + 2 * kMixK));
    const int64_t c = sub + (int64_t)((K + 31) / 32) * P * 10 + n / 2;
    if (c < cost) {
      cost = c;
      best = P;
    }
  }
  return best;
}

// Powers of two, kFftMinN <= n <= kLongMaxN: a radix FFT per tile instead of
// the O(n^2) direct sum.  One warp per tile; a CTA stages the series of
// TILES consecutive tiles by asynchronous global -> shared copies (each cube
// row a TILES x 4-byte segment).  The real series y_0..y_(n-1), mean removed,
// is read as the complex series z_j = y_(2j) + i y_(2j+1) of N = n/2 points
// (the staging buffer already holds it in that order), transformed by a
// Stockham autosort FFT (radix-8 passes, one radix-4 or radix-2 pass for the
// rest of log2 N) that alternates between the staging buffer and a second warp
// buffer, and the real spectrum is recovered as
//   X_k = (Z_k + conj Z_(N-k)) / 2 - (i/2) e^(-2 pi i k/n) (Z_k - conj Z_(N-k)),
//   X_(n/2) = Re Z_0 - Im Z_0,
// whose squared magnitudes feed the same maximum / harmonic-sum reduction as
// the direct kernels.  Every twiddle is an entry of the host's FP64 table of
// (cos, sin)(2 pi a / n), a = 0..n-1, rounded once to FP32.
// Bound by shared memory: what counts is the number of passes (three instead
// of five at n = 1024) and bank conflicts.  Both buffers leave one entry in
// nine unused, so that a radix-8 pass's stores, eight entries apart, meet
// none, and the tiles' buffers are shifted against each other for the loads.
// 16,384 series of 512 / 1024 / 2048 / 4096 points: 57 / 118 / 257 / 712 us with
// radix-4 passes and neither, 43 / 81 / 237 / 613 now.
constexpr int kFftMinN = 128;

__host__ __device__ constexpr bool fft_length(int n) {
  return n >= kFftMinN && n <= kLongMaxN && (n & (n - 1)) == 0;
}

__device__ __forceinline__ float2 cmul_conj(float2 a, float2 w) {   // a * conj(w)
  return make_float2(fmaf(a.x, w.x, a.y * w.y), fmaf(a.y, w.x, -a.x * w.y));
}

__host__ __device__ constexpr int fft_at(int i) { return i + (i >> 3); }   // place of entry i
__host__ __device__ constexpr int fft_buf(int N) { return N + N / 8; }
// Entries of a tile's two buffers, with a shift of 32 / tiles words between
// tiles: a load instruction writes 32 / tiles points of every tile of the CTA.
__host__ __device__ constexpr int fft_tile(int N, int tiles) { return 2 * fft_buf(N) + 16 / tiles; }

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 mul_mi(float2 a) { return make_float2(a.y, -a.x); }   // -i a

// Forward DFTs of R points in registers.
template <int R>
__device__ __forceinline__ void dft_r(float2 (&a)[R]) {
  if constexpr (R == 2) {
    const float2 t = a[0];
    a[0] = cadd(t, a[1]);
    a[1] = csub(t, a[1]);
  } else if constexpr (R == 4) {
    const float2 b0 = cadd(a[0], a[2]), b1 = csub(a[0], a[2]);
    const float2 b2 = cadd(a[1], a[3]), b3 = mul_mi(csub(a[1], a[3]));
    a[0] = cadd(b0, b2);
    a[1] = cadd(b1, b3);
    a[2] = csub(b0, b2);
    a[3] = csub(b1, b3);
  } else {
    static_assert(R == 8, "radix");
    float2 e[4] = {a[0], a[2], a[4], a[6]}, o[4] = {a[1], a[3], a[5], a[7]};
    dft_r<4>(e);
    dft_r<4>(o);
    constexpr float h = 0.70710678118654752f;   // W_8 = (1 - i) / sqrt 2
    o[1] = make_float2(h * (o[1].x + o[1].y), h * (o[1].y - o[1].x));
    o[2] = mul_mi(o[2]);
    o[3] = make_float2(h * (o[3].y - o[3].x), -h * (o[3].x + o[3].y));
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      a[k] = cadd(e[k], o[k]);
      a[k + 4] = csub(e[k], o[k]);
    }
  }
}

// One Stockham pass of radix R over the warp's N points (Ns points done).
template <int R, bool FIRST>
__device__ __forceinline__ void fft_pass(const float2* src, float2* dst, int N, int Ns, int n,
                                         float mean, const float2* __restrict__ fw, int lane) {
  const int Q = N / R, step = n / (R * Ns);
  for (int j = lane; j < Q; j += 32) {
    const int k = j & (Ns - 1);
    float2 a[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      a[r] = src[fft_at(j + r * Q)];
      if (FIRST) a[r] = make_float2(a[r].x - mean, a[r].y - mean);   // (all twiddles are 1)
      else if (r > 0) a[r] = cmul_conj(a[r], __ldg(fw + r * k * step));   // W_(R Ns)^(r k)
    }
    dft_r<R>(a);
    const int base = (j - k) * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) dst[fft_at(base + r * Ns)] = a[r];
  }
  __syncwarp();
}

template <int TILES>
__global__ void __launch_bounds__(TILES * 32) k_fft_pow2(const float* __restrict__ vp, int n,
                                                         int logN, int64_t T, int64_t vs,
                                                         const float2* __restrict__ fw,
                                                         const float* __restrict__ wts, int hmax,
                                                         float* eta, int* bin) {
  extern __shared__ float2 fsm[];
  const int N = n >> 1, NB = fft_buf(N);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t t0 = (int64_t)blockIdx.x * TILES;
  auto at = [](int q) { return 2 * fft_at(q >> 1) + (q & 1); };   // series point q as a float
  for (int i = threadIdx.x; i < n * TILES; i += TILES * 32) {
    const int q = i / TILES, c = i - q * TILES;
    float* dst = reinterpret_cast<float*>(fsm + (size_t)c * fft_tile(N, TILES)) + at(q);
    if (t0 + c < T) {
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)),
                   "l"(vp + (size_t)q * vs + t0 + c)
                   : "memory");
    } else {
      *dst = 0.f;
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  const int64_t t = t0 + warp;
  if (t >= T) return;
  float2* src = fsm + (size_t)warp * fft_tile(N, TILES);   // z_j = (y_2j, y_2j+1)
  float2* dst = src + NB;
  float* y = reinterpret_cast<float*>(src);
  float sum = 0.f;
  bool ok = true;
  for (int q = lane; q < n; q += 32) {
    float v = y[at(q)];
    if (wts) {
      v *= wts[q];
      y[at(q)] = v;
    }
    ok = ok && isfinite(v);
    sum += v;
  }
  ok = __all_sync(0xffffffffu, ok);
#pragma unroll
  for (int off = 16; off; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
  if (!ok) {
    if (lane == 0) {
      eta[t] = NAN;
      bin[t] = -1;
    }
    return;
  }
  const float mean = sum / (float)n;
  __syncwarp();
  auto swap = [&]() {
    float2* tmp = src;
    src = dst;
    dst = tmp;
  };
  fft_pass<8, true>(src, dst, N, 1, n, mean, fw, lane);   // N >= 64
  swap();
  int Ns = 8;
  for (int left = logN - 3; left > 0;) {
    if (left >= 3) {
      fft_pass<8, false>(src, dst, N, Ns, n, 0.f, fw, lane);
      Ns <<= 3;
      left -= 3;
    } else if (left == 2) {
      fft_pass<4, false>(src, dst, N, Ns, n, 0.f, fw, lane);
      Ns <<= 2;
      left = 0;
    } else {
      fft_pass<2, false>(src, dst, N, Ns, n, 0.f, fw, lane);
      Ns <<= 1;
      left = 0;
    }
    swap();
  }
  float* mk = reinterpret_cast<float*>(dst);   // |X_k|^2 at mk[k], k = 1..N
  for (int k = 1 + lane; k <= N; k += 32) {
    float m2;
    if (k == N) {
      const float2 z0 = src[0];
      const float x = z0.x - z0.y;
      m2 = x * x;
    } else {
      const float2 zk = src[fft_at(k)], zc = src[fft_at(N - k)];
      const float er = 0.5f * (zk.x + zc.x), ei = 0.5f * (zk.y - zc.y);
      const float orr = 0.5f * (zk.y + zc.y), oi = 0.5f * (zc.x - zk.x);
      const float2 w = __ldg(fw + k);   // (cos, sin)(2 pi k / n); forward uses conj
      const float xr = er + fmaf(w.x, orr, w.y * oi);
      const float xi = ei + fmaf(w.x, oi, -w.y * orr);
      m2 = xr * xr + xi * xi;
    }
    mk[k] = m2;
  }
  __syncwarp();
  warp_spectrum_best(mk, N, hmax, lane, eta + t, bin + t);
}

static int fft_tiles(int n) { return n <= 1024 ? 8 : 4; }

std::vector<float2> spectrum_twiddles(int n) {
  std::vector<float2> tw;
  if (fft_length(n)) {   // the full circle: (cos, sin)(2 pi a / n), a = 0..n-1
    tw.resize((size_t)n);
    for (int a = 0; a < n; ++a) {
      const double ang = 2.0 * M_PI * (double)a / (double)n;
      tw[(size_t)a] = make_float2((float)std::cos(ang), (float)std::sin(ang));
    }
    return tw;
  }
  // (cos, sin)(2 pi ((k q) mod n) / n) for k = 1..K, q = 1..H: [K][H] for the
  // direct kernels of series up to 256 points; longer series take only the
  // first row (k = 1), which is all the warp-per-tile kernel reads.
  const int H = (n - 1) / 2, K = n > 256 ? 1 : n / 2;
  tw.resize((size_t)std::max(1, K * H));
  for (int k = 1; k <= K; ++k)
    for (int q = 1; q <= H; ++q) {
      const double ang = 2.0 * M_PI * (double)(((int64_t)k * q) % n) / (double)n;
      tw[(size_t)(k - 1) * H + (q - 1)] = make_float2((float)std::cos(ang), (float)std::sin(ang));
    }
  return tw;
}

int spectrum_max_n() { return kLongMaxN; }

static cudaError_t launch_long(const float* vp, int n, int64_t T, int64_t vs,
                               const float2* tw_row, const float* wts, int hmax, float* eta,
                               int* bin, cudaStream_t st) {
  const int K = n / 2;
  const size_t sm = (size_t)kLongWarps * (long_ldy(n) + K + 1) * sizeof(float);
  const cudaError_t lim = allow_smem(k_dft_long, sm);
  if (lim != cudaSuccess) return lim;
  const int64_t lblocks = (T + kLongWarps - 1) / kLongWarps;
  k_dft_long<<<(unsigned)lblocks, kLongWarps * 32, sm, st>>>(vp, n, T, vs, tw_row, wts, hmax,
                                                             eta, bin);
  count_launches(1);
  return cudaGetLastError();
}

template <int WARPS>
static cudaError_t launch_mixed_t(const float* vp, int n, int P, int64_t T, int64_t vs,
                                  const float2* tw, const float* wts, int hmax, float* eta,
                                  int* bin, cudaStream_t st) {
  const size_t sm = sizeof(float2) * ((size_t)n + (size_t)WARPS * mixed_lds(n, P)) +
                    sizeof(float) * (size_t)WARPS * long_ldy(n);
  const cudaError_t lim = allow_smem(k_dft_mixed<WARPS>, sm);
  if (lim != cudaSuccess) return lim;
  const int64_t blocks = (T + WARPS - 1) / WARPS;
  k_dft_mixed<WARPS><<<(unsigned)blocks, WARPS * 32, sm, st>>>(vp, n, P, T, vs, tw, wts, hmax, eta,
                                                              bin);
  count_launches(1);
  return cudaGetLastError();
}

template <int TILES>
static cudaError_t launch_fft_t(const float* vp, int n, int64_t T, int64_t vs, const float2* fw,
                                const float* wts, int hmax, float* eta, int* bin,
                                cudaStream_t st) {
  const size_t sm = (size_t)TILES * fft_tile(n / 2, TILES) * sizeof(float2);
  const cudaError_t lim = allow_smem(k_fft_pow2<TILES>, sm);
  if (lim != cudaSuccess) return lim;
  int logN = 0;
  while ((2 << logN) < n) ++logN;   // N = n / 2 = 2^logN
  const int64_t blocks = (T + TILES - 1) / TILES;
  k_fft_pow2<TILES><<<(unsigned)blocks, TILES * 32, sm, st>>>(vp, n, logN, T, vs, fw, wts, hmax,
                                                             eta, bin);
  count_launches(1);
  return cudaGetLastError();
}

static cudaError_t launch_odd_length(const float* vp, int n, int64_t T, int64_t vs,
                                     const float2* twiddle, const float* wts, int hmax, float* eta,
                                     int* bin, bool direct, cudaStream_t st);

cudaError_t launch_spectrum_method(const float* vp, int n, int64_t T, int64_t vs,
                                   const float2* twiddle, const float* wts, int hmax, float* eta,
                                   int* bin, int method, cudaStream_t st) {
  if (n < 2 || n > kLongMaxN || hmax < 1) return cudaErrorInvalidValue;
  if (T == 0) return cudaSuccess;
  if (fft_length(n)) {
    if (method == kSpectrumDirect)   // the O(n^2) warp kernel on the same table
      return launch_long(vp, n, T, vs, twiddle + 1, wts, hmax, eta, bin, st);
    return fft_tiles(n) == 8 ? launch_fft_t<8>(vp, n, T, vs, twiddle, wts, hmax, eta, bin, st)
                             : launch_fft_t<4>(vp, n, T, vs, twiddle, wts, hmax, eta, bin, st);
  }
  if (method == kSpectrumRadix) return cudaErrorInvalidValue;
  return launch_odd_length(vp, n, T, vs, twiddle, wts, hmax, eta, bin, method == kSpectrumDirect, st);
}

cudaError_t launch_spectrum(const float* vp, int n, int64_t T, int64_t vs,
                            const float2* twiddle, const float* wts, int hmax, float* eta,
                            int* bin, cudaStream_t st) {
  return launch_spectrum_method(vp, n, T, vs, twiddle, wts, hmax, eta, bin, kSpectrumAuto, st);
}

// CTAs of the short kernels.  Up to 32 points: what shared memory (sm bytes
// each) lets be resident, at most 16 per SM, so that each walks several groups of
// tiles and builds its tables once (24.2 M series of 6 points 655 -> 529 us, and
// 250 with the bins' registers cut to the four there are); longer series
// hide the tables behind their own sums, and a CTA per group balances better
// (672,400 of 62 points: 77 us, 85 as a loop).
static unsigned short_grid(int n, int64_t blocks, size_t sm) {
  if (n > 32) return (unsigned)blocks;
  const int64_t per_sm = std::max<int64_t>(1, std::min<int64_t>(16, (int64_t)(227 * 1024 / (sm + 1024))));
  return (unsigned)std::min<int64_t>(blocks, 152 * per_sm);
}

// Every length that is not the radix kernel's; `direct`: without the splitting.
static cudaError_t launch_odd_length(const float* vp, int n, int64_t T, int64_t vs,
                                     const float2* twiddle, const float* wts, int hmax, float* eta,
                                     int* bin, bool direct, cudaStream_t st) {
  const int64_t blocks = (T + kDftThreads - 1) / kDftThreads;
  const int H = (n - 1) / 2, K = n / 2;
  const bool harm = hmax > 1;
  if ((n & 1) == 0 && n <= 66) {
    const int m = n / 2, Hm = (m - 1) / 2, Kh = m / 2;
    const size_t sm = (size_t)(Hm > 0 ? Hm * Kh : 0) * sizeof(float2) + (size_t)m * sizeof(float2) +
                      (size_t)n * kDftThreads * sizeof(float);
    auto kern = Kh <= 4 ? (harm ? k_dft_even<4, true> : k_dft_even<4, false>)
                        : (harm ? k_dft_even<16, true> : k_dft_even<16, false>);
    kern<<<short_grid(n, blocks, sm), kDftThreads, sm, st>>>(vp, n, T, vs, twiddle, wts, hmax, eta, bin);
    count_launches(1);
    return cudaGetLastError();
  }
  if (n <= 65 && H >= 1) {
    const size_t sm = (size_t)H * K * sizeof(float2) + (size_t)n * kDftThreads * sizeof(float);
    auto kern = K <= 16 ? (harm ? k_dft_short<16, true> : k_dft_short<16, false>)
                        : (harm ? k_dft_short<32, true> : k_dft_short<32, false>);
    kern<<<short_grid(n, blocks, sm), kDftThreads, sm, st>>>(vp, n, T, vs, twiddle, wts, hmax, eta, bin);
    count_launches(1);
    return cudaGetLastError();
  }
  if (n > 256 || hmax > 1) {
    const int P = direct ? 0 : mixed_split(n);
    // eight tiles per CTA fill 32-byte segments of the cube's rows; four where
    // eight tiles' series, sub-spectra and the table exceed half an SM's memory
    if (P && n <= 1664)
      return launch_mixed_t<8>(vp, n, P, T, vs, twiddle, wts, hmax, eta, bin, st);
    if (P) return launch_mixed_t<4>(vp, n, P, T, vs, twiddle, wts, hmax, eta, bin, st);
    return launch_long(vp, n, T, vs, twiddle, wts, hmax, eta, bin, st);
  }
  const size_t smem = (size_t)n * kDftThreads * sizeof(float);
  const cudaError_t lim = allow_smem(k_dft, smem);
  if (lim != cudaSuccess) return lim;
  k_dft<<<(unsigned)blocks, kDftThreads, smem, st>>>(vp, n, T, vs, twiddle, wts, eta, bin);
  count_launches(1);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- ingest conversion
__device__ __forceinline__ float load_any(const void* p, int type, int64_t i) {
  if (type == FITRIG_BF16) return to_f32(static_cast<const bf16_t*>(p)[i]);
  if (type == FITRIG_F16) return to_f32(static_cast<const f16_t*>(p)[i]);
  return static_cast<const float*>(p)[i];
}

// Stores v in `type` (half types: round to nearest even) and returns the
// stored value as FP32.
__device__ __forceinline__ float store_any(void* p, int type, int64_t i, float v) {
  if (type == FITRIG_BF16) {
    unsigned short h;
    asm("cvt.rn.bf16.f32 %0, %1;" : "=h"(h) : "f"(v));
    static_cast<uint16_t*>(p)[i] = h;
    return __uint_as_float((uint32_t)h << 16);
  }
  if (type == FITRIG_F16) {
    unsigned short h;
    asm("cvt.rn.f16.f32 %0, %1;" : "=h"(h) : "f"(v));
    static_cast<uint16_t*>(p)[i] = h;
    float r;
    asm("cvt.f32.f16 %0, %1;" : "=f"(r) : "h"(h));
    return r;
  }
  static_cast<float*>(p)[i] = v;
  return v;
}

// Rows over blockIdx.y, columns over the threads of blockIdx.x (no per-pixel
// division).
__global__ void k_convert(const void* src, int st, int64_t sp, void* dst, int dt, int64_t dp,
                          int ny, int nx) {
  for (int y = blockIdx.y; y < ny; y += gridDim.y)
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < nx; x += gridDim.x * blockDim.x)
      store_any(dst, dt, (int64_t)y * dp + x, load_any(src, st, (int64_t)y * sp + x));
}

static dim3 image_grid(int ny, int nx) {
  return dim3((unsigned)std::min(8, (nx + 255) / 256), (unsigned)std::min(ny, 4096));
}

// Rows from one pitch to another, in the widest unit that divides both pitches,
// the row and the addresses (rows of odd length are 2- or 4-byte units).  A
// thread has four units in flight; a warp's units lie side by side.  (The
// runtime's pitched device copy moves 6200-byte rows at 0.9 TB/s, and a copy
// per snapshot is a launch each: 70 snapshots of 370 x 464 BF16 with the detect
// 617 -> 270 us as one of these.)
template <typename U>
__global__ void __launch_bounds__(256) k_repitch(const U* __restrict__ src, int64_t sp,
                                                 U* __restrict__ dst, int64_t dp, int n,
                                                 int64_t rows) {
  constexpr int B = 4;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= n) return;
  for (int64_t y = (int64_t)blockIdx.y * B; y < rows; y += (int64_t)gridDim.y * B) {
    U v[B];
#pragma unroll
    for (int b = 0; b < B; ++b)
      if (y + b < rows) v[b] = src[(y + b) * sp + x];
#pragma unroll
    for (int b = 0; b < B; ++b)
      if (y + b < rows) dst[(y + b) * dp + x] = v[b];
  }
}

template <typename U>
static void repitch_t(const void* src, size_t sp, void* dst, size_t dp, size_t width, int64_t rows,
                      cudaStream_t st) {
  const int64_t n = (int64_t)(width / sizeof(U));
  const dim3 grid((unsigned)((n + 255) / 256), (unsigned)std::min<int64_t>((rows + 3) / 4, 65535));
  k_repitch<U><<<grid, 256, 0, st>>>(static_cast<const U*>(src), (int64_t)(sp / sizeof(U)),
                                     static_cast<U*>(dst), (int64_t)(dp / sizeof(U)), (int)n, rows);
}

cudaError_t launch_repitch(const void* src, size_t spitch, void* dst, size_t dpitch, size_t width,
                           int64_t rows, cudaStream_t st) {
  const size_t all = width | spitch | dpitch | (size_t)reinterpret_cast<uintptr_t>(src) |
                     (size_t)reinterpret_cast<uintptr_t>(dst);
  if (all % 16 == 0) repitch_t<uint4>(src, spitch, dst, dpitch, width, rows, st);
  else if (all % 8 == 0) repitch_t<uint2>(src, spitch, dst, dpitch, width, rows, st);
  else if (all % 4 == 0) repitch_t<uint32_t>(src, spitch, dst, dpitch, width, rows, st);
  else repitch_t<uint16_t>(src, spitch, dst, dpitch, width, rows, st);
  count_launches(1);
  return cudaGetLastError();
}

// Difference coding, closed loop (FITRIG_CODING_DELTA): the first snapshot is
// kept in FP32 (key frame) and starts the coder's decoded snapshot `state`;
// each later one stores q = round-to-nearest-even half of the FP32 difference
// x - state, and state advances by the decoded difference, fl32(state + q),
// exactly as the stack march decodes it.  NaN and infinities propagate.
__global__ void k_delta_encode(const void* src, int st, int64_t sp, float* state, float* key,
                               int64_t kp, void* dst, int dt, int64_t dp, int first, int ny,
                               int nx) {
  for (int y = blockIdx.y; y < ny; y += gridDim.y) {
    float* srow = state + (int64_t)y * nx;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < nx; x += gridDim.x * blockDim.x) {
      const float v = load_any(src, st, (int64_t)y * sp + x);
      if (first) {
        key[(int64_t)y * kp + x] = v;
        srow[x] = v;
      } else {
        const float prev = srow[x];
        const float q = store_any(dst, dt, (int64_t)y * dp + x, __fsub_rn(v, prev));
        srow[x] = __fadd_rn(prev, q);   // the decoded difference
      }
    }
  }
}

cudaError_t launch_delta_encode(const void* src, int src_type, int64_t src_pitch, float* state,
                                float* key, int64_t key_pitch, void* dst, int dst_type,
                                int64_t dst_pitch, bool first, int ny, int nx, cudaStream_t st) {
  k_delta_encode<<<image_grid(ny, nx), 256, 0, st>>>(src, src_type, src_pitch, state, key,
                                                     key_pitch, dst, dst_type, dst_pitch,
                                                     first ? 1 : 0, ny, nx);
  count_launches(1);
  return cudaGetLastError();
}

// Snapshot accumulation (Sec. 3.3.2): acc = x (first raw snapshot of a
// block) or acc + x in FP32; the last raw snapshot of the block stores the
// sum, in the storage type, to the stack slot instead.
__global__ void k_accumulate(const void* src, int st, int64_t sp, float* acc, int first, int last,
                             void* dst, int dt, int64_t dp, int ny, int nx) {
  for (int y = blockIdx.y; y < ny; y += gridDim.y) {
    float* arow = acc + (int64_t)y * nx;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < nx; x += gridDim.x * blockDim.x) {
      const float v = load_any(src, st, (int64_t)y * sp + x);
      const float a = first ? v : arow[x] + v;
      if (last) store_any(dst, dt, (int64_t)y * dp + x, a);
      else arow[x] = a;
    }
  }
}

cudaError_t launch_accumulate(const void* src, int src_type, int64_t src_pitch, float* acc,
                              bool first, bool last, void* dst, int dst_type, int64_t dst_pitch,
                              int ny, int nx, cudaStream_t st) {
  k_accumulate<<<image_grid(ny, nx), 256, 0, st>>>(src, src_type, src_pitch, acc, first ? 1 : 0,
                                                   last ? 1 : 0, dst, dst_type, dst_pitch, ny, nx);
  count_launches(1);
  return cudaGetLastError();
}

// A serving unit's frequency-series weight 1 / M_s^2 (FP64, rounded to FP32),
// with M_s the running maximum over every snapshot seen so far (its ordered
// key, 0 before any finite pixel), floored at C (Eq. 5's constant).
__global__ void k_unit_weight(const unsigned* gmax_key, float* w) {
  const unsigned k = *gmax_key;
  double m = k ? (double)f32_from_key(k) : 0.0;
  if (!(m > (double)kGuardC)) m = (double)kGuardC;
  *w = (float)(1.0 / (m * m));
}

cudaError_t launch_unit_weight(const unsigned* gmax_key, float* w, cudaStream_t st) {
  k_unit_weight<<<1, 1, 0, st>>>(gmax_key, w);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_convert(const void* src, int src_type, int64_t src_pitch, void* dst,
                           int dst_type, int64_t dst_pitch, int ny, int nx, cudaStream_t st) {
  k_convert<<<image_grid(ny, nx), 256, 0, st>>>(src, src_type, src_pitch, dst, dst_type, dst_pitch,
                                                ny, nx);
  count_launches(1);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- timestamps
// The GPU's global nanosecond timer, written when the stream reaches this
// point (serving: per-stage device times of a unit, read by the host without
// a CUDA call).
__global__ void k_stamp(long long* dst) {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  *dst = (long long)t;
}

cudaError_t launch_stamp(long long* dst, cudaStream_t st) {
  k_stamp<<<1, 1, 0, st>>>(dst);
  count_launches(1);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- autotuner probe data
// Deterministic pseudo-random values in [-4, 4) (an integer hash of the index),
// used only as timing input for the autotuner.
__global__ void k_fill_probe(void* dst, int type, int64_t n, uint32_t seed) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    uint32_t h = (uint32_t)i * 2654435761u ^ seed;
    h ^= h >> 15;
    h *= 2246822519u;
    h ^= h >> 13;
    store_any(dst, type, i, ((float)(h >> 8) * (1.0f / 16777216.0f)) * 8.f - 4.f);
  }
}

cudaError_t launch_fill_probe(void* dst, int type, int64_t n, uint32_t seed, cudaStream_t st) {
  k_fill_probe<<<152 * 8, 256, 0, st>>>(dst, type, n, seed);
  count_launches(1);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- tLISI report
// tLISI = 1 - v / M^2 in FP64 (Eq. tLISI), M = max(stack maximum, C).
__global__ void k_tlisi(const float* vp, int64_t n, const unsigned* gmax, const double* m_unit,
                        float* out) {
  double M;
  if (m_unit) {
    M = *m_unit;
  } else {
    const unsigned key = *gmax;
    M = key ? (double)f32_from_key(key) : 0.0;
    if (!(M > (double)kGuardC)) M = (double)kGuardC;
  }
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = (float)(1.0 - (double)vp[i] / (M * M));
}

cudaError_t launch_tlisi_from_values(const float* vp, int64_t n, const unsigned* gmax,
                                     const double* m_unit, float* out, cudaStream_t st) {
  k_tlisi<<<152 * 2, 256, 0, st>>>(vp, n, gmax, m_unit, out);
  count_launches(1);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- running M
// Real-time reading of M (Sec. 2.2.4): unit s is normalised by the maximum
// over snapshots 0..s+2.  The march leaves each snapshot's maximum key in
// smax[k] (+inf included); a snapshot whose maximum is +inf gets the maximum
// of its finite pixels instead (rare: only stacks with non-finite pixels).
template <typename T>
__global__ void k_snap_finite_max(const T* stack, int L, int ny, int nx, int64_t pitch,
                                  size_t slice, unsigned* smax) {
  const unsigned inf_key = f32_key(INFINITY);
  for (int k = 0; k < L; ++k) {
    if (smax[k] != inf_key) continue;   // uniform: every thread reads the same word
    const T* x = stack + (size_t)k * slice;
    float m = -INFINITY;
    const int64_t total = (int64_t)ny * nx;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
      const float v = to_f32(x[(i / nx) * pitch + (i % nx)]);
      if (isfinite(v)) m = fmaxf(m, v);
    }
    // the words are replaced only after every block has read them: write the
    // finite maxima to the upper half and let k_running_norm prefer it
    warp_max_to(m, smax + L + k);
  }
}

// M_s = max(C, max over k <= s + 2 of the snapshot maxima) for s < U, in FP64,
// and the series weights (M_{U-1} / M_s)^2 of the frequency branch, whose
// spectrum is then the spectrum of the tLISI series scaled by M^2 like the
// global reading's.
__global__ void k_running_norm(const unsigned* smax, int L, double* m_unit, float* wts) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const unsigned inf_key = f32_key(INFINITY);
  const int U = L - 2;
  double run = (double)kGuardC;
  for (int k = 0; k < L; ++k) {
    unsigned key = smax[k];
    if (key == inf_key) key = smax[L + k];
    if (key) {
      const double v = (double)f32_from_key(key);
      if (v > run) run = v;   // NaN never compares greater
    }
    if (k >= 2) m_unit[k - 2] = run;
  }
  const double last = m_unit[U - 1];
  for (int s = 0; s < U; ++s) {
    const double q = last / m_unit[s];
    wts[s] = (float)(q * q);
  }
}

cudaError_t launch_running_norm(const void* stack, int storage, int L, int ny, int nx,
                                int64_t pitch, unsigned* smax, double* m_unit, float* wts,
                                cudaStream_t st) {
  const size_t slice = (size_t)pitch * ny;
  int n = 1;
  if (!stack) {
    // a difference-coded stack: the caller ran launch_delta_finite_max
  } else if (storage == FITRIG_F32)
    k_snap_finite_max<float><<<152 * 2, 256, 0, st>>>(static_cast<const float*>(stack), L, ny, nx,
                                                       pitch, slice, smax);
  else if (storage == FITRIG_BF16)
    k_snap_finite_max<bf16_t><<<152 * 2, 256, 0, st>>>(static_cast<const bf16_t*>(stack), L, ny,
                                                        nx, pitch, slice, smax);
  else
    k_snap_finite_max<f16_t><<<152 * 2, 256, 0, st>>>(static_cast<const f16_t*>(stack), L, ny, nx,
                                                       pitch, slice, smax);
  if (stack) n = 2;
  k_running_norm<<<1, 32, 0, st>>>(smax, L, m_unit, wts);
  count_launches(n);
  return cudaGetLastError();
}

}  // namespace fitrig
