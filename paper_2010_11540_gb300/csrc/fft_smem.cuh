// Radix-2 Stockham FFT in shared memory, float64, shared by the float64
// solves (open boundary and conducting pipe).
//
// A transform waits for its barriers and shared-memory trips and for the FP64
// pipe of the SM it runs on (two instructions per clock, 64 clocks of a
// sub-partition per warp instruction), so FP64 instructions per butterfly
// count.  a +- w b with w = c + i s takes six fused multiply-adds instead of
// eight instructions when w is factored by its larger part (E. Linzer and
// E. Feig, IEEE Trans. Signal Process. 41 (1993) 93): w b = c (b + i t b),
// t = s/c, or w b = i s (b + i u b), u = -c/s; |t|, |u| <= 1, so no accuracy is
// lost.
#pragma once

#include <cmath>
#include <vector>

#include "sc_internal.cuh"

namespace sc {

// Twiddle t of M (angle -2 pi t / M, t < M/2) as (ratio, larger part): the
// larger part is the sine for M/8 < t < 3M/8.
inline std::vector<double2> fft_twiddles(int M) {
  std::vector<double2> w(M / 2);
  for (int t = 0; t < M / 2; ++t) {
    const double ang = -2.0 * M_PI * (double)t / (double)M;
    const double c = std::cos(ang), s = std::sin(ang);
    w[t] = (8 * t > M && 8 * t < 3 * M) ? make_double2(-c / s, s) : make_double2(s / c, c);
  }
  return w;
}

// Butterfly of v0, v1 with twiddle index t: lo = v0 + w v1 and, unless HALF,
// hi = v0 - w v1 (INV: the conjugate w).
template <bool INV, bool HALF>
__device__ __forceinline__ void fft_butterfly(double2 v0, double2 v1, int t, int M, const double2* __restrict__ tw,
                                              double2& lo, double2& hi) {
  const double2 w = __ldg(tw + t);
  const bool swap = 8 * t > M && 8 * t < 3 * M;
  const double r = INV ? -w.x : w.x, m = (INV && swap) ? -w.y : w.y;
  const double bx = fma(-r, v1.y, v1.x), by = fma(r, v1.x, v1.y);
  const double x = swap ? -by : bx, y = swap ? bx : by;
  lo = make_double2(fma(m, x, v0.x), fma(m, y, v0.y));
  if (!HALF) hi = make_double2(fma(-m, x, v0.x), fma(-m, y, v0.y));
}

// The stages Ns = first, 2 first, ... M/2 of a transform of length M by the
// M/2 threads j (every thread of the block calls it; several transforms may
// run side by side, each in its own pair of buffers).  a: the data after the
// stages before `first`; the caller has synchronised.  HALF: only the first
// half of the result is formed.  Returns the buffer that holds the result.
template <bool INV, bool HALF>
__device__ __forceinline__ double2* fft_stages(double2* a, double2* b, int M, int first, int j,
                                               const double2* __restrict__ tw) {
  const int half = M >> 1;
  for (int Ns = first; Ns < half; Ns <<= 1) {
    const int k = j & (Ns - 1), idx = ((j - k) << 1) + k;
    double2 lo, hi;
    fft_butterfly<INV, false>(a[j], a[j + half], k * (half / Ns), M, tw, lo, hi);
    b[idx] = lo;
    b[idx + Ns] = hi;
    __syncthreads();
    double2* t = a;
    a = b;
    b = t;
  }
  double2 lo, hi;  // Ns = M/2
  fft_butterfly<INV, HALF>(a[j], a[j + half], j, M, tw, lo, hi);
  b[j] = lo;
  if (!HALF) b[j + half] = hi;
  __syncthreads();
  return b;
}

// A whole transform, blockDim.x == M/2 (M >= 4).  The first stage has no
// twiddles.  Caller synchronises before.
template <bool INV>
__device__ __forceinline__ double2* fft_smem(double2* a, double2* b, int M, const double2* __restrict__ tw) {
  const int j = threadIdx.x, half = M >> 1;
  const double2 v0 = a[j], v1 = a[j + half];
  b[2 * j] = make_double2(v0.x + v1.x, v0.y + v1.y);
  b[2 * j + 1] = make_double2(v0.x - v1.x, v0.y - v1.y);
  __syncthreads();
  return fft_stages<INV, false>(b, a, M, 2, j, tw);
}

}  // namespace sc
