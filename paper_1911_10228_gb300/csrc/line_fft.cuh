// Complex FFTs of one line held in a thread's registers (lengths up to 32)
// with twiddles known at compile time, and the pieces of the pruned transforms
// of length 2H whose second half of the inputs is zero (forward) or of the
// outputs is not kept (inverse): the even outputs of the forward transform are
// the length-H transform of the inputs, the odd ones the same at frequencies
// k + 1/2; the kept outputs of the inverse are E + w^-j O with E and O the
// transforms of the even and odd inputs.
#pragma once
#include <cuda_runtime.h>

namespace flgf {

// cos(2 pi j / 64), sin(2 pi j / 64)
__host__ __device__ constexpr double cos64(int j) {
  constexpr double c[17] = {  // the first quadrant
      1.0,
      0.995184726672196886245,
      0.980785280403230449126,
      0.956940335732208864936,
      0.923879532511286756128,
      0.881921264348355029713,
      0.831469612302545237079,
      0.773010453362736960811,
      0.707106781186547524401,
      0.634393284163645498215,
      0.555570233019602224743,
      0.471396736825997648556,
      0.382683432365089771728,
      0.290284677254462367636,
      0.195090322016128267848,
      0.0980171403295606019942,
      0.0};
  j &= 63;
  if (j > 32) j = 64 - j;
  return j <= 16 ? c[j] : -c[32 - j];
}
__host__ __device__ constexpr double sin64(int j) { return cos64(j - 16); }

// (xr + i xi) *= e^{-2 pi i j / 64} (DIR < 0) or its conjugate
template <int DIR, typename R>
__device__ __forceinline__ void rotate64(int j, R& xr, R& xi) {
  const R c = (R)cos64(j), s = DIR < 0 ? (R)-sin64(j) : (R)sin64(j);
  const R tr = c * xr - s * xi;
  xi = c * xi + s * xr;
  xr = tr;
}

// (u, v) -> (u + w v, u - w v), w = e^{-2 pi i j / 64} (DIR < 0) or its
// conjugate: six fused multiply-adds with tan or cot, whichever is at most 1,
// factored out of w v.
template <int DIR, typename R>
__device__ __forceinline__ void butterfly64(int j, R ur, R ui, R vr, R vi, R& ar, R& ai, R& br, R& bi) {
  const double c = cos64(j), s = DIR < 0 ? -sin64(j) : sin64(j);  // w = c + i s
  if (s == 0.0 || c == 0.0) {                                      // +-1, +-i
    const R tr = s == 0.0 ? (c > 0 ? vr : -vr) : (s > 0 ? -vi : vi);
    const R ti = s == 0.0 ? (c > 0 ? vi : -vi) : (s > 0 ? vr : -vr);
    ar = ur + tr; ai = ui + ti;
    br = ur - tr; bi = ui - ti;
    return;
  }
  const bool big = c * c >= s * s;
  const R t = (R)(big ? s / c : c / s), f = (R)(big ? c : s);
  const R p = big ? fma(-t, vi, vr) : fma(t, vr, -vi), q = big ? fma(t, vr, vi) : fma(t, vi, vr);
  ar = fma(f, p, ur); ai = fma(f, q, ui);
  br = fma(-f, p, ur); bi = fma(-f, q, ui);
}

// In-register FFT of length L (a power of two up to 32), natural order in and
// out, unnormalised; DIR = -1 forward, +1 inverse.  ODD: the odd outputs of the
// transform of length 2L whose inputs L.. are zero (frequencies k + 1/2).
template <int L, int DIR, typename R, bool ODD = false>
struct LineFFT {
  static __device__ __forceinline__ void run(R* re, R* im) {
    constexpr int H = L / 2;
    R er[H], ei[H], odr[H], odi[H];
#pragma unroll
    for (int j = 0; j < H; ++j) {
      er[j] = re[2 * j]; ei[j] = im[2 * j];
      odr[j] = re[2 * j + 1]; odi[j] = im[2 * j + 1];
    }
    LineFFT<H, DIR, R, ODD>::run(er, ei);
    LineFFT<H, DIR, R, ODD>::run(odr, odi);
#pragma unroll
    for (int k = 0; k < H; ++k)
      butterfly64<DIR>((2 * k + ODD) * (32 / L), er[k], ei[k], odr[k], odi[k], re[k], im[k], re[k + H], im[k + H]);
  }
};
template <int DIR, typename R, bool ODD>
struct LineFFT<1, DIR, R, ODD> {
  static __device__ __forceinline__ void run(R*, R*) {}
};

}  // namespace flgf
