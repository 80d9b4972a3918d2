// Complex FFTs of one line held in a thread's registers (lengths up to 32)
// with twiddles known at compile time, and the pieces of the pruned transforms
// of length 2H whose second half of the inputs is zero (forward) or of the
// outputs is not kept (inverse): the even outputs of the forward transform are
// the length-H transform of the inputs, the odd ones that of the inputs times
// w^j; the kept outputs of the inverse are E + w^-j O with E and O the
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

// In-register FFT of length L (a power of two up to 32), natural order in and
// out, unnormalised; DIR = -1 forward, +1 inverse.
template <int L, int DIR, typename R>
struct LineFFT {
  static __device__ __forceinline__ void run(R* re, R* im) {
    constexpr int H = L / 2;
    R er[H], ei[H], odr[H], odi[H];
#pragma unroll
    for (int j = 0; j < H; ++j) {
      er[j] = re[2 * j]; ei[j] = im[2 * j];
      odr[j] = re[2 * j + 1]; odi[j] = im[2 * j + 1];
    }
    LineFFT<H, DIR, R>::run(er, ei);
    LineFFT<H, DIR, R>::run(odr, odi);
#pragma unroll
    for (int k = 0; k < H; ++k) {
      R tr = odr[k], ti = odi[k];
      if (4 * k == L) {  // w = -i (forward) or +i (inverse)
        tr = DIR < 0 ? odi[k] : -odi[k];
        ti = DIR < 0 ? -odr[k] : odr[k];
      } else if (k > 0) {
        rotate64<DIR>(k * (64 / L), tr, ti);
      }
      re[k] = er[k] + tr; im[k] = ei[k] + ti;
      re[k + H] = er[k] - tr; im[k + H] = ei[k] - ti;
    }
  }
};
template <int DIR, typename R>
struct LineFFT<1, DIR, R> {
  static __device__ __forceinline__ void run(R*, R*) {}
};

}  // namespace flgf
