// a2-a4 between parents, for the finest octree level: the near field and the
// influence lists of a finest-level target (Sec. 2.1) are together all the
// children of its parent's 27 neighbours, so the level's interaction is a
// convolution between PARENT blocks of H = 2N cells a side.  One zero-padded
// FFT of P = 4N points an axis per parent replaces eight of 2N: a neighbour
// pair then costs 8 NW complex products (NW frequencies of a child's padded
// spectrum) where the child pairs cost 64 NW.
//
// Coarser octree levels exclude the near field, which depends on the child.  In
// FP64 they run between parents all the same: the parent kernels are zero for
// |displacement|_inf <= N (reached by near pairs only; a block's siblings, e = 0,
// need no product at all), and what the near pairs of neighbour parents still
// get is taken out block by block: at most 19 pair-list entries a target with
// the kernel -G where |displacement|_inf > N, added by the inverse transform.
// The parts that cancel are no larger than those that stay, so the error is
// the same (11 x 9 x 13 blocks of 16^3: 2.4e-14 from 64-bit values both ways).
// FP64's FMA rate bounds it: 27 x 8 + 152 products instead of 1512 a parent.
// Whole solves: 11 x 9 x 13 blocks of 16^3 17.6 -> 12.7 ms, three-level torus of
// 8^3 blocks 10.5 -> 7.4 ms.  FP32 keeps the child-pair kernels there: their
// spectra go through float-float inverse transforms.
//
// The transform along axis 0 is fused with the products (FP64: only the
// inverse), so HBM only holds spectra of the two transformed axes, half as long
// as padded ones:
//   pf_forward_kernel   planes z of a source parent: axis 2, axis 1
//   pf_axis0_kernel     FP64: axis 0 forward, into fully padded spectra
//   pf_mac_kernel       axis 0 forward (FP32), products, axis 0 inverse
//   pf_inverse_kernel   planes z of a target parent: axis 1, axis 2
// Layout between them: lines l = k1 (H + 1) + k2 (P (H + 1) of them); a unit
// is the 32 / H lines that fill a warp, stored [unit][parent][32] (FP64
// sources: [unit][parity][parent][32]) with lane (l % (32 / H)) H + z, so the
// product kernel reads 256-byte (FP32) or 512-byte rows.
//
// The axis-0 transform is pruned by parity: the even (odd) outputs are the
// H-point transform of the H inputs (times w^z), and the kept inverse outputs
// are the sum of the inverses of the two halves (the odd one times w^-z).  The
// product kernel takes the two parities one after the other, so its shared
// memory holds H values per line and parent.
//
// Measured against the child-pair kernels (finest level only; GB300): 16^3
// blocks of 16^3 cells, FP32: products 2.42 -> 0.81 ms, its transforms 0.31 ->
// 0.17 ms; 11 x 9 x 13 blocks, FP64: 32.5 -> 9.2 ms and 2.4 -> 2.2 ms.
#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "line_fft.cuh"

namespace flgf {

namespace {

template <typename R> struct Vec2;
template <> struct Vec2<float> { using type = float2; };
template <> struct Vec2<double> { using type = double2; };

constexpr int kPfStride = 33;  // complex values between two parents' lines in shared memory (odd: no conflicts)

template <int N> struct PfDims {
  static constexpr int H = 2 * N, P = 4 * N, NX = H + 1, L = P * NX, S = 32 / H, U = L / S;
  static_assert(L % S == 0, "whole units");
};

// a row of N values of block gid in 16-byte vectors, zero for no block (gid < 0)
template <typename R, int N>
__device__ __forceinline__ void load_row(const R* __restrict__ nodes, int gid, size_t off, R* x) {
  constexpr int V = 16 / (int)sizeof(R);
  const int4* p = reinterpret_cast<const int4*>(nodes + (size_t)max(gid, 0) * N * N * N + off);
#pragma unroll
  for (int u = 0; u < N / V; ++u) {
    const int4 v = gid >= 0 ? __ldg(p + u) : make_int4(0, 0, 0, 0);
    const R* r = reinterpret_cast<const R*>(&v);
#pragma unroll
    for (int j = 0; j < V; ++j) x[u * V + j] = r[j];
  }
}

template <typename R>
__device__ __forceinline__ void cp_async_complex(void* dst, const void* src) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  if constexpr (sizeof(R) == 4)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
// keeps the compiler from moving one half's shared-memory reads above the
// other half's work (a thread has the registers for one half)
__device__ __forceinline__ void half_barrier() { asm volatile("" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

}  // namespace

// Plane padding of the [ZP][H][NX] buffer of the plane kernels: the lanes of
// a shared-memory access (16 complex floats or 8 complex doubles) are ZP
// planes of consecutive columns, so planes are offset to fill all banks.
template <typename R, int N, int ZP>
constexpr int pf_plane_stride() {
  constexpr int B = 128 / (2 * (int)sizeof(R));
  constexpr int want = ZP >= B ? 1 : B / ZP;
  return PfDims<N>::H * PfDims<N>::NX + ((want - PfDims<N>::H * PfDims<N>::NX % B) % B + B) % B;
}

constexpr int kPfPlaneThreads = 288;
// Halves of a source parent's spectrum in memory: FP64 both parities of the
// transformed axis 0, FP32 the planes.
template <typename R> constexpr int pf_halves() { return sizeof(R) == 8 ? 2 : 1; }

// ---------------------------------------------------------------------------
// Axes 2 and 1 of ZP planes of a source parent.  Axis 2 transforms the real
// rows y and y + N (children of different b1) as one complex line and splits
// the two spectra; axis 1 writes its outputs straight to HBM, ZP consecutive
// z per line.
// ---------------------------------------------------------------------------
template <typename R, int N, int ZP>
__global__ void __launch_bounds__(kPfPlaneThreads, sizeof(R) == 4 ? 2 : 1)
    pf_forward_kernel(const R* __restrict__ nodes, const int* __restrict__ cell_ch, typename Vec2<R>::type* __restrict__ out,
                      int ncol) {
  using D = PfDims<N>;
  using C2 = typename Vec2<R>::type;
  constexpr int H = D::H, NX = D::NX, ZS = pf_plane_stride<R, N, ZP>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2* buf = reinterpret_cast<C2*>(smem_raw);
  const int col = blockIdx.x / (H / ZP), z0 = (blockIdx.x % (H / ZP)) * ZP;
  // a thread per (parity, row pair), then per (parity, column)
  auto rows = [&](auto parity, int i) {
    constexpr int par = decltype(parity)::value;
    const int zl = i / N, y = i % N, z = z0 + zl;
    const int* ch = cell_ch + col * 8 + (z >= N ? 4 : 0);
    const size_t roff = (size_t)((z % N) * N + y) * N;
    C2* r0 = buf + zl * ZS + y * NX;
    C2* r1 = r0 + N * NX;
    R xr[H], xi[H];
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      load_row<R, N>(nodes, __ldg(ch + b), roff, xr + b * N);
      load_row<R, N>(nodes, __ldg(ch + 2 + b), roff, xi + b * N);
    }
    LineFFT<H, -1, R, par == 1>::run(xr, xi);
    // row y: (Z[k] + conj Z[P-k]) / 2, row y + N: (Z[k] - conj Z[P-k]) / 2i
#pragma unroll
    for (int m = 0; m <= H / 2 - par; ++m) {
      const int q = par ? H - 1 - m : (H - m) % H, k = 2 * m + par;
      r0[k] = C2{R(0.5) * (xr[m] + xr[q]), R(0.5) * (xi[m] - xi[q])};
      r1[k] = C2{R(0.5) * (xi[m] + xi[q]), R(0.5) * (xr[q] - xr[m])};
    }
  };
  for (int i = threadIdx.x; i < 2 * ZP * N; i += kPfPlaneThreads) {
    if (i < ZP * N) rows(std::integral_constant<int, 0>{}, i);
    else rows(std::integral_constant<int, 1>{}, i - ZP * N);
  }
  __syncthreads();
  auto columns = [&](auto parity, int i) {
    constexpr int par = decltype(parity)::value;
    const int zl = i % ZP, kx = i / ZP;
    const C2* src = buf + zl * ZS + kx;
    R xr[H], xi[H];
#pragma unroll
    for (int y = 0; y < H; ++y) {
      const C2 v = src[y * NX];
      xr[y] = v.x; xi[y] = v.y;
    }
    LineFFT<H, -1, R, par == 1>::run(xr, xi);
#pragma unroll
    for (int m = 0; m < H; ++m) {
      const int l = (2 * m + par) * NX + kx;
      out[((size_t)(l / D::S) * pf_halves<R>() * ncol + col) * 32 + (l % D::S) * H + z0 + zl] = C2{xr[m], xi[m]};
    }
  };
  for (int i = threadIdx.x; i < 2 * ZP * NX; i += kPfPlaneThreads) {
    if (i < ZP * NX) columns(std::integral_constant<int, 0>{}, i);
    else columns(std::integral_constant<int, 1>{}, i - ZP * NX);
  }
}

// ---------------------------------------------------------------------------
// FP64: axis 0 of every source parent, once, into the two parities' halves of
// its fully padded spectrum ([unit][parity][parent][32], the planes in parity
// 0's place).  Fused with the products, as in FP32, a parent's lines would be
// transformed by every group that reads them (up to three times), and the FP64
// pipe bounds it; the doubled spectra cost less.  A thread per line, rows
// staged through shared memory; 64 threads leave three CTAs an SM.
// Whole solves: 11 x 9 x 13 blocks of 16^3 12.7 -> 11.1 ms, three-level torus
// of 8^3 blocks 7.44 -> 7.02 ms.
// ---------------------------------------------------------------------------
constexpr int kPfAxisThreads = 64;
template <typename R, int N>
__global__ void __launch_bounds__(kPfAxisThreads) pf_axis0_kernel(typename Vec2<R>::type* __restrict__ spec, int ncol) {
  using D = PfDims<N>;
  using C2 = typename Vec2<R>::type;
  constexpr int H = D::H, RC = kPfAxisThreads / D::S;  // parents per CTA
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2* A = reinterpret_cast<C2*>(smem_raw);  // [RC][33] planes, then the odd half
  C2* B = A + RC * kPfStride;               // [RC][33] the even half
  const int nch = (ncol + RC - 1) / RC, unit = blockIdx.x / nch, c0 = blockIdx.x % nch * RC, n = min(RC, ncol - c0);
  C2* even = spec + ((size_t)unit * 2 * ncol + c0) * 32;
  C2* odd = even + (size_t)ncol * 32;
  for (int i = threadIdx.x; i < n * 32; i += kPfAxisThreads) A[(i / 32) * kPfStride + i % 32] = even[i];
  __syncthreads();
  if (threadIdx.x < n * D::S) {
    const int off = (threadIdx.x / D::S) * kPfStride + (threadIdx.x % D::S) * H;
    auto half = [&](auto parity, C2* out) {
      constexpr int par = decltype(parity)::value;
      R xr[H], xi[H];
#pragma unroll
      for (int z = 0; z < H; ++z) { const C2 v = A[off + z]; xr[z] = v.x; xi[z] = v.y; }
      LineFFT<H, -1, R, par == 1>::run(xr, xi);
#pragma unroll
      for (int k = 0; k < H; ++k) out[off + k] = C2{xr[k], xi[k]};
    };
    half(std::integral_constant<int, 0>{}, B);
    half_barrier();
    half(std::integral_constant<int, 1>{}, A);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n * 32; i += kPfAxisThreads) {
    even[i] = B[(i / 32) * kPfStride + i % 32];
    odd[i] = A[(i / 32) * kPfStride + i % 32];
  }
}

// ---------------------------------------------------------------------------
// Axes 1 and 2 back, of ZP planes of a target parent: keep H outputs an axis,
// write the children that are targets.  The halves of a pruned inverse are
// combined through the buffer, so a thread holds one H-point line.
// ---------------------------------------------------------------------------
template <typename R, int N, int ZP>
__global__ void __launch_bounds__(kPfPlaneThreads, sizeof(R) == 4 ? 2 : 1)
    pf_inverse_kernel(const typename Vec2<R>::type* __restrict__ in, int ncol, const int* __restrict__ tgt_ch,
                      const double* __restrict__ scales, R* __restrict__ unodes) {
  using D = PfDims<N>;
  using C2 = typename Vec2<R>::type;
  constexpr int H = D::H, NX = D::NX, P = D::P, ZS = pf_plane_stride<R, N, ZP>(), TW = 64 / P;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2* buf = reinterpret_cast<C2*>(smem_raw);
  const int col = blockIdx.x / (H / ZP), z0 = (blockIdx.x % (H / ZP)) * ZP;
  for (int i = threadIdx.x; i < ZP * NX; i += kPfPlaneThreads) {
    const int zl = i % ZP, kx = i / ZP;
    C2* dst = buf + zl * ZS + kx;
    auto half = [&](auto parity) {
      constexpr int par = decltype(parity)::value;
      R xr[H], xi[H];
#pragma unroll
      for (int m = 0; m < H; ++m) {
        const int l = (2 * m + par) * NX + kx;
        const C2 v = in[((size_t)(l / D::S) * ncol + col) * 32 + (l % D::S) * H + z0 + zl];
        xr[m] = v.x; xi[m] = v.y;
      }
      LineFFT<H, +1, R>::run(xr, xi);
#pragma unroll
      for (int y = 0; y < H; ++y) {
        if constexpr (par == 0) {
          dst[y * NX] = C2{xr[y], xi[y]};
        } else {
          if (y > 0) rotate64<+1>(y * TW, xr[y], xi[y]);
          const C2 v = dst[y * NX];
          dst[y * NX] = C2{v.x + xr[y], v.y + xi[y]};
        }
      }
    };
    half(std::integral_constant<int, 0>{});
    half_barrier();
    half(std::integral_constant<int, 1>{});
  }
  __syncthreads();
  const R scale = (R)(scales[col] / ((double)P * P * P));
  for (int i = threadIdx.x; i < ZP * N; i += kPfPlaneThreads) {
    const int zl = i / N, y = i % N, z = z0 + zl;
    C2* r0 = buf + zl * ZS + y * NX;
    C2* r1 = r0 + N * NX;
    R xr[H], xi[H];
    // Z = A + i B of the rows y and y + N, whose upper halves are Hermitian;
    // the even half's outputs wait in the rows' own even slots
#pragma unroll
    for (int m = 0; m < H; ++m) {
      const int k = 2 * m;
      const C2 a = r0[k <= H ? k : P - k], b = r1[k <= H ? k : P - k];
      xr[m] = k <= H ? a.x - b.y : a.x + b.y;
      xi[m] = k <= H ? a.y + b.x : b.x - a.y;
    }
    LineFFT<H, +1, R>::run(xr, xi);
#pragma unroll
    for (int n = 0; n < H; ++n) (n <= N ? r0[2 * n] : r1[2 * (n - N - 1)]) = C2{xr[n], xi[n]};
    half_barrier();
#pragma unroll
    for (int m = 0; m < H; ++m) {
      const int k = 2 * m + 1;
      const C2 a = r0[k < H ? k : P - k], b = r1[k < H ? k : P - k];
      xr[m] = k < H ? a.x - b.y : a.x + b.y;
      xi[m] = k < H ? a.y + b.x : b.x - a.y;
    }
    LineFFT<H, +1, R>::run(xr, xi);
#pragma unroll
    for (int n = 0; n < H; ++n) {
      if (n > 0) rotate64<+1>(n * TW, xr[n], xi[n]);
      const C2 v = n <= N ? r0[2 * n] : r1[2 * (n - N - 1)];
      xr[n] += v.x;
      xi[n] += v.y;
    }
    const int* ch = tgt_ch + col * 8 + (z >= N ? 4 : 0);
    const size_t roff = (size_t)((z % N) * N + y) * N;
    constexpr int V = 16 / (int)sizeof(R);
#pragma unroll
    for (int b1 = 0; b1 < 2; ++b1)
#pragma unroll
      for (int b2 = 0; b2 < 2; ++b2) {
        const int gid = __ldg(ch + 2 * b1 + b2);
        if (gid < 0) continue;
        int4* o = reinterpret_cast<int4*>(unodes + (size_t)gid * N * N * N + roff);
#pragma unroll
        for (int u = 0; u < N / V; ++u) {
          int4 v;
          R* r = reinterpret_cast<R*>(&v);
#pragma unroll
          for (int j = 0; j < V; ++j) r[j] = scale * (b1 ? xi : xr)[b2 * N + u * V + j];
          o[u] = v;
        }
      }
  }
}

// ---------------------------------------------------------------------------
// Axis 0 and the products.  A CTA takes a group of target parents (consecutive
// in tile order, so they share neighbour cells) and upc units of lines (one,
// unless the groups are small: mac_units); lane = (line, k0).  Per parity of k0
// the group's source lines are copied to shared memory and, in FP32,
// transformed in place (a thread per line); a warp then takes two
// parents that are neighbours along axis 2 (or one) at a time, its lane's 27
// kernel values in registers: the pair's 36 distinct source values feed 54
// products (shared-memory bandwidth bounds the kernel with 27 reads each, and
// longer runs lost more to their short parts than they saved: 20 sparse
// problems 7.6 ms with single parents, 8.2 ms with runs).  FP32 joins two pairs
// that are neighbours along axis 1 where both exist: 48 reads for 108 products
// and a third fewer table entries to unpack; whole solves, 16^3 blocks of 16^3
// 1.487 -> 1.438 ms, three-level torus 4.33 -> 4.27 ms, two-level vector torus
// 2.13 -> 2.09 ms.  FP32 now, 16^3 blocks of 16^3 (0.65 ms): issue slots 62 %, L1
// 64 %, the FMA pipe 39 %, the ALU pipe (unpacking, addresses) 24 %, 4 warps a
// scheduler; copies, line transforms and products take turns behind barriers.
// FP64, 11 x 9 x 13 blocks (6.3 ms): the FP64 pipe 80 %.  FP32 multiplies absent
// neighbours of an item as zeros: 1.2 (that box) to 1.5 times (torus, sparse
// problems) the products that exist.  The sums are
// transformed back (a thread per line) and the two parities added.
// FP64 products take the three-multiplication form (kr (fr + fi), (kr + ki)
// fi, (ki - kr) fr) with fr + fi kept beside the sources, and skip absent cells
// one by one: the FP64 pipe is the bound.
// ---------------------------------------------------------------------------
// kOne: one unit a CTA (known at compile time: 703 us against 735 for 16^3
// blocks of 16^3, FP32).
template <typename R, int N, bool kOne>
__global__ void __launch_bounds__(kPfMacThreads, sizeof(R) == 4 ? 2 : 1)
    pf_mac_kernel(const PfGroup* __restrict__ groups, int ngroups, const PfLimits lim,
                  const uint16_t* __restrict__ items, const int* __restrict__ cell_col, const int* __restrict__ tgt_col,
                  const typename Vec2<R>::type* __restrict__ src, int nsrc, typename Vec2<R>::type* __restrict__ dst,
                  int ndst, const typename Vec2<R>::type* __restrict__ kspec, int src_stride, int dst_stride, int units) {
  using D = PfDims<N>;
  using C2 = typename Vec2<R>::type;
  constexpr int H = D::H, TW = 64 / D::P;
  constexpr bool G3 = sizeof(R) == 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int upc = kOne ? 1 : units, NW = kPfMacThreads / 32 / upc;  // warps per unit
  const int g = blockIdx.x % ngroups, sub = kOne ? 0 : threadIdx.x / 32 / NW, unit = blockIdx.x / ngroups * upc + sub;
  const PfGroup gp = groups[g];
  const int nc = gp.ncell, nt = gp.nact;
  const int tid = threadIdx.x, lane = tid & 31, warp = (tid >> 5) % NW;
  // per unit: the cells' lines (line nc is zero) and the parents' (FP64: of both parities); FP64: fr + fi
  constexpr int kT = G3 ? 2 : 1;
  const int xs = (lim.cells + 1) * kPfStride, ts = kT * lim.parents * kPfStride;
  C2* const X0 = reinterpret_cast<C2*>(smem_raw);                   // [upc][cells + 1][33]
  C2* const T0 = X0 + (size_t)upc * xs;                             // [upc][kT][parents][33]
  R* const S0 = reinterpret_cast<R*>(smem_raw + pf_sum_offset<R>(lim, upc));  // [upc][cells + 1][33]
  C2* const X = X0 + sub * xs;
  C2* const T = T0 + sub * ts;
  R* const Sm = S0 + (G3 ? sub * xs : 0);
  uint4* IT = reinterpret_cast<uint4*>(smem_raw + pf_table_offset<R>(lim, upc));  // [items][5]
  int* CC = reinterpret_cast<int*>(IT + (size_t)lim.items * (kPfItem / 8));
  int* TC = CC + lim.cells;

  for (int i = tid; i < nc; i += kPfMacThreads) CC[i] = __ldg(cell_col + gp.cell_off + i) + (int)blockIdx.y * src_stride;
  if (warp == 0) {
    X[(size_t)nc * kPfStride + lane] = C2{R(0), R(0)};
    if constexpr (G3) Sm[(size_t)nc * kPfStride + lane] = R(0);
  }
  __syncthreads();
  const C2* sbase = src + (size_t)unit * pf_halves<R>() * nsrc * 32 + lane;
  auto fill = [&](int par) {
    const C2* sp = sbase + (G3 ? (size_t)par * nsrc * 32 : 0);
    for (int c = warp; c < nc; c += NW) cp_async_complex<R>(X + c * kPfStride + lane, sp + (size_t)CC[c] * 32);
  };
  fill(0);
  for (int i = tid; i < nt; i += kPfMacThreads) TC[i] = __ldg(tgt_col + gp.row_off + i) + (int)blockIdx.y * dst_stride;
  for (int i = tid; i < gp.nitem * (kPfItem / 8); i += kPfMacThreads)
    IT[i] = __ldg(reinterpret_cast<const uint4*>(items) + (size_t)gp.item_off * (kPfItem / 8) + i);
  C2* dbase = dst + (size_t)unit * ndst * 32 + lane;
  // FP64 keeps both parities' sums and transforms them back at once (few lines
  // a group: more of them in flight); FP32 transforms and writes each parity's,
  // the second adding to the first, which leaves room for larger groups
  constexpr bool kBoth = G3;
  auto inverse = [&](int last) {
    for (int i = tid; i < upc * kT * nt * D::S; i += kPfMacThreads) {
      const int j = kOne && kT * D::S == 1 ? 0 : i / nt, m = i - j * nt, par = kBoth ? j / D::S % 2 : last;  // j: (unit, parity, line of the unit)
      C2* line = T0 + (j / D::S / kT) * ts + ((kBoth ? par * lim.parents : 0) + m) * kPfStride + (j % D::S) * H;
      R xr[H], xi[H];
#pragma unroll
      for (int k = 0; k < H; ++k) { const C2 v = line[k]; xr[k] = v.x; xi[k] = v.y; }
      LineFFT<H, +1, R>::run(xr, xi);
      if (par)
#pragma unroll
        for (int z = 1; z < H; ++z) rotate64<+1>(z * TW, xr[z], xi[z]);
#pragma unroll
      for (int z = 0; z < H; ++z) line[z] = C2{xr[z], xi[z]};
    }
  };
#pragma unroll 1
  for (int par = 0; par < 2; ++par) {
    cp_async_wait();
    if constexpr (G3) {
      // the values that this thread copied
      for (int c = warp; c < nc; c += NW) {
        const C2 v = X[c * kPfStride + lane];
        Sm[c * kPfStride + lane] = v.x + v.y;
      }
    } else {
      __syncthreads();
      for (int i = tid; i < upc * nc * D::S; i += kPfMacThreads) {
        const int j = kOne && D::S == 1 ? 0 : i / nc, c = i - j * nc;
        C2* line = X0 + (j / D::S) * xs + c * kPfStride + (j % D::S) * H;
        R xr[H], xi[H];
#pragma unroll
        for (int z = 0; z < H; ++z) { const C2 v = line[z]; xr[z] = v.x; xi[z] = v.y; }
        if (par)
          LineFFT<H, -1, R, true>::run(xr, xi);
        else
          LineFFT<H, -1, R>::run(xr, xi);
#pragma unroll
        for (int k = 0; k < H; ++k) line[k] = C2{xr[k], xi[k]};
      }
    }
    R k0[27], k1[27], k2[G3 ? 27 : 1];
    {
      const C2* kp = kspec + (((size_t)gp.level * D::U + unit) * 2 + par) * 27 * 32 + lane;
#pragma unroll
      for (int e = 0; e < 27; ++e) {
        const C2 k = __ldg(kp + e * 32);
        k0[e] = k.x;
        k1[e] = G3 ? k.x + k.y : k.y;
        if constexpr (G3) k2[e] = k.y - k.x;
      }
    }
    __syncthreads();
    C2* Tp = T + (G3 ? (size_t)par * lim.parents * kPfStride : 0) + lane;
    constexpr int NA = G3 ? 3 : 4;
    auto product = [&](R (&s)[NA], int e, const C2& f, const R& sum) {
      if constexpr (G3) {
        s[0] = fma(k0[e], sum, s[0]);
        s[1] = fma(k1[e], f.y, s[1]);
        s[2] = fma(k2[e], f.x, s[2]);
      } else {
        s[0] = fma(k0[e], f.x, s[0]);
        s[1] = fma(k0[e], f.y, s[1]);
        s[2] = fma(k1[e], f.y, s[2]);
        s[3] = fma(k1[e], f.x, s[3]);
      }
    };
    auto result = [&](const R (&s)[NA]) {
      return G3 ? C2{s[0] - s[1], s[0] + s[2]} : C2{s[0] - s[2], s[1] + s[NA - 1]};
    };
    const C2* Xl = X + lane;
    const R* Sl = Sm + lane;
    int it0 = warp;
    if constexpr (!G3) {
      for (int iq = warp; iq < gp.nquad; iq += NW) {
        const uint4* I = IT + 2 * iq * (kPfItem / 8);
        const uint4 meta = I[6];
        R a[4][NA];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int t = 0; t < NA; ++t) a[i][t] = R(0);
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          if (!(meta.y >> r & 1)) continue;  // no sources at this e0 (uniform)
          const uint4 v0 = I[2 * r], v1 = I[2 * r + 1];
          const uint32_t w[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const C2 f = Xl[(i & 1) ? w[i / 2] >> 16 : w[i / 2] & 0xFFFFu];
#pragma unroll
            for (int m = 0; m < 4; ++m) {
              const int e1 = i / 4 - m / 2, e2 = i % 4 - m % 2;
              if (e1 >= 0 && e1 < 3 && e2 >= 0 && e2 < 3) product(a[m], 9 * r + 3 * e1 + e2, f, R(0));
            }
          }
        }
        const int m0 = meta.x & 0xFFFF, m1 = meta.x >> 16;
        Tp[m0 * kPfStride] = result(a[0]);
        Tp[(m0 + 1) * kPfStride] = result(a[1]);
        Tp[m1 * kPfStride] = result(a[2]);
        Tp[(m1 + 1) * kPfStride] = result(a[3]);
      }
      it0 = 2 * gp.nquad + (warp + NW - gp.nquad % NW) % NW;  // the warps go on in turn
    }
    for (int it = it0; it < gp.nitem; it += NW) {
      uint32_t w[kPfItem / 2];
#pragma unroll
      for (int q = 0; q < kPfItem / 8; ++q) {
        const uint4 v = IT[it * (kPfItem / 8) + q];
        w[4 * q] = v.x; w[4 * q + 1] = v.y; w[4 * q + 2] = v.z; w[4 * q + 3] = v.w;
      }
      auto entry = [&](int i) { return (i & 1) ? w[i / 2] >> 16 : w[i / 2] & 0xFFFFu; };
      const uint32_t m0 = entry(36), flags = entry(38);
      R a[2][NA];
#pragma unroll
      for (int t = 0; t < NA; ++t) a[0][t] = a[1][t] = R(0);
      // all forms take a parent's 27 products in the same order
      if (entry(37) == 2) {
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          if (!(flags >> r & 1)) continue;  // no sources at this e0 (uniform)
#pragma unroll
          for (int c = 3 * r; c < 3 * r + 3; ++c)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const uint32_t o = entry(9 * q + c);
              if (G3 && o == (uint32_t)nc * kPfStride) continue;
              const C2 f = Xl[o];
              const R s = G3 ? Sl[o] : R(0);
              if (q < 3) product(a[0], 3 * c + q, f, s);
              if (q > 0) product(a[1], 3 * c + q - 1, f, s);
            }
        }
        Tp[(m0 + 1) * kPfStride] = result(a[1]);
      } else {
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          if (!(flags >> r & 1)) continue;
#pragma unroll
          for (int c = 3 * r; c < 3 * r + 3; ++c)
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              const uint32_t o = entry(9 * q + c);
              if (G3 && o == (uint32_t)nc * kPfStride) continue;
              product(a[0], 3 * c + q, Xl[o], G3 ? Sl[o] : R(0));
            }
        }
      }
      Tp[m0 * kPfStride] = result(a[0]);
    }
    __syncthreads();
    if (par == 0) fill(1);  // the second parity's copy of the sources
    if (!kBoth || par == 1) {
      inverse(par);
      __syncthreads();
      for (int m = warp; m < nt; m += NW) {
        C2 v = T[m * kPfStride + lane];
        C2* o = dbase + (size_t)TC[m] * 32;
        if (par) {  // the first parity's part: beside this one, or written by this thread
          const C2 h = kBoth ? T[((size_t)lim.parents + m) * kPfStride + lane] : *o;
          v.x += h.x;
          v.y += h.y;
        }
        *o = v;
      }
    }
  }
}
// ---------------------------------------------------------------------------
// Setup (FP64): parent kernel arrays to spectra, one axis per pass by plain
// discrete Fourier sums.  G is even in every component, so the array of a
// negative e_a is the mirror image along that axis of the positive one's: only
// the 8 arrays with e_a >= 0 are transformed, and the packing reads the others
// at negated frequencies (their negative k2 by Hermitian symmetry).
// ---------------------------------------------------------------------------
// axis 2: real rows [rows][P] -> [rows][NX]
__global__ void pf_setup_axis2(const double* __restrict__ in, double2* __restrict__ out, int P, int NX, int rows) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* w = reinterpret_cast<double2*>(smem_raw);
  double* x = reinterpret_cast<double*>(w + P);
  for (int j = threadIdx.x; j < P; j += blockDim.x) {
    double s, c;
    sincospi(2.0 * j / P, &s, &c);
    w[j] = make_double2(c, -s);
    x[j] = in[(size_t)blockIdx.x * P + j];
  }
  __syncthreads();
  for (int k = threadIdx.x; k < NX; k += blockDim.x) {
    double re = 0.0, im = 0.0;
    for (int j = 0; j < P; ++j) {
      const double2 t = w[(j * k) & (P - 1)];
      re = fma(x[j], t.x, re);
      im = fma(x[j], t.y, im);
    }
    out[(size_t)blockIdx.x * NX + k] = make_double2(re, im);
  }
}
// a strided axis of P points: in[a][j][b] -> out[a][k][b] (b < nb), block = (a, chunk of b), one thread per (b, k)
__global__ void pf_setup_axis(const double2* __restrict__ in, double2* __restrict__ out, int P, int nb) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* w = reinterpret_cast<double2*>(smem_raw);
  double2* x = w + P;  // [P]
  const int b = blockIdx.x % nb;
  const size_t a = blockIdx.x / nb;
  for (int j = threadIdx.x; j < P; j += blockDim.x) {
    double s, c;
    sincospi(2.0 * j / P, &s, &c);
    w[j] = make_double2(c, -s);
    x[j] = in[(a * P + j) * nb + b];
  }
  __syncthreads();
  for (int k = threadIdx.x; k < P; k += blockDim.x) {
    double re = 0.0, im = 0.0;
    for (int j = 0; j < P; ++j) {
      const double2 t = w[(j * k) & (P - 1)];
      re = fma(x[j].x, t.x, fma(-x[j].y, t.y, re));
      im = fma(x[j].x, t.y, fma(x[j].y, t.x, im));
    }
    out[(a * P + k) * nb + b] = make_double2(re, im);
  }
}
// [8][k0][l] -> [unit][parity][27][32] in precision R
template <typename R, int N>
__global__ void pf_setup_pack(const double2* __restrict__ in, typename Vec2<R>::type* __restrict__ out) {
  using D = PfDims<N>;
  constexpr int P = D::P, NX = D::NX;
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (size_t)D::U * 2 * 27 * 32) return;
  const int lane = i % 32, e = (i / 32) % 27, par = (i / (32 * 27)) % 2, u = (int)(i / (32 * 27 * 2));
  const int l = u * D::S + lane / D::H, k2 = l % NX;
  int k0 = 2 * (lane % D::H) + par, k1 = l / NX;
  const int e0 = e / 9 - 1, e1 = (e / 3) % 3 - 1, e2 = e % 3 - 1;
  const bool conj = e2 < 0;  // K(k0, k1, -k2) = conj K(-k0, -k1, k2)
  if ((e0 < 0) != conj) k0 = (P - k0) % P;
  if ((e1 < 0) != conj) k1 = (P - k1) % P;
  const int base = (e0 != 0) * 4 + (e1 != 0) * 2 + (e2 != 0);
  const double2 v = in[((size_t)base * P + k0) * D::L + k1 * NX + k2];
  out[i] = typename Vec2<R>::type{(R)v.x, (R)(conj ? -v.y : v.y)};
}

template <typename R, int N>
static cudaError_t setup_spectra(const double* karr, void* tmp, void* kspec, cudaStream_t s) {
  using D = PfDims<N>;
  constexpr int P = D::P, NX = D::NX;
  double2* t0 = reinterpret_cast<double2*>(tmp);
  double2* t1 = t0 + (size_t)8 * P * P * NX;
  pf_setup_axis2<<<8 * P * P, 64, P * 24, s>>>(karr, t0, P, NX, 8 * P * P);
  pf_setup_axis<<<8 * P * NX, 64, P * 32, s>>>(t0, t1, P, NX);       // axis 1: a = (e, i0), b = k2
  pf_setup_axis<<<8 * P * NX, 64, P * 32, s>>>(t1, t0, P, P * NX);   // axis 0: a = e, b = (k1, k2)
  const size_t total = (size_t)D::U * 2 * 27 * 32;
  pf_setup_pack<R, N><<<(unsigned)((total + 255) / 256), 256, 0, s>>>(t0, reinterpret_cast<typename Vec2<R>::type*>(kspec));
  return cudaGetLastError();
}

size_t pf_kernel_values(int N) { return (size_t)4 * N * (2 * N + 1) * 2 * N * 2 * 27; }
size_t pf_setup_bytes(int N) { return (size_t)2 * 16 * 8 * 4 * N * 4 * N * (2 * N + 1); }
size_t pf_parent_values(int N) { return (size_t)4 * N * (2 * N + 1) * 2 * N; }
size_t pf_source_values(int N, bool fp64) { return pf_parent_values(N) * (fp64 ? pf_halves<double>() : pf_halves<float>()); }

template <typename R>
cudaError_t launch_pf_setup(int N, const double* karr, void* tmp, void* kspec, cudaStream_t s) {
  if (N == 16) return setup_spectra<R, 16>(karr, tmp, kspec, s);
  if (N == 8) return setup_spectra<R, 8>(karr, tmp, kspec, s);
  return cudaErrorInvalidValue;
}

// Planes per CTA of the plane kernels: FP32 8 of 32 (16 at N = 8, whole
// parents), FP64 half of that: about 68 KB of shared memory.  Two CTAs an SM
// hold FP32 at N = 16 to 96 registers, of which the forward kernel spills 88
// bytes a thread and the inverse 60.
template <typename R, int N> constexpr int pf_planes() { return (N == 16 ? 8 : 16) / (sizeof(R) == 8 ? 2 : 1); }

template <typename R, int N>
static cudaError_t forward_n(const R* nodes, const int* cell_ch, int n, void* out, int ncol, cudaStream_t s) {
  constexpr int ZP = pf_planes<R, N>();
  const size_t sm = sizeof(R) * 2 * ZP * pf_plane_stride<R, N, ZP>();
  auto k = pf_forward_kernel<R, N, ZP>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  using C2 = typename Vec2<R>::type;
  k<<<n * (PfDims<N>::H / ZP), kPfPlaneThreads, sm, s>>>(nodes, cell_ch, reinterpret_cast<C2*>(out), ncol);
  if constexpr (pf_halves<R>() == 2) {
    constexpr int RC = kPfAxisThreads / PfDims<N>::S, sa = 2 * RC * kPfStride * (int)sizeof(C2);
    const long long ctas = (long long)PfDims<N>::U * ((ncol + RC - 1) / RC);
    if (ctas >= (1ll << 31)) return cudaErrorInvalidConfiguration;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(pf_axis0_kernel<R, N>, cudaFuncAttributeMaxDynamicSharedMemorySize, sa)) != cudaSuccess) return e;
    pf_axis0_kernel<R, N><<<(unsigned)ctas, kPfAxisThreads, sa, s>>>(reinterpret_cast<C2*>(out), ncol);
  }
  return cudaGetLastError();
}
template <typename R, int N>
static cudaError_t inverse_n(const void* in, const int* tgt_ch, const double* scales, int n, R* unodes, cudaStream_t s) {
  constexpr int ZP = pf_planes<R, N>();
  const size_t sm = sizeof(R) * 2 * ZP * pf_plane_stride<R, N, ZP>();
  auto k = pf_inverse_kernel<R, N, ZP>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  k<<<n * (PfDims<N>::H / ZP), kPfPlaneThreads, sm, s>>>(reinterpret_cast<const typename Vec2<R>::type*>(in), n, tgt_ch, scales,
                                                        unodes);
  return cudaGetLastError();
}
// Units per CTA of the product kernel: small groups leave most threads without
// a line to transform, so up to 8 units share a CTA while every line has a
// thread, the shared memory stays below half an SM's, and every SM gets a CTA.
template <typename R, int N>
static int mac_units(int ngroups, int ncomp, const PfLimits& lim) {
  int upc = 1;
  while (upc < 8 && 2 * upc * lim.cells * PfDims<N>::S <= kPfMacThreads && pf_smem_bytes<R>(lim, 2 * upc) <= 100 * 1024 &&
         (long long)PfDims<N>::U / (2 * upc) * ngroups * ncomp >= 152)
    upc *= 2;
  return upc;
}
template <typename R, int N>
static cudaError_t mac_n(const PfGroup* groups, int ngroups, const PfLimits& lim, const uint16_t* items, const int* cell_col,
                         const int* tgt_col, const void* src, int nsrc, void* dst, int ndst,
                         const void* kspec, int ncomp, int src_stride, int dst_stride, cudaStream_t s) {
  using C2 = typename Vec2<R>::type;
  static_assert(PfDims<N>::U % 8 == 0, "whole CTAs of 8 units");
  const int upc = mac_units<R, N>(ngroups, ncomp, lim);
  const size_t sm = pf_smem_bytes<R>(lim, upc);
  if (sm > kFlSmemBytes || (size_t)PfDims<N>::U * ngroups >= (1u << 31)) return cudaErrorInvalidConfiguration;
  auto k = upc == 1 ? pf_mac_kernel<R, N, true> : pf_mac_kernel<R, N, false>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  k<<<dim3((unsigned)(PfDims<N>::U / upc * ngroups), ncomp), kPfMacThreads, sm, s>>>(
      groups, ngroups, lim, items, cell_col, tgt_col, reinterpret_cast<const C2*>(src), nsrc, reinterpret_cast<C2*>(dst),
      ndst, reinterpret_cast<const C2*>(kspec), src_stride, dst_stride, upc);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_pf_forward(int N, const R* nodes, const int* cell_ch, int n, void* out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (N == 16) return forward_n<R, 16>(nodes, cell_ch, n, out, n, s);
  if (N == 8) return forward_n<R, 8>(nodes, cell_ch, n, out, n, s);
  return cudaErrorInvalidValue;
}
template <typename R>
cudaError_t launch_pf_mac(int N, const PfGroup* groups, int ngroups, const PfLimits& lim, const uint16_t* items,
                          const int* cell_col, const int* tgt_col, const void* src, int nsrc, void* dst,
                          int ndst, const void* kspec, int ncomp, int src_stride, int dst_stride, cudaStream_t s) {
  if (ngroups <= 0) return cudaSuccess;
  if (N == 16)
    return mac_n<R, 16>(groups, ngroups, lim, items, cell_col, tgt_col, src, nsrc, dst, ndst, kspec, ncomp, src_stride,
                        dst_stride, s);
  if (N == 8)
    return mac_n<R, 8>(groups, ngroups, lim, items, cell_col, tgt_col, src, nsrc, dst, ndst, kspec, ncomp, src_stride,
                       dst_stride, s);
  return cudaErrorInvalidValue;
}
template <typename R>
cudaError_t launch_pf_inverse(int N, const void* in, const int* tgt_ch, const double* scales, int n, R* unodes,
                              cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (N == 16) return inverse_n<R, 16>(in, tgt_ch, scales, n, unodes, s);
  if (N == 8) return inverse_n<R, 8>(in, tgt_ch, scales, n, unodes, s);
  return cudaErrorInvalidValue;
}

#define FLGF_PF_INST(R)                                                                                             \
  template cudaError_t launch_pf_setup<R>(int, const double*, void*, void*, cudaStream_t);                          \
  template cudaError_t launch_pf_forward<R>(int, const R*, const int*, int, void*, cudaStream_t);                   \
  template cudaError_t launch_pf_mac<R>(int, const PfGroup*, int, const PfLimits&, const uint16_t*, const int*,       \
                                        const int*, const void*, int, void*, int, const void*, int, int, \
                                        int, cudaStream_t);                                                         \
  template cudaError_t launch_pf_inverse<R>(int, const void*, const int*, const double*, int, R*, cudaStream_t);
FLGF_PF_INST(float)
FLGF_PF_INST(double)
#undef FLGF_PF_INST

}  // namespace flgf
