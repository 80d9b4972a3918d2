// On-device refinement of one mesh level (Sec. 3.1, Eq. ref_crit): a block of
// level l is refined where its source exceeds alpha^(L_R - l) times the
// largest |source| on the level.  The refined blocks' children form the next
// level, and the closure of the mesh needs every refined block's 26 same-level
// neighbours (Sec. 3: the buffer around a refined region), so the neighbours
// missing from the level are listed too.  Outputs are in Morton order.
//
// Morton order: blocks compare by the key that interleaves the bits of
// (x + 2^20, y + 2^20, z + 2^20), bit i of x at key bit 3i + 2, of y at 3i + 1,
// of z at 3i (|coordinates| < 2^20, 21 bits per axis).  Bit 63 carries a
// block's flag.
//
// The step is bound by launches and host round trips, not by its data (16^3
// blocks: the 67 MB of source are read in 10 us), so: the level's keys are
// sorted once, by a radix sort of 8 bits a pass over the bits that can vary;
// the children of the sorted flagged blocks are then in order as they are
// (halving the coordinates keeps the order of the keys); of the neighbours only
// those missing from the level are listed and sorted.  4096 blocks with 459
// flagged, none of whose neighbours is missing, a call: 1.65 ms with a stable
// split of five launches per varying bit of three sorts, 459 x 26 candidates
// sorted and an allocation per scratch array; 0.18 ms (84 us of kernels and two
// round trips; a third where neighbours are missing).
#include <algorithm>
#include <cstdint>
#include <utility>

#include "flgf.h"
#include "internal.h"

namespace flgf {

namespace {

constexpr int kMgThreads = 1024;
// keys per CTA of a radix pass: 1024 for lists of up to 2^18 keys (more CTAs:
// the passes are latency-bound), 4096 beyond (fewer digit counts to scan)
constexpr int mg_tile(size_t n) { return n <= (1u << 18) ? 1024 : 4096; }
constexpr size_t kMgKeepBytes = 64u << 20;  // scratch kept by the context between calls
constexpr int kMgDigits = 256;
constexpr int kMgCoordBias = 1 << 20;    // coordinates + bias are in [0, 2^21)
constexpr int kMgMaxKeys = 1 << 24;
constexpr uint64_t kMgFlag = 1ull << 63;

__host__ __device__ inline uint64_t spread3(uint32_t v) {
  uint64_t x = v & 0x1fffffu;
  x = (x | (x << 32)) & 0x1f00000000ffffull;
  x = (x | (x << 16)) & 0x1f0000ff0000ffull;
  x = (x | (x << 8)) & 0x100f00f00f00f00full;
  x = (x | (x << 4)) & 0x10c30c30c30c30c3ull;
  x = (x | (x << 2)) & 0x1249249249249249ull;
  return x;
}
__host__ __device__ inline uint32_t compact3(uint64_t x) {
  x &= 0x1249249249249249ull;
  x = (x | (x >> 2)) & 0x10c30c30c30c30c3ull;
  x = (x | (x >> 4)) & 0x100f00f00f00f00full;
  x = (x | (x >> 8)) & 0x1f0000ff0000ffull;
  x = (x | (x >> 16)) & 0x1f00000000ffffull;
  x = (x | (x >> 32)) & 0x1fffffull;
  return (uint32_t)x;
}
__host__ __device__ inline uint64_t morton_key(int x, int y, int z) {
  return (spread3((uint32_t)(x + kMgCoordBias)) << 2) | (spread3((uint32_t)(y + kMgCoordBias)) << 1) |
         spread3((uint32_t)(z + kMgCoordBias));
}
__device__ inline void morton_decode(uint64_t k, int32_t* c) {
  c[0] = (int32_t)compact3(k >> 2) - kMgCoordBias;
  c[1] = (int32_t)compact3(k >> 1) - kMgCoordBias;
  c[2] = (int32_t)compact3(k) - kMgCoordBias;
}

// What the host needs to know of a level.
struct MgInfo {
  unsigned long long maxbits;  // largest |f| (bits of a non-negative number order like it)
  int lo[3], hi[3];            // range of the coordinates
  uint32_t bad, nflag, nparent, ncand, nbuf;  // nparent: flagged blocks, each coordinate once
};

__global__ void info_init_kernel(MgInfo* info) {
  *info = MgInfo{0ull, {1 << 20, 1 << 20, 1 << 20}, {-(1 << 20), -(1 << 20), -(1 << 20)}, 0u, 0u, 0u, 0u, 0u};
}

__device__ __forceinline__ unsigned long long abs_bits(float v) { return (unsigned long long)__float_as_uint(v); }
__device__ __forceinline__ unsigned long long abs_bits(double v) { return (unsigned long long)__double_as_longlong(v); }
template <typename R> __device__ __forceinline__ double from_bits(unsigned long long b);
template <> __device__ __forceinline__ double from_bits<float>(unsigned long long b) { return (double)__uint_as_float((unsigned)b); }
template <> __device__ __forceinline__ double from_bits<double>(unsigned long long b) { return __longlong_as_double((long long)b); }

// max |f| over each block (one CTA per block; NaN counts as absent, as in fmax),
// the level's maximum and coordinate range, the block's key; bad = 1 when a
// coordinate is outside (-2^19, 2^19) (children must fit the keys)
template <typename R>
__global__ void __launch_bounds__(256) block_kernel(const R* __restrict__ f, int n3, const int32_t* __restrict__ coords,
                                                    R* __restrict__ bmax, uint64_t* __restrict__ keys, MgInfo* info) {
  __shared__ R red[8];
  const R* b = f + (size_t)blockIdx.x * n3;
  R m = R(0);
  if (reinterpret_cast<uintptr_t>(f) % 16 == 0) {  // a block is a multiple of 16 bytes
    constexpr int V = 16 / (int)sizeof(R);
    for (int i = threadIdx.x; i < n3 / V; i += 256) {
      const int4 q = __ldg(reinterpret_cast<const int4*>(b) + i);
      const R* r = reinterpret_cast<const R*>(&q);
#pragma unroll
      for (int j = 0; j < V; ++j) m = fmax(m, fabs(r[j]));
    }
  } else {
    for (int i = threadIdx.x; i < n3; i += 256) m = fmax(m, fabs(b[i]));
  }
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) m = fmax(m, red[w]);
    bmax[blockIdx.x] = m;
    if (m > R(0)) atomicMax(&info->maxbits, abs_bits(m));
    int c[3];
    for (int a = 0; a < 3; ++a) {
      c[a] = coords[3 * (size_t)blockIdx.x + a];
      if (c[a] <= -(kMgCoordBias >> 1) || c[a] >= (kMgCoordBias >> 1)) {
        info->bad = 1u;
        c[a] = 0;
      }
      if (c[a] < info->lo[a]) atomicMin(&info->lo[a], c[a]);
      if (c[a] > info->hi[a]) atomicMax(&info->hi[a], c[a]);
    }
    keys[blockIdx.x] = morton_key(c[0], c[1], c[2]);
  }
}

// the flags (compared in FP64), also into bit 63 of the keys, and their number
template <typename R>
__global__ void flag_kernel(const R* __restrict__ bmax, int n, double rel, uint8_t* __restrict__ flags,
                            uint64_t* __restrict__ keys, MgInfo* info) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const double top = from_bits<R>(info->maxbits);
  const bool v = i < n && top > 0.0 && (double)bmax[i] > rel * top;
  if (i < n) {
    flags[i] = v;
    if (v) keys[i] |= kMgFlag;
  }
  const unsigned w = __ballot_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0 && w) atomicAdd(&info->nflag, (uint32_t)__popc(w));
}

// Exclusive scan over the CTA (kMgThreads threads, one value each, replaced by
// its prefix); returns the total.
__device__ __forceinline__ uint32_t block_scan(uint32_t& v, uint32_t* ws) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t x = v;
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += t;
  }
  if (lane == 31) ws[warp] = x;
  __syncthreads();
  if (warp == 0) {
    uint32_t y = ws[lane];
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= o) y += t;
    }
    ws[32 + lane] = y;
  }
  __syncthreads();
  const uint32_t total = ws[63];
  v = x - v + (warp ? ws[32 + warp - 1] : 0u);
  __syncthreads();
  return total;
}

__device__ __forceinline__ uint32_t radix_digit(uint64_t k, int shift) {
  return (uint32_t)((k & ~kMgFlag) >> shift) & (kMgDigits - 1);
}

// Radix pass, 8 bits at `shift`: digit counts per tile [digit][tile], one CTA's
// exclusive scan of them, stable scatter.
__global__ void __launch_bounds__(kMgThreads) radix_count_kernel(const uint64_t* __restrict__ keys, int n, int shift,
                                                                 uint32_t* __restrict__ counts, int ntiles, int tile) {
  __shared__ uint32_t h[kMgDigits];
  if (threadIdx.x < kMgDigits) h[threadIdx.x] = 0;
  __syncthreads();
  for (int j = 0; j < tile; j += kMgThreads) {
    const int i = blockIdx.x * tile + j + threadIdx.x;
    if (i < n) atomicAdd(&h[radix_digit(keys[i], shift)], 1u);
  }
  __syncthreads();
  if (threadIdx.x < kMgDigits) counts[(size_t)threadIdx.x * ntiles + blockIdx.x] = h[threadIdx.x];
}
__global__ void __launch_bounds__(kMgThreads) scan_kernel(uint32_t* __restrict__ v, int n, uint32_t* __restrict__ total) {
  __shared__ uint32_t ws[64];
  uint32_t carry = 0;
  for (int base = 0; base < n; base += 4 * kMgThreads) {
    uint32_t x[4], sum = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int i = base + 4 * (int)threadIdx.x + j;
      x[j] = i < n ? v[i] : 0u;
      sum += x[j];
    }
    uint32_t at = sum;
    const uint32_t t = block_scan(at, ws);
    at += carry;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int i = base + 4 * (int)threadIdx.x + j;
      if (i < n) v[i] = at;
      at += x[j];
    }
    carry += t;
  }
  if (total && threadIdx.x == 0) *total = carry;
}
__global__ void __launch_bounds__(kMgThreads) radix_scatter_kernel(const uint64_t* __restrict__ in, int n, int shift,
                                                                   const uint32_t* __restrict__ offs, int ntiles, int tile,
                                                                   uint64_t* __restrict__ out) {
  __shared__ uint32_t at[kMgDigits];           // next slot of each digit
  __shared__ uint16_t cnt[32][kMgDigits];      // per warp, then its exclusive prefix over the warps
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x < kMgDigits) at[threadIdx.x] = offs[(size_t)threadIdx.x * ntiles + blockIdx.x];
  for (int j = 0; j < tile; j += kMgThreads) {
    const int i = blockIdx.x * tile + j + threadIdx.x;
    if (blockIdx.x * tile + j >= n) break;  // uniform
    for (int q = threadIdx.x; q < 32 * kMgDigits; q += kMgThreads) cnt[0][q] = 0;
    __syncthreads();
    const uint64_t k = i < n ? in[i] : 0ull;
    const uint32_t d = i < n ? radix_digit(k, shift) : kMgDigits;  // 256: past the end
    const unsigned same = __match_any_sync(0xffffffffu, d);
    const uint32_t rank = __popc(same & ((1u << lane) - 1u));
    if (d < kMgDigits && rank == 0) cnt[warp][d] = (uint16_t)__popc(same);
    __syncthreads();
    if (threadIdx.x < kMgDigits) {
      uint32_t run = 0;
      for (int w = 0; w < 32; ++w) {
        const uint32_t c = cnt[w][threadIdx.x];
        cnt[w][threadIdx.x] = (uint16_t)run;
        run += c;
      }
      cnt[0][threadIdx.x] = (uint16_t)run;  // warp 0's prefix is zero: its slot carries the total
    }
    __syncthreads();
    if (d < kMgDigits) out[at[d] + (warp ? cnt[warp][d] : 0u) + rank] = k;
    __syncthreads();
    if (threadIdx.x < kMgDigits) at[threadIdx.x] += cnt[0][threadIdx.x];
    __syncthreads();
  }
}

// mark[i] = 1 where sorted key i carries the flag as the first flagged one of
// its coordinates (flagged = 1: the parents of the children), or is the first of
// its run of equal keys (flagged = 0: neighbours)
__device__ __forceinline__ bool marked(const uint64_t* __restrict__ keys, int i, int flagged) {
  const uint64_t k = keys[i];
  if (!flagged) return i == 0 || keys[i - 1] != k;
  if (!(k & kMgFlag)) return false;
  for (int j = i - 1; j >= 0 && ((keys[j] ^ k) & ~kMgFlag) == 0; --j)
    if (keys[j] & kMgFlag) return false;
  return true;
}
__global__ void mark_kernel(const uint64_t* __restrict__ keys, int n, int flagged, uint32_t* __restrict__ mark) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) mark[i] = marked(keys, i, flagged);
}

// children of the flagged blocks in the order of their sorted keys
__global__ void children_kernel(const uint64_t* __restrict__ keys, int n, const uint32_t* __restrict__ rank,
                                int32_t* __restrict__ out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x, i = t / 8, a = t % 8;
  if (i >= n || !marked(keys, i, 1)) return;
  int32_t c[3];
  morton_decode(keys[i] & ~kMgFlag, c);
  int32_t* o = out + 3 * ((size_t)rank[i] * 8 + a);
  o[0] = 2 * c[0] + (a >> 2);
  o[1] = 2 * c[1] + ((a >> 1) & 1);
  o[2] = 2 * c[2] + (a & 1);
}

// keys of the flagged blocks' neighbours that are not blocks of the level (any order)
__global__ void missing_kernel(const uint64_t* __restrict__ keys, int n, uint64_t* __restrict__ out, MgInfo* info) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x, i = t / 32, e = t % 32;  // a warp per block
  if (i >= n || !(keys[i] & kMgFlag)) return;                                   // uniform
  bool miss = e < 27 && e != 13;
  uint64_t k = 0;
  if (miss) {
    int32_t c[3];
    morton_decode(keys[i] & ~kMgFlag, c);
    k = morton_key(c[0] + e / 9 - 1, c[1] + (e / 3) % 3 - 1, c[2] + e % 3 - 1);
    int lo = 0, hi = n;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if ((keys[mid] & ~kMgFlag) < k) lo = mid + 1; else hi = mid;
    }
    miss = !(lo < n && (keys[lo] & ~kMgFlag) == k);
  }
  const unsigned w = __ballot_sync(0xffffffffu, miss);
  if (!w) return;
  uint32_t base = 0;
  if (e == 0) base = atomicAdd(&info->ncand, (uint32_t)__popc(w));
  base = __shfl_sync(0xffffffffu, base, 0);
  if (miss) out[base + __popc(w & ((1u << e) - 1u))] = k;
}

__global__ void unique_kernel(const uint64_t* __restrict__ keys, int n, const uint32_t* __restrict__ rank,
                              int32_t* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n && marked(keys, i, 0)) morton_decode(keys[i], out + 3 * (size_t)rank[i]);
}

inline int ceil_div(size_t n, int t) { return (int)((n + t - 1) / t); }

// stable sort of keys[0..n) by their low `bits` bits (result in *keys; *other and counts are scratch)
void sort_keys(uint64_t** keys, uint64_t** other, int n, int bits, uint32_t* counts, cudaStream_t s) {
  if (n <= 1) return;
  const int tile = mg_tile(n), nt = ceil_div((size_t)n, tile);
  for (int shift = 0; shift < bits; shift += 8) {
    radix_count_kernel<<<nt, kMgThreads, 0, s>>>(*keys, n, shift, counts, nt, tile);
    scan_kernel<<<1, kMgThreads, 0, s>>>(counts, kMgDigits * nt, nullptr);
    radix_scatter_kernel<<<nt, kMgThreads, 0, s>>>(*keys, n, shift, counts, nt, tile, *other);
    std::swap(*keys, *other);
  }
}

}  // namespace

template <typename R>
static cudaError_t refine_level(int N, const R* f, int nblk, const int32_t* coords, double rel, uint8_t* flags,
                                int32_t* children, int32_t* buffer, int* counts, MgScratch& keep, cudaStream_t s) {
  counts[0] = counts[1] = 0;
  // one array: level keys (two), neighbour keys (two), ranks, digit counts, block maxima, info
  const size_t n = (size_t)nblk, ncap = 26 * n;
  auto up = [](size_t b) { return (b + 255) / 256 * 256; };
  const size_t o_lvl0 = 0, o_lvl1 = o_lvl0 + up(8 * n), o_c0 = o_lvl1 + up(8 * n), o_c1 = o_c0 + up(8 * ncap);
  const size_t o_rank = o_c1 + up(8 * ncap), o_cnt = o_rank + up(4 * ncap);
  const size_t o_max = o_cnt + up(4 * (size_t)kMgDigits * std::max(ceil_div(ncap, mg_tile(ncap)), ceil_div(std::min<size_t>(ncap, 1u << 18), 1024))), o_info = o_max + up(sizeof(R) * n);
  cudaError_t e = cudaSuccess;
  if (keep.bytes < o_info + 256) {
    cudaFree(keep.ptr);
    keep = MgScratch();
    e = cudaMalloc(&keep.ptr, o_info + 256);
    if (e != cudaSuccess) return e;
    keep.bytes = o_info + 256;
  }
  char* base = (char*)keep.ptr;
  uint64_t* lvl = (uint64_t*)(base + o_lvl0);
  uint64_t* lvl1 = (uint64_t*)(base + o_lvl1);
  uint64_t* cand = (uint64_t*)(base + o_c0);
  uint64_t* cand1 = (uint64_t*)(base + o_c1);
  uint32_t* rank = (uint32_t*)(base + o_rank);
  uint32_t* cnt = (uint32_t*)(base + o_cnt);
  R* bmax = (R*)(base + o_max);
  MgInfo* info = (MgInfo*)(base + o_info);
  MgInfo h{};
  auto read_info = [&]() {
    cudaError_t r = cudaGetLastError();
    if (r == cudaSuccess) r = cudaMemcpyAsync(&h, info, sizeof(h), cudaMemcpyDeviceToHost, s);
    return r == cudaSuccess ? cudaStreamSynchronize(s) : r;
  };
  info_init_kernel<<<1, 1, 0, s>>>(info);
  block_kernel<R><<<nblk, 256, 0, s>>>(f, N * N * N, coords, bmax, lvl, info);
  flag_kernel<R><<<ceil_div(n, 256), 256, 0, s>>>(bmax, nblk, rel, flags, lvl, info);
  e = read_info();
  if (e == cudaSuccess && h.bad) e = cudaErrorInvalidValue;
  if (e == cudaSuccess && h.nflag > 0) {
    // key bits that can vary among the level's blocks and their neighbours
    int bits = 1;
    for (int a = 0; a < 3; ++a) {
      const uint32_t x = (uint32_t)(h.lo[a] - 1 + kMgCoordBias) ^ (uint32_t)(h.hi[a] + 1 + kMgCoordBias);
      int b = 0;
      while (x >> b) ++b;
      bits = std::max(bits, 3 * b);
    }
    sort_keys(&lvl, &lvl1, nblk, bits, cnt, s);
    mark_kernel<<<ceil_div(n, 256), 256, 0, s>>>(lvl, nblk, 1, rank);
    scan_kernel<<<1, kMgThreads, 0, s>>>(rank, nblk, &info->nparent);
    children_kernel<<<ceil_div(8 * n, 256), 256, 0, s>>>(lvl, nblk, rank, children);
    missing_kernel<<<ceil_div(32 * n, 256), 256, 0, s>>>(lvl, nblk, cand, info);
    e = read_info();
    const int nc = (int)h.ncand;
    if (e == cudaSuccess && nc > 0) {
      sort_keys(&cand, &cand1, nc, bits, cnt, s);
      mark_kernel<<<ceil_div((size_t)nc, 256), 256, 0, s>>>(cand, nc, 0, rank);
      scan_kernel<<<1, kMgThreads, 0, s>>>(rank, nc, &info->nbuf);
      unique_kernel<<<ceil_div((size_t)nc, 256), 256, 0, s>>>(cand, nc, rank, buffer);
      e = read_info();
    }
    if (e == cudaSuccess) {
      counts[0] = 8 * (int)h.nparent;
      counts[1] = (int)h.nbuf;
    }
  }
  if (keep.bytes > kMgKeepBytes) {
    cudaFree(keep.ptr);
    keep = MgScratch();
  }
  return e;
}

cudaError_t launch_refine_level(int N, int prec_fp64, const void* f, int nblk, const int32_t* coords, double rel,
                                uint8_t* flags, int32_t* children, int32_t* buffer, int* counts, MgScratch& keep,
                                cudaStream_t s) {
  if ((size_t)nblk * 26 > (size_t)kMgMaxKeys) return cudaErrorInvalidValue;
  return prec_fp64 ? refine_level<double>(N, (const double*)f, nblk, coords, rel, flags, children, buffer, counts, keep, s)
                   : refine_level<float>(N, (const float*)f, nblk, coords, rel, flags, children, buffer, counts, keep, s);
}

}  // namespace flgf
