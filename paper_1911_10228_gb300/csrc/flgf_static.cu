// flgf_convolve_static: the exact block convolution without any device
// allocation.
//
// Who needs it: callers that must not allocate device memory while they
// compute -- code that runs inside a memory pool owned by another framework,
// latency-critical loops that cannot afford cudaMalloc's implicit
// synchronisation, or processes whose device memory is fully reserved up
// front.  The block-set API allocates its spectra at flgf_blockset_create;
// this entry point instead keeps its scratch (the forward and accumulated
// spectra and the launch lists) in one file-scope __device__ array of fixed
// size that every GPU loading the library holds until the process exits.
//
// It computes u = h^2 (G * f) over at most kStaticMaxBlocks blocks whose
// octree has a single level (all blocks within a 4 x 4 x 4 box aligned to
// even coordinates), so every pair is an exact zero-padded FFT convolution:
// the products between parents of flgf_solve (parent.cu; at most 8 parents,
// neighbours of each other), with their scratch in the static array.  27 blocks
// of 16^3, FP32, a call: 122 us with the child-pair kernel (104 us of it), 50 us.
#include <algorithm>
#include <array>
#include <cstring>
#include <mutex>
#include <vector>

#include "../../include/flgf.h"
#include "common.cuh"
#include "internal.h"

namespace {

using namespace flgf;

constexpr int kStaticMaxBlocks = 32;
constexpr size_t kSpecBytes = (size_t)kStaticMaxBlocks * nfreq(16) * 16;  // half-transformed spectra of 8 parents (complex double, N = 16: 8.65 MB)
constexpr size_t kListBytes = 512 * 1024;
constexpr size_t kScratchBytes = 3 * kSpecBytes + kListBytes;             // sources (FP64: two halves) and targets, ~27.3 MB

// Shared by every call on a device; see the header for the concurrency rule.
static __device__ __align__(256) unsigned char g_scratch[kScratchBytes];

constexpr int kMaxDevices = 64;
std::mutex g_mu;
void* g_scratch_ptr[kMaxDevices] = {nullptr};

// Device address of g_scratch on the current device (set up once per device).
cudaError_t scratch_address(void** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_scratch);
    if (e != cudaSuccess) return e;
    g_scratch_ptr[dev] = p;
  }
  *out = g_scratch_ptr[dev];
  return cudaSuccess;
}

// Launch lists of one call, passed to the list-writing kernel by value (the
// kernel's parameters are copied at launch, so nothing is read from host
// memory afterwards).  At most 8 parents, all sources and targets: the blocks
// lie in one aligned 4x4x4 box.  Laid out as in the scratch array.
constexpr int kMaxParents = 8;
struct __align__(16) StaticLists {
  uint16_t items[kMaxParents * kPfItem];
  int child[kMaxParents * 8];
  int col[kMaxParents];
  double scale[kMaxParents];
  PfGroup group;
};
static_assert(sizeof(StaticLists) <= kListBytes, "lists fit the scratch");
static_assert(sizeof(StaticLists) % sizeof(int) == 0, "copied by words");

__global__ void static_lists_kernel(const StaticLists L, int* __restrict__ dl) {
  for (int i = threadIdx.x; i < (int)(sizeof(L) / sizeof(int)); i += blockDim.x) dl[i] = reinterpret_cast<const int*>(&L)[i];
}

}  // namespace

extern "C" int flgf_convolve_static(flgf_ctx* ctx, int nblk, const int32_t* coords, const void* f, void* u,
                                    double h) {
  CtxView cv;
  if (!flgf::ctx_view(ctx, &cv)) return FLGF_EINVAL;
  auto bad = [&](int code, const char* m) {
    flgf::ctx_set_error(ctx, m);
    return code;
  };
  if (nblk < 1 || nblk > kStaticMaxBlocks || !coords || !f || !u || !(h > 0.0))
    return bad(FLGF_EINVAL, "convolve_static: need 1..32 blocks, coordinates, device f and u, h > 0");
  if (reinterpret_cast<uintptr_t>(f) % 16 || reinterpret_cast<uintptr_t>(u) % 16)
    return bad(FLGF_EINVAL, "convolve_static: f and u must be 16-byte aligned");
  const int N = cv.N;
  // one octree level: the parents of all blocks lie within one block of each other
  std::array<int, 3> plo = {INT32_MAX, INT32_MAX, INT32_MAX}, phi = {INT32_MIN, INT32_MIN, INT32_MIN};
  std::vector<std::array<int, 3>> c(nblk);
  for (int b = 0; b < nblk; ++b)
    for (int a = 0; a < 3; ++a) {
      c[b][a] = coords[3 * b + a];
      if (c[b][a] < -(1 << 19) || c[b][a] >= (1 << 19)) return bad(FLGF_EINVAL, "convolve_static: coordinate range");
      plo[a] = std::min(plo[a], c[b][a] >> 1);
      phi[a] = std::max(phi[a], c[b][a] >> 1);
    }
  for (int a = 0; a < 3; ++a)
    if (phi[a] - plo[a] > 1)
      return bad(FLGF_EINVAL, "convolve_static: blocks must lie in one 4x4x4 box aligned to even coordinates");
  {
    std::vector<std::array<int, 3>> s = c;
    std::sort(s.begin(), s.end());
    if (std::adjacent_find(s.begin(), s.end()) != s.end()) return bad(FLGF_EMESH, "convolve_static: duplicate block");
  }
  // the box's blocks by their place in it, and its parents
  int at[4][4][4];
  std::fill(&at[0][0][0], &at[0][0][0] + 64, -1);
  for (int b = 0; b < nblk; ++b) at[c[b][0] - 2 * plo[0]][c[b][1] - 2 * plo[1]][c[b][2] - 2 * plo[2]] = b;
  StaticLists L;
  std::memset(&L, 0, sizeof(L));
  int col[2][2][2], np = 0;
  for (int p = 0; p < 8; ++p) {
    const int x = p >> 2, y = (p >> 1) & 1, z = p & 1;
    bool any = false;
    for (int a = 0; a < 8; ++a) {
      L.child[np * 8 + a] = at[2 * x + (a >> 2)][2 * y + ((a >> 1) & 1)][2 * z + (a & 1)];
      any |= L.child[np * 8 + a] >= 0;
    }
    col[x][y][z] = any ? np++ : -1;
  }
  // one item per parent: its neighbours in the box (the entries of PfGroup's items)
  for (int p = 0; p < 8; ++p) {
    const int q[3] = {p >> 2, (p >> 1) & 1, p & 1}, m = col[q[0]][q[1]][q[2]];
    if (m < 0) continue;
    uint16_t* it = L.items + m * kPfItem;
    for (int i = 0; i < 36; ++i) it[i] = (uint16_t)(33 * np);
    it[36] = (uint16_t)m;
    it[37] = 1;
    for (int e = 0; e < 27; ++e) {
      const int x = q[0] + e / 9 - 1, y = q[1] + (e / 3) % 3 - 1, z = q[2] + e % 3 - 1;
      if (x < 0 || x > 1 || y < 0 || y > 1 || z < 0 || z > 1 || col[x][y][z] < 0) continue;
      it[9 * (e % 3) + e / 3] = (uint16_t)(33 * col[x][y][z]);
      it[38] |= (uint16_t)(1 << (e / 9));
    }
    L.col[m] = m;
    L.scale[m] = h * h;
  }
  L.group = PfGroup{np, np, np, 0, 0, 0, 0, 0};
  const PfLimits lim{np, np, np};

  void* base = nullptr;
  cudaError_t e = scratch_address(&base);
  if (e != cudaSuccess) return bad(FLGF_ECUDA, cudaGetErrorString(e));
  unsigned char* sp = static_cast<unsigned char*>(base);
  void* spec = sp;
  void* acc = sp + 2 * kSpecBytes;
  unsigned char* dl = sp + 3 * kSpecBytes;
  cudaStream_t s = cv.stream;
  // the lists travel as kernel parameters, written into the scratch on the stream
  static_lists_kernel<<<1, 256, 0, s>>>(L, reinterpret_cast<int*>(dl));
  e = cudaGetLastError();
  const StaticLists* d = reinterpret_cast<const StaticLists*>(dl);
  auto run = [&](auto zero) {
    using R = decltype(zero);
    cudaError_t r = launch_pf_forward<R>(N, static_cast<const R*>(f), d->child, np, spec, s);
    if (r == cudaSuccess)
      r = launch_pf_mac<R>(N, &d->group, 1, lim, d->items, d->col, d->col, spec, np, acc, np, cv.pspec, 1, 0, 0, s);
    return r == cudaSuccess ? launch_pf_inverse<R>(N, acc, d->child, d->scale, np, static_cast<R*>(u), s) : r;
  };
  if (e == cudaSuccess) e = cv.fp64 ? run(0.0) : run(0.0f);
  if (e != cudaSuccess) return bad(FLGF_ECUDA, cudaGetErrorString(e));
  return FLGF_OK;
}
