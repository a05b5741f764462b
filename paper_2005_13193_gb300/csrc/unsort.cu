// Rows of results written in bin order -> rows in the particles' own order.
// A brick kernel that follows a permutation stores every value of a particle
// at a random place of its row; with more rows than the L2 holds, each 4-byte
// store goes to DRAM as a sector of its own.  Here the brick kernel stores in
// bin order (full lines), and the rows are then scattered a few at a time, so
// that the group of rows being written stays in the L2 until its sectors are
// whole.  256^3, 4 M particles: 28 to 30 us a float row; a double row 46 us
// scattered.
#include <algorithm>

#include "ps_internal.cuh"

namespace ps {
namespace {

constexpr int kUnsortThreads = 256, kUnsortItems = 4;
// Bytes of result rows in flight: well under the 129 MB L2, of which the two
// dies hold a part each (4 M particles: three rows).
constexpr int64_t kUnsortGroupBytes = 48ll << 20;

// Rows [blockIdx.y * group, + group): entry perm[s] of row r takes entry s of
// src row r, or (GATHER) entry s takes entry perm[s].  Rows r < n0 go to d0,
// the others to d1.
template <typename T, bool GATHER>
__global__ void __launch_bounds__(kUnsortThreads)
    permute_rows(int64_t np, const int64_t* __restrict__ perm, const T* __restrict__ src,
                 T* __restrict__ d0, int n0, T* __restrict__ d1, int rows, int group) {
  int64_t p[kUnsortItems];
  const int64_t s0 = (int64_t)blockIdx.x * (kUnsortThreads * kUnsortItems) + threadIdx.x;
#pragma unroll
  for (int u = 0; u < kUnsortItems; ++u) {
    const int64_t s = s0 + u * kUnsortThreads;
    p[u] = s < np ? __ldg(perm + s) : -1;
    if (p[u] >= np) p[u] = -1;  // not a permutation: such an entry is left out
  }
  const int r1 = min(rows, ((int)blockIdx.y + 1) * group);
  for (int r = blockIdx.y * group; r < r1; ++r) {
    const T* sr = src + r * np;
    T* dr = r < n0 ? d0 + r * np : d1 + (r - n0) * np;
    T v[kUnsortItems];
#pragma unroll
    for (int u = 0; u < kUnsortItems; ++u)
      if (p[u] >= 0) v[u] = GATHER ? __ldg(sr + p[u]) : __ldcs(sr + s0 + u * kUnsortThreads);
#pragma unroll
    for (int u = 0; u < kUnsortItems; ++u)
      if (p[u] >= 0) dr[GATHER ? s0 + u * kUnsortThreads : p[u]] = v[u];
  }
}

template <typename T, bool GATHER>
ps_status permute_launch(int64_t np, const int64_t* perm, const T* src, T* d0, int n0, T* d1,
                         int n1, cudaStream_t st) {
  const int rows = n0 + n1;
  if (np <= 0 || rows <= 0) return PS_OK;
  const int group = (int)std::min<int64_t>(
      rows, std::max<int64_t>(1, kUnsortGroupBytes / ((int64_t)sizeof(T) * np)));
  const int64_t per = kUnsortThreads * kUnsortItems;
  const dim3 grid((unsigned)((np + per - 1) / per), (unsigned)((rows + group - 1) / group));
  permute_rows<T, GATHER><<<grid, kUnsortThreads, 0, st>>>(np, perm, src, d0, n0, d1, rows, group);
  return check_launch("permute_rows");
}

}  // namespace

ps_status unsort_launch(int64_t np, const int64_t* perm, const float* src, float* d0, int n0,
                        float* d1, int n1, cudaStream_t st) {
  return permute_launch<float, false>(np, perm, src, d0, n0, d1, n1, st);
}

}  // namespace ps

using namespace ps;

extern "C" ps_status ps_permute_rows(int64_t np, int rows, int elem_bytes, const int64_t* perm,
                                     const void* src, void* dst, int to_bins, void* stream) {
  if (np < 0 || rows < 0 || rows > 64)
    return fail(PS_ERR_INVALID_ARG, "np >= 0 and 0..64 rows are taken");
  if (elem_bytes != 4 && elem_bytes != 8)
    return fail(PS_ERR_INVALID_ARG, "elements of 4 or 8 bytes are taken");
  if (np == 0 || rows == 0) return PS_OK;
  if (!perm || !src || !dst || src == dst)
    return fail(PS_ERR_INVALID_ARG, "perm, src and dst are required, src != dst");
  cudaStream_t st = as_stream(stream);
  auto go = [&](auto tag) {
    using T = decltype(tag);
    const T* s = static_cast<const T*>(src);
    T* d = static_cast<T*>(dst);
    return to_bins ? permute_launch<T, true>(np, perm, s, d, rows, nullptr, 0, st)
                   : permute_launch<T, false>(np, perm, s, d, rows, nullptr, 0, st);
  };
  return elem_bytes == 4 ? go(float{}) : go(double{});
}

extern "C" size_t ps_unsort_workspace_size(int64_t np, int rows) {
  if (np < 0 || rows < 0) return 0;
  return align_up((size_t)np * (size_t)rows * sizeof(float), 256);
}
