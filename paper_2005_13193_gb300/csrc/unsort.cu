// Rows of results written in bin order -> rows in the particles' own order.
// A brick kernel that follows a permutation stores every value of a particle
// at a random place of its row; with more rows than the L2 holds, each 4-byte
// store goes to DRAM as a sector of its own.  Here the brick kernel stores in
// bin order (full lines), and the rows are then put in place: eight or four at
// a time by way of whole sectors (interleave_rows, split_rows), what is left a
// few rows at a time by words (permute_rows), so that the rows being written
// stay in the L2 until their sectors are whole.
#include <algorithm>

#include "ps_internal.cuh"

namespace ps {
namespace {

constexpr int kUnsortThreads = 256, kUnsortItems = 4;

// Slots [lo, hi) that the bins hold: the others, and particles that no slot
// names, keep what their result rows held.
struct Slots {
  const int32_t* first;  // bin_offsets, NULL: all np slots
  const int32_t* last;   // bin_offsets + bins
  __device__ __forceinline__ bool has(int64_t s, int64_t np) const {
    return s < np && (!first || (s >= __ldg(first) && s < __ldg(last)));
  }
};
// Bytes of result rows in flight: well under the 129 MB L2, of which the two
// dies hold a part each (4 M particles: three rows).
constexpr int64_t kUnsortGroupBytes = 48ll << 20;

// What bounds it is the L2's rate of sectors touched, one per value: 28 to 30 us
// a float row of 4 M particles, a double row 46, gathered 18.
// Rows [blockIdx.y * group, + group): entry perm[s] of row r takes entry s of
// src row r, or (GATHER) entry s takes entry perm[s].  Rows r < n0 go to d0,
// the others to d1.
template <typename T, bool GATHER>
__global__ void __launch_bounds__(kUnsortThreads)
    permute_rows(int64_t np, const int64_t* __restrict__ perm, Slots slots,
                 const T* __restrict__ src, T* __restrict__ d0, int n0, T* __restrict__ d1,
                 int rows, int group) {
  int64_t p[kUnsortItems];
  const int64_t s0 = (int64_t)blockIdx.x * (kUnsortThreads * kUnsortItems) + threadIdx.x;
#pragma unroll
  for (int u = 0; u < kUnsortItems; ++u) {
    const int64_t s = s0 + u * kUnsortThreads;
    p[u] = slots.has(s, np) ? __ldg(perm + s) : -1;
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
ps_status permute_launch(int64_t np, const int64_t* perm, Slots slots, const T* src, T* d0, int n0,
                         T* d1, int n1, cudaStream_t st) {
  const int rows = n0 + n1;
  if (np <= 0 || rows <= 0) return PS_OK;
  const int group = (int)std::min<int64_t>(
      rows, std::max<int64_t>(1, kUnsortGroupBytes / ((int64_t)sizeof(T) * np)));
  const int64_t per = kUnsortThreads * kUnsortItems;
  const dim3 grid((unsigned)((np + per - 1) / per), (unsigned)((rows + group - 1) / group));
  permute_rows<T, GATHER><<<grid, kUnsortThreads, 0, st>>>(np, perm, slots, src, d0, n0, d1, rows,
                                                           group);
  return check_launch("permute_rows");
}

// Eight rows at a time in two passes.  permute_rows is bound by the rate of its
// single-word stores, one sector each (1.4e11 a second).  Here interleave_rows
// stores a particle's eight values as one whole sector at its own place of
// `mid` [np][8], two lanes per sector in one store, and split_rows reads `mid`
// in order and writes the rows in full lines.  Four rows alike, as half a
// sector.  256^3, 4 M particles, the whole call by words -> by sectors: second
// derivatives (18 rows) 1005 -> 747 us, velocity and gradient (12) 741 -> 582.
// `mid` is first filled with kUnnamed: split_rows leaves the rows of a place that
// still holds it alone, and marks the others in `named` for a group of four
// that follows.  It is no result in all four words: arithmetic gives the NaN
// 0x7fffffff, a position that is not finite 0x7fc00000.  The fill came later
// and takes 20 us more there (another set of positions: 846 -> 866 and 683 -> 706).
constexpr unsigned kUnnamed = 0xffffffffu;
template <int G>
__global__ void __launch_bounds__(kUnsortThreads)
    interleave_rows(int64_t np, const int64_t* __restrict__ perm, Slots slots,
                    const float* __restrict__ src, float4* __restrict__ mid) {
  const int64_t s = (int64_t)blockIdx.x * kUnsortThreads + threadIdx.x;
  int64_t p = slots.has(s, np) ? __ldg(perm + s) : -1;
  if (p >= np) p = -1;  // not a permutation: such an entry is left out
  float v[G];
#pragma unroll
  for (int r = 0; r < G; ++r) v[r] = s < np ? __ldcs(src + r * np + s) : 0.f;
  if constexpr (G == 4) {
    if (p >= 0) mid[p] = make_float4(v[0], v[1], v[2], v[3]);
  } else {
    // the even lane stores both particles' first halves, the odd lane the second
    const unsigned FULL = 0xffffffffu;
    const bool odd = threadIdx.x & 1;
    float o[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) o[r] = __shfl_xor_sync(FULL, odd ? v[r] : v[4 + r], 1);
    const int64_t q = __shfl_xor_sync(FULL, p, 1);
    const float4 own = odd ? make_float4(v[4], v[5], v[6], v[7]) : make_float4(v[0], v[1], v[2], v[3]);
    const float4 other = make_float4(o[0], o[1], o[2], o[3]);
    const int64_t pe = odd ? q : p, po = odd ? p : q;  // the even and the odd lane's particle
    if (pe >= 0) mid[2 * pe + odd] = odd ? other : own;
    if (po >= 0) mid[2 * po + odd] = odd ? own : other;
  }
}

// Rows [r0, r0 + G) of the result: rows below n0 in d0, the others in d1.  A bit
// of `named` per particle: written by a group of eight, read by one of four
// (NULL: its `mid` was filled).
template <int G>
__global__ void __launch_bounds__(kUnsortThreads)
    split_rows(int64_t np, const float4* __restrict__ mid, float* __restrict__ d0, int n0,
               float* __restrict__ d1, int r0, unsigned* named) {
  const int64_t p = (int64_t)blockIdx.x * kUnsortThreads + threadIdx.x;
  const int lane = threadIdx.x & 31;
  float4 v[G / 4];
#pragma unroll
  for (int h = 0; h < G / 4; ++h)
    v[h] = p < np ? __ldcs(mid + p * (G / 4) + h) : make_float4(0.f, 0.f, 0.f, 0.f);
  bool has = p < np && (__float_as_uint(v[0].x) & __float_as_uint(v[0].y) &
                        __float_as_uint(v[0].z) & __float_as_uint(v[0].w)) != kUnnamed;
  if (G == 8) {
    const unsigned bits = __ballot_sync(0xffffffffu, has);
    if (named && lane == 0 && p < np) named[p >> 5] = bits;
  } else if (named) {
    has = p < np && (__ldg(named + (p >> 5)) >> lane & 1);
  }
  if (!has) return;
#pragma unroll
  for (int h = 0; h < G / 4; ++h) {
    const float a[4] = {v[h].x, v[h].y, v[h].z, v[h].w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int r = r0 + 4 * h + k;
      float* dr = r < n0 ? d0 + r * np : d1 + (r - n0) * np;
      __stcs(dr + p, a[k]);
    }
  }
}

template <int G>
ps_status interleaved(int64_t np, const int64_t* perm, Slots slots, const float* src, float4* mid,
                      float* d0, int n0, float* d1, int r0, unsigned* named, cudaStream_t st) {
  const unsigned blocks = (unsigned)((np + kUnsortThreads - 1) / kUnsortThreads);
  interleave_rows<G><<<blocks, kUnsortThreads, 0, st>>>(np, perm, slots, src + r0 * np, mid);
  ps_status rc = check_launch("interleave_rows");
  if (rc) return rc;
  split_rows<G><<<blocks, kUnsortThreads, 0, st>>>(np, mid, d0, n0, d1, r0, named);
  return check_launch("split_rows");
}

// Bytes of the interleaved places: eight or four values per particle, or none.
size_t mid_bytes(int64_t np, int rows) {
  return align_up((size_t)np * (rows >= 8 ? 8 : rows >= 4 ? 4 : 0) * sizeof(float), 256);
}

}  // namespace

// src: the n0 + n1 rows in a workspace of ps_unsort_workspace_size bytes, of
// which the rest holds a group's interleaved values.
ps_status unsort_launch(int64_t np, const int64_t* perm, const int32_t* offs, int64_t nbins,
                        float* src, float* d0, int n0, float* d1, int n1, cudaStream_t st) {
  const int rows = n0 + n1;
  if (np <= 0 || rows <= 0) return PS_OK;
  const Slots slots{offs, offs + nbins};
  float4* mid = reinterpret_cast<float4*>(reinterpret_cast<char*>(src) +
                                          align_up((size_t)np * rows * sizeof(float), 256));
  ps_status rc = PS_OK;
  int r = 0;
  if (rows >= 4)
    rc = check_cuda(cudaMemsetAsync(mid, 0xff, mid_bytes(np, rows), st), "row places memset");
  unsigned* named = rows >= 8 ? reinterpret_cast<unsigned*>(reinterpret_cast<char*>(mid) +
                                                              mid_bytes(np, rows))
                               : nullptr;
  for (; !rc && rows - r >= 8; r += 8)
    rc = interleaved<8>(np, perm, slots, src, mid, d0, n0, d1, r, named, st);
  if (!rc && rows - r >= 4) {
    rc = interleaved<4>(np, perm, slots, src, mid, d0, n0, d1, r, named, st);
    r += 4;
  }
  if (rc || r == rows) return rc;
  const int m0 = r < n0 ? n0 - r : 0;  // rows still due in d0
  return permute_launch<float, false>(np, perm, slots, src + (int64_t)r * np,
                                      m0 ? d0 + (int64_t)r * np : nullptr, m0,
                                      m0 ? d1 : d1 + (int64_t)(r - n0) * np, rows - r - m0, st);
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
    return to_bins ? permute_launch<T, true>(np, perm, Slots{}, s, d, rows, nullptr, 0, st)
                   : permute_launch<T, false>(np, perm, Slots{}, s, d, rows, nullptr, 0, st);
  };
  return elem_bytes == 4 ? go(float{}) : go(double{});
}

extern "C" size_t ps_unsort_workspace_size(int64_t np, int rows) {
  if (np < 0 || rows < 0) return 0;
  return align_up((size_t)np * (size_t)rows * sizeof(float), 256) +
         mid_bytes(np, rows) + (rows >= 8 ? align_up((size_t)np / 8 + 4, 256) : 0);
}
