// Adjoint of the binned interpolation (Sec. 2.2, Operations 2 and 3 transposed):
// the cotangent's scatter onto the field by bricks of cells.  (The position
// gradients are the unbinned kernel's, over particles in bin order: interp.cu.)
//
// The scatter adds g_vel * basis weights to 64 nodes of three components per
// particle.  Straight to global memory that is 192 atomics per particle, 8
// sectors of the L2's atomic units per row (256^3, 4 M particles: 4447 us).
// Here a block of two warps takes a brick's particles in turn.  Warp w owns the
// halo planes of parity w: of the four planes of any stencil two are its own,
// and its 32 lanes are their 32 nodes, so it adds to a float4 per node in
// shared memory by plain loads and stores, in order within the warp, and no two
// adds ever meet.  The brick's sums then go to the workspace as they are, and a
// second kernel adds up, for every node of the field, the one or two bricks
// per axis that reach it; without a workspace (or where the bricks do not tile
// the grid) they go to the field by atomics, one per node and component
// (1411 us in all at that size, bound by the atomics' rate, about 1.8e11 a
// second).  Measured there: 4447 us of atomics -> 549 us for the bricks and
// 171 us for the sums (875 and 306 us before a round's records held the products
// of the x and y weights, read one particle ahead, and before a thread summed all
// three components of its node).  What bounds it is the chain load, add, store of
// a warp's float4, one per particle.
#include <algorithm>

#include "brick.cuh"

namespace ps {
namespace {

constexpr int kSegment = 512;    // particles of one brick that one block takes
constexpr int kMinSegment = 16;  // fewer go to global memory directly
constexpr int kScatterThreads = 64;

struct ScatterArgs {
  GridArgs g;
  BrickArgs b;
  int S[3], SX, PS;  // halo extents, row and plane stride in nodes
  int64_t np;
  double ih32[3];
  const double* pos;
  const int64_t* perm;
  const int32_t* offs;
  const float* gvel;
  float* gfield;
  float* sums;  // [nbins][3][S2][S1][SX], or NULL: atomics on gfield
  int32_t* status;
};

// Records of a round's particles: the 16 products of the x and y weights (in
// the order of the lanes), the z weights in the order 0, 2, 1, 3 (a lane finds
// its plane's at 2 * first row + plane), (g_u, g_v, g_w, twice the stencil's
// first node plus the parity of its first plane; -1 outside the halo, -2 not
// finite).
struct ScatterRecs {
  float4 wxy[kScatterThreads][4];
  float4 bz[kScatterThreads], gi[kScatterThreads];
};

__device__ __forceinline__ void add_global(const ScatterArgs& a, int cx, int cy, int cz, float w,
                                           const float4& g) {
  const int nx = padded_to_node(cx, a.g.n[0]), ny = padded_to_node(cy, a.g.n[1]),
            nz = padded_to_node(cz, a.g.n[2]);
  const int64_t vol = (int64_t)a.g.n[0] * a.g.n[1] * a.g.n[2];
  float* o = a.gfield + ((int64_t)nz * a.g.n[1] + ny) * a.g.n[0] + nx;
  atomicAdd(o, w * g.x);
  atomicAdd(o + vol, w * g.y);
  atomicAdd(o + 2 * vol, w * g.z);
}

// Slots [lo, hi) of brick `bin` by the block, into the brick's sums in the
// workspace (to_sums, also when there are few or none) or into the field.
__device__ __forceinline__ void scatter_segment(const ScatterArgs& a, int bin, int lo, int hi,
                                                bool to_sums, float4* acc, ScatterRecs& R) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int li = lane & 3, lj = (lane >> 2) & 3, lk = lane >> 4;
  const int nbx = a.b.nb[0], nby = a.b.nb[1];
  const int bz = bin / (nbx * nby), rem = bin - bz * nbx * nby, by = rem / nbx, bx = rem - by * nbx;
  const int P0[3] = {bx * a.b.B[0], by * a.b.B[1], bz * a.b.B[2]};
  const bool staged = to_sums || hi - lo >= kMinSegment;
  if (staged) {
    for (int e = tid; e < a.PS * a.S[2]; e += kScatterThreads)
      acc[e] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  float4* mine = acc + 2 * lk * a.PS + lj * a.SX + li;  // + the warp's first plane of a stencil
  const float* wz = reinterpret_cast<const float*>(R.bz) + lk;
  const float* wxy = reinterpret_cast<const float*>(R.wxy) + (lane & 15);
  for (unsigned c0 = lo; c0 < (unsigned)hi; c0 += kScatterThreads) {  // (to beyond 2^31)
    const int m = (int)min((unsigned)kScatterThreads, (unsigned)hi - c0);
    if (tid < m) {
      const int64_t p = a.perm ? a.perm[c0 + tid] : (int64_t)(c0 + tid);
      float4 gi;
      gi.x = a.gvel[p];
      gi.y = a.gvel[a.np + p];
      gi.z = a.gvel[2 * a.np + p];
      int cell[3];
      float t[3];
      bool ok = true;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const double x = a.pos[d * a.np + p];
        const long long s = __double2ll_rd(__dmul_rn(x, a.ih32[d]));
        cell[d] = (int)(s >> 32);
        t[d] = (float)((unsigned)s >> 8) * 0x1p-24f;
        if ((unsigned)cell[d] >= (unsigned)a.g.n[d])
          ok &= locate(x, a.g.inv_h[d], a.g.n[d], cell[d], t[d]);
      }
      const int l0 = cell[0] - P0[0], l1 = cell[1] - P0[1], l2 = cell[2] - P0[2];
      int first = -1;
      if (!ok) {
        first = -2;
        flag_status(a.status, PS_DEV_NONFINITE_POS, p);
      } else if (staged && (unsigned)l0 <= (unsigned)(a.S[0] - 4) &&
                 (unsigned)l1 <= (unsigned)(a.S[1] - 4) && (unsigned)l2 <= (unsigned)(a.S[2] - 4)) {
        first = 2 * (l2 * a.PS + l1 * a.SX + l0) + (l2 & 1);
      }
      gi.w = __int_as_float(first);
      float b[4], by4[4];
      qbasis(t[0], b);
      qbasis(t[1], by4);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        R.wxy[tid][j] = make_float4(b[0] * by4[j], b[1] * by4[j], b[2] * by4[j], b[3] * by4[j]);
      qbasis(t[2], b);
      R.bz[tid] = make_float4(zscale(b[0]), zscale(b[2]), zscale(b[1]), zscale(b[3]));
      R.gi[tid] = gi;
    }
    __syncthreads();
    // the records of one particle ahead of the sums
    float4 gn = R.gi[0];
    float wn = wxy[0];
#pragma unroll 2
    for (int i = 0; i < m; ++i) {
      const float4 g = gn;
      const float wp = wn;
      const int first = __float_as_int(g.w);
      if (first >= 0) {  // (uniform over the warp)
        const int row0 = (first & 1) ^ warp;  // the stencil's first plane of this warp
        float4* q = mine + ((first >> 1) + row0 * a.PS);
        float4 v = *q;
        const float w = wp * wz[4 * i + 2 * row0];
        if (i + 1 < m) {
          gn = R.gi[i + 1];
          wn = wxy[16 * (i + 1)];
        }
        v.x = fmaf(w, g.x, v.x);
        v.y = fmaf(w, g.y, v.y);
        v.z = fmaf(w, g.z, v.z);
        *q = v;
        __syncwarp();  // the next stencil's nodes may be other lanes'
      } else {
        if (first == -1) {  // planes warp and warp + 2 of the stencil
          const int64_t p = a.perm ? a.perm[c0 + i] : (int64_t)(c0 + i);
          int cell[3];
          float t;
#pragma unroll
          for (int d = 0; d < 3; ++d)
            locate(a.pos[d * a.np + p], a.g.inv_h[d], a.g.n[d], cell[d], t);
          add_global(a, cell[0] + li, cell[1] + lj, cell[2] + warp + 2 * lk,
                     wp * wz[4 * i + 2 * warp], g);
        }
        if (i + 1 < m) {
          gn = R.gi[i + 1];
          wn = wxy[16 * (i + 1)];
        }
      }
    }
    __syncthreads();  // the records are refilled, or the sums are complete
  }
  if (!staged) return;
  if (lo >= hi) __syncthreads();  // (no round above ordered the cleared sums)
  if (to_sums) {
    const int e1 = a.PS * a.S[2];
    float* o = a.sums + (int64_t)bin * 3 * e1;
    for (int e = tid; e < e1; e += kScatterThreads) {
      const float4 v = acc[e];
      o[e] = v.x;
      o[e1 + e] = v.y;
      o[2 * e1 + e] = v.z;
    }
    return;
  }
  // the sums to the field: 16 (or 32) lanes along a row
  const int W = a.S[0] <= 16 ? 16 : 32, tx = tid & (W - 1);
  const int64_t vol = (int64_t)a.g.n[0] * a.g.n[1] * a.g.n[2];
  int nx = P0[0] + tx - 1;  // node of padded index P0 + tx
  nx = nx < 0 ? nx + a.g.n[0] : nx % a.g.n[0];
  const int rows = a.S[1] * a.S[2];
  for (int r = tid / W; r < rows; r += kScatterThreads / W) {
    const int lz = r / a.S[1], ly = r - lz * a.S[1];
    int ny = P0[1] + ly - 1, nz = P0[2] + lz - 1;
    ny = ny < 0 ? ny + a.g.n[1] : ny % a.g.n[1];
    nz = nz < 0 ? nz + a.g.n[2] : nz % a.g.n[2];
    if (tx < a.S[0]) {
      const float4 v = acc[lz * a.PS + ly * a.SX + tx];
      float* o = a.gfield + ((int64_t)nz * a.g.n[1] + ny) * a.g.n[0] + nx;
      if (v.x != 0.f) atomicAdd(o, v.x);
      if (v.y != 0.f) atomicAdd(o + vol, v.y);
      if (v.z != 0.f) atomicAdd(o + 2 * vol, v.z);
    }
  }
}

// Blocks [0, nbins): a brick's first kSegment particles.  The blocks after
// them cut all slots into ranges of kSegment and take what bricks hold beyond
// their first kSegment (nothing, at a uniform density below it), so that a
// crowded brick is shared by many blocks.
__global__ void __launch_bounds__(kScatterThreads) scatter_bricks(const __grid_constant__ ScatterArgs a) {
  extern __shared__ __align__(16) float4 acc_sh[];
  __shared__ ScatterRecs R;
  const int nbins = (int)a.b.nbins;
  const int64_t blk = blockIdx.x;
  if (blk < nbins) {
    const int beg = a.offs[blk];
    const int end = (int)min((int64_t)a.offs[blk + 1], (int64_t)beg + kSegment);
    if (beg < end || a.sums) scatter_segment(a, (int)blk, beg, end, a.sums != nullptr, acc_sh, R);
    return;
  }
  const int s0 = (int)((blk - nbins) * kSegment);
  const int s1 = (int)min((int64_t)s0 + kSegment, a.np);
  int lo = 0, hi = nbins;  // offs[lo] <= s0 < offs[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (a.offs[mid] <= s0) lo = mid;
    else hi = mid;
  }
  for (int b = lo; b < nbins && a.offs[b] < s1; ++b) {
    const int from = (int)max((int64_t)s0, (int64_t)a.offs[b] + kSegment);
    const int to = min(s1, a.offs[b + 1]);
    if (from < to) {
      scatter_segment(a, b, from, to, false, acc_sh, R);
      __syncthreads();
    }
  }
}

// gfield += the bricks' sums.  Node i of an axis lies in the halo of the bricks
// b with b B - 1 <= i <= b B + B + 1 (mod n): floor((i + 1) / B), and the one
// before where i + 1 - b B <= 2.  A block per (z, y) row (the bricks along y
// and z and their offsets are the block's), a thread per node and all three
// components.
struct Reach {
  int brick[2], l[2];
  bool two;
};
__device__ __forceinline__ Reach reach(int node, int B, int nb) {
  const int P = node + 1, b = P / B, l = P - b * B;
  Reach r;
  r.brick[0] = b == nb ? 0 : b;  // P = n: halo index 0 of brick 0
  r.l[0] = l;
  r.two = l <= 2;
  r.brick[1] = b == 0 ? nb - 1 : b - 1;
  r.l[1] = l + B;
  return r;
}
__global__ void __launch_bounds__(128) gather_sums(const __grid_constant__ ScatterArgs a) {
  const int nx = a.g.n[0], ny = a.g.n[1], z = blockIdx.x / ny, y = blockIdx.x - z * ny;
  const int e1 = a.PS * a.S[2];
  const Reach rz = reach(z, a.b.B[2], a.b.nb[2]), ry = reach(y, a.b.B[1], a.b.nb[1]);
  const int64_t vol = (int64_t)a.g.n[2] * ny * nx;
  float* o = a.gfield + (int64_t)blockIdx.x * nx;
  const float* base[2][2];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j)
      base[i][j] = a.sums + ((int64_t)rz.brick[i] * a.b.nb[1] + ry.brick[j]) * a.b.nb[0] * 3 * e1 +
                   rz.l[i] * a.PS + ry.l[j] * a.SX;
  for (int x = threadIdx.x; x < nx; x += blockDim.x) {
    const Reach rx = reach(x, a.b.B[0], a.b.nb[0]);
    const int x0 = rx.brick[0] * 3 * e1 + rx.l[0], x1 = rx.brick[1] * 3 * e1 + rx.l[1];
    float s[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) s[c] = o[c * vol + x];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j)
        if ((i == 0 || rz.two) && (j == 0 || ry.two)) {
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            s[c] += __ldg(base[i][j] + c * e1 + x0);
            if (rx.two) s[c] += __ldg(base[i][j] + c * e1 + x1);
          }
        }
#pragma unroll
    for (int c = 0; c < 3; ++c) o[c * vol + x] = s[c];
  }
}

// Bricks whose sums gather_sums finds: they tile the grid, each axis is long
// enough that a brick's halo does not meet itself, and at most two reach a node.
bool sums_apply(const ps_grid* g, const int32_t brick[3]) {
  for (int d = 0; d < 3; ++d)
    if (brick[d] < 3 || g->n[d] % brick[d] || g->n[d] < 2 * brick[d]) return false;
  return true;
}
int sums_row(int S0) { return S0 + ((12 - S0 % 8) % 8); }

}  // namespace

// The scatter of a binned cotangent (three components) onto a cleared field;
// *done stays false where a brick's sums do not fit in shared memory.
ps_status scatter_bricks_launch(const ps_grid* grid, const int32_t brick[3], int64_t np,
                                const double* pos, const int64_t* perm, const int32_t* offs,
                                const float* gvel, float* gfield, int32_t* status,
                                void* ws, size_t ws_bytes, cudaStream_t st, bool* done) {
  *done = false;
  ScatterArgs a{};
  ps_status rc = make_brick_args(grid, brick, &a.b);
  if (rc) return rc;
  a.g = make_grid_args(grid);
  for (int d = 0; d < 3; ++d) {
    a.S[d] = a.b.B[d] + 3;
    a.ih32[d] = a.g.inv_h[d] * 4294967296.0;
  }
  if (a.S[0] > 32) return PS_OK;
  // rows of 4 (mod 8) nodes: the eight lanes of a load phase (four nodes of
  // two rows) read different banks
  a.SX = sums_row(a.S[0]);
  a.PS = a.SX * a.S[1];
  const size_t smem = (size_t)a.PS * a.S[2] * sizeof(float4);
  if (smem + sizeof(ScatterRecs) > 226 * 1024 || a.b.nbins > (1ll << 30)) return PS_OK;
  a.np = np;
  a.pos = pos;
  a.perm = perm;
  a.offs = offs;
  a.gvel = gvel;
  a.gfield = gfield;
  a.status = status;
  if (smem > 40 * 1024) {
    rc = check_cuda(cudaFuncSetAttribute(scatter_bricks,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
                    "scatter smem attribute");
    if (rc) return rc;
  }
  *done = true;
  const size_t need = ps_backward_workspace_size(grid, brick);
  if (need && ws && ws_bytes >= need && (reinterpret_cast<uintptr_t>(ws) & 255) == 0)
    a.sums = static_cast<float*>(ws);
  const int64_t blocks = a.b.nbins + (np + kSegment - 1) / kSegment;
  scatter_bricks<<<(unsigned)blocks, kScatterThreads, smem, st>>>(a);
  if ((rc = check_launch("scatter_bricks")) || !a.sums) return rc;
  gather_sums<<<(unsigned)(a.g.n[1] * a.g.n[2]), 128, 0, st>>>(a);
  return check_launch("gather_sums");
}

}  // namespace ps

extern "C" size_t ps_backward_workspace_size(const ps_grid* grid, const int32_t brick[3]) {
  ps::BrickArgs b;
  if (ps::validate_grid(grid) || ps::make_brick_args(grid, brick, &b)) return 0;
  if (!ps::sums_apply(grid, brick) || brick[0] + 3 > 32) return 0;
  const size_t per = (size_t)ps::sums_row(brick[0] + 3) * (brick[1] + 3) * (brick[2] + 3);
  return ps::align_up((size_t)b.nbins * 3 * per * sizeof(float), 256);
}
