// One brick of particles by the warps of a block, each on its own: the body of
// the single-field kernels (quad.cu) and of the many-field ones (batch_step.cu).
//
// The brick's coefficient halo (the union of the stencils of its cells,
// (B+3)^3 nodes) is brought into shared memory by one tensor copy (nodes,
// planar FP32) or by plain loads, in the coefficients' own layout: float4 (u,
// v, w, 0) per node, three planes of floats, or 16-bit nodes beside their rows'
// scales (planar 16-bit coefficients are widened to float4).  Each warp takes
// 32 of the brick's particles at a time:
//
//  1  lane i loads particle i's position (the next 32 are loaded before the
//     current ones are processed), locates it exactly (FP64 index arithmetic)
//     and takes a slot: particles are dealt to the quads of lanes so that the
//     quads of one shared-memory load phase read different banks;
//  2  eight particles at a time, a quad of lanes per particle, lane k owning
//     stencil z-row k: the 16 nodes of the row go into registers, the lane
//     sums its (y, x) terms, the quad its four rows.  Heun step: the predictor
//     is located in FP32 from the stage-1 cell, and when it stays in that cell
//     (about 80% of particles at Courant numbers near 0.1) the second sum
//     reuses the nodes held in registers;
//  3  the results return to lane i by shuffles, which finishes the particle:
//     FP64 position update, the next step's bin, full-width stores.
//
// The location, the update and the stores run once per particle, not once per
// (particle, axis) or per quad, and nothing is exchanged between warps: the
// only block barrier publishes the copy's mbarrier.  Figures in quad.cu.
//
// Particles whose stencil is not inside the staged halo (stale bins, a
// predictor that left the brick, bricks below the staging threshold, a halo
// copy that did not complete in time) read their nodes from global memory, so
// results never depend on the bins being fresh.
#pragma once

#include "staged.cuh"

namespace ps {
namespace {

// Halo geometry.  CT > 0: the compile-time 8^3 brick (11 nodes per axis) with
// rows of CT nodes: 14 for float4 nodes (planes of 154 = 2 mod 8 nodes), 12 for
// 16-bit nodes (planes of 132 = 4 mod 16 nodes) and for planar floats (planes
// of 132 = 4 mod 32 words); CT = 0 reads the launch arguments.
template <int CT> struct QGeo {
  static constexpr int Sx = 11, Sy = 11, Sz = 11, SX = CT, PS = CT * 11;
  __device__ __forceinline__ explicit QGeo(const StagedArgs&) {}
};
template <> struct QGeo<0> {
  int Sx, Sy, Sz, SX, PS;
  __device__ __forceinline__ explicit QGeo(const StagedArgs& a)
      : Sx(a.S[0]), Sy(a.S[1]), Sz(a.S[2]), SX(a.SX), PS(a.PS) {}
};

// Planar FP32 coefficients keep three planes of floats in shared memory.
template <typename Tc> struct IsPlanar { static constexpr bool value = false; };
template <> struct IsPlanar<float> { static constexpr bool value = true; };

// Bytes of one halo, a multiple of 128 (16-bit nodes: followed at a 128-byte
// boundary by the rows' float4 scales).
__host__ __device__ constexpr int scale_off_bytes(int Sz, int PS) {
  return (Sz * PS * 8 + 127) & ~127;
}
template <typename Tc>
__host__ __device__ constexpr int halo_bytes(int Sz, int Sy, int PS) {
  return ((IsNode16<Tc>::value  ? scale_off_bytes(Sz, PS) + Sz * Sy * 16
           : IsPlanar<Tc>::value ? 3 * Sz * PS * 4
                                 : Sz * PS * 16) +
          127) & ~127;
}

// The 16 nodes (j, i) of one stencil z-row from the staged halo: `node` the
// row's first node, `row` its halo row (for the scales of 16-bit nodes: each
// value is widened and multiplied by its row's power-of-two scale, exact).
template <typename Tc, int CT>
__device__ __forceinline__ void fetch_halo(float v[16][3], const unsigned char* halo, int node,
                                           int row, const QGeo<CT>& geo) {
  if constexpr (IsNode16<Tc>::value) {
    const Tc* hp = reinterpret_cast<const Tc*>(halo) + node;
    const float4* sp =
        reinterpret_cast<const float4*>(halo + scale_off_bytes(geo.Sz, geo.PS)) + row;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float4 sc = sp[j];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const Tc n = hp[j * geo.SX + i];
        v[4 * j + i][0] = __fmul_rn(node16_value(n.v[0]), sc.x);
        v[4 * j + i][1] = __fmul_rn(node16_value(n.v[1]), sc.y);
        v[4 * j + i][2] = __fmul_rn(node16_value(n.v[2]), sc.z);
      }
    }
  } else if constexpr (IsPlanar<Tc>::value) {
    const float* hp = reinterpret_cast<const float*>(halo) + node;
    const int cs = geo.Sz * geo.PS;
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < 3; ++c) v[4 * j + i][c] = hp[c * cs + j * geo.SX + i];
  } else {
    const float4* hp = reinterpret_cast<const float4*>(halo) + node;
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 q = hp[j * geo.SX + i];
        v[4 * j + i][0] = q.x;
        v[4 * j + i][1] = q.y;
        v[4 * j + i][2] = q.z;
      }
  }
}
// The same nodes from global memory (padded stencil start = cell).
template <typename Tc>
__device__ __forceinline__ void fetch_global(float v[16][3], const int cell[3], int k,
                                             const GridArgs& g, const Tc* __restrict__ coef,
                                             const float* __restrict__ scale) {
  const int Pz = cell[2] + k;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if constexpr (IsNode4<Tc>::value) {
      const int64_t row = (int64_t)Pz * g.m[1] + cell[1] + j;
      if constexpr (IsNode16<Tc>::value) {
        const float4 sc = __ldg(reinterpret_cast<const float4*>(scale) + row);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const Tc n = coef[row * g.rx + cell[0] + i];
          v[4 * j + i][0] = __fmul_rn(node16_value(n.v[0]), sc.x);
          v[4 * j + i][1] = __fmul_rn(node16_value(n.v[1]), sc.y);
          v[4 * j + i][2] = __fmul_rn(node16_value(n.v[2]), sc.z);
        }
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 q = __ldg(reinterpret_cast<const float4*>(coef) + row * g.rx + cell[0] + i);
          v[4 * j + i][0] = q.x;
          v[4 * j + i][1] = q.y;
          v[4 * j + i][2] = q.z;
        }
      }
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < 3; ++c)
          v[4 * j + i][c] = (float)load_coef<Tc>(coef, scale, g, c, Pz, cell[1] + j, cell[0] + i);
    }
  }
}

// Six times the uniform cubic B-spline weights (Sec. 2.2, Operation 2) and
// their derivatives, with every rounding explicit, so that each instantiation
// evaluates them identically.  With s = 1 - t: s^3, 4 + t^2 (3t - 6), the same
// in s, t^3.  The factors 1/6 of the three axes are applied once, on the z
// weight, as the other kernels apply them: 1/6 rounded to FP32 on each axis, in
// all 8.9e-8 above 1/216.  (The FP32 solves' pole and gain round so that their
// coefficients come out about as much low, and a velocity's error against 64
// bits is 7.9e-8 of the rms at 512^3; with 1/216 itself it is 1.2e-7.)
__device__ __forceinline__ float b_outer(float r) { return __fmul_rn(__fmul_rn(r, r), r); }
__device__ __forceinline__ float b_inner(float r) {
  return __fmaf_rn(__fmul_rn(r, r), __fmaf_rn(3.f, r, -6.f), 4.f);
}
__device__ __forceinline__ void qbasis(float t, float b[4]) {
  const float s = __fsub_rn(1.f, t);
  b[0] = b_outer(s);
  b[1] = b_inner(t);
  b[2] = b_inner(s);
  b[3] = b_outer(t);
}
__device__ __forceinline__ float d_inner(float r) { return __fmul_rn(r, __fmaf_rn(9.f, r, -12.f)); }
__device__ __forceinline__ void qdbasis(float t, float d[4]) {
  const float s = __fsub_rn(1.f, t);
  d[0] = __fmul_rn(__fmul_rn(s, s), -3.f);
  d[1] = d_inner(t);
  d[2] = -d_inner(s);
  d[3] = __fmul_rn(__fmul_rn(t, t), 3.f);
}
// d2 b / dt2 (piecewise linear: the spline is twice continuously
// differentiable, Sec. 2.2).
__device__ __forceinline__ void qddbasis(float t, float d[4]) {
  d[0] = __fmaf_rn(-6.f, t, 6.f);
  d[1] = __fmaf_rn(18.f, t, -12.f);
  d[2] = __fmaf_rn(-18.f, t, 6.f);
  d[3] = __fmul_rn(6.f, t);
}
// (1/6)^3 as above in two factors, since no single float is that near: the first one
// short, so that its products with the constants of the derivatives are exact and cost
// nothing, the second a multiplication.
constexpr float kZ0 = 1365.f / 2048.f;
constexpr double kSixth3 = (double)(1.f / 6.f) * (double)(1.f / 6.f) * (double)(1.f / 6.f);
constexpr float kZ1 = (float)(kSixth3 / (double)kZ0);
static_assert((double)kZ0 * (double)kZ1 / kSixth3 - 1.0 < 1e-10 &&
                  1.0 - (double)kZ0 * (double)kZ1 / kSixth3 < 1e-10,
              "the two factors give (1/6)^3");
__device__ __forceinline__ float zscale(float b) { return __fmul_rn(__fmul_rn(b, kZ0), kZ1); }
// Weight k of the z axis alone (a lane's z-row), scaled, and its first and second
// derivative: in r = s for even k, t for odd k.
__device__ __forceinline__ float zbasis(float t, int k) {
  const float r = (k & 1) ? t : __fsub_rn(1.f, t);
  const bool in = k == 1 || k == 2;
  const float b = __fmaf_rn(__fmul_rn(r, r), in ? __fmaf_rn(3.f, r, -6.f) : r, in ? 4.f : 0.f);
  return zscale(b);  // (with kZ0 in the constants a Heun step took 4% longer)
}
__device__ __forceinline__ float zdbasis(float t, int k) {
  const float r = (k & 1) ? t : __fsub_rn(1.f, t);
  const bool in = k == 1 || k == 2;
  const float q = __fmaf_rn(in ? 9.f * kZ0 : 3.f * kZ0, r, in ? -12.f * kZ0 : 0.f);
  return __fmul_rn(__fmul_rn((k & 1) ? r : -r, q), kZ1);
}
__device__ __forceinline__ float zddbasis(float t, int k) {
  const float r = (k & 1) ? t : __fsub_rn(1.f, t);
  const bool in = k == 1 || k == 2;
  return __fmul_rn(__fmaf_rn(in ? 18.f * kZ0 : 6.f * kZ0, r, in ? -12.f * kZ0 : 0.f), kZ1);
}

// z sum over the quad of one value (xor butterfly: every lane ends with the
// same bits) and of a packed pair.
__device__ __forceinline__ float quad_add(float v) {
  v = __fadd_rn(v, __shfl_xor_sync(FULL, v, 1));
  return __fadd_rn(v, __shfl_xor_sync(FULL, v, 2));
}

// Sum of the quad's stencil with the basis at (t_x, t_y, t_z): every lane
// returns the three components, with the same bits in all four lanes.  GRAD
// also returns the three derivatives (in cells): out[3 r + c], r = value,
// d/dx, d/dy, d/dz.
template <bool GRAD>
__device__ __forceinline__ void quad_sum(const float v[16][3], const float t[3], int k,
                                         float* out) {
  float bx[4], by[4];
  qbasis(t[0], bx);
  qbasis(t[1], by);
  const float bz = zbasis(t[2], k);
  float dbx[4], dby[4], dbz = 0.f;
  if (GRAD) {
    qdbasis(t[0], dbx);
    qdbasis(t[1], dby);
    dbz = zdbasis(t[2], k);
  }
  float A = 0.f, Bx = 0.f, By = 0.f;
  // u and v as packed pairs (two FP32 operations per instruction, each
  // rounded as its scalar form), w alone
  float2 A2 = make_float2(0.f, 0.f), Bx2 = A2, By2 = A2;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float2 vr[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) vr[i] = make_float2(v[4 * j + i][0], v[4 * j + i][1]);
    float2 sx2 = __fmul2_rn(make_float2(bx[0], bx[0]), vr[0]);
#pragma unroll
    for (int i = 1; i < 4; ++i) sx2 = __ffma2_rn(make_float2(bx[i], bx[i]), vr[i], sx2);
    A2 = j == 0 ? __fmul2_rn(make_float2(by[0], by[0]), sx2)
                : __ffma2_rn(make_float2(by[j], by[j]), sx2, A2);
    float sx = __fmul_rn(bx[0], v[4 * j][2]);
#pragma unroll
    for (int i = 1; i < 4; ++i) sx = __fmaf_rn(bx[i], v[4 * j + i][2], sx);
    A = j == 0 ? __fmul_rn(by[0], sx) : __fmaf_rn(by[j], sx, A);
    if (GRAD) {
      float2 dx2 = __fmul2_rn(make_float2(dbx[0], dbx[0]), vr[0]);
#pragma unroll
      for (int i = 1; i < 4; ++i) dx2 = __ffma2_rn(make_float2(dbx[i], dbx[i]), vr[i], dx2);
      Bx2 = __ffma2_rn(make_float2(by[j], by[j]), dx2, Bx2);
      By2 = __ffma2_rn(make_float2(dby[j], dby[j]), sx2, By2);
      float dx = __fmul_rn(dbx[0], v[4 * j][2]);
#pragma unroll
      for (int i = 1; i < 4; ++i) dx = __fmaf_rn(dbx[i], v[4 * j + i][2], dx);
      Bx = __fmaf_rn(by[j], dx, Bx);
      By = __fmaf_rn(dby[j], sx, By);
    }
  }
  auto row = [&](int r, float w, float2 uv, float c) {
    const float2 q = group_sum2<4>(__fmul2_rn(make_float2(w, w), uv));
    out[3 * r] = q.x;
    out[3 * r + 1] = q.y;
    out[3 * r + 2] = quad_add(__fmul_rn(w, c));
  };
  row(0, bz, A2, A);
  if (GRAD) {
    row(1, bz, Bx2, Bx);
    row(2, bz, By2, By);
    row(3, dbz, A2, A);
  }
}

// The six second derivatives (in cells^-2) of the three components: out[3 e +
// c], e = xx, yy, zz, xy, xz, yz; every lane of the quad returns them.
__device__ __forceinline__ void quad_sum_hess(const float v[16][3], const float t[3], int k,
                                              float* out) {
  float bx[4], by[4], dbx[4], dby[4], ddbx[4], ddby[4];
  qbasis(t[0], bx);
  qbasis(t[1], by);
  qdbasis(t[0], dbx);
  qdbasis(t[1], dby);
  qddbasis(t[0], ddbx);
  qddbasis(t[1], ddby);
  const float bz = zbasis(t[2], k);
  const float dbz = zdbasis(t[2], k), ddbz = zddbasis(t[2], k);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    // y sums of the x sums: A = by s0, Bx = by s1, By = dby s0, Cxx = by s2,
    // Cyy = ddby s0, Cxy = dby s1 (s0, s1, s2: x sums with b, b', b'')
    float A = 0.f, Bx = 0.f, By = 0.f, Cxx = 0.f, Cyy = 0.f, Cxy = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float s0 = __fmul_rn(bx[0], v[4 * j][c]), s1 = __fmul_rn(dbx[0], v[4 * j][c]),
            s2 = __fmul_rn(ddbx[0], v[4 * j][c]);
#pragma unroll
      for (int i = 1; i < 4; ++i) {
        s0 = __fmaf_rn(bx[i], v[4 * j + i][c], s0);
        s1 = __fmaf_rn(dbx[i], v[4 * j + i][c], s1);
        s2 = __fmaf_rn(ddbx[i], v[4 * j + i][c], s2);
      }
      A = __fmaf_rn(by[j], s0, A);
      Bx = __fmaf_rn(by[j], s1, Bx);
      By = __fmaf_rn(dby[j], s0, By);
      Cxx = __fmaf_rn(by[j], s2, Cxx);
      Cyy = __fmaf_rn(ddby[j], s0, Cyy);
      Cxy = __fmaf_rn(dby[j], s1, Cxy);
    }
    out[c] = quad_add(__fmul_rn(bz, Cxx));
    out[3 + c] = quad_add(__fmul_rn(bz, Cyy));
    out[6 + c] = quad_add(__fmul_rn(ddbz, A));
    out[9 + c] = quad_add(__fmul_rn(bz, Cxy));
    out[12 + c] = quad_add(__fmul_rn(dbz, Bx));
    out[15 + c] = quad_add(__fmul_rn(dbz, By));
  }
}

// The brick's halo of `coef` by plain loads, in the layout the gathers read.
// Indices beyond the array are clamped: no stencil reaches those nodes.  No
// barrier.
template <typename Tc, int CT>
__device__ __forceinline__ void stage_loads(const StagedArgs& a, const QGeo<CT>& geo,
                                            const int P0[3], const Tc* coef, const float* scale,
                                            unsigned char* halo) {
  const int tid = threadIdx.x;
  const GridArgs& g = a.g;
  const int nrow = geo.Sy * geo.Sz;
  if constexpr (IsNode16<Tc>::value) {
    Tc* h16 = reinterpret_cast<Tc*>(halo);
    float4* scl = reinterpret_cast<float4*>(halo + scale_off_bytes(geo.Sz, geo.PS));
    for (int it = tid; it < nrow * geo.Sx; it += blockDim.x) {
      const int r = it / geo.Sx, x = it - r * geo.Sx;
      const int lz = r / geo.Sy, ly = r - lz * geo.Sy;
      const int64_t row = (int64_t)min(P0[2] + lz, g.m[2] - 1) * g.m[1] + min(P0[1] + ly, g.m[1] - 1);
      h16[lz * geo.PS + ly * geo.SX + x] = coef[row * g.rx + min(P0[0] + x, g.rx - 1)];
    }
    for (int r = tid; r < nrow; r += blockDim.x) {
      const int lz = r / geo.Sy, ly = r - lz * geo.Sy;
      const int64_t row = (int64_t)min(P0[2] + lz, g.m[2] - 1) * g.m[1] + min(P0[1] + ly, g.m[1] - 1);
      scl[r] = __ldg(reinterpret_cast<const float4*>(scale) + row);
    }
  } else if constexpr (IsPlanar<Tc>::value) {
    // 16 (or 32) lanes walk x within a row
    float* h = reinterpret_cast<float*>(halo);
    const int W = geo.Sx <= 16 ? 16 : 32, tx = tid & (W - 1);
    const int Px = min(P0[0] + tx, g.rx - 1);
    if (tx < geo.Sx) {
#pragma unroll 4
      for (int r = tid / W; r < 3 * nrow; r += blockDim.x / W) {
        const int c = r / nrow, r2 = r - c * nrow, lz = r2 / geo.Sy, ly = r2 - lz * geo.Sy;
        const int64_t row = ((int64_t)c * g.m[2] + min(P0[2] + lz, g.m[2] - 1)) * g.m[1] +
                            min(P0[1] + ly, g.m[1] - 1);
        h[c * geo.Sz * geo.PS + lz * geo.PS + ly * geo.SX + tx] = __ldg(coef + row * g.rx + Px);
      }
    }
  } else if (a.vec) {
    stage_halo_vec<Tc, 3>(a, coef, P0, reinterpret_cast<float4*>(halo), false, scale);
  } else {
    stage_halo<Tc, 3>(a, coef, P0, reinterpret_cast<float4*>(halo), false, scale);
  }
}

// Values a lane keeps per particle until it finishes it: MODE 0 velocities; 1
// and the gradient tensor; 2 the velocities of both stages of a Heun step; 3
// second derivatives; 4 Lagrangian acceleration from two fields (u, its
// gradient, the later field's u); 5 from one (u, its gradient).
template <int MODE> struct NOut {
  static constexpr int v =
      MODE == 0 ? 3 : MODE == 1 || MODE == 5 ? 12 : MODE == 2 ? 6 : MODE == 3 ? 18 : 15;
};

// A particle's stencil start in the halo in one word (negative: outside): the
// node index and, for the moves of a Heun step, the three coordinates.
template <int CT> struct WPack {  // 8^3 bricks: coordinates below 8, nodes below 2^11
  static __device__ __forceinline__ int make(int l0, int l1, int l2, const QGeo<CT>& g) {
    return ((l2 * g.PS + l1 * g.SX + l0) << 12) | (l2 << 8) | (l1 << 4) | l0;
  }
  static __device__ __forceinline__ int node(int w, const QGeo<CT>&) { return w >> 12; }
  static __device__ __forceinline__ int l0(int w) { return w & 15; }
  static __device__ __forceinline__ int l1(int w) { return (w >> 4) & 15; }
  static __device__ __forceinline__ int l2(int w) { return (w >> 8) & 15; }
};
template <> struct WPack<0> {
  static __device__ __forceinline__ int make(int l0, int l1, int l2, const QGeo<0>&) {
    return l0 | (l1 << 5) | (l2 << 15);
  }
  static __device__ __forceinline__ int node(int w, const QGeo<0>& g) {
    return l2(w) * g.PS + l1(w) * g.SX + l0(w);
  }
  static __device__ __forceinline__ int l0(int w) { return w & 31; }
  static __device__ __forceinline__ int l1(int w) { return (w >> 5) & 1023; }
  static __device__ __forceinline__ int l2(int w) { return (w >> 15) & 1023; }
};

// The mbarriers of a block's halo copies: the halo, a second field's halo, the
// test knob's (which nothing completes).  A block that takes one brick
// initialises them in warp_brick (ONCE); one that takes brick after brick
// initialises them once, by one thread, with a block barrier before the first
// brick, and each copy completes the next phase, whose parity every thread
// keeps in `phase` (bit i: barrier i).
struct CopyBarriers {
  unsigned long long b[3];
};
__device__ __forceinline__ void init_copy_barriers(CopyBarriers& mb) {
#pragma unroll
  for (int i = 0; i < 3; ++i) tma_init_barrier(&mb.b[i]);
}

// Returns whether this thread saw every copy of the brick land (false: the
// block's shared memory must not be used again).
template <typename Tc, int MODE, int CT, bool ONCE = true>
__device__ __forceinline__ bool warp_brick(const StagedArgs& a, int bin, int bxi, int byi,
                                           int bzi, unsigned char* smem, const StagedArgs* maps,
                                           CopyBarriers& mb, unsigned& phase) {
  const int beg = a.offs[bin], end = a.offs[bin + 1];
  if (beg >= end) return true;
  const QGeo<CT> geo(a);
  const GridArgs& g = a.g;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned per_trip = blockDim.x;
  const int k = lane & 3, quad = lane >> 2;
  const int64_t np = a.np;
  const Tc* coef = static_cast<const Tc*>(a.coef);
  const bool second = MODE == 4 || (MODE == 2 && a.coef2 != nullptr);
  const Tc* coef2 = second ? static_cast<const Tc*>(a.coef2) : coef;
  const float* scale2 = second ? a.scale2 : a.scale;

  // the first particles' positions are on their way before anything else (slots
  // as unsigned: the trip after the last one lies beyond 2^31 in the largest sets)
  const unsigned last = (unsigned)end;
  unsigned c0 = (unsigned)beg + 32 * warp;
  int p = 0;
  double x[3] = {0.0, 0.0, 0.0};
  auto load = [&](unsigned c) {
    if (c + lane < last) {
      p = a.perm ? (int)a.perm[c + lane] : (int)(c + lane);
#pragma unroll
      for (int d = 0; d < 3; ++d) x[d] = a.pos_in[d * np + p];
    }
  };
  load(c0);

  const int P0[3] = {bxi * a.b.B[0], byi * a.b.B[1], bzi * a.b.B[2]};
  const int hbytes = halo_bytes<Tc>(geo.Sz, geo.Sy, geo.PS);
  unsigned char* halo = smem;
  unsigned char* halo2 = smem + hbytes;
  unsigned long long* mbar = mb.b;
  const unsigned par = ONCE ? 0 : phase & 1, par2 = ONCE ? 0 : phase >> 1 & 1;
  __shared__ unsigned char slot_lane[4][32];

  // use1, use2: the halos of coef and coef2 hold the brick's nodes
  bool use1 = end - beg >= a.min_stage && !a.chunked;
  bool use2 = use1 && second && a.two;
  const bool tma = use1 && a.tma && (smem_u32(halo) & 127) == 0;
  const bool tma2 = tma && use2 && a.tma == 2;
  if (use1) {
    if (tid == 0 && tma) {
      if (ONCE) {
        if (a.wait_probe > 0) tma_init_barrier(&mbar[2]);
        tma_init_barrier(&mbar[0]);
      } else {  // the last brick's accesses to the halo before this one's copy
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      }
      if constexpr (IsNode16<Tc>::value) {
        // the nodes and the rows' scales, both on one barrier
        tma_copy_node16(&maps->tmap, &maps->tmap2, halo,
                        halo + scale_off_bytes(geo.Sz, geo.PS), &mbar[0], P0,
                        (unsigned)(geo.Sz * (geo.PS * 8 + geo.Sy * 16)));
      } else if constexpr (IsNode4<Tc>::value || IsPlanar<Tc>::value) {
        const unsigned bytes =
            (unsigned)((IsPlanar<Tc>::value ? 12 : 16) * geo.PS * geo.Sz);
        tma_copy<IsPlanar<Tc>::value>(&maps->tmap, halo, &mbar[0], P0, bytes);
        if (tma2) {
          if (ONCE) tma_init_barrier(&mbar[1]);
          tma_copy<IsPlanar<Tc>::value>(&maps->tmap2, halo2, &mbar[1], P0, bytes);
        }
      }
    }
    if (!tma) stage_loads<Tc, CT>(a, geo, P0, coef, a.scale, halo);
    if (use2 && !tma2) stage_loads<Tc, CT>(a, geo, P0, coef2, scale2, halo2);
    __syncthreads();  // barrier initialisation, halos staged by loads
  }
  bool waited = !tma, landed = !tma, landed2 = !tma2;
  // largest stencil start in the halo along each axis (the last brick of an
  // axis may hold fewer cells than the others)
  const int lmax[3] = {min(geo.Sx - 4, g.n[0] - 1 - P0[0]), min(geo.Sy - 4, g.n[1] - 1 - P0[1]),
                       min(geo.Sz - 4, g.n[2] - 1 - P0[2])};
  int stays = 0;

  for (; c0 < last; c0 += per_trip) {
    const int m = (int)min(32u, last - c0);
    const bool v = lane < m;
    // -- 1: location, and the slot among the warp's particles
    const double xp[3] = {x[0], x[1], x[2]};
    const int pp = p;
    int cell[3];
    float t[3];
    bool inside = true;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      // floor and fraction of x n / L in 32.32 fixed point (the scaling by
      // 2^32 is exact, so both are those of the rounded product x n / L)
      const long long s = __double2ll_rd(__dmul_rn(xp[d], a.ih32[d]));
      cell[d] = (int)(s >> 32);
      t[d] = (float)((unsigned)s >> 8) * 0x1p-24f;
      inside = inside && (unsigned)cell[d] < (unsigned)g.n[d];
    }
    bool ok = v;
    if (v && !inside) {  // another image of the box, or not finite
#pragma unroll
      for (int d = 0; d < 3; ++d) ok &= locate(xp[d], g.inv_h[d], g.n[d], cell[d], t[d]);
    }
    load(c0 + per_trip);
    // packed stencil start in the halo, -1 outside it
    int w = -1;
    {
      const int l0 = cell[0] - P0[0], l1 = cell[1] - P0[1], l2 = cell[2] - P0[2];
      if (ok && use1 && (unsigned)l0 <= (unsigned)lmax[0] && (unsigned)l1 <= (unsigned)lmax[1] &&
          (unsigned)l2 <= (unsigned)lmax[2])
        w = WPack<CT>::make(l0, l1, l2, geo);
    }
    // Slots in classes of the stencil start's bank group: the lanes k of a
    // quad read groups of one parity (float4 nodes, two quads per load phase)
    // or one residue mod 4 (16-bit nodes, four quads per phase; planar words,
    // eight), so neighbouring slots take different classes: rank 0 of every
    // class, then rank 1, ...
    int slot = -1;
    {
      const unsigned lt = (1u << lane) - 1u;
      const int first = WPack<CT>::node(w, geo);
      if constexpr (IsNode16<Tc>::value || IsPlanar<Tc>::value) {
        const int cls = w < 0 ? 0 : first & 3;
        const unsigned bv = __ballot_sync(FULL, v);
        const unsigned b0 = __ballot_sync(FULL, cls & 1), b1 = __ballot_sync(FULL, cls & 2);
        const unsigned in[4] = {bv & ~b0 & ~b1, bv & b0 & ~b1, bv & ~b0 & b1, bv & b0 & b1};
        const unsigned mine = cls == 0 ? in[0] : cls == 1 ? in[1] : cls == 2 ? in[2] : in[3];
        const int r = __popc(mine & lt);
        int s = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int cq = __popc(in[q]);
          s += min(cq, r) + ((q < cls && cq > r) ? 1 : 0);
        }
        slot = v ? s : -1;
      } else {
        const bool odd = w >= 0 && (first & 1);
        const unsigned bo = __ballot_sync(FULL, v && odd), be = __ballot_sync(FULL, v && !odd);
        const int ne = __popc(be), no = __popc(bo), nm = min(ne, no);
        const int r = __popc((odd ? bo : be) & lt);
        slot = !v ? -1 : (r < nm ? 2 * r + (odd ? 1 : 0) : nm + r);
      }
    }
    __syncwarp();
    if (v) slot_lane[warp][slot] = (unsigned char)lane;
    __syncwarp();
    const int src = slot_lane[warp][lane];
    if (!waited) {
      // a copy that does not complete in time is reported and the particles
      // read global memory
      waited = true;
      landed = tma_wait(&mbar[0], par);
      bool done = landed;
      if (done && a.wait_probe > 0) done = tma_wait(&mbar[2], 0, a.wait_probe);
      if (tma2) {
        landed2 = tma_wait(&mbar[1], par2);
        done = done && landed2;
      }
      if (!__all_sync(FULL, done)) {
        use1 = use2 = false;
        if (lane == 0) flag_status(a.status, PS_DEV_TIMEOUT, beg);
      }
    }
    if (!use1) w = -1;
    const bool some_out = __any_sync(FULL, v && w < 0);

    // -- 2: eight particles at a time, a quad each
    float res[NOut<MODE>::v];
#pragma unroll
    for (int i = 0; i < NOut<MODE>::v; ++i) res[i] = 0.f;
    for (int ch = 0; 8 * ch < m; ++ch) {
      const int sj = __shfl_sync(FULL, src, min(8 * ch + quad, m - 1));
      const int wq = __shfl_sync(FULL, w, sj);
      const float tq[3] = {__shfl_sync(FULL, t[0], sj), __shfl_sync(FULL, t[1], sj),
                           __shfl_sync(FULL, t[2], sj)};
      int cq[3] = {0, 0, 0};
      // (the cell of stencils read from global memory: outside the halo, or of a
      // later field that is not staged)
      if (some_out || (MODE == 4 && !use2)) {
#pragma unroll
        for (int d = 0; d < 3; ++d) cq[d] = __shfl_sync(FULL, cell[d], sj);
      }
      const int node = WPack<CT>::node(wq, geo) + k * geo.PS;
      const int hrow = IsNode16<Tc>::value ? (WPack<CT>::l2(wq) + k) * geo.Sy + WPack<CT>::l1(wq) : 0;
      float vq[16][3];
      float out[NOut<MODE>::v];
      if (wq >= 0) fetch_halo<Tc, CT>(vq, halo, node, hrow, geo);
      else fetch_global<Tc>(vq, cq, k, g, coef, a.scale);
      if constexpr (MODE == 0) quad_sum<false>(vq, tq, k, out);
      if constexpr (MODE == 1 || MODE == 5) quad_sum<true>(vq, tq, k, out);
      if constexpr (MODE == 3) quad_sum_hess(vq, tq, k, out);
      if constexpr (MODE == 4) {
        quad_sum<true>(vq, tq, k, out);
        if (wq >= 0 && use2) fetch_halo<Tc, CT>(vq, halo2, node, hrow, geo);
        else fetch_global<Tc>(vq, cq, k, g, coef2, scale2);
        quad_sum<false>(vq, tq, k, out + 12);
      }
      if constexpr (MODE == 2) {
        quad_sum<false>(vq, tq, k, out);
        // predictor x* = x + dt u1, located in FP32 from the stage-1 cell
        float t2[3];
        bool stay = true;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          t2[d] = __fmaf_rn(out[d], a.dtih[d], tq[d]);
          stay = stay && t2[d] >= 0.f && t2[d] < 1.f;
        }
        if (!stay || second) {
          const int l[3] = {WPack<CT>::l0(wq), WPack<CT>::l1(wq), WPack<CT>::l2(wq)};
          int f3[3], c2[3];
          bool inh2 = wq >= 0 && (second ? use2 : use1);
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            float f = floorf(t2[d]);
            if (!(fabsf(f) < 1.0e9f)) f = 0.f;  // non-finite velocity: keep the cell
            t2[d] = fminf(fmaxf(__fsub_rn(t2[d], f), 0.f), 1.f);
            f3[d] = (int)f;
            inh2 = inh2 && (unsigned)(l[d] + f3[d]) <= (unsigned)lmax[d];
          }
          if (inh2) {
            const int shift = f3[2] * geo.PS + f3[1] * geo.SX + f3[0];
            fetch_halo<Tc, CT>(vq, second ? halo2 : halo, node + shift,
                               hrow + f3[2] * geo.Sy + f3[1], geo);
          } else {
#pragma unroll
            for (int d = 0; d < 3; ++d) {
              int c = (wq >= 0 ? P0[d] + l[d] : cq[d]) + f3[d];
              if (c < 0 || c >= g.n[d]) {
                c %= g.n[d];
                if (c < 0) c += g.n[d];
              }
              c2[d] = c;
            }
            fetch_global<Tc>(vq, c2, k, g, coef2, scale2);
          }
        }
        quad_sum<false>(vq, t2, k, out + 3);
      }
      // back to the particle's lane
      const int from = (slot & 7) << 2;
      const bool mine = (slot >> 3) == ch;  // slot = -1: never
#pragma unroll
      for (int i = 0; i < NOut<MODE>::v; ++i) {
        const float y = __shfl_sync(FULL, out[i], from);
        if (mine) res[i] = y;
      }
    }

    // -- 3: lane i finishes particle i
    const float nanf_ = __int_as_float(0x7fc00000);
    if (v && !ok) flag_status(a.status, PS_DEV_NONFINITE_POS, pp);
    const int oo = a.slot_out ? (int)(c0 + lane) : pp;  // where the results go
    if constexpr (MODE <= 1) {
      if (v) {
#pragma unroll
        for (int c = 0; c < 3; ++c) a.vel[c * np + oo] = ok ? res[c] : nanf_;
        if (MODE == 1) {
#pragma unroll
          for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int d = 0; d < 3; ++d)
              a.grad[(c * 3 + d) * np + oo] =
                  ok ? __fmul_rn(res[(MODE == 1 ? 3 : 0) * (1 + d) + c], g.inv_hf[d]) : nanf_;
        }
      }
    }
    if constexpr (MODE == 3) {
      // hess [3][6][np] (a.grad), scaled by n_a/L_a n_b/L_b
      if (v) {
        const float hx = g.inv_hf[0], hy = g.inv_hf[1], hz = g.inv_hf[2];
        const float sc[6] = {__fmul_rn(hx, hx), __fmul_rn(hy, hy), __fmul_rn(hz, hz),
                             __fmul_rn(hx, hy), __fmul_rn(hx, hz), __fmul_rn(hy, hz)};
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int e = 0; e < 6; ++e)
            a.grad[(c * 6 + e) * np + oo] = ok ? __fmul_rn(res[3 * e + c], sc[e]) : nanf_;
      }
    }
    if constexpr (MODE == 4 || MODE == 5) {
      // a = (u . grad) u [+ (u(coef2) - u) / dt_field] (a.dt = 1 / dt_field) -> a.grad [3][np]
      if (v) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          float acc = __fmul_rn(__fmul_rn(res[3 + c], g.inv_hf[0]), res[0]);
          acc = __fmaf_rn(__fmul_rn(res[6 + c], g.inv_hf[1]), res[1], acc);
          acc = __fmaf_rn(__fmul_rn(res[9 + c], g.inv_hf[2]), res[2], acc);
          if (MODE == 4)
            acc = __fmaf_rn(__fsub_rn(res[MODE == 4 ? 12 + c : 0], res[c]), (float)a.dt, acc);
          a.grad[c * np + oo] = ok ? acc : nanf_;
          if (a.vel) a.vel[c * np + oo] = ok ? res[c] : nanf_;
        }
      }
    }
    if constexpr (MODE == 2) {
      int bc[3] = {-1, -1, -1};
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const float u1 = res[d], u2 = res[3 + d], us = __fadd_rn(u1, u2);
        const double xn = ok ? fma(a.half_dt, (double)us, xp[d])
                             : __longlong_as_double(0x7ff8000000000000ll);
        if (v) {
          a.pos_out[d * np + pp] = xn;
          if (a.vel) a.vel[d * np + pp] = ok ? u1 : nanf_;
        }
        if (a.next_counts) {
          // The new cell: the stage-1 cell plus the floor of its fraction
          // plus the step's displacement dt (u1 + u2) / 2 in cells, in FP32.
          // That floor is the exact one wherever the sum lies 2^-10 or more
          // from a cell face and |x n/L| < 2^30 (displacements of up to four
          // cells: the FP32 and FP64 roundings on both routes stay below 1e-6
          // cell).  Elsewhere, and for positions that are not finite, the
          // FP64 location decides.
          const float wn = __fmaf_rn(0.5f * a.dtih[d], us, t[d]);
          const float f = floorf(wn), fr = wn - f;
          int c;
          if (ok && fr >= 0x1p-10f && fr <= 1.f - 0x1p-10f && fabsf(f) <= 2.f &&
              (__double2hiint(xp[d]) & 0x7fffffff) < a.xguard_hi[d]) {
            const int nd = g.n[d];
            c = cell[d] + (int)f;  // in [-2, n + 1], n >= 3
            c = c < 0 ? c + nd : (c >= nd ? c - nd : c);
          } else {
            float tn;
            if (!v || !locate(xn, g.inv_h[d], g.n[d], c, tn)) c = -1;
          }
          bc[d] = c < 0 ? -1 : (a.bshift[d] >= 0 ? c >> a.bshift[d] : c / a.b.B[d]);
        }
      }
      if (v && a.ids_out) a.ids_out[pp] = a.ids_in[pp];
      if (a.next_counts) {
        // The bin goes to next_bin[p]; the counters take the totals only (the
        // scatter takes the ranks).  Particles that stay in this bin are
        // counted per warp and added once; the others add one each.  A
        // rejected position is counted in bin 0 and reported, as the counting
        // pass of the sort does.
        int key = bin_of_coords(a.b, bc[0], bc[1], bc[2]);
        if (a.next_runs > 0 && key >= 0) key = (int)((int64_t)key * a.next_runs / a.b.nbins);
        if (v && key < 0) {
          flag_status(a.status, PS_DEV_NONFINITE_POS, pp);
          key = 0;
        }
        if (v) a.next_bin[pp] = a.next_key_base + key;
        const bool stay = v && key == bin;
        stays += __popc(__ballot_sync(FULL, stay));
        if (v && !stay) atomicAdd(&a.next_counts[key], 1);
      }
    }
  }
  if (MODE == 2 && a.next_counts && lane == 0 && stays) atomicAdd(&a.next_counts[bin], stays);
  // a copy still in flight must land before the block's memory is released
  if (tma && !(waited && landed)) landed = tma_wait(&mbar[0], par);
  if (tma2 && !(waited && landed2)) landed2 = tma_wait(&mbar[1], par2);
  if (!ONCE) phase ^= (tma ? 1u : 0u) | (tma2 ? 2u : 0u);
  return landed && landed2;
}

}  // namespace
}  // namespace ps
