// Operations 2 and 3 of Sec. 2.2 (basis functions and the 64-term sum of
// Eq. (spline)), their adjoint, and the second-order Runge-Kutta particle
// advance of Sec. 2.1 / Sec. 4.3.
//
// Two gather strategies:
//  * direct: a quad of lanes per particle, lane q owning stencil column
//    x = a_x + q; every (j,k) row is one 16-byte segment per quad.  Works for
//    any particle order (the "unsorted" path).
//  * staged: particles stored in brick order (Sec. 3's dynamic mapping read as
//    a bin sort); one CTA per brick copies the brick's coefficient halo once
//    into shared memory.  This is the GPU form of the paper's "fetch only the
//    coefficients a particle needs": the halo is the union of the stencils of
//    the brick's particles.  Three components: brick.cuh and quad.cu.  Here:
//    one component, as float4 in shared memory and 8 lanes per particle, and
//    the thread-per-particle form of both.
//
// FP64 work per particle is one multiply per axis (done by three lanes in
// parallel); floor and fraction come from the bits of the product, the RK2
// predictor position is located in FP32 relative to the stage-1 cell, and the
// position update is one FMA per axis.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include <mutex>

#include <cuda.h>
#include <cudaTypedefs.h>

#include "bin_device.cuh"
#include "staged.cuh"

namespace ps {
namespace {

// The first three lanes of each group of G lanes locate one axis each; the
// cell indices and fractions are broadcast to the whole group.  xd returns
// the FP64 coordinate of the lane's own axis (lanes 0..2 of the group).
template <int G, typename A>
__device__ __forceinline__ bool locate_group(const GridArgs& g, const double* pos, int64_t np,
                                             int64_t p, int lane, int cell[3], A t[3],
                                             double& xd) {
  const int sub = lane & (G - 1), base = lane & ~(G - 1);
  int cd = 0;
  A td = A(0);
  xd = 0.0;
  if (sub < 3) {
    xd = pos[sub * np + p];
    bool okd;
    if constexpr (std::is_same<A, double>::value)
      okd = locate_f64(xd, g.inv_h[sub], g.n[sub], cd, td);
    else
      okd = locate(xd, g.inv_h[sub], g.n[sub], cd, td);
    if (!okd) cd = -1;
  }
  bool ok = true;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    cell[d] = __shfl_sync(FULL, cd, base + d);
    t[d] = __shfl_sync(FULL, td, base + d);
    ok &= cell[d] >= 0;
    cell[d] = max(cell[d], 0);
  }
  return ok;
}

template <typename A, bool GRAD>
struct Basis {
  int a[3];
  A b[3][4];
  A db[3][4];
  __device__ __forceinline__ void set(const int cell[3], const A t[3]) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      a[d] = cell[d];
      bspline<A>(t[d], b[d]);
      if (GRAD) dbspline<A>(t[d], db[d]);
    }
  }
};

// Predictor position of a Heun step located in FP32 relative to the stage-1
// cell: t* = t + u dt n/L, cell* = cell + floor(t*) (mod n).
__device__ __forceinline__ void advance_cell(int n, int cell, float t, float du, int& c2,
                                             float& t2) {
  float tt = t + du;
  float fl = floorf(tt);
  if (!(fabsf(fl) < 1.0e9f)) fl = 0.f;  // non-finite velocity: keep the cell
  tt -= fl;
  int c = cell + (int)fl;
  if (c < 0 || c >= n) {
    c %= n;
    if (c < 0) c += n;
  }
  c2 = c;
  t2 = fminf(fmaxf(tt, 0.f), 1.f);
}

// Direct gather by a quad: lane q accumulates its column over the 16 rows.
template <typename Tc, int NC, bool GRAD, typename A>
__device__ __forceinline__ void quad_rows(const GridArgs& g, const Tc* __restrict__ coef,
                                          const float* __restrict__ scale,
                                          const Basis<A, GRAD>& B, int q, A acc[NC],
                                          A accy[NC], A accz[NC]) {
#pragma unroll
  for (int c = 0; c < NC; ++c) acc[c] = accy[c] = accz[c] = A(0);
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const A w = B.b[1][j] * B.b[2][k];
      A wy = A(0), wz = A(0);
      if (GRAD) {
        wy = B.db[1][j] * B.b[2][k];
        wz = B.b[1][j] * B.db[2][k];
      }
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const A v = load_coef<Tc>(coef, scale, g, c, B.a[2] + k, B.a[1] + j, B.a[0] + q);
        acc[c] += w * v;
        if (GRAD) {
          accy[c] += wy * v;
          accz[c] += wz * v;
        }
      }
    }
}

// MODE 0: vel; 1: vel + grad; 2: g_pos = sum_c g_vel[c] grad[c][.]
template <typename Tc, int NC, int MODE>
__global__ void __launch_bounds__(256) interp_direct(GridArgs g, const Tc* __restrict__ coef,
                                                     const float* __restrict__ scale,
                                                     int64_t np,
                                                     const double* __restrict__ pos,
                                                     const int64_t* __restrict__ perm,
                                                     float* __restrict__ vel,
                                                     float* __restrict__ grad,
                                                     const float* __restrict__ gvel,
                                                     double* __restrict__ gpos,
                                                     int32_t* status) {
  using A = typename AccOf<Tc>::type;
  constexpr bool GRAD = MODE >= 1;
  const int lane = threadIdx.x & 31, q = lane & 3;
  const int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 2;
  const bool valid = s < np;
  const int64_t p = valid ? (perm ? perm[s] : s) : 0;
  int cell[3];
  A t[3];
  double xd;
  const bool ok = locate_group<4, A>(g, pos, valid ? np : 0, p, lane, cell, t, xd) || !valid;
  Basis<A, GRAD> B;
  B.set(cell, t);
  A acc[NC], accy[NC], accz[NC];
  quad_rows<Tc, NC, GRAD, A>(g, coef, scale, B, q, acc, accy, accz);
  const A bq = pick4(B.b[0], q);
  A u[NC], gx[NC], gy[NC], gz[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    u[c] = group_sum<4>(bq * acc[c]);
    if (GRAD) {
      const A dbq = pick4(B.db[0], q);
      gx[c] = group_sum<4>(dbq * acc[c]) * (A)g.inv_h[0];
      gy[c] = group_sum<4>(bq * accy[c]) * (A)g.inv_h[1];
      gz[c] = group_sum<4>(bq * accz[c]) * (A)g.inv_h[2];
    }
  }
  if (!valid || q != 0) return;
  if (!ok) flag_status(status, PS_DEV_NONFINITE_POS, p);
  const float nanf_ = __int_as_float(0x7fc00000);
  if (MODE <= 1) {
#pragma unroll
    for (int c = 0; c < NC; ++c) vel[(int64_t)c * np + p] = ok ? (float)u[c] : nanf_;
    if (MODE == 1 && grad) {
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        grad[((int64_t)c * 3 + 0) * np + p] = ok ? (float)gx[c] : nanf_;
        grad[((int64_t)c * 3 + 1) * np + p] = ok ? (float)gy[c] : nanf_;
        grad[((int64_t)c * 3 + 2) * np + p] = ok ? (float)gz[c] : nanf_;
      }
    }
  } else {
    A sx = A(0), sy = A(0), sz = A(0);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const A w = (A)gvel[(int64_t)c * np + p];
      sx += w * gx[c];
      sy += w * gy[c];
      sz += w * gz[c];
    }
    const double nand = __longlong_as_double(0x7ff8000000000000ll);
    gpos[p] = ok ? (double)sx : nand;
    gpos[np + p] = ok ? (double)sy : nand;
    gpos[2 * np + p] = ok ? (double)sz : nand;
  }
}

// Scatter-add of g_vel * basis weights onto the periodic nodes: the adjoint
// of the 64-term sum followed by the adjoint of the periodic padding (fold).
template <int NC>
__global__ void __launch_bounds__(256) scatter_field(GridArgs g, int64_t np,
                                                    const double* __restrict__ pos,
                                                    const float* __restrict__ gvel,
                                                    float* __restrict__ gfield,
                                                    int32_t* status) {
  const int lane = threadIdx.x & 31, q = lane & 3;
  const int64_t p0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 2;
  const bool valid = p0 < np;
  const int64_t p = valid ? p0 : 0;
  int cell[3];
  float t[3];
  double xd;
  const bool ok = locate_group<4, float>(g, pos, valid ? np : 0, p, lane, cell, t, xd);
  if (!valid) return;  // no shuffles below
  if (!ok) {
    if (q == 0) flag_status(status, PS_DEV_NONFINITE_POS, p);
    return;
  }
  Basis<float, false> B;
  B.set(cell, t);
  float gc[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) gc[c] = gvel[(int64_t)c * np + p] * pick4(B.b[0], q);
  const int64_t vol = (int64_t)g.n[0] * g.n[1] * g.n[2];
  const int nodex = padded_to_node(B.a[0] + q, g.n[0]);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int nodez = padded_to_node(B.a[2] + k, g.n[2]);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int nodey = padded_to_node(B.a[1] + j, g.n[1]);
      const float w = B.b[1][j] * B.b[2][k];
      const int64_t off = ((int64_t)nodez * g.n[1] + nodey) * g.n[0] + nodex;
#pragma unroll
      for (int c = 0; c < NC; ++c) atomicAdd(gfield + c * vol + off, w * gc[c]);
    }
  }
}

// Second derivatives of Eq. (spline) by a quad of lanes per particle (lane q
// owns stencil column a_x + q): six sums per component over the 16 (j, k)
// rows with the y and z factors of each derivative, the x factor applied per
// lane before the quad reduction.  hess [ncomp][6][np]: xx, yy, zz, xy, xz, yz.
template <typename Tc, int NC>
__global__ void __launch_bounds__(256) interp_hessian_direct(GridArgs g,
                                                             const Tc* __restrict__ coef,
                                                             const float* __restrict__ scale,
                                                             int64_t np,
                                                             const double* __restrict__ pos,
                                                             float* __restrict__ hess,
                                                             int32_t* status) {
  using A = typename AccOf<Tc>::type;
  const int lane = threadIdx.x & 31, q = lane & 3;
  const int64_t p0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 2;
  const bool valid = p0 < np;
  const int64_t p = valid ? p0 : 0;
  int cell[3];
  A t[3];
  double xd;
  const bool ok = locate_group<4, A>(g, pos, valid ? np : 0, p, lane, cell, t, xd) || !valid;
  A b[3][4], db[3][4], d2[3][4];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    bspline<A>(t[d], b[d]);
    dbspline<A>(t[d], db[d]);
    ddbspline<A>(t[d], d2[d]);
  }
  A s0[NC], sy[NC], sz[NC], syy[NC], szz[NC], syz[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) s0[c] = sy[c] = sz[c] = syy[c] = szz[c] = syz[c] = A(0);
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const A v = load_coef<Tc>(coef, scale, g, c, cell[2] + k, cell[1] + j, cell[0] + q);
        s0[c] += b[1][j] * b[2][k] * v;
        sy[c] += db[1][j] * b[2][k] * v;
        sz[c] += b[1][j] * db[2][k] * v;
        syy[c] += d2[1][j] * b[2][k] * v;
        szz[c] += b[1][j] * d2[2][k] * v;
        syz[c] += db[1][j] * db[2][k] * v;
      }
    }
  const A bq = pick4(b[0], q), dbq = pick4(db[0], q), d2q = pick4(d2[0], q);
  const A hx = (A)g.inv_h[0], hy = (A)g.inv_h[1], hz = (A)g.inv_h[2];
  A h[NC][6];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    h[c][0] = group_sum<4>(d2q * s0[c]) * (hx * hx);
    h[c][1] = group_sum<4>(bq * syy[c]) * (hy * hy);
    h[c][2] = group_sum<4>(bq * szz[c]) * (hz * hz);
    h[c][3] = group_sum<4>(dbq * sy[c]) * (hx * hy);
    h[c][4] = group_sum<4>(dbq * sz[c]) * (hx * hz);
    h[c][5] = group_sum<4>(bq * syz[c]) * (hy * hz);
  }
  if (!valid || q != 0) return;
  if (!ok) flag_status(status, PS_DEV_NONFINITE_POS, p);
  const float nanf_ = __int_as_float(0x7fc00000);
#pragma unroll
  for (int c = 0; c < NC; ++c)
#pragma unroll
    for (int e = 0; e < 6; ++e) hess[((int64_t)c * 6 + e) * np + p] = ok ? (float)h[c][e] : nanf_;
}

// Lagrangian acceleration a = du/dt + (u . grad) u by a quad per particle:
// u and its gradient from c0, u from c1 (if given) for the time difference.
template <typename Tc>
__global__ void __launch_bounds__(256) lagrangian_accel_direct(
    GridArgs g, const Tc* __restrict__ c0, const float* __restrict__ s0,
    const Tc* __restrict__ c1, const float* __restrict__ s1, double inv_dt, int64_t np,
    const double* __restrict__ pos, float* __restrict__ acc, float* __restrict__ vel,
    int32_t* status) {
  using A = typename AccOf<Tc>::type;
  const int lane = threadIdx.x & 31, q = lane & 3;
  const int64_t p0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 2;
  const bool valid = p0 < np;
  const int64_t p = valid ? p0 : 0;
  int cell[3];
  A t[3];
  double xd;
  const bool ok = locate_group<4, A>(g, pos, valid ? np : 0, p, lane, cell, t, xd) || !valid;
  Basis<A, true> B;
  B.set(cell, t);
  A a0[3], ay[3], az[3];
  quad_rows<Tc, 3, true, A>(g, c0, s0, B, q, a0, ay, az);
  const A bq = pick4(B.b[0], q), dbq = pick4(B.db[0], q);
  A u[3], gx[3], gy[3], gz[3], u1[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    u[c] = group_sum<4>(bq * a0[c]);
    gx[c] = group_sum<4>(dbq * a0[c]) * (A)g.inv_h[0];
    gy[c] = group_sum<4>(bq * ay[c]) * (A)g.inv_h[1];
    gz[c] = group_sum<4>(bq * az[c]) * (A)g.inv_h[2];
    u1[c] = u[c];
  }
  if (c1) {
    Basis<A, false> B1;
    B1.set(cell, t);
    quad_rows<Tc, 3, false, A>(g, c1, s1, B1, q, a0, ay, az);
#pragma unroll
    for (int c = 0; c < 3; ++c) u1[c] = group_sum<4>(bq * a0[c]);
  }
  if (!valid || q != 0) return;
  if (!ok) flag_status(status, PS_DEV_NONFINITE_POS, p);
  const float nanf_ = __int_as_float(0x7fc00000);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const A a = gx[c] * u[0] + gy[c] * u[1] + gz[c] * u[2] + (u1[c] - u[c]) * (A)inv_dt;
    acc[(int64_t)c * np + p] = ok ? (float)a : nanf_;
    if (vel) vel[(int64_t)c * np + p] = ok ? (float)u[c] : nanf_;
  }
}

// Fused Heun step with direct gathers (any particle order).
template <typename Tc>
__global__ void __launch_bounds__(256) rk2_direct(GridArgs g, const Tc* __restrict__ c0,
                                                  const float* __restrict__ s0,
                                                  const Tc* __restrict__ c1,
                                                  const float* __restrict__ s1, int64_t np,
                                                  double* pos, float* __restrict__ vel_out,
                                                  double dt, float3 dtih, int32_t* status) {
  using A = typename AccOf<Tc>::type;
  const int lane = threadIdx.x & 31, q = lane & 3;
  const int64_t p0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 2;
  const bool valid = p0 < np;
  const int64_t p = valid ? p0 : 0;
  int cell[3];
  A t[3];
  double xd;
  bool ok = locate_group<4, A>(g, pos, valid ? np : 0, p, lane, cell, t, xd);
  Basis<A, false> B;
  B.set(cell, t);
  A acc[3], ay[3], az[3];
  quad_rows<Tc, 3, false, A>(g, c0, s0, B, q, acc, ay, az);
  A bq = pick4(B.b[0], q);
  A u1[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) u1[c] = group_sum<4>(bq * acc[c]);
  const float dti[3] = {dtih.x, dtih.y, dtih.z};
  int c2[3];
  A t2[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    if constexpr (std::is_same<A, double>::value) {
      // FP64 coefficients: locate the predictor exactly as x + dt u1
      double xs = __shfl_sync(FULL, xd, (lane & ~3) + d) + dt * u1[d];
      double tt;
      ok &= locate_f64(xs, g.inv_h[d], g.n[d], c2[d], tt);
      t2[d] = tt;
    } else {
      float tt;
      advance_cell(g.n[d], cell[d], t[d], ok ? (float)u1[d] * dti[d] : 0.f, c2[d], tt);
      t2[d] = tt;
    }
  }
  B.set(c2, t2);
  quad_rows<Tc, 3, false, A>(g, c1, s1, B, q, acc, ay, az);
  bq = pick4(B.b[0], q);
  A u2[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) u2[c] = group_sum<4>(bq * acc[c]);
  if (!valid) return;
  if (!ok && q == 0) flag_status(status, PS_DEV_NONFINITE_POS, p);
  if (q < 3) {
    const double nand = __longlong_as_double(0x7ff8000000000000ll);
    const double w = (double)(sel3(u1, q) + sel3(u2, q));
    pos[(int64_t)q * np + p] = ok ? fma(dt * 0.5, w, xd) : nand;
    if (vel_out)
      vel_out[(int64_t)q * np + p] = ok ? (float)sel3(u1, q) : __int_as_float(0x7fc00000);
  }
}

// Particle records in shared memory, one entry per particle of the current
// round (kRecords), stored field-major so that neither the per-axis writers
// nor the 8-lane readers conflict on banks:
//   b[d][i]    float4  b_0..3(t_d) of particle i along axis d
//   db[d][i]   float4  b'_0..3(t_d)   (gradient mode only)
//   loc[d][i]  int     brick-local stencil start along d, -1 = outside halo
//   cell[d][i] int     global cell along d, -1 = position not finite
// 80 particles per round: a brick of the mid density (64 particles on
// average, Poisson) rarely needs a second, mostly empty round, and the 240
// (particle, axis) tasks still fit two per thread.
constexpr int kRecords = 80;   // particles per round
constexpr int kThreads = 128;  // threads per brick CTA

struct Recs {
  float4* f;  // b[3], then db[3] in gradient mode
  int* ip;    // lw, cell[3]
  __device__ __forceinline__ float4* b(int d) const { return f + d * kRecords; }
  __device__ __forceinline__ float4* db(int d) const { return f + (3 + d) * kRecords; }
  // byte d of lw[i]: brick-local stencil start along d, -1 outside the halo,
  // -2 position not finite
  __device__ __forceinline__ int* lw() const { return ip; }
  __device__ __forceinline__ int* cell(int d) const { return ip + (1 + d) * kRecords; }
};
__host__ __device__ constexpr size_t rec_bytes(bool grad) {
  return (size_t)kRecords * ((grad ? 6 : 3) * sizeof(float4) + 4 * sizeof(int));
}

template <bool GRAD>
__device__ __forceinline__ Recs carve_recs(void* base) {
  Recs r;
  r.f = static_cast<float4*>(base);
  r.ip = reinterpret_cast<int*>(r.f + (GRAD ? 6 : 3) * kRecords);
  return r;
}

// One (particle, axis) task of phases A / A': basis along the axis and the
// brick-local index of the stencil start.  The z basis is stored in the order
// (b0, b2, b1, b3) so that a gather lane reads its pair (b_kh, b_kh+2) at once.
template <bool GRAD>
__device__ __forceinline__ void write_axis(const Recs& R, int i, int d, int cell, float t,
                                           bool ok, int P0, int S) {
  float b[4];
  bspline<float>(t, b);
  R.b(d)[i] = d == 2 ? make_float4(b[0], b[2], b[1], b[3]) : make_float4(b[0], b[1], b[2], b[3]);
  if (GRAD) {
    float db[4];
    dbspline<float>(t, db);
    R.db(d)[i] =
        d == 2 ? make_float4(db[0], db[2], db[1], db[3]) : make_float4(db[0], db[1], db[2], db[3]);
  }
  const int l = cell - P0;
  const int code = !ok ? -2 : ((unsigned)l <= (unsigned)(S - 4) ? l : -1);
  reinterpret_cast<signed char*>(R.lw())[4 * i + d] = (signed char)code;
  R.cell(d)[i] = cell;
}

__device__ __forceinline__ float f4get(const float4 v, int j) {
  return j == 0 ? v.x : (j == 1 ? v.y : (j == 2 ? v.z : v.w));
}

// Phase B: 8 lanes per particle.  Lane (q, kh) covers stencil column
// x = a_x + q and the z rows k = kh, kh + 2, all four y rows; the partial
// sums meet in a 3-level butterfly.  Shared-memory reads of one particle
// (one 8-lane phase of a 128-bit load) are conflict-free because rows k and
// k+2 are PS = 4 (mod 8) float4 apart.  Returns ok (all axes finite).
template <typename Tc, int NC, bool GRAD>
__device__ __forceinline__ bool gather8(const float4* __restrict__ halo, int PS, int Sx,
                                        const Recs& R, int i, const GridArgs& g,
                                        const Tc* __restrict__ coef,
                                        const float* __restrict__ scale, int q, int kh,
                                        float out[NC], float dx[NC], float dy[NC],
                                        float dz[NC]) {
  const float bxq = reinterpret_cast<const float*>(R.b(0))[4 * i + q];
  const float4 by = R.b(1)[i];
  const float2 bzp = reinterpret_cast<const float2*>(R.b(2))[2 * i + kh];
  const float bz[2] = {bzp.x, bzp.y};
  const int w = R.lw()[i];
  const bool ok = (__vcmpeq4(w, 0xfefefefe) & 0x00ffffff) == 0;
  const bool inh = (w & 0x00808080) == 0;
  float4 dby = make_float4(0.f, 0.f, 0.f, 0.f);
  float dbz[2] = {0.f, 0.f};
  if (GRAD) {
    dby = R.db(1)[i];
    const float2 d2 = reinterpret_cast<const float2*>(R.db(2))[2 * i + kh];
    dbz[0] = d2.x;
    dbz[1] = d2.y;
  }
  float acc[NC], accy[NC], accz[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) acc[c] = accy[c] = accz[c] = 0.f;
  if (inh) {
    const int lx = (signed char)(w & 0xff), ly = (signed char)((w >> 8) & 0xff),
              lz = (signed char)((w >> 16) & 0xff);
    const float4* hp = halo + (lz + kh) * PS + ly * Sx + lx + q;
#pragma unroll
    for (int kk = 0; kk < 2; ++kk) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float4 v = hp[2 * kk * PS + j * Sx];
        const float vv[3] = {v.x, v.y, v.z};
        const float w = f4get(by, j) * bz[kk];
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[c] = fmaf(w, vv[c], acc[c]);
        if (GRAD) {
          const float wy = f4get(dby, j) * bz[kk], wz = f4get(by, j) * dbz[kk];
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            accy[c] = fmaf(wy, vv[c], accy[c]);
            accz[c] = fmaf(wz, vv[c], accz[c]);
          }
        }
      }
    }
  } else {
    const int ax = max(R.cell(0)[i], 0), ay = max(R.cell(1)[i], 0), az = max(R.cell(2)[i], 0);
#pragma unroll
    for (int kk = 0; kk < 2; ++kk) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float w = f4get(by, j) * bz[kk];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const float v = (float)load_coef<Tc>(coef, scale, g, c, az + kh + 2 * kk, ay + j, ax + q);
          acc[c] = fmaf(w, v, acc[c]);
          if (GRAD) {
            accy[c] = fmaf(f4get(dby, j) * bz[kk], v, accy[c]);
            accz[c] = fmaf(f4get(by, j) * dbz[kk], v, accz[c]);
          }
        }
      }
    }
  }
#pragma unroll
  for (int c = 0; c < NC; ++c) out[c] = group_sum<8>(bxq * acc[c]);
  if (GRAD) {
    const float dbxq = reinterpret_cast<const float*>(R.db(0))[4 * i + q];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      dx[c] = group_sum<8>(dbxq * acc[c]) * g.inv_hf[0];
      dy[c] = group_sum<8>(bxq * accy[c]) * g.inv_hf[1];
      dz[c] = group_sum<8>(bxq * accz[c]) * g.inv_hf[2];
    }
  }
  return ok;
}

// Particles [beg, end) of one brick whose halo is in shared memory, in rounds
// of kRecords:
//   A  one thread per (particle, axis): locate (exact FP64 index arithmetic),
//      basis along the axis, brick-local index;
//   B  8 lanes per particle: gather, sum and store.
template <typename Tc, int NC, int MODE, int KS = 0>
__device__ __forceinline__ void process_brick(const StagedArgs& a, int beg, int end,
                                              const int P0[3], const float4* halo,
                                              const Recs& R) {
  constexpr bool GRAD = MODE == 1;
  const GridArgs& g = a.g;
  const Tc* coef = static_cast<const Tc*>(a.coef);
  const int tid = threadIdx.x, lane = tid & 31;
  const int q = lane & 3, kh = (lane >> 2) & 1, sub = lane & 7;
  const int warp = tid >> 5, nwarps = blockDim.x >> 5;
  const int64_t np = a.np;
  const float nanf_ = __int_as_float(0x7fc00000);
  const HaloGeo<KS> hg(a);

  for (unsigned cb = beg; cb < (unsigned)end; cb += kRecords) {  // (to beyond 2^31)
    const int m = (int)min((unsigned)kRecords, (unsigned)end - cb);
    // phase A: tasks (particle i, axis d), task = d * m + i
    for (int task = tid; task < 3 * m; task += kThreads) {
      const int d = task < m ? 0 : (task < 2 * m ? 1 : 2), i = task - d * m;
      const int64_t p = a.perm ? a.perm[cb + i] : (int64_t)(cb + i);
      int cell;
      float t;
      const bool ok = locate(a.pos_in[d * np + p], g.inv_h[d], g.n[d], cell, t);
      write_axis<GRAD>(R, i, d, cell, t, ok, sel3(P0, d),
                       d == 0 ? hg.Sx : (d == 1 ? hg.Sy : hg.Sz));
    }
    __syncthreads();
    // phase B: gathers, 8 lanes per particle; the loop is uniform per warp
    // (the butterfly uses full-warp shuffles), idle groups redo record b4
    for (int b4 = warp * 4; b4 < m; b4 += nwarps * 4) {
      const int i = b4 + (lane >> 3);
      const bool vi = i < m;
      float u[NC], dx[NC], dy[NC], dz[NC];
      const bool oki = gather8<Tc, NC, GRAD>(halo, hg.PS, hg.SX, R, vi ? i : b4, g, coef, a.scale,
                                             q, kh, u, dx, dy, dz);
      if (!vi) continue;
      const int64_t pi = a.perm ? a.perm[cb + i] : (int64_t)(cb + i);
#pragma unroll
      for (int c = 0; c < NC; ++c)
        if (sub == c) a.vel[(int64_t)c * np + pi] = oki ? u[c] : nanf_;
      if (GRAD && a.grad) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          if (sub == 3) a.grad[((int64_t)c * 3 + 0) * np + pi] = oki ? dx[c] : nanf_;
          if (sub == 4) a.grad[((int64_t)c * 3 + 1) * np + pi] = oki ? dy[c] : nanf_;
          if (sub == 5) a.grad[((int64_t)c * 3 + 2) * np + pi] = oki ? dz[c] : nanf_;
        }
      }
      if (sub == 7 && !oki) flag_status(a.status, PS_DEV_NONFINITE_POS, pi);
    }
    __syncthreads();
  }
}

// Phased form of one brick: stage the halo (unless the brick holds fewer than
// min_stage particles, whose stencils are then read from global memory), then
// the location and gather phases of process_brick.
template <typename Tc, int NC, int MODE>
__device__ __forceinline__ void brick_phased(const StagedArgs& a, int bin, float4* smem) {
  const int beg = a.offs[bin], end = a.offs[bin + 1];
  if (beg >= end) return;
  const int nbx = a.b.nb[0], nby = a.b.nb[1];
  const int bzi = bin / (nbx * nby);
  const int rem = bin - bzi * nbx * nby;
  const int byi = rem / nbx, bxi = rem - byi * nbx;
  const int P0[3] = {bxi * a.b.B[0] - a.E, byi * a.b.B[1] - a.E, bzi * a.b.B[2] - a.E};
  const Tc* coef = static_cast<const Tc*>(a.coef);
  float4* halo = smem;
  const Recs R = carve_recs<MODE == 1>(smem + a.S[2] * a.PS);
  if (end - beg < a.min_stage) {
    // an origin far from every cell sends every stencil to global memory
    const int far[3] = {-(1 << 29), -(1 << 29), -(1 << 29)};
    process_brick<Tc, NC, MODE>(a, beg, end, far, halo, R);
    return;
  }
  // no barrier here: phase A of the first round does not read the halo, and
  // the barrier that follows it also publishes the staged halo
  if (a.vec && is_cube11(a)) {
    stage_halo_vec<Tc, NC, 11>(a, coef, P0, halo, false, a.scale);
    process_brick<Tc, NC, MODE, 11>(a, beg, end, P0, halo, R);
    return;
  }
  if (a.vec)
    stage_halo_vec<Tc, NC>(a, coef, P0, halo, false, a.scale);
  else
    stage_halo<Tc, NC>(a, coef, P0, halo, false, a.scale);
  process_brick<Tc, NC, MODE>(a, beg, end, P0, halo, R);
}

// One component.  MODE 0: vel; 1: vel + grad.  One CTA per brick.
template <typename Tc, int NC, int MODE>
__global__ void __launch_bounds__(kThreads, 7) interp_staged(const __grid_constant__ StagedArgs a) {
  extern __shared__ __align__(128) float4 smem_a128[];
  brick_phased<Tc, NC, MODE>(a, blockIdx.x, smem_a128);
}

// ------------------------------------------------- thread per particle ----
// One thread carries a particle through every step: exact location, the 12
// basis values, its 64 stencil points read from the staged halo (128-bit
// loads; lanes of a warp hit random banks, the price of needing no records,
// shuffles or further barriers), the Heun predictor and the FP64 update.

template <int NC, bool GRAD>
struct Sum1 {
  float u[NC], gx[NC], gy[NC], gz[NC];
};

// 64-term sum of Eq. (spline) by one thread; `row(k, j)` returns the four
// x-consecutive points of stencil row (j, k) as float4 (u, v, w, -).
template <int NC, bool GRAD, typename RowFn>
__device__ __forceinline__ void sum64(const float bx[4], const float by[4], const float bz[4],
                                      const float dbx[4], const float dby[4], const float dbz[4],
                                      RowFn row, Sum1<NC, GRAD>& r) {
#pragma unroll
  for (int c = 0; c < NC; ++c) r.u[c] = r.gx[c] = r.gy[c] = r.gz[c] = 0.f;
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float4 v[4];
      row(k, j, v);
      const float w = by[j] * bz[k];
      float wy = 0.f, wz = 0.f;
      if (GRAD) {
        wy = dby[j] * bz[k];
        wz = by[j] * dbz[k];
      }
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const float v0 = c == 0 ? v[0].x : (c == 1 ? v[0].y : v[0].z);
        const float v1 = c == 0 ? v[1].x : (c == 1 ? v[1].y : v[1].z);
        const float v2 = c == 0 ? v[2].x : (c == 1 ? v[2].y : v[2].z);
        const float v3 = c == 0 ? v[3].x : (c == 1 ? v[3].y : v[3].z);
        float sx = bx[0] * v0;
        sx = fmaf(bx[1], v1, sx);
        sx = fmaf(bx[2], v2, sx);
        sx = fmaf(bx[3], v3, sx);
        r.u[c] = fmaf(w, sx, r.u[c]);
        if (GRAD) {
          float dx = dbx[0] * v0;
          dx = fmaf(dbx[1], v1, dx);
          dx = fmaf(dbx[2], v2, dx);
          dx = fmaf(dbx[3], v3, dx);
          r.gx[c] = fmaf(w, dx, r.gx[c]);
          r.gy[c] = fmaf(wy, sx, r.gy[c]);
          r.gz[c] = fmaf(wz, sx, r.gz[c]);
        }
      }
    }
}

template <typename Tc, int NC, bool GRAD>
__device__ __forceinline__ void gather1(const StagedArgs& a, const Tc* __restrict__ coef,
                                        const float* __restrict__ scale,
                                        const float4* __restrict__ halo, const int P0[3],
                                        const int cell[3], const float t[3],
                                        Sum1<NC, GRAD>& r) {
  const GridArgs& g = a.g;
  float bx[4], by[4], bz[4], dbx[4], dby[4], dbz[4];
  bspline<float>(t[0], bx);
  bspline<float>(t[1], by);
  bspline<float>(t[2], bz);
  if (GRAD) {
    dbspline<float>(t[0], dbx);
    dbspline<float>(t[1], dby);
    dbspline<float>(t[2], dbz);
  }
  const int lx = cell[0] - P0[0], ly = cell[1] - P0[1], lz = cell[2] - P0[2];
  const bool inh = (unsigned)lx <= (unsigned)(a.S[0] - 4) &&
                   (unsigned)ly <= (unsigned)(a.S[1] - 4) &&
                   (unsigned)lz <= (unsigned)(a.S[2] - 4);
  if (inh) {
    const float4* base = halo + lz * a.PS + ly * a.SX + lx;
    const int PS = a.PS, Sx = a.SX;
    sum64<NC, GRAD>(bx, by, bz, dbx, dby, dbz,
                    [&](int k, int j, float4 v[4]) {
                      const float4* rp = base + k * PS + j * Sx;
                      v[0] = rp[0];
                      v[1] = rp[1];
                      v[2] = rp[2];
                      v[3] = rp[3];
                    },
                    r);
  } else {
    sum64<NC, GRAD>(bx, by, bz, dbx, dby, dbz,
                    [&](int k, int j, float4 v[4]) {
#pragma unroll
                      for (int i = 0; i < 4; ++i) {
                        float vv[3] = {0.f, 0.f, 0.f};
#pragma unroll
                        for (int c = 0; c < NC; ++c)
                          vv[c] = load_coef<Tc>(coef, scale, g, c, cell[2] + k, cell[1] + j,
                                                cell[0] + i);
                        v[i] = make_float4(vv[0], vv[1], vv[2], 0.f);
                      }
                    },
                    r);
  }
  if (GRAD) {
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      r.gx[c] *= g.inv_hf[0];
      r.gy[c] *= g.inv_hf[1];
      r.gz[c] *= g.inv_hf[2];
    }
  }
}

template <typename Tc, int NC, int MODE>
__global__ void __launch_bounds__(64) interp_thread(StagedArgs a) {
  extern __shared__ float4 smem[];
  constexpr bool GRAD = MODE == 1;
  const int bin = blockIdx.x;
  const int beg = a.offs[bin], end = a.offs[bin + 1];
  if (beg >= end) return;
  const int nbx = a.b.nb[0], nby = a.b.nb[1];
  const int bzi = bin / (nbx * nby);
  const int rem = bin - bzi * nbx * nby;
  const int byi = rem / nbx, bxi = rem - byi * nbx;
  const int P0[3] = {bxi * a.b.B[0] - a.E, byi * a.b.B[1] - a.E, bzi * a.b.B[2] - a.E};
  const Tc* coef = static_cast<const Tc*>(a.coef);
  float4* halo = smem;
  if (a.vec)
    stage_halo_vec<Tc, NC>(a, coef, P0, halo, true, a.scale);
  else
    stage_halo<Tc, NC>(a, coef, P0, halo, true, a.scale);
  const GridArgs& g = a.g;
  const int64_t np = a.np;
  const float nanf_ = __int_as_float(0x7fc00000);
  for (unsigned s = beg + threadIdx.x; s < (unsigned)end; s += blockDim.x) {
    const int64_t p = a.perm ? a.perm[s] : (int64_t)s;
    double x[3];
    int cell[3];
    float t[3];
    bool ok = true;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      x[d] = a.pos_in[d * np + p];
      ok &= locate(x[d], g.inv_h[d], g.n[d], cell[d], t[d]);
    }
    Sum1<NC, GRAD> r;
    gather1<Tc, NC, GRAD>(a, coef, a.scale, halo, P0, cell, t, r);
    if constexpr (MODE <= 1) {
#pragma unroll
      for (int c = 0; c < NC; ++c) a.vel[(int64_t)c * np + p] = ok ? r.u[c] : nanf_;
      if (GRAD && a.grad) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          a.grad[((int64_t)c * 3 + 0) * np + p] = ok ? r.gx[c] : nanf_;
          a.grad[((int64_t)c * 3 + 1) * np + p] = ok ? r.gy[c] : nanf_;
          a.grad[((int64_t)c * 3 + 2) * np + p] = ok ? r.gz[c] : nanf_;
        }
      }
      if (!ok) flag_status(a.status, PS_DEV_NONFINITE_POS, p);
    } else {
      const float u1[3] = {r.u[0], r.u[1], r.u[2]};
      int c2[3];
      float t2[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        float tt = t[d] + (ok ? u1[d] * a.dtih[d] : 0.f);
        float fl = floorf(tt);
        if (!(fabsf(fl) < 1.0e9f)) fl = 0.f;
        t2[d] = fminf(fmaxf(tt - fl, 0.f), 1.f);
        int c = cell[d] + (int)fl;
        if (c < 0 || c >= g.n[d]) {
          c %= g.n[d];
          if (c < 0) c += g.n[d];
        }
        c2[d] = c;
      }
      Sum1<NC, false> r2;
      if (a.coef2) {
        // second field: its coefficients are not staged
        int far[3] = {P0[0] - 1000000, 0, 0};
        gather1<Tc, NC, false>(a, static_cast<const Tc*>(a.coef2), a.scale2, halo, far, c2, t2,
                               r2);
      } else {
        gather1<Tc, NC, false>(a, coef, a.scale, halo, P0, c2, t2, r2);
      }
      const double half_dt = a.dt * 0.5;
      int bc[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const double xn = ok ? fma(half_dt, (double)(u1[d] + r2.u[d]), x[d])
                             : __longlong_as_double(0x7ff8000000000000ll);
        a.pos_out[d * np + p] = xn;
        if (a.vel) a.vel[d * np + p] = ok ? u1[d] : nanf_;
        bc[d] = a.next_counts ? brick_coord(g, a.b, xn, d) : 0;
      }
      if (a.ids_out) a.ids_out[p] = a.ids_in[p];
      if (!ok) flag_status(a.status, PS_DEV_NONFINITE_POS, p);
      if (a.next_counts) {
        // the next step's counting, one atomic per particle (this loop's
        // lanes leave it at different trips)
        int key = bin_of_coords(a.b, bc[0], bc[1], bc[2]);
        if (key < 0) {
          flag_status(a.status, PS_DEV_NONFINITE_POS, p);
          key = 0;
        }
        a.next_bin[p] = key;
        atomicAdd(&a.next_counts[key], 1);
      }
    }
  }
}

// ------------------------------------------------------------------ host ----

template <typename F>
ps_status with_coef_type(ps_dtype t, F&& f) {
  switch (t) {
    case PS_F32: return f(float{});
    case PS_F64: return f(double{});
    case PS_BF16: return f(__nv_bfloat16{});
    case PS_F16: return f(__half{});
    case PS_F32X4: return f(float4{});
    case PS_BF16X4: return f(bf16x4{});
    case PS_F16X4: return f(f16x4{});
  }
  return fail(PS_ERR_INVALID_ARG, "bad coefficient dtype %d", (int)t);
}

ps_status check_coef(ps_dtype coef_t, const void* coef, const float* scale) {
  if (coef_t != PS_F32 && coef_t != PS_F64 && coef_t != PS_BF16 && coef_t != PS_F16 &&
      coef_t != PS_F32X4 && coef_t != PS_BF16X4 && coef_t != PS_F16X4)
    return fail(PS_ERR_INVALID_ARG, "bad coefficient dtype %d", (int)coef_t);
  if (!coef) return fail(PS_ERR_INVALID_ARG, "coef is NULL");
  if ((coef_t == PS_BF16 || coef_t == PS_F16 || coef_t == PS_BF16X4 || coef_t == PS_F16X4) &&
      !scale)
    return fail(PS_ERR_INVALID_ARG, "scale required for BF16/F16 coefficients");
  return PS_OK;
}

unsigned quad_blocks(int64_t np) { return (unsigned)((np * 4 + 255) / 256); }

int plane_stride(int sx, int sy) {
  int ps = sx * sy;
  while ((ps & 7) != 4) ++ps;
  return ps;
}

}  // namespace

ps_status fill_staged(const ps_grid* grid, ps_dtype coef_t, const int32_t brick[3], int E,
                      bool grad, StagedArgs* a, size_t* smem) {
  ps_status rc = make_brick_args(grid, brick, &a->b);
  if (rc) return rc;
  a->g = make_grid_args(grid, coef_t);
  a->E = E;
  for (int d = 0; d < 3; ++d) {
    a->S[d] = a->b.B[d] + 3 + 2 * E;
    const int B = a->b.B[d];
    a->bshift[d] = (B & (B - 1)) ? -1 : __builtin_ctz((unsigned)B);
    const double xg = 1073741824.0 / a->g.inv_h[d];  // 2^30 cells
    int64_t bits;
    memcpy(&bits, &xg, sizeof(bits));
    a->xguard_hi[d] = (int)(bits >> 32);
  }
  if (a->S[0] > 32) return fail(PS_ERR_UNSUPPORTED, "brick x extent above 29 cells");
  a->SX = a->S[0];
  a->PS = plane_stride(a->SX, a->S[1]);
  // vector staging needs E = 0, bricks tiling the grid, 16-byte-aligned halo
  // rows and the last row vector inside the row pitch
  const int V = coef_t == PS_F32 ? 4 : (coef_t == PS_BF16 || coef_t == PS_F16 ? 8 : 0);
  bool vec = E == 0 && V > 0 && a->b.B[0] % V == 0;
  for (int d = 0; d < 3; ++d) vec = vec && grid->n[d] % a->b.B[d] == 0;
  const int qx = (a->S[0] + V - 1) / (V > 0 ? V : 1);
  vec = vec && qx <= 4 && (a->b.nb[0] - 1) * a->b.B[0] + qx * V <= a->g.rx;
  if (coef_t == PS_F32X4 || coef_t == PS_BF16X4 || coef_t == PS_F16X4) {
    // node rows: any x offset is a whole node; the halo stays inside
    // the padded array when the bricks tile the grid
    vec = E == 0;
    for (int d = 0; d < 3; ++d) vec = vec && grid->n[d] % a->b.B[d] == 0;
    // rows padded so that a plane is 4 (mod 8) nodes long
    for (int sx = a->S[0]; vec && sx < a->S[0] + 8; ++sx)
      if ((sx * a->S[1]) % 8 == 4) {
        a->SX = sx;
        a->PS = sx * a->S[1];
        break;
      }
  }
  a->vec = vec ? 1 : 0;
  a->tma = 0;
  a->min_stage = tuning().brick_min_stage;
  a->wait_probe = tuning().wait_probe;
  const size_t halo = (size_t)a->S[2] * a->PS * sizeof(float4);
  *smem = halo + rec_bytes(grad);
  if (halo + (grad ? 10240 : 7360) > 227 * 1024)
    return fail(PS_ERR_UNSUPPORTED, "brick halo exceeds shared memory");
  return PS_OK;
}

// Tensor map of the halo box over the coefficients (nodes: S[2] planes of PS / SX
// rows of SX nodes; planar FP32: rows of SX floats of the three components); the
// driver's encoder is looked up once.
bool encode_node_halo_map(StagedArgs* a, ps_dtype coef_t) {
  static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  static bool looked = false;
  static std::mutex mu;
  {
    std::lock_guard<std::mutex> lock(mu);
    if (!looked) {
      looked = true;
      cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
      void* fn = nullptr;
      if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault,
                                           &q) == cudaSuccess &&
          q == cudaDriverEntryPointSuccess)
        encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
      else
        cudaGetLastError();
    }
  }
  if (!encode) return false;
  const GridArgs& g = a->g;
  const cuuint32_t unit[3] = {1, 1, 1};
  const cuuint64_t m1 = (cuuint64_t)g.m[1], m2 = (cuuint64_t)g.m[2], rx = (cuuint64_t)g.rx;
  // a box holds at most 256 values per axis
  const cuuint32_t rows = (cuuint32_t)(a->PS / a->SX);
  if (rows > 256 || a->S[2] > 256 || (coef_t == PS_F32 ? 1 : 4) * a->SX > 256) return false;
  if (coef_t == PS_F32) {
    // planar: [3][m2][m1][rx] floats, the box's three components one behind the other
    const cuuint64_t pd[4] = {rx, m1, m2, 3};
    const cuuint64_t ps[3] = {rx * 4, rx * m1 * 4, rx * m1 * m2 * 4};
    const cuuint32_t pb[4] = {(cuuint32_t)a->SX, rows, (cuuint32_t)a->S[2], 3};
    const cuuint32_t pu[4] = {1, 1, 1, 1};
    return encode(&a->tmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<void*>(a->coef), pd, ps,
                  pb, pu, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
  }
  const cuuint64_t dims[3] = {4 * rx, m1, m2};
  const cuuint32_t box[3] = {4 * (cuuint32_t)a->SX, rows, (cuuint32_t)a->S[2]};
  const cuuint64_t nb = coef_t == PS_F32X4 ? 16 : 8;  // bytes of a node
  const cuuint64_t strides[2] = {rx * nb, rx * m1 * nb};
  const CUtensorMapDataType t = coef_t == PS_F32X4    ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                : coef_t == PS_BF16X4 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                                      : CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
  if (encode(&a->tmap, t, 3, const_cast<void*>(a->coef), dims, strides, box, unit,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return false;
  if (coef_t == PS_F32X4) return true;
  // 16-bit nodes: the rows' scales (s_u, s_v, s_w, 1), [m2][m1][4] floats
  if (4 * a->S[1] > 256) return false;
  const cuuint64_t sdims[2] = {4 * m1, m2};
  const cuuint64_t sstrides[1] = {m1 * 16};
  const cuuint32_t sbox[2] = {4 * (cuuint32_t)a->S[1], (cuuint32_t)a->S[2]};
  return encode(&a->tmap2, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(a->scale),
                sdims, sstrides, sbox, unit, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

namespace {

template <typename Tc> struct DtypeOf { static constexpr int v = -1; };
template <> struct DtypeOf<float> { static constexpr int v = PS_F32; };
template <> struct DtypeOf<float4> { static constexpr int v = PS_F32X4; };
template <> struct DtypeOf<__nv_bfloat16> { static constexpr int v = PS_BF16; };
template <> struct DtypeOf<__half> { static constexpr int v = PS_F16; };
template <> struct DtypeOf<bf16x4> { static constexpr int v = PS_BF16X4; };
template <> struct DtypeOf<f16x4> { static constexpr int v = PS_F16X4; };

template <typename Tc, int NC, int MODE>
ps_status launch_staged(const StagedArgs& a, size_t smem, cudaStream_t st,
                        float* rows_ws = nullptr) {
  // three components take the quad form (brick_kernel 2: the thread per
  // particle), one the phased kernel
  const int k = tuning().brick_kernel;
  if constexpr (NC == 3 && DtypeOf<Tc>::v >= 0) {
    if (k != 2) return launch_quad(a, (ps_dtype)DtypeOf<Tc>::v, MODE, st, rows_ws);
  }
  if (k == 2) {
    auto tk = interp_thread<Tc, NC, MODE>;
    const size_t hs = (size_t)a.S[2] * a.PS * sizeof(float4);
    if (hs > 48 * 1024) {
      ps_status rc = check_cuda(
          cudaFuncSetAttribute(tk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)hs),
          "thread-kernel smem attribute");
      if (rc) return rc;
    }
    tk<<<(unsigned)a.b.nbins, 64, hs, st>>>(a);
    return check_launch("interp_thread");
  }
  if constexpr (NC == 1 && MODE <= 1) {
    auto kern = interp_staged<Tc, NC, MODE>;
    if (smem > 48 * 1024) {
      ps_status rc = check_cuda(
          cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
          "staged smem attribute");
      if (rc) return rc;
    }
    if (a.b.nbins > 0x7fffffff) return fail(PS_ERR_UNSUPPORTED, "too many bins");
    kern<<<(unsigned)a.b.nbins, kThreads, smem, st>>>(a);
    return check_launch("interp_staged");
  } else {
    return fail(PS_ERR_UNSUPPORTED, "no brick kernel for this case");
  }
}

}  // namespace

float3 dt_over_h(const GridArgs& g, double dt) {
  return make_float3((float)(dt * g.inv_h[0]), (float)(dt * g.inv_h[1]),
                     (float)(dt * g.inv_h[2]));
}

// RK2 kernels used by ps_rk2_step (rk2.cu).
ps_status rk2_launch_direct(const ps_grid* grid, ps_dtype coef_t, const void* c0,
                            const float* s0, const void* c1, const float* s1, int64_t np,
                            double* pos, float* vel_out, double dt, int32_t* status,
                            cudaStream_t st) {
  GridArgs g = make_grid_args(grid, coef_t);
  const float3 dtih = dt_over_h(g, dt);
  return with_coef_type(coef_t, [&](auto tag) -> ps_status {
    using Tc = decltype(tag);
    rk2_direct<Tc><<<quad_blocks(np), 256, 0, st>>>(g, static_cast<const Tc*>(c0), s0,
                                                    static_cast<const Tc*>(c1), s1, np, pos,
                                                    vel_out, dt, dtih, status);
    return check_launch("rk2_direct");
  });
}

ps_status rk2_launch_staged(const ps_grid* grid, const int32_t brick[3], int E,
                            ps_dtype coef_t, const void* c0, const float* s0,
                            const void* c1, const float* s1, int64_t np,
                            const double* pos_in, double* pos_out, const int32_t* offs,
                            float* vel_out, const int64_t* ids_in, int64_t* ids_out,
                            double dt, int32_t* status, int32_t* next_counts,
                            int32_t* next_bin, cudaStream_t st) {
  if (coef_t == PS_F64)
    return fail(PS_ERR_UNSUPPORTED, "staged RK2 needs F32/BF16/F16 coefficients");
  StagedArgs a{};
  size_t smem;
  ps_status rc = fill_staged(grid, coef_t, brick, E, false, &a, &smem);
  if (rc) return rc;
  a.coef = c0;
  a.scale = s0;
  a.coef2 = c1;
  a.scale2 = s1;
  a.np = np;
  a.pos_in = pos_in;
  a.pos_out = pos_out;
  a.offs = offs;
  a.vel = vel_out;
  a.ids_in = ids_in;
  a.ids_out = ids_out;
  a.dt = dt;
  const float3 d = dt_over_h(a.g, dt);
  a.dtih[0] = d.x;
  a.dtih[1] = d.y;
  a.dtih[2] = d.z;
  a.status = status;
  a.next_counts = next_counts;
  a.next_bin = next_bin;
  return with_coef_type(coef_t, [&](auto tag) -> ps_status {
    using Tc = decltype(tag);
    if constexpr (std::is_same<Tc, double>::value) return PS_ERR_UNSUPPORTED;
    else return launch_staged<Tc, 3, 2>(a, smem, st);
  });
}

}  // namespace ps

using namespace ps;

// The workspace for `rows` result rows in bin order, if the caller gave one
// that holds them and there is a permutation to undo; else NULL (the results
// are stored where they belong, one particle at a time).
static float* result_rows(const int64_t* perm, int64_t np, int rows, void* ws, size_t ws_bytes) {
  if (!perm || !ws || (reinterpret_cast<uintptr_t>(ws) & 255)) return nullptr;
  return ws_bytes >= ps_unsort_workspace_size(np, rows) ? static_cast<float*>(ws) : nullptr;
}

extern "C" ps_status ps_interp(const ps_grid* grid, int ncomp, ps_dtype coef_t,
                               const void* coef, const float* scale, int64_t np,
                               const double* pos, const int64_t* perm,
                               const int32_t* bin_offsets, const int32_t brick[3],
                               float* vel, float* grad, int32_t* status, void* stream) {
  return ps_interp_ws(grid, ncomp, coef_t, coef, scale, np, pos, perm, bin_offsets, brick, vel,
                      grad, nullptr, 0, status, stream);
}

extern "C" ps_status ps_interp_ws(const ps_grid* grid, int ncomp, ps_dtype coef_t,
                                  const void* coef, const float* scale, int64_t np,
                                  const double* pos, const int64_t* perm,
                                  const int32_t* bin_offsets, const int32_t brick[3],
                                  float* vel, float* grad, void* ws, size_t ws_bytes,
                                  int32_t* status, void* stream) {
  ps_status rc = validate_grid(grid);
  if (rc) return rc;
  if (ncomp != 1 && ncomp != 3) return fail(PS_ERR_INVALID_ARG, "ncomp must be 1 or 3");
  if ((coef_t == PS_F32X4 || coef_t == PS_BF16X4 || coef_t == PS_F16X4) && ncomp != 3)
    return fail(PS_ERR_INVALID_ARG, "node coefficients need ncomp == 3");
  if ((rc = check_coef(coef_t, coef, scale))) return rc;
  if (np < 0) return fail(PS_ERR_INVALID_ARG, "np < 0");
  if (np == 0) return PS_OK;
  if (!pos || !vel) return fail(PS_ERR_INVALID_ARG, "pos and vel are required");
  if (perm && !bin_offsets) return fail(PS_ERR_INVALID_ARG, "perm needs bin_offsets");
  if (bin_offsets && !brick) return fail(PS_ERR_INVALID_ARG, "bin_offsets needs brick");
  cudaStream_t st = as_stream(stream);
  GridArgs g = make_grid_args(grid, coef_t);
  const bool staged = bin_offsets && coef_t != PS_F64;
  if (!staged) {
    return with_coef_type(coef_t, [&](auto tag) -> ps_status {
      using Tc = decltype(tag);
      const Tc* c = static_cast<const Tc*>(coef);
      if (ncomp == 3) {
        if (grad)
          interp_direct<Tc, 3, 1><<<quad_blocks(np), 256, 0, st>>>(
              g, c, scale, np, pos, perm, vel, grad, nullptr, nullptr, status);
        else
          interp_direct<Tc, 3, 0><<<quad_blocks(np), 256, 0, st>>>(
              g, c, scale, np, pos, perm, vel, nullptr, nullptr, nullptr, status);
      } else {
        if (grad)
          interp_direct<Tc, 1, 1><<<quad_blocks(np), 256, 0, st>>>(
              g, c, scale, np, pos, perm, vel, grad, nullptr, nullptr, status);
        else
          interp_direct<Tc, 1, 0><<<quad_blocks(np), 256, 0, st>>>(
              g, c, scale, np, pos, perm, vel, nullptr, nullptr, nullptr, status);
      }
      return check_launch("interp_direct");
    });
  }
  StagedArgs a{};
  size_t smem;
  if ((rc = fill_staged(grid, coef_t, brick, 0, grad != nullptr, &a, &smem))) return rc;
  a.coef = coef;
  a.scale = scale;
  a.np = np;
  a.pos_in = pos;
  a.perm = perm;
  a.offs = bin_offsets;
  a.vel = vel;
  a.grad = grad;
  a.status = status;
  return with_coef_type(coef_t, [&](auto tag) -> ps_status {
    using Tc = decltype(tag);
    if constexpr (std::is_same<Tc, double>::value) {
      return PS_ERR_UNSUPPORTED;
    } else {
      if (ncomp == 3)
        return grad ? launch_staged<Tc, 3, 1>(a, smem, st,
                                              result_rows(perm, np, 12, ws, ws_bytes))
                    : launch_staged<Tc, 3, 0>(a, smem, st,
                                              result_rows(perm, np, 3, ws, ws_bytes));
      return grad ? launch_staged<Tc, 1, 1>(a, smem, st) : launch_staged<Tc, 1, 0>(a, smem, st);
    }
  });
}

extern "C" ps_status ps_interp_backward(const ps_grid* grid, int ncomp, ps_dtype coef_t,
                                        const void* coef, const float* scale, int64_t np,
                                        const double* pos, const float* g_vel,
                                        double* g_pos, float* g_field, void* ws,
                                        size_t ws_bytes, int32_t* status, void* stream) {
  (void)ws;
  (void)ws_bytes;
  ps_status rc = validate_grid(grid);
  if (rc) return rc;
  if (ncomp != 1 && ncomp != 3) return fail(PS_ERR_INVALID_ARG, "ncomp must be 1 or 3");
  if ((coef_t == PS_F32X4 || coef_t == PS_BF16X4 || coef_t == PS_F16X4) && ncomp != 3)
    return fail(PS_ERR_INVALID_ARG, "node coefficients need ncomp == 3");
  if (np < 0) return fail(PS_ERR_INVALID_ARG, "np < 0");
  if (np > 0 && (!pos || !g_vel)) return fail(PS_ERR_INVALID_ARG, "pos and g_vel required");
  cudaStream_t st = as_stream(stream);
  GridArgs g = make_grid_args(grid, coef_t);
  if (g_pos && np > 0) {
    if ((rc = check_coef(coef_t, coef, scale))) return rc;
    rc = with_coef_type(coef_t, [&](auto tag) -> ps_status {
      using Tc = decltype(tag);
      const Tc* c = static_cast<const Tc*>(coef);
      if (ncomp == 3)
        interp_direct<Tc, 3, 2><<<quad_blocks(np), 256, 0, st>>>(
            g, c, scale, np, pos, nullptr, nullptr, nullptr, g_vel, g_pos, status);
      else
        interp_direct<Tc, 1, 2><<<quad_blocks(np), 256, 0, st>>>(
            g, c, scale, np, pos, nullptr, nullptr, nullptr, g_vel, g_pos, status);
      return check_launch("interp_backward_pos");
    });
    if (rc) return rc;
  }
  if (g_field) {
    const int64_t vol = grid_volume(grid);
    rc = check_cuda(cudaMemsetAsync(g_field, 0, sizeof(float) * vol * ncomp, st),
                    "g_field memset");
    if (rc) return rc;
    if (np > 0) {
      if (ncomp == 3)
        scatter_field<3><<<quad_blocks(np), 256, 0, st>>>(g, np, pos, g_vel, g_field, status);
      else
        scatter_field<1><<<quad_blocks(np), 256, 0, st>>>(g, np, pos, g_vel, g_field, status);
      if ((rc = check_launch("scatter_field"))) return rc;
    }
    rc = solve_unpadded_inplace_f32(grid, ncomp, g_field, st);
    if (rc) return rc;
  }
  return PS_OK;
}

extern "C" ps_status ps_interp_backward_binned(
    const ps_grid* grid, int ncomp, ps_dtype coef_t, const void* coef, const float* scale,
    int64_t np, const double* pos, const int64_t* perm, const int32_t* bin_offsets,
    const int32_t brick[3], const float* g_vel, double* g_pos, float* g_field, void* ws,
    size_t ws_bytes, int32_t* status, void* stream) {
  ps_status rc = validate_grid(grid);
  if (rc) return rc;
  if (bin_offsets && !brick) return fail(PS_ERR_INVALID_ARG, "bin_offsets needs brick");
  if (!bin_offsets) return fail(PS_ERR_INVALID_ARG, "bin_offsets is required");
  BrickArgs ba;
  if ((rc = make_brick_args(grid, brick, &ba))) return rc;
  cudaStream_t st = as_stream(stream);
  const bool three = ncomp == 3 && np > 0 && np < ((int64_t)1 << 31) && pos && g_vel;
  bool have_pos = false, have_field = false;
  if (three && g_pos) {
    // the unbinned kernel, its particles taken in bin order: neighbouring
    // quads then find one another's rows in the caches
    if ((rc = check_coef(coef_t, coef, scale))) return rc;
    const GridArgs g = make_grid_args(grid, coef_t);
    rc = with_coef_type(coef_t, [&](auto tag) -> ps_status {
      using Tc = decltype(tag);
      interp_direct<Tc, 3, 2><<<quad_blocks(np), 256, 0, st>>>(
          g, static_cast<const Tc*>(coef), scale, np, pos, perm, nullptr, nullptr, g_vel, g_pos,
          status);
      return check_launch("interp_backward_pos");
    });
    if (rc) return rc;
    have_pos = true;
  }
  if (three && g_field) {
    rc = check_cuda(cudaMemsetAsync(g_field, 0, sizeof(float) * grid_volume(grid) * ncomp, st),
                    "g_field memset");
    if (rc) return rc;
    if ((rc = scatter_bricks_launch(grid, brick, np, pos, perm, bin_offsets, g_vel, g_field,
                                    status, ws, ws_bytes, st, &have_field)))
      return rc;
    if (have_field && (rc = solve_unpadded_inplace_f32(grid, ncomp, g_field, st))) return rc;
  }
  // what the brick forms do not take (and the argument errors) goes the direct way
  if ((!g_pos || have_pos) && (!g_field || have_field) && three) return PS_OK;
  return ps_interp_backward(grid, ncomp, coef_t, coef, scale, np, pos, g_vel,
                            have_pos ? nullptr : g_pos, have_field ? nullptr : g_field, nullptr, 0,
                            status, stream);
}

// Bricks whose halos are a multiple of four rows high bring further rows into
// shared memory (quad.cu); with few particles each, the second derivatives and the
// acceleration are faster unbinned.  Particles per brick, staged / unbinned, us,
// bricks of 4 x 9 x 4.  128^3, coefficients in the L2, second derivatives: FP32 nodes
// 24 80 / 70, 32 87 / 92; planar 32 91 / 84, 48 99 / 129; planar FP16 64 268 / 206;
// acceleration from two fields: 8 64 / 48, 16 74 / 83; 24 87 / 87.  256^3, second
// derivatives: 16 474 / 358, 492 / 354; at particles in no order (perm given), whose
// unbinned stencils come from DRAM, 8 428 / 343, 435 / 639; acceleration: 8 464 / 305,
// 16 520 / 582; 16 515 / 463; in no order 4 504 / 374, 2 401 / 402.
static bool unbinned_pays(const ps_grid* grid, ps_dtype coef_t, const int32_t brick[3],
                          int64_t np, const int64_t* perm, bool accel) {
  StagedArgs a{};
  size_t smem;
  if ((brick[1] + 3) % 4 || fill_staged(grid, coef_t, brick, 0, false, &a, &smem))
    return false;  // (what the staged form refuses stays refused)
  const bool nodes = coef_t == PS_F32X4 || coef_t == PS_BF16X4 || coef_t == PS_F16X4;
  const bool in_l2 = (double)grid_volume(grid) * (double)dtype_size(coef_t) * (nodes ? 1 : 3) < 64e6;
  double least = in_l2 ? (nodes ? 64.0 : 80.0) : !perm ? 36.0 : nodes ? 20.0 : 10.0;
  if (accel) least *= 0.5;  // per 11^3 halo nodes
  return (double)np * 1331.0 < least * (double)a.S[0] * a.S[1] * a.S[2] * (double)a.b.nbins;
}

// Brick-staged form of the second derivatives (mode 3) or the Lagrangian
// acceleration (mode 4) by the quad kernel.
static ps_status staged_extra(const ps_grid* grid, ps_dtype coef_t, const void* coef,
                              const float* scale, const void* coef2, const float* scale2,
                              double inv_dt, int64_t np, const double* pos,
                              const int64_t* perm, const int32_t* bin_offsets,
                              const int32_t brick[3], float* out, float* vel, float* rows_ws,
                              int32_t* status, int mode, cudaStream_t st) {
  StagedArgs a{};
  size_t smem;
  ps_status rc = fill_staged(grid, coef_t, brick, 0, false, &a, &smem);
  if (rc) return rc;
  a.coef = coef;
  a.scale = scale;
  a.coef2 = coef2;
  a.scale2 = scale2;
  a.np = np;
  a.pos_in = pos;
  a.perm = perm;
  a.offs = bin_offsets;
  a.grad = out;
  a.vel = vel;
  a.dt = inv_dt;
  a.status = status;
  return launch_quad(a, coef_t, mode, st, rows_ws);
}

extern "C" ps_status ps_interp_hessian(const ps_grid* grid, int ncomp, ps_dtype coef_t,
                                       const void* coef, const float* scale, int64_t np,
                                       const double* pos, const int64_t* perm,
                                       const int32_t* bin_offsets, const int32_t brick[3],
                                       float* hess, int32_t* status, void* stream) {
  return ps_interp_hessian_ws(grid, ncomp, coef_t, coef, scale, np, pos, perm, bin_offsets, brick,
                              hess, nullptr, 0, status, stream);
}

extern "C" ps_status ps_interp_hessian_ws(const ps_grid* grid, int ncomp, ps_dtype coef_t,
                                          const void* coef, const float* scale, int64_t np,
                                          const double* pos, const int64_t* perm,
                                          const int32_t* bin_offsets, const int32_t brick[3],
                                          float* hess, void* ws, size_t ws_bytes,
                                          int32_t* status, void* stream) {
  ps_status rc = validate_grid(grid);
  if (rc) return rc;
  if (ncomp != 1 && ncomp != 3) return fail(PS_ERR_INVALID_ARG, "ncomp must be 1 or 3");
  if ((coef_t == PS_F32X4 || coef_t == PS_BF16X4 || coef_t == PS_F16X4) && ncomp != 3)
    return fail(PS_ERR_INVALID_ARG, "node coefficients need ncomp == 3");
  if ((rc = check_coef(coef_t, coef, scale))) return rc;
  if (np < 0) return fail(PS_ERR_INVALID_ARG, "np < 0");
  if (np == 0) return PS_OK;
  if (!pos || !hess) return fail(PS_ERR_INVALID_ARG, "pos and hess are required");
  if (perm && !bin_offsets) return fail(PS_ERR_INVALID_ARG, "perm needs bin_offsets");
  if (bin_offsets && !brick) return fail(PS_ERR_INVALID_ARG, "bin_offsets needs brick");
  cudaStream_t st = as_stream(stream);
  if (bin_offsets && ncomp == 3 && coef_t != PS_F64 &&
      !unbinned_pays(grid, coef_t, brick, np, perm, false)) {
    return staged_extra(grid, coef_t, coef, scale, nullptr, nullptr, 0.0, np, pos, perm,
                        bin_offsets, brick, hess, nullptr, result_rows(perm, np, 18, ws, ws_bytes),
                        status, 3, st);
  }
  GridArgs g = make_grid_args(grid, coef_t);
  return with_coef_type(coef_t, [&](auto tag) -> ps_status {
    using Tc = decltype(tag);
    const Tc* c = static_cast<const Tc*>(coef);
    if (ncomp == 3)
      interp_hessian_direct<Tc, 3><<<quad_blocks(np), 256, 0, st>>>(g, c, scale, np, pos, hess,
                                                                     status);
    else
      interp_hessian_direct<Tc, 1><<<quad_blocks(np), 256, 0, st>>>(g, c, scale, np, pos, hess,
                                                                     status);
    return check_launch("interp_hessian_direct");
  });
}

extern "C" ps_status ps_lagrangian_accel(const ps_grid* grid, ps_dtype coef_t,
                                         const void* coef_n, const float* scale_n,
                                         const void* coef_np1, const float* scale_np1,
                                         double dt_field, int64_t np, const double* pos,
                                         const int64_t* perm, const int32_t* bin_offsets,
                                         const int32_t brick[3], float* acc, float* vel,
                                         int32_t* status, void* stream) {
  return ps_lagrangian_accel_ws(grid, coef_t, coef_n, scale_n, coef_np1, scale_np1, dt_field, np,
                                pos, perm, bin_offsets, brick, acc, vel, nullptr, 0, status,
                                stream);
}

extern "C" ps_status ps_lagrangian_accel_ws(const ps_grid* grid, ps_dtype coef_t,
                                            const void* coef_n, const float* scale_n,
                                            const void* coef_np1, const float* scale_np1,
                                            double dt_field, int64_t np, const double* pos,
                                            const int64_t* perm, const int32_t* bin_offsets,
                                            const int32_t brick[3], float* acc, float* vel,
                                            void* ws, size_t ws_bytes, int32_t* status,
                                            void* stream) {
  ps_status rc = validate_grid(grid);
  if (rc) return rc;
  if ((rc = check_coef(coef_t, coef_n, scale_n))) return rc;
  if (coef_np1 && (rc = check_coef(coef_t, coef_np1, scale_np1))) return rc;
  if (coef_np1 && !(dt_field > 0.0 && std::isfinite(dt_field)))
    return fail(PS_ERR_INVALID_ARG, "dt_field must be finite and > 0");
  if (np < 0) return fail(PS_ERR_INVALID_ARG, "np < 0");
  if (np == 0) return PS_OK;
  if (!pos || !acc) return fail(PS_ERR_INVALID_ARG, "pos and acc are required");
  if (perm && !bin_offsets) return fail(PS_ERR_INVALID_ARG, "perm needs bin_offsets");
  if (bin_offsets && !brick) return fail(PS_ERR_INVALID_ARG, "bin_offsets needs brick");
  cudaStream_t st = as_stream(stream);
  const double inv_dt = coef_np1 ? 1.0 / dt_field : 0.0;
  if (bin_offsets && coef_t != PS_F64 &&
      !unbinned_pays(grid, coef_t, brick, np, perm, true)) {
    return staged_extra(grid, coef_t, coef_n, scale_n, coef_np1, scale_np1, inv_dt, np, pos, perm,
                      bin_offsets, brick, acc, vel, result_rows(perm, np, vel ? 6 : 3, ws, ws_bytes),
                      status, 4, st);
  }
  GridArgs g = make_grid_args(grid, coef_t);
  return with_coef_type(coef_t, [&](auto tag) -> ps_status {
    using Tc = decltype(tag);
    lagrangian_accel_direct<Tc><<<quad_blocks(np), 256, 0, st>>>(
        g, static_cast<const Tc*>(coef_n), scale_n, static_cast<const Tc*>(coef_np1), scale_np1,
        inv_dt, np, pos, acc, vel, status);
    return check_launch("lagrangian_accel_direct");
  });
}
