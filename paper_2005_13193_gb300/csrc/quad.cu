// Brick-staged interpolation (Sec. 2.2, Operations 2 and 3) and the fused
// second-order Runge-Kutta particle advance (Sec. 2.1, Sec. 4.3) for three
// components: one block of two or four warps per brick of cells (brick.cuh).
//
// What bounds it (512^3, 64 particles per brick, ncu at the same density): the
// latency of each warp's chain at 13 warps per SM (37-49% of the issue slots,
// 44-61% of the shared-memory wavefronts; HBM 24-39%).  Eight blocks of 27 KB
// of halo and 64 threads of at most 128 registers fill both the shared memory
// and the register file.  Against the form with (particle, axis) tasks and
// block barriers between its phases: 29 warp instructions per particle instead
// of 61 (interpolation) and 62 instead of 104 (Heun step), 12 and 16
// shared-memory wavefronts instead of 13 and 30.  Measured there, one launch,
// before -> after: interpolation 1427 -> 1020 us, gradient tensor 1938 ->
// 1339, second derivatives 2345 -> 1792, acceleration from two fields 3007 ->
// 2655, re-binned Heun step with its sort 2596 -> 2195.  256^3 with 1.4 M
// particles and FP16 nodes: Heun step with its sort 328 -> 254.  Planar FP32,
// 256^3 with 4 M particles, halo by a planar tensor copy and gathered as three
// planes instead of loaded and interleaved: interpolation 419 -> 257, Heun step
// with its sort 683 -> 501; two snapshots of 180 x 150 x 132 with 500,000
// particles, the second halo staged beside the first instead of gathered from
// global memory: two steps 531 -> 322.  Tried and not faster: three warps of 24
// particles (spills at 96 registers: 1503), two bricks along x per block
// (1055), blocks that walk over the bricks with the next bounds and positions
// loaded ahead (1024, Heun step 2516).
#include <algorithm>
#include <cstring>
#include <type_traits>

#include "brick.cuh"

namespace ps {
namespace {

constexpr int kMaxThreads = 128;

// MODE 0: velocities; 1: velocities and the gradient tensor; 2: fused Heun
// step; 3: second derivatives; 4: Lagrangian acceleration from two fields; 5:
// from one (by itself: with the later field's sums beside it 64^3 with 4 M
// particles took 553 us, 405 now).  CT: the halo
// geometry of the 8^3 brick fixed at compile time.  The argument block is a
// grid constant so that its tensor maps can be named by the tensor copies.
template <typename Tc, int MODE, int CT>
__global__ void __launch_bounds__(kMaxThreads, 4)
    quad_kernel(const __grid_constant__ StagedArgs a) {
  extern __shared__ __align__(128) unsigned char smem_q[];
  __shared__ CopyBarriers mb;
  unsigned phase = 0;
  const int bin = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
  warp_brick<Tc, MODE, CT>(a, bin, blockIdx.x, blockIdx.y, blockIdx.z, smem_q, &a, mb,
                           phase);
}

// The halo as it lies in shared memory: rows of SX >= S[0] nodes and planes of PS
// nodes, PS / SX >= S[1] rows (the further ones are copied too and not read), the
// smallest plane whose stride spreads a quad's four z-rows over the banks.  float4
// nodes: PS = 2 (mod 4), four bank groups of one parity; 16-bit nodes and planar
// floats: rows of whole 16-byte units (`unit` values), PS an odd multiple of 4, so
// that the rows' banks are 4 apart.  Extents S[1] that are a multiple of 4 have
// such planes with further rows only (bricks of 12 x 5 x 8, 128^3, 1.5 M particles,
// interpolation without / with them, us: FP32 nodes 205 / 79, planar 227 / 102).
void halo_plane(StagedArgs* a, int unit, bool words) {
  const int r0 = (a->S[0] + unit - 1) / unit * unit;
  int best = 0;
  for (int sy = a->S[1]; sy < a->S[1] + 4; ++sy)
    for (int r = r0; r < r0 + 16; r += unit) {
      const bool ok = words ? (r & 3) == 0 && ((r * sy) & 7) == 4 : ((r * sy) & 3) == 2;
      if (!ok || (best && r * sy >= best)) continue;
      best = r * sy;
      a->SX = r;
    }
  a->PS = best;
}
template <typename Tc> struct CoefDtype { static constexpr int v = -1; };
template <> struct CoefDtype<float> { static constexpr int v = PS_F32; };
template <> struct CoefDtype<float4> { static constexpr int v = PS_F32X4; };
template <> struct CoefDtype<bf16x4> { static constexpr int v = PS_BF16X4; };
template <> struct CoefDtype<f16x4> { static constexpr int v = PS_F16X4; };

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// Tensor copies of the halo: a box's rows start on 16-byte boundaries (any
// float4 node, an even 16-bit node, every fourth planar float) and its last
// bricks may reach beyond the array (zeros that no stencil uses).
template <typename Tc>
bool halo_map(StagedArgs* a) {
  if constexpr (CoefDtype<Tc>::v < 0) {
    return false;
  } else {
    constexpr ps_dtype t = (ps_dtype)CoefDtype<Tc>::v;
    constexpr int unit = t == PS_F32X4 ? 1 : t == PS_F32 ? 4 : 2;
    if (!tuning().node_tma || a->b.B[0] % unit || a->g.rx % unit || !aligned16(a->coef)) return false;
    if (IsNode16<Tc>::value && !aligned16(a->scale)) return false;
    return encode_node_halo_map(a, t);
  }
}

// Whether a step through two fields (or an acceleration from two) stages both
// halos: from so many particles per brick on (of 11^3 halo nodes, others in
// proportion).  Below, the later field's nodes are read from global memory: one
// halo less to bring in, and twice the blocks.  256^3, one halo / both, us.  Heun
// step: FP32 nodes, 12 particles per brick 267 / 288, 24 382 / 341, 64 680 / 411;
// planar FP32 6 206 / 278, 12 250 / 238, 24 352 / 281; planar FP16 12 520 / 577, 24
// 722 / 648; 16-bit nodes (whose later halo comes by plain loads) 24 300 / 347, 64
// 440 / 457, 96 627 / 611.  Acceleration: 6 198 / 255, 12 246 / 235; 6 148 / 212,
// 12 193 / 177; 12 448 / 519, 24 586 / 589; 24 232 / 278, 64 365 / 356.  Planar 16
// bits in bricks that do not tile the grid, whose rows come value by value (250 x
// 200 x 150, Heun step): 24 493 / 670, 48 644 / 708, 96 824 / 750.
template <typename Tc>
bool second_halo_pays(const StagedArgs& a) {
  const double least = IsNode16<Tc>::value ? 64.0 : !IsQuant<Tc>::value ? 14.0 : a.vec ? 20.0 : 80.0;
  const double nodes = (double)a.S[0] * a.S[1] * a.S[2];
  return (double)a.np * 1331.0 >= least * nodes * (double)a.b.nbins;
}

// Geometry, shared memory and tensor maps of the quad form; *ct: the
// compile-time geometry that applies (0: none).
template <typename Tc>
void setup_t(StagedArgs* a, bool second, size_t* smem, int* ct) {
  constexpr bool n16 = IsNode16<Tc>::value, planar = IsPlanar<Tc>::value;
  halo_plane(a, n16 ? 2 : planar ? 4 : 1, n16 || planar);
  // planar 16-bit halos that do not come in whole vectors are widened value by value,
  // 16 or 32 lanes a row: staged from a particle per four rows on.  128^3 boxes, FP16,
  // interpolation staged / from global memory, us: bricks of 8 x 5 x 8 with 9 particles
  // 68 / 25, 17 85 / 39, 35 89 / 64; 4 x 4 x 4 with 12 255 / 110; 12^3 with 61 56 / 37,
  // 122 60 / 66; 250 x 200 x 150, 8^3 with 12 220 / 103, 24 243 / 205, 48 265 / 442.
  if (IsQuant<Tc>::value && !n16 && !a->vec)
    a->min_stage = std::max(a->min_stage, a->S[1] * a->S[2] * (a->S[0] > 16 ? 2 : 1) / 4);
  a->half_dt = 0.5 * a->dt;
  for (int d = 0; d < 3; ++d) a->ih32[d] = a->g.inv_h[d] * 4294967296.0;
  a->wait_probe = tuning().wait_probe;
  if (halo_bytes<Tc>(a->S[2], a->S[1], a->PS) > 226 * 1024) {
    // the largest halos: without the further rows and the padding
    a->SX = (a->S[0] + (planar ? 3 : n16 ? 1 : 0)) & ~(planar ? 3 : n16 ? 1 : 0);
    a->PS = a->SX * a->S[1];
  }
  *ct = a->S[0] == 11 && a->S[1] == 11 && a->S[2] == 11 && a->SX == (n16 || planar ? 12 : 14)
            ? a->SX
            : 0;
  a->two = 0;
  a->tma = halo_map<Tc>(a) ? 1 : 0;
  *smem = (size_t)halo_bytes<Tc>(a->S[2], a->S[1], a->PS);
  if (*smem > 226 * 1024) {  // no halo: every stencil from global memory
    *smem = 0;
    a->tma = 0;
    a->min_stage = 0x7fffffff;
    return;
  }
  // a second field's halo beside the first where both fit
  if (second && a->coef2 && 2 * *smem <= 226 * 1024 && second_halo_pays<Tc>(*a)) {
    a->two = 1;
    *smem *= 2;
    if constexpr (!n16) {
      // the later field's map in tmap2 (tma = 2)
      StagedArgs t = *a;
      t.coef = a->coef2;
      if (a->tma == 1 && halo_map<Tc>(&t)) {
        a->tmap2 = t.tmap;
        a->tma = 2;
      }
    }
  }
}

// Threads of a brick's block.  64 (two warps) where eight blocks share an SM; the
// registers hold four blocks of 128.  So where the halos' size (as many as fit
// into 227 KB) or the number of bricks leaves at most four blocks on an SM, 128
// take twice the particles at a time.  64^3 FP32 nodes, 64 / 128 threads, us: 512
// particles per brick, interpolation 25 / 20, gradient 33 / 27, Heun step 57 / 46;
// 2048, 78 / 60, 111 / 84, 171 / 127 (32: alike); 72^3, with five blocks on an SM,
// 88 / 91, 130 / 130, 200 / 205.  Bricks of 16^3, 128^3, 1.5 M particles: 348 /
// 189, 503 / 271, 790 / 434.  With five to seven blocks that fit, 128 pay for dense
// bricks (two planar halos, six blocks, Heun step at 256^3: 64 particles per brick
// 404 / 452, 96 565 / 518, 256 1252 / 1189).
int brick_threads(const StagedArgs& a, size_t smem) {
  const int64_t fit = std::min<int64_t>(8, 227 * 1024 / ((int64_t)smem + 1024));
  const int64_t sms = sm_count(), waiting = (a.b.nbins + sms - 1) / sms;
  if (fit <= 4) return 128;
  if (waiting <= 4) return a.np >= 64 * a.b.nbins ? 128 : 64;
  return fit < 8 && a.np >= 96 * a.b.nbins ? 128 : 64;
}

template <typename Tc, int MODE>
ps_status launch_quad_t(const StagedArgs& a0, cudaStream_t st, float* rows_ws) {
  StagedArgs a = a0;
  size_t smem;
  int ct;
  setup_t<Tc>(&a, MODE == 2 || MODE == 4, &smem, &ct);
  if (a.b.nbins > 0x7fffffff || a.b.nb[1] > 65535 || a.b.nb[2] > 65535)
    return fail(PS_ERR_UNSUPPORTED, "too many bins");
  constexpr int kCt = IsNode16<Tc>::value || IsPlanar<Tc>::value ? 12 : 14;
  auto kern = ct == kCt ? quad_kernel<Tc, MODE, kCt> : quad_kernel<Tc, MODE, 0>;
  if (smem > 48 * 1024) {
    ps_status rc = check_cuda(
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
        "quad smem attribute");
    if (rc) return rc;
  }
  const int threads = brick_threads(a, smem);
  // results by way of bin order: vel, then the gradient's or the second
  // derivatives' rows
  constexpr int rows = MODE == 1 ? 9 : MODE == 3 ? 18 : MODE >= 4 ? 3 : 0;
  const bool unsort = rows_ws && a.perm && MODE != 2;
  if (unsort) {
    a.slot_out = 1;
    a.vel = a0.vel ? rows_ws : nullptr;
    a.grad = rows_ws + (a0.vel ? 3 * a.np : 0);
  }
  kern<<<dim3((unsigned)a.b.nb[0], (unsigned)a.b.nb[1], (unsigned)a.b.nb[2]), threads, smem, st>>>(
      a);
  ps_status rc = check_launch("quad_kernel");
  if (rc || !unsort) return rc;
  return unsort_launch(a.np, a.perm, a.offs, a.b.nbins, rows_ws, a0.vel, a0.vel ? 3 : 0, a0.grad,
                       rows, st);
}

}  // namespace

// The quad form for three components: node coefficients or planar
// F32/BF16/F16.
ps_status launch_quad(const StagedArgs& a, ps_dtype coef_t, int mode, cudaStream_t st,
                      float* rows_ws) {
  auto go = [&](auto tag) -> ps_status {
    using Tc = decltype(tag);
    switch (mode) {
      case 0: return launch_quad_t<Tc, 0>(a, st, rows_ws);
      case 1: return launch_quad_t<Tc, 1>(a, st, rows_ws);
      case 2: return launch_quad_t<Tc, 2>(a, st, rows_ws);
      case 3: return launch_quad_t<Tc, 3>(a, st, rows_ws);
      default:
        return a.coef2 ? launch_quad_t<Tc, 4>(a, st, rows_ws) : launch_quad_t<Tc, 5>(a, st, rows_ws);
    }
  };
  return with_quad_type(coef_t, go);
}

ps_status quad_setup(StagedArgs* a, ps_dtype coef_t, size_t* smem, int* ct) {
  return with_quad_type(coef_t, [&](auto tag) -> ps_status {
    setup_t<decltype(tag)>(a, false, smem, ct);
    return PS_OK;
  });
}

}  // namespace ps
