// The many-field Heun step (batch.cu): all steps of a batch in one persistent
// cooperative launch, or a launch per step over the bricks of all fields.  The
// bricks run the single-field kernel's body (brick.cuh).  Measured, 16 fields of
// 64^3 to 256^3 with 7.0 M particles, four steps, with the phased body before ->
// this one: planar FP32 6824 -> 5001 us persistent, 5852 -> 4122 a launch per
// step; FP32 nodes 5972 -> 5218 and 4497 -> 3913.
#include <algorithm>
#include <cstring>
#include <type_traits>

#include "bin_device.cuh"
#include "brick.cuh"

namespace ps {
namespace {

constexpr int kThreads = 64;  // per block, as the single-field kernel

// The brick (or run of particles) `b` of one field by the block.
template <typename Tc, int CT, bool ONCE = true>
__device__ __forceinline__ bool field_brick(const StagedArgs& a, int b, unsigned char* smem,
                                            const StagedArgs* maps, CopyBarriers& mb,
                                            unsigned& phase) {
  const int nbx = a.b.nb[0], nby = a.b.nb[1];
  const int z = b / (nbx * nby), rem = b - z * nbx * nby, y = rem / nbx, x = rem - y * nbx;
  return warp_brick<Tc, 2, CT, ONCE>(a, b, x, y, z, smem, maps, mb, phase);
}

// The field of global brick b: the last f with bin_base[f] <= b.
__device__ __forceinline__ int field_of(const int* __restrict__ bin_base, int nfields, int b) {
  int lo = 0, hi = nfields;  // bin_base[lo] <= b < bin_base[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (bin_base[mid] <= b) lo = mid;
    else hi = mid;
  }
  return lo;
}

// Global brick b of a many-field batch: the field's arguments are copied to
// shared memory (sa; `cur` the field it holds), its tensor maps stay in the
// global table.  Empty bins return at once.  Every thread of the block calls,
// between block barriers.  Returns what warp_brick does.
template <typename Tc, int CT, bool ONCE = true>
__device__ __forceinline__ bool batch_brick(const StagedArgs* __restrict__ tab,
                                            const int* __restrict__ bin_base, int nfields,
                                            int b, unsigned char* smem, StagedArgs& sa, int& cur,
                                            CopyBarriers& mb, unsigned& phase) {
  // field 0's offsets are the global offsets: empty bins leave at once
  const int32_t* goffs = tab[0].offs;
  if (goffs[b] >= goffs[b + 1]) return true;
  const int f = field_of(bin_base, nfields, b);
  if (f != cur) {
    cur = f;
    constexpr int kWords = (int)(sizeof(StagedArgs) / sizeof(int4));
    static_assert(sizeof(StagedArgs) % sizeof(int4) == 0, "argument block copied in 16 bytes");
    for (int i = threadIdx.x; i < kWords; i += blockDim.x)
      reinterpret_cast<int4*>(&sa)[i] = reinterpret_cast<const int4*>(tab + f)[i];
    // the field's tensor maps stay in the global table (a tensor copy cannot
    // name one in shared memory); order their upload before the copy proxy
    if (threadIdx.x == 0 && tab[f].tma) {
      asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(
                       reinterpret_cast<unsigned long long>(&tab[f].tmap))
                   : "memory");
      if (IsNode16<Tc>::value)
        asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(
                         reinterpret_cast<unsigned long long>(&tab[f].tmap2))
                     : "memory");
    }
    __syncthreads();
  }
  return field_brick<Tc, CT, ONCE>(sa, b - bin_base[f], smem, tab + f, mb, phase);
}

// Many fields in one launch: block b handles global brick b.
template <typename Tc, int CT>
__global__ void __launch_bounds__(kThreads, 8)
    batch_table_step(const StagedArgs* __restrict__ tab, const int* __restrict__ bin_base,
                     int nfields) {
  extern __shared__ __align__(128) unsigned char smem_b128[];
  __shared__ StagedArgs sa;
  __shared__ CopyBarriers mb;
  int cur = -1;
  unsigned phase = 0;
  batch_brick<Tc, CT>(tab, bin_base, nfields, blockIdx.x, smem_b128, sa, cur, mb, phase);
}

// (48 x 640 bytes of arguments: within the 32 KB of parameters)
struct BatchParams {
  StagedArgs a[kBatchParamFields];
  int bin_base[kBatchParamFields + 1];
  int nfields;
};
static_assert(sizeof(BatchParams) <= 32764, "kernel parameters are limited to 32764 bytes");

// A batch of at most kBatchParamFields fields passes its argument table as one
// kernel parameter: the brick body then reads each field's arguments from the
// constant bank, as the single-field kernel does, and the tensor maps are named
// in parameter space like the single-field kernel's.
template <typename Tc, int CT>
__global__ void __launch_bounds__(kThreads, 8)
    batch_param_step(const __grid_constant__ BatchParams tab) {
  extern __shared__ __align__(128) unsigned char smem_bp128[];
  __shared__ CopyBarriers mb;
  unsigned phase = 0;
  const int b = blockIdx.x;
  // field 0's offsets are the global offsets: empty bins leave at once
  const int32_t* goffs = tab.a[0].offs;
  if (goffs[b] >= goffs[b + 1]) return;
  const int f = field_of(tab.bin_base, tab.nfields, b);
  field_brick<Tc, CT>(tab.a[f], b - tab.bin_base[f], smem_bp128, &tab.a[f], mb, phase);
}

// ----------------------------------------------------- persistent batch ----
// All Heun steps of a many-field batch in one cooperative launch: per step
// the three scan phases, the scatter into bin order, then the bricks of all
// fields, which count the bins of the positions they write for the next
// step (the first step counts from the positions, scatters by rank and
// clears the counters; later ones scatter from the counts, which end at
// zero); the phases are separated by grid-wide barriers.  Each barrier is an arrival
// counter and a generation word; a wait gives up after about 2^31 clocks,
// sets the block-stop word and PS_DEV_TIMEOUT, and every block leaves at its
// next barrier.  sync[3] is a word nothing sets: with wait_probe > 0 (a test
// knob) every block waits on it after the first barrier, for that many
// clocks, so that the give-up path runs.  sync[4] is the brick pass's claim
// counter: blocks take one global bin at a time.
struct BatchRun {
  const StagedArgs* tab;   // per-field brick-kernel arguments
  const int* bin_base;     // nfields + 1
  const BinField* bintab;  // per-field binning table
  int nfields;
  int nsteps;
  int64_t total_bins, np;
  double* pos;             // the caller's positions (bin order after a step)
  int64_t* ids;
  double* pos_s;           // copies in bin order (workspace)
  int64_t* ids_s;
  int32_t* bin_of;
  int32_t* rank;
  int32_t* counts;         // total_bins + 1, zero at launch
  int32_t* offsets;        // total_bins + 1
  int32_t* scan_tmp;
  int32_t* status;
  unsigned* sync;          // arrivals, generation, stop, never set, claims; zero at launch
  int wait_probe;
};

__device__ __forceinline__ bool grid_barrier(const BatchRun& r, int& nbar) {
  __shared__ int go;
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned* vs = r.sync;
    bool ok = vs[2] == 0;
    if (ok) {
      const unsigned gen = vs[1];
      __threadfence();
      if (atomicAdd(&r.sync[0], 1u) + 1u == gridDim.x) {
        atomicExch(&r.sync[0], 0u);
        __threadfence();
        atomicAdd(&r.sync[1], 1u);
      } else {
        const long long t0 = clock64();
        while (vs[1] == gen) {
          if (vs[2]) {
            ok = false;
            break;
          }
          if (clock64() - t0 > (1ll << 31)) {
            if (atomicExch(&r.sync[2], 1u) == 0u) flag_status(r.status, PS_DEV_TIMEOUT, nbar);
            ok = false;
            break;
          }
          __nanosleep(100);
        }
      }
      __threadfence();
      if (ok && r.wait_probe > 0 && nbar == 0) {
        const long long t0 = clock64();
        while (vs[3] == 0 && clock64() - t0 <= r.wait_probe) __nanosleep(100);
        if (vs[3] == 0) {
          if (atomicExch(&r.sync[2], 1u) == 0u) flag_status(r.status, PS_DEV_TIMEOUT, nbar);
          ok = false;
        }
      }
    }
    go = ok ? 1 : 0;
  }
  __syncthreads();
  ++nbar;
  return go != 0;
}

template <typename Tc, int CT>
__global__ void __launch_bounds__(kThreads, 8) batch_persistent(const __grid_constant__ BatchRun r) {
  extern __shared__ __align__(128) unsigned char smem_bp[];
  __shared__ StagedArgs sa;
  __shared__ int32_t scan_sh[kThreads / 32];
  __shared__ unsigned claim[2];
  __shared__ CopyBarriers mb;
  __shared__ int lost;  // 1: a halo copy of this block did not land
  unsigned phase = 0;
  if (threadIdx.x == 0) {
    init_copy_barriers(mb);
    lost = 0;
  }  // (published by the first grid barrier)
  int nbar = 0, cur = -1;  // cur: the field whose arguments sa holds
  const int lane = threadIdx.x & 31;
  const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t gs = (int64_t)gridDim.x * blockDim.x;
  const int64_t ntiles = (r.total_bins + kScanTile - 1) / kScanTile;
  for (int step = 0; step < r.nsteps; ++step) {
    // the first step counts from the positions; later ones scan the counts
    // the previous step's bricks took
    if (step == 0) {
      batch_count_range(r.bintab, r.nfields, r.np, r.pos, r.bin_of, r.rank, r.counts, r.status,
                        gt - lane, gs);
      if (!grid_barrier(r, nbar)) return;
    }
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x)
      scan_tile_sum<kThreads>(r.counts, r.total_bins, t, r.scan_tmp, scan_sh);
    if (!grid_barrier(r, nbar)) return;
    if (blockIdx.x == 0) scan_tile_offsets_block<kThreads>(r.scan_tmp, ntiles, scan_sh);
    if (!grid_barrier(r, nbar)) return;
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x)
      scan_tile<kThreads>(r.counts, r.total_bins, r.scan_tmp, r.offsets, -1, t, ntiles,
                          scan_sh);
    if (!grid_barrier(r, nbar)) return;
    if (step == 0) {
      scatter_range(r.np, r.pos, r.bin_of, r.rank, r.offsets, nullptr, r.pos_s, r.ids,
                    r.ids ? r.ids_s : nullptr, gt, gs);
      for (int64_t i = gt; i <= r.total_bins; i += gs) r.counts[i] = 0;
    } else {  // the counters end at zero, ready for this step's counting
      scatter_counted_range(r.np, r.pos, r.bin_of, r.counts, r.offsets, nullptr, r.pos_s,
                            r.ids, r.ids ? r.ids_s : nullptr, r.total_bins, r.status, gt >> 5,
                            gs >> 5);
    }
    if (gt == 0) atomicExch(&r.sync[4], 0u);
    if (!grid_barrier(r, nbar)) return;
    // bricks claimed one at a time (their costs vary with their particles: at
    // four per claim a block could end a step on four of the densest), the next
    // claim on its way while the current brick is processed
    unsigned c = 0;
    if (threadIdx.x == 0) c = atomicAdd(&r.sync[4], 1u);
    for (int it = 0;; it ^= 1) {
      if (threadIdx.x == 0) claim[it] = c;
      __syncthreads();  // the claim; and the last brick is done with sa and the shared memory
      const unsigned b = claim[it];
      if (lost) {  // the copy may yet write to the halo: the run ends here
        if (threadIdx.x == 0) atomicExch(&r.sync[2], 1u);
        break;
      }
      if (b >= r.total_bins) break;
      if (threadIdx.x == 0) c = atomicAdd(&r.sync[4], 1u);
      if (!batch_brick<Tc, CT, false>(r.tab, r.bin_base, r.nfields, (int)b, smem_bp, sa, cur, mb,
                                      phase))
        lost = 1;  // (after the brick's block barrier, so behind every thread's read above)
    }
    if (!grid_barrier(r, nbar)) return;
  }
}

}  // namespace

// ---------------------------------------------------------------- batch ----
// Helpers of the many-field form (batch.cu, where a field's StagedArgs travel as
// opaque bytes).

size_t staged_args_size() { return sizeof(StagedArgs); }

namespace {
// The coefficient type, and the compile-time geometry of the 8^3 brick where
// every field has it (the fields share the brick shape).
template <typename F>
ps_status with_step_type(ps_dtype t, bool cube, F&& f) {
  return with_quad_type(t, [&](auto tag) -> ps_status {
    using Tc = decltype(tag);
    constexpr int kCt = IsNode16<Tc>::value || IsPlanar<Tc>::value ? 12 : 14;
    return cube ? f(tag, std::integral_constant<int, kCt>{})
                : f(tag, std::integral_constant<int, 0>{});
  });
}
}  // namespace

// Arguments of one field's fused Heun step inside a batch: positions are the
// concatenated [3][np_total] arrays, offs points at the field's first bin.
ps_status staged_fill_rk2(const ps_grid* grid, ps_dtype coef_t, const int32_t brick[3],
                          const void* coef, const float* scale, int64_t np_total,
                          const double* pos_in, double* pos_out, const int32_t* offs,
                          float* vel, const int64_t* ids_in, int64_t* ids_out, double dt,
                          int32_t* status, int chunked, int32_t* next_counts, int32_t* next_bin,
                          int next_key_base, int next_runs, void* out, size_t* smem) {
  if (coef_t == PS_F64) return fail(PS_ERR_UNSUPPORTED, "batched RK2 needs F32/BF16/F16");
  StagedArgs a{};
  ps_status rc = fill_staged(grid, coef_t, brick, 0, false, &a, smem);
  if (rc) return rc;
  a.coef = coef;
  a.scale = scale;
  a.np = np_total;
  a.pos_in = pos_in;
  a.pos_out = pos_out;
  a.offs = offs;
  a.vel = vel;
  a.ids_in = ids_in;
  a.ids_out = ids_out;
  a.dt = dt;
  const float3 d = dt_over_h(a.g, dt);
  a.dtih[0] = d.x;
  a.dtih[1] = d.y;
  a.dtih[2] = d.z;
  a.status = status;
  a.chunked = chunked;
  a.next_counts = next_counts;
  a.next_bin = next_bin;
  a.next_key_base = next_key_base;
  a.next_runs = next_runs;
  int ct;
  if ((rc = quad_setup(&a, coef_t, smem, &ct))) return rc;
  memcpy(out, &a, sizeof(a));
  return PS_OK;
}

// Launch the batched fused Heun step over total_bins bricks of nfields
// fields.  Set prepare = true once before any stream capture (it only sets the
// shared-memory limit of the kernel).
ps_status staged_batch_launch(ps_dtype coef_t, bool cube, const void* d_tab, const int* d_bin_base,
                              const void* h_tab, const int* h_bin_base, int nfields,
                              int64_t total_bins, size_t smem, bool prepare, cudaStream_t st) {
  return with_step_type(coef_t, cube, [&](auto tag, auto ct) -> ps_status {
    using Tc = decltype(tag);
    {
      auto kern = batch_table_step<Tc, ct>;
      auto kern_p = batch_param_step<Tc, ct>;
      if (prepare) {
        ps_status rc = PS_OK;
        if (smem > 48 * 1024) {
          rc = check_cuda(
              cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
              "batch smem attribute");
          if (!rc)
            rc = check_cuda(cudaFuncSetAttribute(
                                kern_p, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
                            "batch smem attribute");
        }
        return rc;
      }
      if (total_bins <= 0) return PS_OK;
      if (h_tab && h_bin_base && nfields <= kBatchParamFields) {
        // the table by value (a graph captures it with the launch)
        BatchParams tab;
        memcpy(tab.a, h_tab, (size_t)nfields * sizeof(StagedArgs));
        memcpy(tab.bin_base, h_bin_base, (size_t)(nfields + 1) * sizeof(int));
        tab.nfields = nfields;
        kern_p<<<(unsigned)total_bins, kThreads, smem, st>>>(tab);
        return check_launch("batch_param_step");
      }
      kern<<<(unsigned)total_bins, kThreads, smem, st>>>(
          static_cast<const StagedArgs*>(d_tab), d_bin_base, nfields);
      return check_launch("batch_table_step");
    }
  });
}

// All nsteps Heun steps of a batch in one cooperative launch (batch_persistent):
// a grid of every block the device holds at once.  counts and sync must be
// zero at launch (the caller clears them on the same stream).
ps_status staged_batch_persistent(ps_dtype coef_t, bool cube, const void* d_tab, const int* d_bin_base,
                                  const BinField* d_bintab, int nfields, int64_t total_bins,
                                  int64_t np, int nsteps, double* pos, int64_t* ids,
                                  double* pos_s, int64_t* ids_s, int32_t* bin_of, int32_t* rank,
                                  int32_t* counts, int32_t* offsets, int32_t* scan_tmp,
                                  int32_t* status, unsigned* sync, size_t smem,
                                  cudaStream_t st) {
  return with_step_type(coef_t, cube, [&](auto tag, auto ct) -> ps_status {
    using Tc = decltype(tag);
    {
      auto kern = batch_persistent<Tc, ct>;
      if (smem > 48 * 1024) {
        ps_status rc = check_cuda(
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
            "persistent batch smem attribute");
        if (rc) return rc;
      }
      int per_sm = 0;
      ps_status rc = check_cuda(
          cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, smem),
          "persistent batch occupancy");
      if (rc) return rc;
      if (per_sm < 1) return fail(PS_ERR_UNSUPPORTED, "persistent batch kernel does not fit an SM");
      BatchRun r;
      r.tab = static_cast<const StagedArgs*>(d_tab);
      r.bin_base = d_bin_base;
      r.bintab = d_bintab;
      r.nfields = nfields;
      r.nsteps = nsteps;
      r.total_bins = total_bins;
      r.np = np;
      r.pos = pos;
      r.ids = ids;
      r.pos_s = pos_s;
      r.ids_s = ids_s;
      r.bin_of = bin_of;
      r.rank = rank;
      r.counts = counts;
      r.offsets = offsets;
      r.scan_tmp = scan_tmp;
      r.status = status;
      r.sync = sync;
      r.wait_probe = tuning().wait_probe;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)(per_sm * sm_count()));
      cfg.blockDim = dim3(kThreads);
      cfg.dynamicSmemBytes = smem;
      cfg.stream = st;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeCooperative;
      attr[0].val.cooperative = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      return check_cuda(cudaLaunchKernelEx(&cfg, kern, r), "persistent batch launch");
    }
  });
}

}  // namespace ps
