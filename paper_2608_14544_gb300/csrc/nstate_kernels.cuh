// nstate_kernels.cuh -- models with N_s = 3..8 electronic states: the per-N_s
// launchers over the FP64 path (nstate_f64.cuh), the FP32-bulk kernels
// (nstate_bulk.cuh) and FP32 spawning (nstate_spawn32.cuh).
#pragma once
#include <mutex>

#include "nstate_f64.cuh"
#include "nstate_spawn32.cuh"

namespace qcl {

// ------------------------------------------------------- per-N_s launchers --
// Instantiated one N_s per translation unit; the FP64 sampling and step
// kernels in their own units (kernels_nstate64_*.cu, compiled without FMA
// contraction so that their arithmetic is the oracle's).
template <int NS>
struct NStateOps {
  static void sample64(const DevModel* dm, const SampleParams& sp, void* buf, cudaStream_t st) {
    const int64_t nb = (sp.n_traj + 127) / 128;
    k_sampleN_f64<NS><<<(unsigned)(nb > 0 ? nb : 1), 128, 0, st>>>(dm, sp, buf);
  }
  static void sample32(const SampleN32& sp, void* buf, cudaStream_t st) {
    const int64_t nb = (sp.n_traj + 127) / 128;
    k_sampleN_f32<NS><<<(unsigned)(nb > 0 ? nb : 1), 128, 0, st>>>(sp, buf);
  }
  static void step64(const DevModel* dm, int repr, void* buf, int64_t nt, int n, int64_t step0,
                     int64_t step, int32_t len, double dt, uint64_t seed, uint64_t traj_off,
                     cudaStream_t st) {
    const unsigned nb = (unsigned)((nt + 31) / 32);
    if (repr == QCL_REPR_DIABATIC)
      k_stepsN_dia_f64<NS><<<nb, 32, 0, st>>>(dm, buf, nt, n, step0, step, len, dt, seed, traj_off);
    else
      k_stepsN_f64<NS><<<nb, 32, 0, st>>>(dm, buf, nt, n, step0, step, len, dt, seed, traj_off);
  }
  static void observe64(const DevModel* dm, const void* buf, int64_t nt, int n, double* part,
                        cudaStream_t st) {
    k_observeN_f64<NS><<<(unsigned)((nt + 255) / 256), 256, 0, st>>>(dm, buf, nt, n, part);
  }
  static void spawn_sample64(const DevModel* dm, const SampleParams& sp, int64_t cap, void* buf,
                             cudaStream_t st) {
    const int64_t nb = (sp.n_traj + 127) / 128;
    k_spawnN_sample<NS><<<(unsigned)(nb > 0 ? nb : 1), 128, 0, st>>>(dm, sp, cap, buf);
    launches_add(1);
  }
  // one spawning step: step kernel, scan, scatter (set step & 1 -> the other)
  static void spawn_step64(const DevModel* dm, void* buf, int64_t cap, int n, int64_t n0,
                           int64_t step0, int64_t step, double dt, uint64_t seed,
                           cudaStream_t st) {
    const unsigned nb = spawn_grid(cap);
    k_spawnN_step<NS><<<nb, 256, 0, st>>>(dm, buf, cap, n, n0, step0, step, dt, seed);
    launch_spawn_scan(buf, cap, n, n0, QCL_PREC_FP64, NS, step0, step, st);
    k_spawnN_scatter<NS><<<nb, 256, 0, st>>>(buf, cap, n, n0, step0, step, seed);
    launches_add(2);
  }
  static void spawn_sample32(const SampleN32& sp, int64_t cap, void* buf, cudaStream_t st) {
    const int64_t nb = (sp.n_traj + 127) / 128;
    k_spawnN_sample32<NS><<<(unsigned)(nb > 0 ? nb : 1), 128, 0, st>>>(sp, cap, buf);
    launches_add(1);
  }
  // (false: the launch was refused)
  template <int NPL>
  static bool spawn_step32_npl(const BulkParams& bp, const CoefN& cf, void* buf, int64_t cap,
                               int64_t n0, int64_t step, cudaStream_t st) {
    // (NPL = 0: the mode table in dynamic shared memory)
    size_t dyn = 0;
    if constexpr (NPL == 0) {
      dyn = ModeRow<NS>::bytes(bp.n);
      if (!allow_dynamic_shared(k_spawnN_step32<NS, NPL>, ModeRow<NS>::bytes(kMaxN))) return false;
    }
    k_spawnN_step32<NS, NPL><<<spawn_grid(cap), 256, dyn, st>>>(bp, cf, buf, cap, n0, step);
    return true;
  }
  // one FP32 spawning step (step kernel, scan, scatter): up to 8 modes in
  // registers, beyond (or under the modes-in-memory option) in memory
  static int spawn_step32(const BulkParams& bp, const CoefN& cf, void* buf, int64_t cap,
                          int64_t n0, int64_t step0, int64_t step, cudaStream_t st) {
    // (without the step's counts nothing may be scanned or scattered)
    if (!(cf.modes_in_memory == 1 || bp.n > 8 ? spawn_step32_npl<0>(bp, cf, buf, cap, n0, step, st)
          : bp.n <= 4 ? spawn_step32_npl<4>(bp, cf, buf, cap, n0, step, st)
                      : spawn_step32_npl<8>(bp, cf, buf, cap, n0, step, st)))
      return 0;
    launch_spawn_scan(buf, cap, bp.n, n0, QCL_PREC_FP32_BULK, NS, step0, step, st);
    k_spawnN_scatter32<NS><<<spawn_grid(cap), 256, 0, st>>>(buf, cap, bp.n, n0, step0, step,
                                                            bp.seed);
    launches_add(2);
    return 1;
  }
  static void spawn_observe32(const BulkParams& bp, const CoefN& cf, const void* buf, int64_t cap,
                              int64_t n0, int set, double* part, cudaStream_t st) {
    launch_spawn_fstart(buf, cap, bp.n, n0, QCL_PREC_FP32_BULK, NS, set, st);
    k_spawnN_observe32<NS><<<(unsigned)((n0 + 127) / 128), 128, 0, st>>>(bp, cf, buf, cap, n0,
                                                                         set, part);
    launches_add(1);
  }
  static void spawn_observe64(const DevModel* dm, const void* buf, int64_t cap, int n,
                              int64_t n0, int set, double* part, cudaStream_t st) {
    launch_spawn_fstart(buf, cap, n, n0, QCL_PREC_FP64, NS, set, st);
    k_spawnN_observe<NS><<<(unsigned)((n0 + 255) / 256), 256, 0, st>>>(dm, buf, cap, n, n0, set,
                                                                       part);
    launches_add(1);
  }
  // (NM > 0: the modes-in-memory form with its coefficient rows as a kernel
  // parameter)
  template <int NPL, int WPT = 1, int NM = 0, int SM = 0>
  static int bulk_npl(const BulkParams& bp, const CoefN& cf, const ModeHost& mh, void* buf,
                      double* part, int grid_cap, cudaStream_t st) {
    // (occupancy cached per kernel: [0] adiabatic, [1] diabatic; NPL = 0: the mode
    // table, or R and P, in dynamic shared memory, at most dyn_max of it)
    static int per_sm[2] = {-1, -1}, n_sm[2] = {0, 0};
    const size_t dyn = NPL != 0  ? 0
                       : NM == 0 ? ModeRow<NS>::bytes(bp.n)
                                 : (size_t)SM * bp.n * 128 * sizeof(float);
    const size_t dyn_max = NM == 0 ? ModeRow<NS>::bytes(kMaxN) : (size_t)64 * 128 * sizeof(float);
    if constexpr (NM == 0) {
      if (bp.repr == QCL_REPR_DIABATIC) {
        CoefArg<(NPL > 8)> ca{};
        ca.c = cf;
        return launch_persistent(k_bulkN_dia<NS, NPL>, per_sm[1], n_sm[1], bp, grid_cap, 1, dyn,
                                 dyn_max, st, bp, ca, buf, part);
      }
    }
    if constexpr (NPL == 0 && NM == 0 && NS <= 4) {
      return 0;  // (adiabatic models of N_s <= 4 take NM > 0)
    } else {
      CoefMem<NS, NM> cm;
      if constexpr (NM > 0) make_coef_mem(mh, bp.n, cm);
      return launch_persistent(k_bulkN<NS, NPL, WPT, NM, SM>, per_sm[0], n_sm[0], bp,
                               grid_cap, WPT, dyn, dyn_max, st, bp, cf, buf, part, cm);
    }
  }
  // one persistent grid: the occupancy limit of resident blocks on every SM
  // (capped), at most one block per WPT tiles
  // (dyn > 0, the modes-in-memory kernels: the occupancy is computed for this
  // call's table)
  template <typename Fn, typename... Args>
  static int launch_persistent(Fn fn, int& per_sm, int& n_sm, const BulkParams& bp, int grid_cap,
                               int WPT, size_t dyn, size_t dyn_max, cudaStream_t st,
                               const Args&... args) {
    int blocks = per_sm;
    if (dyn > 0) {
      static std::mutex mu;
      std::lock_guard<std::mutex> lock(mu);
      if (n_sm == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
      }
      if (!allow_dynamic_shared(fn, dyn_max)) return 1;
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, fn, 128, dyn) != cudaSuccess ||
          blocks < 1)
        blocks = 1;
    } else if (per_sm < 0) {
      int dev = 0;
      cudaGetDevice(&dev);
      cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, fn, 128, 0) != cudaSuccess ||
          blocks < 1)
        blocks = 1;
      per_sm = blocks;
    }
    int64_t grid = (int64_t)blocks * n_sm;
    if (grid_cap > 0 && grid > grid_cap) grid = grid_cap;
    const int64_t units = (bp.n_tiles + WPT - 1) / WPT;
    if (grid > units) grid = units;
    if (grid < 1) grid = 1;
    fn<<<(unsigned)grid, 128, dyn, st>>>(args...);
    return (int)grid;
  }
  // wpt: walkers per thread asked for.  The kernel takes one or two, but only
  // one is instantiated: two walkers per thread (packed lanes, 205-245
  // registers, 8 resident warps per SM) measured 10 % slower on a four-state
  // six-mode model than one (114 registers, 16 warps), with the same bits.
  static int bulk(const BulkParams& bp, const CoefN& cf, const ModeHost& mh, void* buf,
                  double* part, int grid_cap, int wpt, cudaStream_t st) {
    (void)wpt;
    // Register forms exist up to 8 modes for any N_s and up to 32 modes for
    // N_s <= 4 (larger N_s x modes would not fit a walker in registers); the
    // modes-in-memory form takes any mode count with the same bits.  The
    // automatic choice follows measured solve rates on GB300 (1e6 walkers,
    // 200 steps, random LVC models): registers for N_s = 3 (except adiabatic
    // models of 9-24 modes, where the 32-mode register form is 10-50 % slower)
    // and for N_s = 4 up to 8 modes (10-20 % faster); the memory form beyond
    // (N_s = 4 with 12-32 modes: 1.2-2x faster) and for N_s >= 5 at every
    // mode count (1.0-2.2x, the register forms there run one or two blocks per
    // SM).  Models of at most 4 or 6 modes get their own instantiations,
    // which skip the padding modes' arithmetic (padding modes have zero
    // coefficients and stay at zero).
    const int reg_max = NS <= 4 ? 32 : 8;
    bool mem;
    if (cf.modes_in_memory == 1) mem = true;
    else if (cf.modes_in_memory == 2) mem = bp.n > reg_max;
    else if (NS == 3) mem = bp.n > 32 || (bp.repr != QCL_REPR_DIABATIC && bp.n > 8 && bp.n <= 24);
    else if (NS == 4) mem = bp.n > 8;
    else mem = true;
    // The adiabatic memory form of N_s <= 4 takes its coefficients as a kernel
    // parameter and keeps R and P in shared memory up to 32 modes, P alone up
    // to 64 (32 KB a block in either case, so that four blocks still fit an SM;
    // at 128 modes P alone left two, and was 40 % slower than no arrays).
    // N_s = 4, 300011 walkers x 30 steps: 12 modes 0.81 -> 0.74 ms, 32 modes
    // 1.53 -> 1.25, 64 modes 2.72 -> 2.29, 128 modes 5.63 -> 5.13.
    // Ensembles of one turn (at most four tiles on every SM) wait for one walker's
    // chain instead, and their R and P stay in L1: the form without arrays is
    // faster there, for N_s = 4 from 24 modes and N_s = 3 from 48.  N_s = 4, 40
    // steps, arrays / none: 3000 walkers 32 modes 233 / 200 us, 64 modes 524 / 342;
    // 77824 walkers 436 / 398 and 703 / 645; 100001 walkers 630 / 695 and 1338 /
    // 1417.  N_s = 3, 3000 walkers, 40 modes 189 / 195, 48 modes 252 / 223.
    if constexpr (NS <= 4) {
      if (mem && bp.repr != QCL_REPR_DIABATIC) {
        static const int n_sm = [] {
          int dev = 0, n = 0;
          cudaGetDevice(&dev);
          cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
          return n;
        }();
        const bool one_turn = bp.n >= (NS == 4 ? 24 : 48) && bp.n_tiles <= 4 * (int64_t)n_sm;
        if (bp.n > 64 || one_turn) return bulk_npl<0, 1, 256, 0>(bp, cf, mh, buf, part, grid_cap, st);
        if (bp.n <= 32) return bulk_npl<0, 1, 64, 2>(bp, cf, mh, buf, part, grid_cap, st);
        return bulk_npl<0, 1, 64, 1>(bp, cf, mh, buf, part, grid_cap, st);
      }
    }
    if (mem) return bulk_npl<0>(bp, cf, mh, buf, part, grid_cap, st);
    if constexpr (NS <= 5) {
      if (bp.n <= 4) return bulk_npl<4>(bp, cf, mh, buf, part, grid_cap, st);
      if (bp.n <= 6) return bulk_npl<6>(bp, cf, mh, buf, part, grid_cap, st);
    }
    if (bp.n <= 8) return bulk_npl<8>(bp, cf, mh, buf, part, grid_cap, st);
    if (NS <= 4 && bp.n <= 32) return bulk_npl<(NS <= 4 ? 32 : 8)>(bp, cf, mh, buf, part, grid_cap, st);
    return 0;
  }
};

}  // namespace qcl
