// kernels_f64.cu -- FP64 path of two-state models: walker state in contiguous
// GPU arrays (the paper's Sec. II B), three output times a launch, in double
// precision.  It is also the per-trajectory parity path against the CPU oracle.
#include <algorithm>
#include <climits>

#include "f64_2state.cuh"
#include "kernels.h"
#include "reduce.cuh"

namespace qcl {


// ---------------------------------------------------------------- sampling --
__global__ void __launch_bounds__(256) k_sample_f64(const DevModel* __restrict__ M,
                                                    SampleParams sp, void* buf) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nt = sp.n_traj;
  const int n = sp.n, ns = sp.ns;
  W64 w = view64(buf, nt, ns, n);
  if (i == 0) {
    w.hdr->magic = kEnsMagic;
    w.hdr->n_traj = nt;
    w.hdr->precision = QCL_PREC_FP64;
    w.hdr->ns = ns;
    w.hdr->n = n;
    w.hdr->step = 0;
    w.hdr->flags = 0;
    w.hdr->n_degenerate = 0;
    w.hdr->n_nonfinite = 0;
  }
  if (i >= nt) return;
  uint16_t ab;
  sample_walker_f64(M, sp, sp.traj_offset + (uint64_t)i, w.R + i, w.P + i, nt, w.m[i], ab);
  w.phi[i] = 0.0;
  w.ab[i] = ab;
}

// -------------------------------------------------------------------- step --
// Steps of one walker per thread (velocity Verlet on the pair's mean force,
// trapezoid phase, one transition from the coupling term of Eq. 1, or of its
// diabatic form when DIA) with up to kOuts64 output times, the walker in
// registers and the decomposition carried from step to step.  The index-pair
// word carries the quarter-turn count of a diabatic walker in bits 4-5.  At an
// output time each warp reduces its 32 walkers' contributions and their squares
// to one group's sums: the first level of the reduction tree, folded to tiles by
// k_group_tiles, so that the block can be smaller than a tile.
//
// Bound by the FP64 unit (85 % busy at 1e6 walkers, 56 FP64 instructions a step
// of the three-mode spin-boson form, 264 with two decompositions and a division
// for each mode), below 2e4 walkers by the latency of a step's chain.  Blocks of
// one warp: 1e4 walkers then spread evenly over all SMs (blocks of 256 left 112
// of 152 idle).
constexpr int kOuts64 = 3;
constexpr int kBlock64 = 32;

struct Steps64 {
  int64_t nt, step0, step;
  uint64_t seed, traj_off;
  int32_t len, stride, to_out, obs_first;
};

template <int NP, int NC, int KIND, bool DIA>
__global__ void __launch_bounds__(kBlock64) k_steps_f64(const Coef64<NC> c, const Steps64 sp, void* buf,
                                                  double* __restrict__ groups) {
  const int64_t nt = sp.nt;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  W64 w = view64(buf, nt, 2, c.n);
  // (at another step than the call expects nothing moves; the output times still
  // observe the walkers as they are)
  const bool moves = w.hdr->step == sp.step0;
  if (!moves && i == 0) atomicOr(&w.hdr->flags, QCL_FLAG_STEP_MISMATCH);
  const int lane = threadIdx.x & 31;
  const int64_t n_groups = (nt + 31) / 32, group = i >> 5;
  if (group >= n_groups) return;  // (a whole warp)
  const bool live = i < nt;       // (only the last group's lanes differ)
  const int64_t ii = live ? i : nt - 1;
  const uint16_t ab = w.ab[ii];
  int al = ab & 0xf, be = (ab >> 8) & 0xf, q = (ab >> 4) & 3;
  double m = w.m[ii], phi = w.phi[ii];
  double R[NP > 0 ? NP : 1], P[NP > 0 ? NP : 1];
  Dec64 d;
  walker_load_f64<NP, NC, KIND, DIA>(c, w.R + ii, w.P + ii, nt, R, P, d);
  unsigned int n_deg = 0, n_bad = 0;
  auto observe = [&](int slot) {
    Dec64 e = d;
    if (DIA) decompose64<0, false>(e);
    double v[32];
    contrib_f64(e, live ? m : 0.0, phi, (uint16_t)(al | (q << 4) | (be << 8)), DIA, v);
    groups[((int64_t)slot * n_groups + group) * 32 + lane] = warp_transpose_sum<double>(v);
  };
  int slot = sp.obs_first, to_out = sp.to_out;
  if (sp.obs_first) observe(0);
  u4 wd;
  for (int32_t t = 0; t < sp.len; ++t) {
    const int64_t s = sp.step + t;
    if (live && moves) {
      if (t == 0 || (s & 3) == 0)
        wd = philox_draw(sp.seed, (uint32_t)(s >> 2), sp.traj_off + (uint64_t)i, kPurposeHop);
      bool deg;
      const Step64 o = walker_step_f64<NP, NC, KIND, DIA>(
          c, NP > 0 ? R : w.R + i, NP > 0 ? P : w.P + i, nt, d, al, be, phi,
          word_of(wd, (int)(s & 3)) >> 8, deg);
      m = weight64(m, o);
      al ^= o.ev & 1;
      be ^= o.ev >> 1;
      if (DIA) q = (q + o.dq) & 3;
      n_deg += deg ? 1u : 0u;
      n_bad += (nonfinite64(m) || nonfinite64(phi)) ? 1u : 0u;
    }
    if (--to_out == 0) {
      __syncwarp();
      observe(slot++);
      to_out = sp.stride;
    }
  }
  if (!live || !moves || sp.len == 0) return;
  walker_store_f64<NP>(c.n, R, P, w.R + i, w.P + i, nt);
  w.m[i] = m;
  w.phi[i] = phi;
  w.ab[i] = (uint16_t)(al | (q << 4) | (be << 8));
  if (n_deg) {
    atomicAdd(&w.hdr->n_degenerate, (unsigned long long)n_deg);
    atomicOr(&w.hdr->flags, QCL_FLAG_DEGENERATE);
  }
  if (n_bad) {
    atomicAdd(&w.hdr->n_nonfinite, (unsigned long long)n_bad);
    atomicOr(&w.hdr->flags, QCL_FLAG_NONFINITE);
  }
}

// Tile partials from group sums: the binary tree over a tile's 8 groups (zero
// past the last one) of each column, for every output of a launch.
__global__ void __launch_bounds__(256) k_group_tiles(const double* __restrict__ groups,
                                                     int64_t n_groups, int64_t n_tiles,
                                                     double* __restrict__ part) {
  const int col = threadIdx.x & 31;
  const int64_t tile = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (tile >= n_tiles) return;
  const double* in = groups + ((int64_t)blockIdx.y * n_groups + tile * 8) * 32 + col;
  const int64_t left = n_groups - tile * 8;
  double g[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) g[k] = k < left ? in[k * 32] : 0.0;
  part[((int64_t)blockIdx.y * n_tiles + tile) * 32 + col] =
      ((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + (g[6] + g[7]));
}

// ------------------------------------------------------------------ launch --
void launch_sample_f64(const DevModel* dm, const SampleParams& sp, void* buf, cudaStream_t st) {
  const int64_t nb = (sp.n_traj + 255) / 256;
  k_sample_f64<<<(unsigned)(nb > 0 ? nb : 1), 256, 0, st>>>(dm, sp, buf);
  launches_add(1);
}

// The steps of a launch: at most 256, and as many as keep it near a quarter of a
// second, since work on other streams waits for its blocks to be handed out.  A
// step takes up to 35 ps for each walker and mode and as much again for two modes
// (2e5 walkers: 20 ps with 256 modes of the spin-boson form, 35 of the general one;
// 1.1 of 3 with one mode).  What a launch adds, a load and a store of the walkers
// and one decomposition, is small against the ten steps and more that all but
// the largest ensembles take.
static int64_t steps_per_launch(int64_t nt, int n) {
  const double steps = 0.25 / (35e-12 * (double)nt * (double)(n + 2));
  return steps >= 256.0 ? 256 : std::max<int64_t>((int64_t)steps, 1);
}

// Steps from `step` with at most kOuts64 output times: returns the steps taken
// (0 with obs_first alone at the end) and leaves the tile partials of *outs output
// times in part's first slots.  The group sums lie behind them in the same array
// (its kChunkOut slots hold 9 kOuts64 of a tile's 32 doubles).
int64_t launch_steps_f64(const DevModel& host, void* buf, int64_t nt, int64_t step0, int64_t step,
                         int64_t end, int32_t stride, bool obs_first, double dt, uint64_t seed,
                         uint64_t traj_off, double* part, int* outs, cudaStream_t st) {
  static_assert(9 * kOuts64 <= kChunkOut, "room for the group sums");
  const int64_t next = (step / stride + 1) * stride;  // the first output time after step
  const int room = kOuts64 - (obs_first ? 1 : 0);
  const int64_t e = std::min(std::min(end, step + steps_per_launch(nt, host.n)),
                             next + (int64_t)(room - 1) * stride);
  *outs = (obs_first ? 1 : 0) + (e >= next ? (int)((e - next) / stride) + 1 : 0);
  const int64_t n_tiles = (nt + kTile - 1) / kTile, n_groups = (nt + 31) / 32;
  double* groups = part + (size_t)kOuts64 * n_tiles * 32;
  const Steps64 sp{nt, step0, step, seed, traj_off, (int32_t)(e - step), stride,
                   (int32_t)std::min<int64_t>(next - step, INT_MAX), obs_first ? 1 : 0};
  const unsigned nb = (unsigned)((nt + kBlock64 - 1) / kBlock64);
  dispatch_f64(host, [&](auto NP, auto NC, auto KIND, auto DIA) {
    constexpr int nc = decltype(NC)::value;
    Coef64<nc> c;
    make_coef64<nc>(host, dt, c);
    k_steps_f64<decltype(NP)::value, nc, decltype(KIND)::value, decltype(DIA)::value>
        <<<nb, kBlock64, 0, st>>>(c, sp, buf, groups);
  });
  launches_add(1);
  if (*outs > 0) {
    const dim3 grid((unsigned)((n_tiles + 7) / 8), (unsigned)*outs);
    k_group_tiles<<<grid, 256, 0, st>>>(groups, n_groups, n_tiles, part);
    launches_add(1);
  }
  return e - step;
}

}  // namespace qcl
