// kernels_f64.cu -- FP64 path of two-state models: walker state in contiguous
// GPU arrays (the paper's Sec. II B), one launch per output time, in double
// precision.  It is also the per-trajectory parity path against the CPU oracle.
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
// `len` full steps of one walker per thread (velocity Verlet on the pair's
// mean force, trapezoid phase, one transition from the coupling term of Eq. 1,
// or of its diabatic form when DIA) between two output times, with the walker
// in registers and the decomposition carried from step to step.  The index-pair
// word carries the quarter-turn count of a diabatic walker in bits 4-5.
template <int NP, int NC, int KIND, bool DIA>
__global__ void __launch_bounds__(64) k_steps_f64(const Coef64<NC> c, void* buf, int64_t nt,
                                                  int64_t step0, int64_t step, int32_t len,
                                                  uint64_t seed, uint64_t traj_off) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  W64 w = view64(buf, nt, 2, c.n);
  if (i >= nt) return;
  if (w.hdr->step != step0) {
    if (i == 0) atomicOr(&w.hdr->flags, QCL_FLAG_STEP_MISMATCH);
    return;
  }
  const uint16_t ab = w.ab[i];
  int al = ab & 0xf, be = (ab >> 8) & 0xf, q = (ab >> 4) & 3;
  double m = w.m[i], phi = w.phi[i];
  double R[NP > 0 ? NP : 1], P[NP > 0 ? NP : 1];
  Dec64 d;
  walker_load_f64<NP, NC, KIND, DIA>(c, w.R + i, w.P + i, nt, R, P, d);
  unsigned int n_deg = 0, n_bad = 0;
  u4 wd;
  for (int32_t t = 0; t < len; ++t) {
    const int64_t s = step + t;
    if (t == 0 || (s & 3) == 0)
      wd = philox_draw(seed, (uint32_t)(s >> 2), traj_off + (uint64_t)i, kPurposeHop);
    bool deg;
    const Step64 o = walker_step_f64<NP, NC, KIND, DIA>(c, NP > 0 ? R : w.R + i,
                                                        NP > 0 ? P : w.P + i, nt, d, al, be, phi,
                                                        word_of(wd, (int)(s & 3)) >> 8, deg);
    m = __dmul_rn(m, o.factor);
    al ^= o.ev & 1;
    be ^= o.ev >> 1;
    if (DIA) q = (q + o.dq) & 3;
    n_deg += deg ? 1u : 0u;
    n_bad += (nonfinite64(m) || nonfinite64(phi)) ? 1u : 0u;
  }
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

// ------------------------------------------------------------- observation --
// Walker contributions m exp(-i phi) U_ia U_jb (diabatic) and m exp(-i phi) at
// (a, b) (adiabatic), and their squares, summed per 256-walker tile.
__global__ void __launch_bounds__(256) k_observe_f64(const DevModel* __restrict__ M,
                                                     const void* buf, int64_t nt, int n,
                                                     double* __restrict__ part) {
  __shared__ double red[8][32];
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  W64 w = view64((void*)buf, nt, 2, n);
  double v[32];
#pragma unroll
  for (int q = 0; q < 32; ++q) v[q] = 0.0;
  if (i < nt) contrib_f64(M, w.R + i, nt, n, w.m[i], w.phi[i], w.ab[i], v);
  const double x = warp_transpose_sum<double>(v);
  red[threadIdx.x >> 5][threadIdx.x & 31] = x;
  __syncthreads();
  if (threadIdx.x < 32) part[(int64_t)blockIdx.x * 32 + threadIdx.x] =
      tile_tree8(&red[0][0], 32, threadIdx.x);
}

// ------------------------------------------------------------------ launch --
void launch_sample_f64(const DevModel* dm, const SampleParams& sp, void* buf, cudaStream_t st) {
  const int64_t nb = (sp.n_traj + 255) / 256;
  k_sample_f64<<<(unsigned)(nb > 0 ? nb : 1), 256, 0, st>>>(dm, sp, buf);
  launches_add(1);
}

void launch_steps_f64(const DevModel& host, void* buf, int64_t nt, int64_t step0, int64_t step,
                      int32_t len, double dt, uint64_t seed, uint64_t traj_off, cudaStream_t st) {
  const unsigned nb = (unsigned)((nt + 63) / 64);
  dispatch_f64(host, [&](auto NP, auto NC, auto KIND, auto DIA) {
    constexpr int nc = decltype(NC)::value;
    Coef64<nc> c;
    make_coef64<nc>(host, dt, c);
    k_steps_f64<decltype(NP)::value, nc, decltype(KIND)::value, decltype(DIA)::value>
        <<<nb, 64, 0, st>>>(c, buf, nt, step0, step, len, seed, traj_off);
  });
  launches_add(1);
}

void launch_observe_f64(const DevModel* dm, const void* buf, int64_t nt, int n, double* part,
                        cudaStream_t st) {
  const unsigned nb = (unsigned)((nt + 255) / 256);
  k_observe_f64<<<nb, 256, 0, st>>>(dm, buf, nt, n, part);
  launches_add(1);
}

}  // namespace qcl
