// spawn32.cu -- trajectory spawning in FP32 bulk precision (two states, any
// mode count, either representation).  The same scheme and walker order as the
// FP64 spawning kernels (spawn.cu), a child inserted right after its parent; the
// walker's arithmetic is that of the FP32-bulk kernels (compensated phase and
// weight pairs with a carried exponent), with the state read from and written to
// memory every step.  Family observation in FP64 from the walkers' FP32 contributions.
#include "bulk2.cuh"
#include "model.h"
#include "reduce.cuh"

namespace qcl {

namespace {

struct Set32 {
  float* R;
  float* P;
  float* mh;
  float* ml;
  int32_t* me;
  float* ph;
  float* pl;
  uint16_t* ab;
  uint64_t* id;
  uint32_t* fam;
};

__device__ __forceinline__ Set32 set32(void* buf, const SpawnLayout& L, int set) {
  char* b = (char*)buf + (set ? L.set_off[1] : L.set_off[0]);
  return {(float*)(b + L.R),     (float*)(b + L.P),    (float*)(b + L.m),
          (float*)(b + L.mlo),   (int32_t*)(b + L.mexp), (float*)(b + L.phi),
          (float*)(b + L.philo), (uint16_t*)(b + L.ab), (uint64_t*)(b + L.id),
          (uint32_t*)(b + L.fam)};
}

__device__ __forceinline__ SpawnHeader* hdr_spawn(void* buf) {
  return (SpawnHeader*)((char*)buf + kSpawnHeaderOff);
}

// the child's random-stream id (the definition used by the FP64 kernels)
__device__ __forceinline__ uint64_t child_id32(uint64_t seed, int64_t step, uint64_t parent) {
  const u4 w = philox_draw(seed, (uint32_t)step, parent, 3u);
  return (((uint64_t)w.y << 32) | w.x) | (1ull << 63);
}

__global__ void __launch_bounds__(256) k_spawn_sample32(const Sample32 sp, int64_t cap, void* buf) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t n0 = sp.n_traj;
  const SpawnLayout L = SpawnLayout::make(cap, sp.n, n0, QCL_PREC_FP32_BULK);
  EnsHeader* hdr = (EnsHeader*)buf;
  SpawnHeader* sh = hdr_spawn(buf);
  if (i == 0) {
    hdr->magic = kEnsMagic;
    hdr->n_traj = n0;
    hdr->precision = QCL_PREC_FP32_BULK;
    hdr->ns = 2;
    hdr->n = sp.n;
    hdr->step = 0;
    hdr->flags = 0;
    hdr->n_degenerate = 0;
    hdr->n_nonfinite = 0;
    sh->capacity = cap;
    sh->n0 = n0;
    sh->n_live[0] = n0;
    sh->n_live[1] = 0;
    sh->drop = 0;
  }
  // the families' starts: an observation finds indexes within the buffer whatever
  // the steps before it did (a step mismatch moves nothing)
  int64_t* const fstart = (int64_t*)((char*)buf + L.fstart);
  if (i == 0) fstart[n0] = n0;
  if (i >= n0) return;
  fstart[i] = i;
  const Set32 w = set32(buf, L, 0);
  const uint64_t traj = sp.traj_offset + (uint64_t)i;
  float mh;
  uint16_t ab;
  sample_walker_f32(sp, traj, w.R + i, w.P + i, cap, mh, ab);
  w.mh[i] = mh;
  w.ml[i] = 0.0f;
  w.me[i] = 0;
  w.ph[i] = 0.0f;
  w.pl[i] = 0.0f;
  w.ab[i] = ab;
  w.id[i] = traj;
  w.fam[i] = (uint32_t)i;
}

__device__ __forceinline__ uint16_t pair_word(const Scal& z) {
  return (uint16_t)((z.sa > 0.0f ? 1 : 0) | ((z.q & 3) << 4) | ((z.sb > 0.0f ? 1 : 0) << 8));
}

// The phase pair is renormalised, and wrapped past 2^10 rad, at the end of
// every Philox block (absolute steps 4k + 3).
__device__ __forceinline__ void spawn_phase_end(Scal& z, int64_t step) {
  if ((step & 3) == 3) {
    z.ph = two_sum(z.ph.hi, z.ph.lo);
    phase_wrap(z);
  }
}

// What a step reports: non-finite children or phases, a degenerate gap.
__device__ __forceinline__ void spawn_report(EnsHeader* hdr, unsigned int bad, unsigned int deg) {
  if (bad) {
    atomicAdd(&hdr->n_nonfinite, (unsigned long long)bad);
    atomicOr(&hdr->flags, QCL_FLAG_NONFINITE);
  }
  if (deg) {
    atomicAdd(&hdr->n_degenerate, 1ull);
    atomicOr(&hdr->flags, QCL_FLAG_DEGENERATE);
  }
}

// A walker of the chained steps, modes in registers.
template <int NPL>
struct SWalker {
  Walker<NPL> w;
  f2 m, ph;
  int32_t me;
  uint16_t ab;
};

template <int NPL>
__device__ __forceinline__ void put_walker(const Set32& s, int64_t cap, int n, int64_t pos,
                                           const SWalker<NPL>& x, uint64_t id, uint32_t fam) {
#pragma unroll
  for (int j = 0; j < NPL; ++j)
    if (j < n) {
      s.R[(int64_t)j * cap + pos] = x.w.R[j];
      s.P[(int64_t)j * cap + pos] = x.w.P[j];
    }
  s.mh[pos] = x.m.hi;
  s.ml[pos] = x.m.lo;
  s.me[pos] = x.me;
  s.ph[pos] = x.ph.hi;
  s.pl[pos] = x.ph.lo;
  s.ab[pos] = x.ab;
  s.id[pos] = id;
  s.fam[pos] = fam;
}

// The weight, phase and pair of x as the step's scalars, and a and b at its R.
template <int NPL, int KIND, bool DIA>
__device__ __forceinline__ Scal walker_scal(const BulkParams& bp, const CoefLocal<NPL>& cf,
                                            const SWalker<NPL>& x) {
  Scal z;
  z.m = x.m;
  z.mexp = x.me;
  z.ph = x.ph;
  z.sa = sgn(x.ab & 0xf);
  z.sb = sgn((x.ab >> 8) & 0xf);
  z.q = DIA ? (int)((x.ab >> 4) & 3u) : 0;
  z.A = bp.a0;
  z.B = bp.b0;
#pragma unroll
  for (int j = 0; j < NPL; ++j) {
    z.A = __fmaf_rn(cf.a[j], x.w.R[j], z.A);
    if (KIND == 1) z.B = __fmaf_rn(cf.b[j], x.w.R[j], z.B);
  }
  return z;
}

// The couplings' sums over P.
template <int NPL, int KIND>
__device__ __forceinline__ void coupling_sums(const CoefLocal<NPL>& cf, const Walker<NPL>& w,
                                              float& Av, float& Bv) {
  Av = Bv = 0.0f;
#pragma unroll
  for (int j = 0; j < NPL; ++j) {
    Av = __fmaf_rn(cf.am[j], w.P[j], Av);
    if (KIND == 1) Bv = __fmaf_rn(cf.bm[j], w.P[j], Bv);
  }
}

// One step of the walker x (random stream id) in registers: x moves to the next
// step (its weight and pair stay); returns the event its test fires for (0 none).
// `report` counts degenerate gaps and non-finite phases in the header.
template <int NPL, int KIND, bool DIA>
__device__ __forceinline__ int step_walker(const BulkParams& bp, const CoefLocal<NPL>& cf,
                                           EnsHeader* hdr, int64_t step, SWalker<NPL>& x,
                                           uint64_t id, bool report) {
  using CF = CoefLocal<NPL>;
  Walker<NPL>& w = x.w;
  Scal z = walker_scal<NPL, KIND, DIA>(bp, cf, x);
  closed_form(z);
  const u4 wd = philox_draw(bp.seed, (uint32_t)(step >> 2), id, kPurposeHop);
  const uint32_t word = word_of(wd, (int)(step & 3));
  unsigned int deg = 0;
  uint32_t T;
  float fac;
  int ev;
  const float hsab = __fmul_rn(__fmul_rn(bp.hdt, 0.5f), __fadd_rn(z.sa, z.sb));
  if (DIA) {
    kick_dia<NPL, KIND, CF>(w, cf, hsab);
#pragma unroll
    for (int j = 0; j < NPL; ++j) w.R[j] = __fmaf_rn(cf.dtm[j], w.P[j], w.R[j]);
    const float a_old = z.A;
    z.A = bp.a0;
    if (KIND == 1) z.B = bp.b0;
#pragma unroll
    for (int j = 0; j < NPL; ++j) {
      z.A = __fmaf_rn(cf.a[j], w.R[j], z.A);
      if (KIND == 1) z.B = __fmaf_rn(cf.b[j], w.R[j], z.B);
    }
    kick_dia<NPL, KIND, CF>(w, cf, hsab);
    ev = spawn_event<KIND, true>(z, a_old, 0.0f, z.B, word, bp, deg, T, fac);
  } else {
    kick<NPL, KIND, CF>(w, cf, __fmul_rn(hsab, z.c2), __fmul_rn(hsab, z.s2));
#pragma unroll
    for (int j = 0; j < NPL; ++j) w.R[j] = __fmaf_rn(cf.dtm[j], w.P[j], w.R[j]);
    const float r_old = z.r;
    z.A = bp.a0;
    z.B = bp.b0;
#pragma unroll
    for (int j = 0; j < NPL; ++j) {
      z.A = __fmaf_rn(cf.a[j], w.R[j], z.A);
      if (KIND == 1) z.B = __fmaf_rn(cf.b[j], w.R[j], z.B);
    }
    closed_form(z);
    kick<NPL, KIND, CF>(w, cf, __fmul_rn(hsab, z.c2), __fmul_rn(hsab, z.s2));
    float Av, Bv;
    coupling_sums<NPL, KIND>(cf, w, Av, Bv);
    ev = spawn_event<KIND, false>(z, r_old, Av, Bv, word, bp, deg, T, fac);
  }
  spawn_phase_end(z, step);
  x.ph = z.ph;
  if (report) spawn_report(hdr, !isfinite(z.ph.hi) ? 1u : 0u, deg);
  return ev;
}

// The child of the walker x whose step has fired for event ev, from x after that
// step: the test's threshold follows from R and P again.  Returns false when its
// weight is not finite.
template <int NPL, int KIND, bool DIA>
__device__ __forceinline__ bool make_child(const BulkParams& bp, const CoefLocal<NPL>& cf,
                                           const SWalker<NPL>& x, int ev, SWalker<NPL>& c) {
  Scal z = walker_scal<NPL, KIND, DIA>(bp, cf, x);
  float Av = 0.0f, Bv = z.B;
  if (!DIA) {
    closed_form(z);
    coupling_sums<NPL, KIND>(cf, x.w, Av, Bv);
  }
  uint32_t T;
  float fac;
  spawn_rate<KIND, DIA>(z, Av, Bv, bp, T, fac);
  spawn_child<DIA>(z, ev, T, fac);
  renorm(z.m, z.mexp);
  c = x;
  c.m = z.m;
  c.me = z.mexp;
  c.ab = pair_word(z);
  return isfinite(z.m.hi);
}

// The chained steps' counts: children of each 256-walker group of the current
// set at step s in array s mod 3 (the space of bsum and boff), their sum in
// total[s mod 3].
__device__ __forceinline__ unsigned int* chain_counts(void* buf, const SpawnLayout& L, int k) {
  char* b = (char*)buf;
  return (unsigned int*)(k == 0 ? b + L.bsum : (k == 1 ? b + L.boff : b + L.boff + 4 * L.n_blocks));
}

// Adds this warp's firing walkers (bal, lane l at position pos0 + rank) to the
// counts of the groups their positions fall in.
__device__ __forceinline__ void add_counts(unsigned int* cnt, bool fires, int64_t pos) {
  const int lane = threadIdx.x & 31;
  const unsigned act = __ballot_sync(0xffffffffu, fires);
  if (!act) return;
  // positions ascend over the lanes and span at most two groups
  const int64_t g = pos >> 8;
  const int64_t g_lo = __shfl_sync(0xffffffffu, g, __ffs(act) - 1);
  const unsigned lo = __ballot_sync(0xffffffffu, fires && g == g_lo);
  if (lane == __ffs(act) - 1) atomicAdd(cnt + g_lo, (unsigned)__popc(lo));
  const unsigned up = act & ~lo;
  if (up && lane == __ffs(up) - 1) atomicAdd(cnt + g, (unsigned)__popc(up));
}

// One spawning step of the whole ensemble in one pass: set s & 1 to the other.
// The children of this step are known before it starts: the launch before has
// evaluated, beside its own step, which of its walkers fire at the next one, and
// counted them by the group of 256 positions they stand in.  So a block learns
// the children before its walkers by adding the counts of the groups before
// them, writes each walker with its child straight to its place, and evaluates
// the step after for the counts of the next launch (FIRST only counts, for a
// call's first step).  Nothing waits inside a launch, and an overflow is known at
// its start: then the step's children are dropped.
//
// `out`: the walkers are written as the step after leaves them, with the event
// that fired (0, 1, 2) in the top two bits of the pair word, and the next launch
// (`in`) has only to place them and to make the children of the few that fired.
// So a step is evaluated once; at the ends of an interval between output times,
// where the set has to hold the plain state, the step is evaluated for its counts
// and again by the next launch.  A launch that writes the plain state also writes
// the families' starts for the observation (a kernel of its own took 11 us).
//
// What bounds it: instruction issue at 1e6 walkers, launch latency below some 1e5
// (3.8 us a step at 1e3, 5.7 at 1e5).  1e5 initial one-mode walkers growing to
// 1.57e6 over 400 steps with an output every 10: 7.0 ms of device time; 10.0 ms
// when every launch evaluated its own step again, 15.9 ms with a step in place, a
// one-block scan and a scatter.  One cooperative launch for many steps, with a
// decoupled look-back over the groups' counts and a grid barrier, was slower (13.6
// ms): a poll of another die's word costs about a microsecond, and a step needs
// several in a row.
template <int NPL, int KIND, bool DIA, bool FIRST>
__global__ void __launch_bounds__(256, NPL <= 4 ? 3 : (NPL <= 8 ? 2 : 1))
    k_spawn_chain32(const BulkParams bp, const CoefLocal<NPL> cf, const SpawnLayout L, void* buf,
                    int64_t cap, int64_t n0, int64_t step, int in, int out) {
  __shared__ int wcnt[2][8];
  __shared__ unsigned long long wsum[8];
  if (!FIRST) {
    // the launch after may bring its blocks in; this one goes on when the launch
    // before has finished and its writes can be seen
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();
  }
  EnsHeader* hdr = (EnsHeader*)buf;
  SpawnHeader* sh = hdr_spawn(buf);
  // (FIRST counts the step itself; otherwise the step after it)
  const int src = (int)(step & 1), k3 = (int)(step % 3);
  const int64_t n_live = sh->n_live[src];
  const int64_t total = FIRST ? 0 : (int64_t)sh->total[k3];
  if (hdr->step != bp.step0) {  // uniform over the grid
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&hdr->flags, QCL_FLAG_STEP_MISMATCH);
    return;
  }
  const int kn = FIRST ? k3 : (k3 + 1) % 3, kz = (k3 + 2) % 3;
  unsigned int* const cnt = chain_counts(buf, L, k3);
  unsigned int* const nxt = chain_counts(buf, L, kn);
  unsigned int* const clr = chain_counts(buf, L, kz);
  const bool drop = n_live + total > cap;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // a contiguous run of groups for each block
  const int64_t groups = (n_live + 255) / 256;
  const int64_t per = (groups + gridDim.x - 1) / gridDim.x;
  const int64_t g0 = min((int64_t)blockIdx.x * per, groups), g1 = min(g0 + per, groups);
  const Set32 s = set32(buf, L, src), d = set32(buf, L, src ^ 1);
  int64_t* const fstart = (int64_t*)((char*)buf + L.fstart);
  SWalker<NPL> x;
  uint64_t id = 0;
  uint32_t fam = 0;
  int ev = 0;  // the event x's step fired for
  auto load = [&](int64_t g) {
    const int64_t i = g * 256 + threadIdx.x;
    const int64_t ii = i < n_live ? i : 0;
#pragma unroll
    for (int j = 0; j < NPL; ++j) {
      const bool on = j < bp.n;
      x.w.R[j] = on ? s.R[(int64_t)j * cap + ii] : 0.0f;
      x.w.P[j] = on ? s.P[(int64_t)j * cap + ii] : 0.0f;
    }
    x.m = {s.mh[ii], s.ml[ii]};
    x.me = s.me[ii];
    x.ph = {s.ph[ii], s.pl[ii]};
    const unsigned ab = s.ab[ii];
    x.ab = (uint16_t)(ab & 0x3fffu);
    ev = (int)(ab >> 14);
    id = s.id[ii];
    fam = s.fam[ii];
  };
  if (g0 < g1) load(g0);  // (in flight while the prefix is added up)
  int64_t prefix = 0;
  if (!FIRST) {
    for (int64_t k = (int64_t)blockIdx.x * 256 + threadIdx.x; k < L.n_blocks;
         k += (int64_t)gridDim.x * 256)
      clr[k] = 0u;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      sh->total[kz] = 0;
      sh->n_live[src ^ 1] = drop ? n_live : n_live + total;
      if (!out) fstart[n0] = drop ? n_live : n_live + total;
      if (drop) atomicOr(&hdr->flags, QCL_FLAG_SPAWN_OVERFLOW);
    }
    if (!drop && g0 < g1) {
      unsigned long long sum = 0;
      for (int64_t k = threadIdx.x; k < g0; k += 256) sum += cnt[k];
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
      if (lane == 0) wsum[warp] = sum;
      __syncthreads();
#pragma unroll
      for (int k = 0; k < 8; ++k) prefix += (int64_t)wsum[k];
    }
  }
  unsigned int found = 0;  // firing walkers this thread's warp counted (lane 0)
  for (int64_t g = g0; g < g1; ++g) {
    const int64_t i = g * 256 + threadIdx.x;
    bool live = i < n_live;
    if (g > g0) load(g);
    // phase 0: the step itself, of walkers not moved yet; 1: the walkers' next
    // step; 2: their children's.  One copy of the step's code, of a third of the
    // size.  A walker's test comes out the same when it is counted (a call's
    // first step by the FIRST kernel) and when it is taken, since every rounding
    // in it is explicit.
    SWalker<NPL> xc;      // the children
    uint64_t idc = 0;
    bool hop = false;
    int64_t pos = i;
#pragma unroll 1
    for (int phase = FIRST || in ? 1 : 0; phase < 3; ++phase) {
      if (!FIRST && phase == 1) {  // the walkers have moved: children and places
        hop = ev != 0 && live;
        if (hop && !make_child<NPL, KIND, DIA>(bp, cf, x, ev, xc)) spawn_report(hdr, 1u, 0u);
        hop = hop && !drop;
        const unsigned bal = __ballot_sync(0xffffffffu, hop);
        int* const wc = wcnt[(g - g0) & 1];  // (two in turn: one barrier a group)
        if (lane == 0) wc[warp] = __popc(bal);
        __syncthreads();
        int before = __popc(bal & ((1u << lane) - 1u)), c = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          before += k < warp ? wc[k] : 0;
          c += wc[k];
        }
        pos = i + prefix + before;
        prefix += c;
        // (with tests that agree with their counts a group's places lie in the buffer;
        // should they ever differ, nothing is written past its end and the step
        // counts as one that did not fit)
        if (min(g * 256 + 256, n_live) + prefix > cap) {
          if (threadIdx.x == 0) atomicOr(&hdr->flags, QCL_FLAG_SPAWN_OVERFLOW);
          live = hop = false;
        }
        if (hop) idc = child_id32(bp.seed, step, id);
        if (!out) {
          // a family's first walker stays its first: children follow parents
          const uint32_t left = __shfl_up_sync(0xffffffffu, fam, 1);
          if (live && (i == 0 || (lane > 0 ? left : s.fam[i - 1]) != fam) && (int64_t)fam < n0)
            fstart[fam] = pos;
          if (live) put_walker(d, cap, bp.n, pos, x, id, fam);
          if (hop) put_walker(d, cap, bp.n, pos + 1, xc, idc, fam);
        }
      }
      bool on = live;
      if (phase == 2) {
        if (FIRST || !__any_sync(0xffffffffu, hop)) break;
        x = xc;
        id = idc;
        on = hop;
        ++pos;
      }
      ev = step_walker<NPL, KIND, DIA>(bp, cf, hdr, FIRST || phase == 0 ? step : step + 1, x, id,
                                       on && (phase == 0 || (!FIRST && out)));
      if (phase > 0) {
        const bool f = on && ev != 0;
        add_counts(nxt, f, pos);
        found += __popc(__ballot_sync(0xffffffffu, f));
        if (!FIRST && out && on) {
          x.ab |= (uint16_t)(ev << 14);
          put_walker(d, cap, bp.n, pos, x, id, fam);
        }
      }
    }
  }
  if (lane == 0 && found) atomicAdd(&sh->total[kn], (unsigned long long)found);
}

// The counts and totals of a call's first step start at zero.
__global__ void __launch_bounds__(256) k_spawn_chain_clear(void* buf, int64_t cap, int n,
                                                           int64_t n0) {
  const SpawnLayout L = SpawnLayout::make(cap, n, n0, QCL_PREC_FP32_BULK);
  for (int64_t k = (int64_t)blockIdx.x * 256 + threadIdx.x; k < L.n_blocks;
       k += (int64_t)gridDim.x * 256)
    for (int a = 0; a < 3; ++a) chain_counts(buf, L, a)[k] = 0u;
  if (blockIdx.x == 0 && threadIdx.x < 3) hdr_spawn(buf)->total[threadIdx.x] = 0;
}

// Any mode count, the modes in memory: one step of every live walker of set
// `src` (in place); children to the per-parent staging, each block's child count
// to bsum.  R and P are read and written back mode by mode with the
// register form's operations in its order (the same bits): one pass for the diabatic
// step, three for the adiabatic one (a(R_n), b(R_n); first half kick, drift, a
// and b at R_{n+1}; second half kick and the coupling sums).
template <int KIND, bool DIA>
__global__ void __launch_bounds__(256) k_spawn_step32(const BulkParams bp, const Coef2 cf,
                                                      void* buf, int64_t cap, int64_t n0,
                                                      int64_t step) {
  const SpawnLayout L = SpawnLayout::make(cap, bp.n, n0, QCL_PREC_FP32_BULK);
  EnsHeader* hdr = (EnsHeader*)buf;
  const int src = (int)(step & 1);
  const int64_t n_live = hdr_spawn(buf)->n_live[src];
  const bool ok = hdr->step == bp.step0;
  if (!ok) {
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&hdr->flags, QCL_FLAG_STEP_MISMATCH);
    return;
  }
  // a grid of a few blocks per SM walks the live walkers in groups of 256
  const int64_t nvb = (n_live + 255) / 256;
  for (int64_t vb = blockIdx.x; vb < nvb; vb += gridDim.x) {
    const int64_t i = vb * 256 + threadIdx.x;
    int flag = 0;
    if (i < n_live) {
      const Set32 s = set32(buf, L, src);
      Scal z;
      z.m = {s.mh[i], s.ml[i]};
      z.mexp = s.me[i];
      z.ph = {s.ph[i], s.pl[i]};
      const uint32_t ab = s.ab[i];
      z.sa = sgn(ab & 0xf);
      z.sb = sgn((ab >> 8) & 0xf);
      z.q = DIA ? (int)((ab >> 4) & 3u) : 0;
      z.A = bp.a0;
      z.B = bp.b0;
      for (int j = 0; j < bp.n; ++j) {
        const float r = s.R[(int64_t)j * cap + i];
        z.A = __fmaf_rn(cf.a[j], r, z.A);
        if (KIND == 1) z.B = __fmaf_rn(cf.b[j], r, z.B);
      }
      closed_form(z);
      const u4 wd = philox_draw(bp.seed, (uint32_t)(step >> 2), s.id[i], kPurposeHop);
      const uint32_t word = word_of(wd, (int)(step & 3));
      unsigned int deg = 0;
      uint32_t T;
      float fac;
      int ev;
      const float hsab = __fmul_rn(__fmul_rn(bp.hdt, 0.5f), __fadd_rn(z.sa, z.sb));
      // P += dt/2 F with the pair's force (kick / kick_dia of one mode)
      auto kick1 = [&](int j, float r, float p, float hu, float hv) {
        p = __fmaf_rn(-cf.hk[j], r, p);
        if (KIND == 1) p = __fadd_rn(p, -cf.hs[j]);
        if (DIA) return __fmaf_rn(hsab, cf.a[j], p);
        p = __fmaf_rn(hu, -cf.a[j], p);
        if (KIND == 1) p = __fmaf_rn(hv, -cf.b[j], p);
        return p;
      };
      if (DIA) {
        const float a_old = z.A;
        z.A = bp.a0;
        if (KIND == 1) z.B = bp.b0;
        for (int j = 0; j < bp.n; ++j) {
          float r = s.R[(int64_t)j * cap + i], p = s.P[(int64_t)j * cap + i];
          p = kick1(j, r, p, 0.0f, 0.0f);
          r = __fmaf_rn(cf.dtm[j], p, r);
          z.A = __fmaf_rn(cf.a[j], r, z.A);
          if (KIND == 1) z.B = __fmaf_rn(cf.b[j], r, z.B);
          s.R[(int64_t)j * cap + i] = r;
          s.P[(int64_t)j * cap + i] = kick1(j, r, p, 0.0f, 0.0f);
        }
        ev = spawn_event<KIND, true>(z, a_old, 0.0f, z.B, word, bp, deg, T, fac);
      } else {
        const float hu = __fmul_rn(hsab, z.c2), hv = __fmul_rn(hsab, z.s2);
        const float r_old = z.r;
        z.A = bp.a0;
        z.B = bp.b0;
        for (int j = 0; j < bp.n; ++j) {
          float r = s.R[(int64_t)j * cap + i], p = s.P[(int64_t)j * cap + i];
          p = kick1(j, r, p, hu, hv);
          r = __fmaf_rn(cf.dtm[j], p, r);
          z.A = __fmaf_rn(cf.a[j], r, z.A);
          if (KIND == 1) z.B = __fmaf_rn(cf.b[j], r, z.B);
          s.R[(int64_t)j * cap + i] = r;
          s.P[(int64_t)j * cap + i] = p;
        }
        closed_form(z);
        const float hu2 = __fmul_rn(hsab, z.c2), hv2 = __fmul_rn(hsab, z.s2);
        float Av = 0.0f, Bv = 0.0f;
        for (int j = 0; j < bp.n; ++j) {
          const float r = s.R[(int64_t)j * cap + i];
          const float p = kick1(j, r, s.P[(int64_t)j * cap + i], hu2, hv2);
          Av = __fmaf_rn(cf.am[j], p, Av);
          if (KIND == 1) Bv = __fmaf_rn(cf.bm[j], p, Bv);
          s.P[(int64_t)j * cap + i] = p;
        }
        ev = spawn_event<KIND, false>(z, r_old, Av, Bv, word, bp, deg, T, fac);
      }
      Scal child = z;
      const bool hop = ev != 0;
      if (hop) spawn_child<DIA>(child, ev, T, fac);
      spawn_phase_end(z, step);
      s.ph[i] = z.ph.hi;
      s.pl[i] = z.ph.lo;
      flag = hop ? 1 : 0;
      uint8_t* fl = (uint8_t*)((char*)buf + L.flag);
      fl[i] = (uint8_t)flag;
      if (hop) {
        renorm(child.m, child.mexp);
        ((float*)((char*)buf + L.cm))[i] = child.m.hi;
        ((float*)((char*)buf + L.cmlo))[i] = child.m.lo;
        ((int32_t*)((char*)buf + L.cmexp))[i] = child.mexp;
        ((uint16_t*)((char*)buf + L.cab))[i] = pair_word(child);
      }
      spawn_report(hdr, (hop && !isfinite(child.m.hi) ? 1u : 0u) + (!isfinite(z.ph.hi) ? 1u : 0u), deg);
    }
    const int cnt = __syncthreads_count(flag);
    if (threadIdx.x == 0) ((int32_t*)((char*)buf + L.bsum))[vb] = cnt;
  }
}

// Moves every live walker of set src to its place in the other set and writes
// each child right after its parent.
__global__ void __launch_bounds__(256) k_spawn_scatter32(void* buf, int64_t cap, int n, int64_t n0,
                                                         int64_t step0, int64_t step,
                                                         uint64_t seed) {
  __shared__ int wcnt[8];
  const SpawnLayout L = SpawnLayout::make(cap, n, n0, QCL_PREC_FP32_BULK);
  EnsHeader* hdr = (EnsHeader*)buf;
  SpawnHeader* sh = hdr_spawn(buf);
  if (hdr->step != step0) return;  // uniform over the grid
  const int src = (int)(step & 1);
  const int64_t n_live = sh->n_live[src];
  const bool drop = sh->drop != 0;
  const uint8_t* fl = (const uint8_t*)((char*)buf + L.flag);
  const int64_t nvb = (n_live + 255) / 256;
  for (int64_t vb = blockIdx.x; vb < nvb; vb += gridDim.x) {
    const int64_t i = vb * 256 + threadIdx.x;
    const bool live = i < n_live;
    const int flag = (live && !drop) ? fl[i] : 0;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned bal = __ballot_sync(0xffffffffu, flag);
    if (lane == 0) wcnt[wid] = __popc(bal);
    __syncthreads();
    int before = __popc(bal & ((1u << lane) - 1u));
    for (int k = 0; k < wid; ++k) before += wcnt[k];
    if (live) {
      const int64_t boff = drop ? 0 : ((const int64_t*)((char*)buf + L.boff))[vb];
      const int64_t pos = i + boff + before;
      const Set32 s = set32(buf, L, src);
      const Set32 d = set32(buf, L, src ^ 1);
      for (int j = 0; j < n; ++j) {
        const float r = s.R[(int64_t)j * cap + i], p = s.P[(int64_t)j * cap + i];
        d.R[(int64_t)j * cap + pos] = r;
        d.P[(int64_t)j * cap + pos] = p;
        if (flag) {
          d.R[(int64_t)j * cap + pos + 1] = r;
          d.P[(int64_t)j * cap + pos + 1] = p;
        }
      }
      const float ph = s.ph[i], pl = s.pl[i];
      const uint64_t id = s.id[i];
      const uint32_t fam = s.fam[i];
      d.mh[pos] = s.mh[i];
      d.ml[pos] = s.ml[i];
      d.me[pos] = s.me[i];
      d.ph[pos] = ph;
      d.pl[pos] = pl;
      d.ab[pos] = s.ab[i];
      d.id[pos] = id;
      d.fam[pos] = fam;
      if (flag) {
        d.mh[pos + 1] = ((const float*)((char*)buf + L.cm))[i];
        d.ml[pos + 1] = ((const float*)((char*)buf + L.cmlo))[i];
        d.me[pos + 1] = ((const int32_t*)((char*)buf + L.cmexp))[i];
        d.ph[pos + 1] = ph;
        d.pl[pos + 1] = pl;
        d.ab[pos + 1] = ((const uint16_t*)((char*)buf + L.cab))[i];
        d.id[pos + 1] = child_id32(seed, step, id);
        d.fam[pos + 1] = fam;
      }
    }
    __syncthreads();  // wcnt is rewritten by the next group
  }
}

// a += x f with the product's own rounding error: the rounded product enters the
// sum, the exact one its error term.  (Written out: with a fused product in both,
// as the compiler may have it, the error term misses up to 2^-25 of the terms;
// this form is exact to 2^-48.)
__device__ __forceinline__ void add_product(f2& a, float x, float f) {
  const float s = __fadd_rn(__fmul_rn(x, f), a.hi), bb = __fsub_rn(s, a.hi);
  const float err = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fmaf_rn(x, f, -bb));
  a = {s, __fadd_rn(a.lo, err)};
}

// Family observation: for each family the sum X of its walkers' contributions
// and X^2.  A block takes a tile of 256 families.  A family shares one power of
// two (its largest weight exponent), so each walker's contribution is an FP32
// value, summed as a compensated FP32 pair per lane (lane l of the family's w
// takes walkers l, l + w, ...) and then over the lanes by a reduce-scatter of
// pairs; X is rebuilt in FP64 from the pair and the exponent exactly.  (Accumulating
// every walker in FP64 kept the FP64 pipe 84 % busy: FP64 is slow on this part.)
//
// w = 1 up to `per` walkers, twice as many lanes for every doubling, 32 beyond 16
// `per`.  per = 8 up to 24 modes, since the reduce-scatter over the lanes and the
// conversion cost as much as two walkers, and more in a row would leave small
// ensembles waiting on one lane's chain; 4 up to 64 modes and 1 beyond, where a
// walker's own loads outweigh the reduction and lanes of one family read
// neighbouring walkers.  An output of 200000 families by 8, 4, 2 and 1: 13.8
// walkers of 32 modes 411, 338, 348 and 378 us, 5.2 of 40 modes 273, 230, 203 and
// 215, 5.4 of 100 modes 689, 567, 492 and 458; of 16 modes 203, 206, 223 and 244.
//
// 32 / w families go side by side, the block's families ordered by size so that
// those of a warp are alike and few lanes idle, and the block's warps take such
// groups in turn, widest first.  The X of the tile's families then meet in shared
// memory, where the even lane of a pair adds X, the odd lane X^2, of one quantity
// over a warp's 32 families in order, and the 8 warps are folded by the fixed tree
// of the observation kernels.
//
// A family of more than kFamWide walkers is taken by the whole block (a walker of
// 256 a lane, the warps' pairs added in order), so that the few large families of
// a model whose walkers multiply near a crossing do not leave the launch waiting
// for one warp.  200000 families of 13.9 walkers on average, the largest tens of
// thousands, 16 modes, an output: 1518 us by one warp a family, 338, 324 and 299
// with the line at 1024, 512 and 256; families without such a tail are unchanged.
// At 512 the block's eight reductions weigh as much as its sixteen walkers a warp.
//
// Bound by instruction issue, the FP64 pipe (48 operations a family) for small
// families.  1e5 families growing from 1 to 15.7 walkers: 30 to 93 us, 36 to
// 160 with one walker a lane and the families of a warp in its own order.
constexpr int kFamClasses = 9;
constexpr int64_t kFamWide = 512;  // (half of it above 64 modes, `per` = 1)
template <int KIND, bool DIA>
__global__ void __launch_bounds__(256, 4) k_spawn_observe32(const BulkParams bp, const Coef2 cf,
                                                         const void* buf, int64_t cap, int64_t n0,
                                                         int set, int per,
                                                         double* __restrict__ part) {
  __shared__ double red[8][32];
  __shared__ double xs[8][32][17];  // (rows of 17: no bank conflicts between families)
  __shared__ uint8_t ord[256];      // families by class, widest first
  __shared__ int cnt[kFamClasses][8];
  __shared__ int wide_em[8];        // a family of the whole block: its warps' exponents
  __shared__ f2 wide_sum[8][16];    // and sums
  const SpawnLayout L = SpawnLayout::make(cap, bp.n, n0, QCL_PREC_FP32_BULK);
  const Set32 s = set32((void*)buf, L, set);
  const int64_t* fstart = (const int64_t*)((const char*)buf + L.fstart);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t f0 = (int64_t)blockIdx.x * 256;
  // this thread's family and its class: 0 for the whole block, 1 (beyond 16 `per`
  // walkers) to 5 (beyond `per`) for 32 to 2 lanes, 6 to 8 one lane (beyond half of
  // it, 2 or more, at most 1)
  const bool real = f0 + threadIdx.x < n0;
  const int64_t size = real ? fstart[f0 + threadIdx.x + 1] - fstart[f0 + threadIdx.x] : 0;
  const int cls = !real ? kFamClasses
                        : size > (per > 1 ? kFamWide : kFamWide / 2) ? 0
                        : size > 16 * per ? 1 : size > 8 * per ? 2 : size > 4 * per ? 3
                        : size > 2 * per ? 4 : size > per ? 5 : size > (per >> 1) ? 6
                        : size > 1 ? 7 : 8;
  unsigned mates = 0;
#pragma unroll
  for (int c = 0; c < kFamClasses; ++c) {
    const unsigned in = __ballot_sync(0xffffffffu, cls == c);
    if (cls == c) mates = in;
    if (lane == c) cnt[c][warp] = __popc(in);
  }
  __syncthreads();
  if (real) {
    int at = __popc(mates & ((1u << lane) - 1u));
    for (int c = 0; c <= cls; ++c)
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (c < cls || k < warp) at += cnt[c][k];
    ord[at] = (uint8_t)threadIdx.x;
  }
  __syncthreads();
  // the sum over family f (of the tile) by the w lanes of which this one is `sl`
  // (WIDE: by the whole block); lanes without a family (on false) only take part
  auto family = [&](auto wide, int f, bool on, int w, int sl) {
    constexpr bool WIDE = decltype(wide)::value;
    const int off0 = WIDE ? threadIdx.x : sl, step = WIDE ? 256 : w;
    const int64_t j0 = fstart[f0 + f];
    const int64_t j1 = on ? fstart[f0 + f + 1] : j0;
    int em = -(1 << 28);
    for (int64_t j = j0 + off0; j < j1; j += step)
      if (s.mh[j] != 0.0f) em = max(em, s.me[j]);
    for (int off = w >> 1; off > 0; off >>= 1)
      em = max(em, __shfl_xor_sync(0xffffffffu, em, off));
    if constexpr (WIDE) {
      if (lane == 0) wide_em[warp] = em;
      __syncthreads();
      for (int k = 0; k < 8; ++k) em = max(em, wide_em[k]);
    }
    f2 acc[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) acc[q] = {0.0f, 0.0f};
    for (int64_t j = j0 + off0; j < j1; j += step) {
      Scal z;
      z.A = bp.a0;
      z.B = bp.b0;
      for (int m = 0; m < bp.n; ++m) {
        const float r = s.R[(int64_t)m * cap + j];
        z.A = __fmaf_rn(cf.a[m], r, z.A);
        if (KIND == 1) z.B = __fmaf_rn(cf.b[m], r, z.B);
      }
      closed_form(z);
      const uint32_t ab = s.ab[j];
      z.sa = sgn(ab & 0xf);
      z.sb = sgn((ab >> 8) & 0xf);
      z.q = DIA ? (int)((ab >> 4) & 3u) : 0;
      z.ph = {s.ph[j], s.pl[j]};
      const float mh = s.mh[j];
      const float mm = mh == 0.0f ? 0.0f : (mh + s.ml[j]) * pow2i(s.me[j] - em);
      const Contrib c = contrib_factors<DIA>(z, mm);
      const float fac[4] = {c.f00, c.f01, c.f10, c.f11};
      constexpr int other = DIA ? 8 : 0, own = DIA ? 0 : 8;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const float x = (q & 1) ? c.zi : c.zr;
        f2& ao = acc[own + q];
        const f2 t = two_sum(ao.hi, (q >> 1) == c.k ? x : 0.0f);
        ao = {t.hi, ao.lo + t.lo};
        add_product(acc[other + q], x, fac[q >> 1]);
      }
    }
    __syncwarp();
    // reduce-scatter of the pairs: at the step with offset `off`, the lane with
    // that bit set keeps the upper half of its values (q0: the first it keeps)
    int q0 = 0, keep = 16, off = w >> 1;
#pragma unroll
    for (int half = 8; half >= 1; half >>= 1) {
      if (off > 0) {
        const bool upper = (lane & off) != 0;
#pragma unroll
        for (int i2 = 0; i2 < half; ++i2) {
          const f2 snd = upper ? acc[i2] : acc[half + i2];
          const f2 kp = upper ? acc[half + i2] : acc[i2];
          const float rh = __shfl_xor_sync(0xffffffffu, snd.hi, off);
          const float rl = __shfl_xor_sync(0xffffffffu, snd.lo, off);
          const f2 t = two_sum(kp.hi, rh);
          acc[i2] = {t.hi, t.lo + (kp.lo + rl)};
        }
        q0 += upper ? half : 0;
        keep = half;
        off >>= 1;
      }
    }
    if (off > 0) {  // (w = 32: lanes 2q and 2q + 1 both end with quantity q)
      const float rh = __shfl_xor_sync(0xffffffffu, acc[0].hi, 1);
      const float rl = __shfl_xor_sync(0xffffffffu, acc[0].lo, 1);
      const f2 t = two_sum(acc[0].hi, rh);
      acc[0] = {t.hi, t.lo + (acc[0].lo + rl)};
    }
    const int ex = (em < -(1 << 27)) ? 0 : em;
    if constexpr (WIDE) {  // the warps' sums, in order
      if (!(lane & 1)) wide_sum[warp][lane >> 1] = acc[0];
      __syncthreads();
      if (threadIdx.x < 16) {
        f2 t = wide_sum[0][threadIdx.x];
        for (int k = 1; k < 8; ++k) {
          const f2 x = wide_sum[k][threadIdx.x], u = two_sum(t.hi, x.hi);
          t = {u.hi, u.lo + (t.lo + x.lo)};
        }
        xs[f >> 5][f & 31][threadIdx.x] = scaled_double(t.hi, ex) + scaled_double(t.lo, ex);
      }
    } else {
#pragma unroll
      for (int i2 = 0; i2 < 16; ++i2)
        if (on && i2 < keep)
          xs[f >> 5][f & 31][q0 + i2] =
              scaled_double(acc[i2].hi, ex) + scaled_double(acc[i2].lo, ex);
    }
  };
  int first = 0;  // the class's first place in ord
  for (int k = 0; k < 8; ++k) first += cnt[0][k];
  for (int k = 0; k < first; ++k) family(std::true_type{}, ord[k], true, 32, lane);
  int turn = warp;  // groups until this warp's next
#pragma unroll 1
  for (int c = 0; c <= 5; ++c) {
    int count = 0;
    for (int c2 = c + 1; c2 < (c == 5 ? kFamClasses : c + 2); ++c2)  // (one-lane classes together)
#pragma unroll
      for (int k = 0; k < 8; ++k) count += cnt[c2][k];
    const int w = 32 >> c, side = 32 / w, groups = (count + side - 1) / side;
    const int sub = lane / w, sl = lane - sub * w;
#pragma unroll 1
    for (; turn < groups; turn += 8) {
      const int at = turn * side;
      const bool on = at + sub < count;
      family(std::false_type{}, ord[first + (on ? at + sub : at)], on, w, sl);
    }
    first += count;
    turn -= groups;
  }
  __syncthreads();
  const int nf = (int)max((int64_t)0, min((int64_t)32, n0 - (f0 + warp * 32)));
  double T = 0.0;
  for (int f = 0; f < nf; ++f) {
    const double X = xs[warp][f][lane >> 1];
    T = fma(X, (lane & 1) ? X : 1.0, T);  // (X 1 + T is T + X: one FP64 instruction for both)
  }
  red[warp][(lane & 1) ? 16 + (lane >> 1) : (lane >> 1)] = T;
  __syncthreads();
  if (threadIdx.x < 32)
    part[(int64_t)blockIdx.x * 32 + threadIdx.x] = tile_tree8(&red[0][0], 32, threadIdx.x);
}

template <int NPL, int KIND, bool DIA>
void run_steps32(const BulkParams& bp, const Coef2& c2, void* buf, int64_t cap, int64_t n0,
                 int64_t step, int64_t len, cudaStream_t st) {
  CoefLocal<NPL> cf{};
  for (int j = 0; j < NPL && j < bp.n; ++j) {
    cf.hk[j] = c2.hk[j];
    cf.hs[j] = c2.hs[j];
    cf.dtm[j] = c2.dtm[j];
    cf.a[j] = c2.a[j];
    cf.b[j] = c2.b[j];
    cf.am[j] = c2.am[j];
    cf.bm[j] = c2.bm[j];
  }
  const SpawnLayout L = SpawnLayout::make(cap, bp.n, n0, QCL_PREC_FP32_BULK);
  // every block resident at once (at most one group a block)
  static const int per_sm = [] {
    int b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_spawn_chain32<NPL, KIND, DIA, false>, 256, 0);
    return b < 1 ? 1 : b;
  }();
  const unsigned grid = spawn_grid(cap, per_sm);
  if (step == bp.step0) {
    k_spawn_chain_clear<<<grid, 256, 0, st>>>(buf, cap, bp.n, n0);
    k_spawn_chain32<NPL, KIND, DIA, true><<<grid, 256, 0, st>>>(bp, cf, L, buf, cap, n0, step, 0, 0);
    launches_add(2);
  }
  // A step's launch after another step's is a programmatic dependent one: its
  // blocks come in while the last ones of the step before finish.
  cudaLaunchAttribute dep{};
  dep.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  dep.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t lc{};
  lc.gridDim = dim3(grid);
  lc.blockDim = dim3(256);
  lc.stream = st;
  lc.attrs = &dep;
  for (int64_t t = step; t < step + len; ++t) {
    lc.numAttrs = t > step ? 1 : 0;
    cudaLaunchKernelEx(&lc, k_spawn_chain32<NPL, KIND, DIA, false>, bp, cf, L, buf, cap, n0, t,
                       (int)(t > step), (int)(t + 1 < step + len));
  }
  launches_add(len);
}

// Chained steps with the modes in registers up to 32 modes; beyond that (or under
// QCL_OPT_MODES_IN_MEMORY = 1) in memory, three launches a step.
template <int KIND, bool DIA>
void dispatch_steps32(const BulkParams& bp, const Coef2& cf, void* buf, int64_t cap, int64_t n0,
                      int64_t step0, int64_t step, int64_t len, bool chain, cudaStream_t st) {
  const int n = bp.n;
  if (!chain) {
    for (int64_t t = step; t < step + len; ++t) {
      k_spawn_step32<KIND, DIA><<<spawn_grid(cap), 256, 0, st>>>(bp, cf, buf, cap, n0, t);
      launch_spawn_scan(buf, cap, n, n0, QCL_PREC_FP32_BULK, 2, step0, t, st);
      k_spawn_scatter32<<<spawn_grid(cap), 256, 0, st>>>(buf, cap, n, n0, step0, t, bp.seed);
      launches_add(2);
    }
    return;
  }
  if (n <= 1) run_steps32<1, KIND, DIA>(bp, cf, buf, cap, n0, step, len, st);
  else if (n <= 2) run_steps32<2, KIND, DIA>(bp, cf, buf, cap, n0, step, len, st);
  else if (n <= 4) run_steps32<4, KIND, DIA>(bp, cf, buf, cap, n0, step, len, st);
  else if (n <= 8) run_steps32<8, KIND, DIA>(bp, cf, buf, cap, n0, step, len, st);
  else if (n <= 16) run_steps32<16, KIND, DIA>(bp, cf, buf, cap, n0, step, len, st);
  else run_steps32<32, KIND, DIA>(bp, cf, buf, cap, n0, step, len, st);
}

}  // namespace

void launch_spawn_sample32(const DevModel& host, const SampleParams& sp, int64_t capacity, void* buf,
                           cudaStream_t st) {
  const int64_t nb = (sp.n_traj + 255) / 256;
  Sample32 s32;
  make_sample32(host, sp, s32);
  k_spawn_sample32<<<(unsigned)(nb > 0 ? nb : 1), 256, 0, st>>>(s32, capacity, buf);
  launches_add(1);
}

bool spawn_chained32(int n) { return n <= 32 && option_modes_in_memory() != 1; }

void launch_spawn_steps32(const BulkParams& bp, const Coef2& cf, void* buf, int64_t capacity,
                          int64_t n0, int64_t step0, int64_t step, int64_t len, bool chain,
                          cudaStream_t st) {
  auto run = [&](auto f) { f(bp, cf, buf, capacity, n0, step0, step, len, chain, st); };
  if (bp.repr == QCL_REPR_DIABATIC) run(bp.kind == 0 ? dispatch_steps32<0, true> : dispatch_steps32<1, true>);
  else run(bp.kind == 0 ? dispatch_steps32<0, false> : dispatch_steps32<1, false>);
}

void launch_spawn_observe32(const BulkParams& bp, const Coef2& cf, const void* buf, int64_t capacity,
                            int64_t n0, int set, bool starts, double* part, cudaStream_t st) {
  // (starts: chained steps have left the families' starts)
  if (!starts)
    launch_spawn_fstart(buf, capacity, bp.n, n0, QCL_PREC_FP32_BULK, 2, set, st);
  const unsigned nf = (unsigned)((n0 + 255) / 256);
  const bool dia = bp.repr == QCL_REPR_DIABATIC;
  const int per = bp.n <= 24 ? 8 : (bp.n <= 64 ? 4 : 1);  // walkers a lane
  if (dia)
    (bp.kind == 0 ? k_spawn_observe32<0, true> : k_spawn_observe32<1, true>)
        <<<nf, 256, 0, st>>>(bp, cf, buf, capacity, n0, set, per, part);
  else
    (bp.kind == 0 ? k_spawn_observe32<0, false> : k_spawn_observe32<1, false>)
        <<<nf, 256, 0, st>>>(bp, cf, buf, capacity, n0, set, per, part);
  launches_add(1);
}

}  // namespace qcl
