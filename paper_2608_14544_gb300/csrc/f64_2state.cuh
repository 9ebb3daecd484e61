// f64_2state.cuh -- device code of the FP64 two-state walker shared by the step
// kernels (kernels_f64.cu: many steps a launch) and the spawning kernels
// (spawn.cu): SoA views, the closed-form decomposition, the half kicks, one
// whole step of one walker (Verlet, phase, transition test) and the walker's
// observable contributions.
#pragma once
#include <type_traits>

#include "kernels.h"

namespace qcl {

constexpr double kDegTol = 1e-12;  // |e_b - e_a| below this: coupling set to 0

struct W64 {
  double* R;
  double* P;
  double* m;
  double* phi;
  uint16_t* ab;
  EnsHeader* hdr;
};

__device__ __forceinline__ W64 view64(void* buf, int64_t nt, int ns, int n) {
  const EnsLayout L = EnsLayout::make(nt, ns, n, QCL_PREC_FP64);
  char* b = (char*)buf;
  return {(double*)(b + L.off_R), (double*)(b + L.off_P), (double*)(b + L.off_m),
          (double*)(b + L.off_phi), (uint16_t*)(b + L.off_ab), (EnsHeader*)b};
}

// Closed-form two-state decomposition at R: W = s + a sigma_z + b sigma_x,
// r = |(a, b)|, theta = atan2(b, a)/2 (0 at r = 0); the eigenvector angle (c, s) =
// (cos theta, sin theta) by the cancellation-free half-angle formulas.
struct Ad2 {
  double a, b, r;
};

__device__ __forceinline__ void half_angle(const Ad2& d, double& c, double& s) {
  if (d.r == 0.0) {
    c = 1.0;
    s = 0.0;
    return;
  }
  // the larger of cos, sin theta and, from it, the smaller
  const double big = sqrt((d.r + fabs(d.a)) / (2.0 * d.r));
  const double small = fabs(d.b) / (2.0 * d.r * big);
  c = d.a >= 0.0 ? big : small;
  s = copysign(d.a >= 0.0 ? small : big, d.b);
}

// (x + 1/2) 2^-32, exactly: the low bits of 2^19 + u, whose last place is 2^-33,
// less 2^19 (one FP64 operation for a conversion, a sum and a product).
__device__ __forceinline__ double uniform64(uint32_t x) {
  return __dadd_rn(__hiloint2double((int)(0x41200000u | (x >> 31)), (int)(2u * x + 1u)), -0x1p19);
}

template <typename T>
__device__ __forceinline__ void pick_pair(const double* rho_ad, int ns, uint32_t word,
                                          int& al, int& be, double& m0) {
  double tot = 0.0;
  for (int k = 0; k < ns * ns; ++k) tot += fabs(rho_ad[k]);
  uint32_t Tk[kMaxNS * kMaxNS];
  uint64_t sumT = 0;
  int last = -1;
  for (int k = 0; k < ns * ns; ++k) {
    Tk[k] = (uint32_t)floor(fabs(rho_ad[k]) / tot * kP24);
    sumT += Tk[k];
    if (rho_ad[k] != 0.0) last = k;
  }
  Tk[last] += (uint32_t)(16777216ull - sumT);
  const uint32_t y = word >> 8;
  uint64_t cum = 0;
  int pick = last;
  for (int k = 0; k < ns * ns; ++k) {
    cum += Tk[k];
    if ((uint64_t)y < cum) {
      pick = k;
      break;
    }
  }
  al = pick / ns;
  be = pick % ns;
  m0 = rho_ad[pick] / ((double)Tk[pick] / kP24);
}

// Initial sample of one walker with random-stream id `traj`: (R, P) from the
// harmonic Wigner distribution (Box-Muller pair of Philox block (c0 = j,
// purpose INIT) per mode), then the index pair drawn from |rho| in the
// walkers' representation (adiabatic: U^T rho_el0 U at the walker's R;
// diabatic: rho_el0) with word 0 of block (c0 = n, purpose INIT), m0 = rho_ab /
// p_hat.  R, P written at Rg[j * stride], Pg[j * stride].
__device__ __forceinline__ void sample_walker_f64(const DevModel* __restrict__ M,
                                                  const SampleParams& sp, uint64_t traj,
                                                  double* Rg, double* Pg, int64_t stride,
                                                  double& m0, uint16_t& ab) {
  const int n = sp.n;
  double a = M->a0, b = M->b0;
  for (int j = 0; j < n; ++j) {
    double R = sp.R0[j], P = sp.P0[j];
    if (sp.wigner) {
      const u4 wd = philox_draw(sp.seed, (uint32_t)j, traj, kPurposeInit);
      const double u0 = uniform64(wd.x);
      const double u1 = uniform64(wd.y);
      const double rad = sqrt(-2.0 * log(u0));
      double sn, cs;
      sincospi(2.0 * u1, &sn, &cs);
      R += sp.sR[j] * rad * cs;
      P += sp.sP[j] * rad * sn;
    }
    Rg[(int64_t)j * stride] = R;
    Pg[(int64_t)j * stride] = P;
    a += M->a[j] * R;
    b += M->b[j] * R;
  }
  Ad2 d;
  d.a = a;
  d.b = b;
  d.r = sqrt(a * a + b * b);
  double c, s;
  half_angle(d, c, s);
  const double U[4] = {-s, c, c, s};  // U[i*2 + alpha]
  double rho_ad[4];  // the density in the walkers' representation
  for (int al = 0; al < 2; ++al)
    for (int be = 0; be < 2; ++be) {
      double acc = 0.0;
      if (M->repr == QCL_REPR_DIABATIC) {
        acc = sp.rho[al * 2 + be];
      } else {
        // (zero elements of the density, most of a pure state's, add nothing)
        for (int k = 0; k < 2; ++k)
          for (int l = 0; l < 2; ++l)
            if (sp.rho[k * 2 + l] != 0.0) acc += U[k * 2 + al] * sp.rho[k * 2 + l] * U[l * 2 + be];
      }
      rho_ad[al * 2 + be] = acc;
    }
  const u4 wd = philox_draw(sp.seed, (uint32_t)n, traj, kPurposeInit);
  int al, be;
  pick_pair<double>(rho_ad, 2, wd.x, al, be, m0);
  ab = (uint16_t)(al | (be << 8));
}

// --------------------------------------------------------------- FP64 step --
// The FP64 unit is the narrow resource here (2 lanes per clock per SM; the
// kernels below keep it 80-90 % busy), so a step is written for few FP64
// operations: per-mode constants made on the host and read as constant-bank
// operands, one reciprocal square root in place of a square root and two
// divisions, the decomposition at R_n carried from the step before, the
// spin-boson form without the terms that are zero there, thresholds and weight
// factors from integers, signs and selections in integer registers.  Every
// operation is an explicit round-to-nearest one, so that the bits do not
// depend on where the step is inlined (one launch or several, moving or
// spawning walkers).

// Per-mode and per-launch constants (kernel parameter; NC modes).
template <int NC>
struct Coef64 {
  double hk[NC], hs[NC];  // dt/2 k_j, dt/2 s_j
  double dtm[NC];         // dt / M_j
  double a[NC], b[NC];    // d a / d R_j, d b / d R_j
  double am[NC], bm[NC];  // a_j / M_j, b_j / M_j
  double a0, b0;
  double hdt;    // dt / 2
  double wph;    // dt / hbar: dt/2 (w_n + w_{n+1}) = +-wph (r_n + r_{n+1}) off the diagonal
  double cg;     // event amplitude |A_e| = |dt g|: cg Av ir^2 (spin-boson form,
                 // cg = -b0 dt/2), cg (a Bv - b Av) ir^2 (cg = dt/2), or cg b (diabatic,
                 // cg = dt / hbar)
  double kamp;   // hop_scale 2^24
  uint32_t tmax2;  // floor(floor(p_max 2^24) / 2)
  int32_t n;
};

template <int NC>
inline void make_coef64(const DevModel& h, double dt, Coef64<NC>& c) {
  for (int j = 0; j < NC; ++j) {
    const bool on = j < h.n;
    c.hk[j] = on ? 0.5 * dt * h.k[j] : 0.0;
    c.hs[j] = on ? 0.5 * dt * h.s[j] : 0.0;
    c.dtm[j] = on ? dt / h.mass[j] : 0.0;
    c.a[j] = on ? h.a[j] : 0.0;
    c.b[j] = on ? h.b[j] : 0.0;
    c.am[j] = on ? h.a[j] / h.mass[j] : 0.0;
    c.bm[j] = on ? h.b[j] / h.mass[j] : 0.0;
  }
  c.a0 = h.a0;
  c.b0 = h.b0;
  c.hdt = 0.5 * dt;
  c.wph = dt / h.hbar;
  c.cg = h.repr == QCL_REPR_DIABATIC ? dt / h.hbar : (h.kind == 0 ? -0.5 * h.b0 * dt : 0.5 * dt);
  c.kamp = h.hop_scale * kP24;
  c.tmax2 = (uint32_t)std::floor(h.p_max * kP24) >> 1;
  c.n = h.n;
}

// An integer below 2^32 as a double (bits of 2^52 + i, less 2^52).
__device__ __forceinline__ double int_double(uint32_t i) {
  return __dadd_rn(__hiloint2double(0x43300000, (int)i), -0x1p52);
}

// 1 / sqrt(x) for x in the normal range: the hardware approximation y and one
// third-order step.  With e = 1 - x y^2 the root is y (1 - e)^(-1/2), of which the
// binomial series gives y (1 + e/2 + 3/8 e^2); the first term left out is 5/16 e^3,
// below 2^-56 of y.  Within 2^-52 of the root (a test: every exponent from -500 to
// 500).
__device__ __forceinline__ double rsqrt64(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = __fma_rn(-__dmul_rn(x, y), y, 1.0);
  return __fma_rn(__fma_rn(e, 0.375, 0.5), __dmul_rn(e, y), y);
}

// The decomposition a walker carries between steps: a(R), b(R), r, 1/r^2 (0
// where the gap is degenerate, which sets the coupling to 0), cos and sin
// 2theta, and whether the gap is degenerate.
struct Dec64 {
  double a, b, r, ir2, c2, s2;
  bool deg;
};

// (r^2 below (kDegTol / 2)^2: the exact square root and quotients, theta = 0
// at r = 0.)
template <int KIND, bool DIA>
__device__ __forceinline__ void decompose64(Dec64& d) {
  d.deg = false;
  if (DIA) return;
  const double r2 = __fma_rn(d.a, d.a, __dmul_rn(d.b, d.b));
  const double ir = rsqrt64(r2);
  d.r = __dmul_rn(r2, ir);
  d.ir2 = __dmul_rn(ir, ir);
  d.c2 = __dmul_rn(d.a, ir);
  if (KIND == 1) d.s2 = __dmul_rn(d.b, ir);
  if (__double_as_longlong(r2) < __double_as_longlong(0.25 * kDegTol * kDegTol)) {
    d.deg = true;
    d.r = sqrt(r2);
    d.ir2 = 0.0;
    d.c2 = d.r > 0.0 ? d.a / d.r : 1.0;
    if (KIND == 1) d.s2 = d.r > 0.0 ? d.b / d.r : 0.0;
  }
}

// Outcome of one step's transition test: event 0 (none), 1 (first index) or
// 2 (second index); num / den, the factor the event puts on the weight (A_e /
// p_hat_e for an event, 1 / (1 - sum p_hat) for none); the event's quarter turns.
struct Step64 {
  int ev;
  double num, den;
  int dq;
};

// P += dt/2 F_ab for one mode with hu = dt/2 sab cos 2theta, hv = dt/2 sab sin
// 2theta (diabatic: hu = -dt/2 sab).  The force's terms are added up before they
// meet P, so that a kick rounds P once (one operation more than subtracting them
// one by one in the spin-boson form, and half the trajectory error against quad
// precision).
template <int KIND, bool DIA>
__device__ __forceinline__ double kick64(double hk, double hs, double a, double b, double R,
                                         double P, double hu, double hv) {
  double f = KIND == 1 ? __fma_rn(hk, R, hs) : __dmul_rn(hk, R);
  f = __fma_rn(hu, a, f);
  if (KIND == 1 && !DIA) f = __fma_rn(hv, b, f);
  return __dadd_rn(P, -f);
}

// One step n -> n+1 of one two-state walker in FP64: velocity Verlet on the
// pair's mean force (adiabatic: Hellmann-Feynman diagonal; diabatic: the
// diagonal of W), the trapezoid phase, and the transition test with the hop
// word `y` (24 bits).  R and P of NP > 0 modes in registers, or (NP = 0) at
// Rg[j * stride], Pg[j * stride] in two passes; d is the decomposition at R_n
// on entry and at R_{n+1} on return; deg reports a degenerate gap at either.
template <int NP, int NC, int KIND, bool DIA>
__device__ __forceinline__ Step64 walker_step_f64(const Coef64<NC>& c, double* R, double* P,
                                                  int64_t stride, Dec64& d, int al, int be,
                                                  double& phi, uint32_t y, bool& deg) {
  // dt/2 (sig_a + sig_b)/2 and dt/hbar (sig_a - sig_b)/2 of the pair
  const bool same = al == be;
  const double hsab = same ? (al ? c.hdt : -c.hdt) : 0.0;
  const double wab = same ? 0.0 : (al ? c.wph : -c.wph);
  const double hu = DIA ? -hsab : __dmul_rn(hsab, d.c2);
  const double hv = (KIND == 1 && !DIA) ? __dmul_rn(hsab, d.s2) : 0.0;
  const double w0 = DIA ? d.a : d.r;
  deg = d.deg;
  d.a = c.a0;
  d.b = c.b0;
  double Av = 0.0, Bv = 0.0;
  if constexpr (NP > 0) {
#pragma unroll
    for (int j = 0; j < NP; ++j)
      if (NP <= 4 || j < c.n) {
        P[j] = kick64<KIND, DIA>(c.hk[j], c.hs[j], c.a[j], c.b[j], R[j], P[j], hu, hv);
        R[j] = __fma_rn(c.dtm[j], P[j], R[j]);
        d.a = __fma_rn(c.a[j], R[j], d.a);
        if (KIND == 1) d.b = __fma_rn(c.b[j], R[j], d.b);
      }
    decompose64<KIND, DIA>(d);
    const double hu2 = DIA ? hu : __dmul_rn(hsab, d.c2);
    const double hv2 = (KIND == 1 && !DIA) ? __dmul_rn(hsab, d.s2) : 0.0;
#pragma unroll
    for (int j = 0; j < NP; ++j)
      if (NP <= 4 || j < c.n) {
        P[j] = kick64<KIND, DIA>(c.hk[j], c.hs[j], c.a[j], c.b[j], R[j], P[j], hu2, hv2);
        if (!DIA) {
          Av = __fma_rn(c.am[j], P[j], Av);
          if (KIND == 1) Bv = __fma_rn(c.bm[j], P[j], Bv);
        }
      }
  } else {
    for (int j = 0; j < c.n; ++j) {
      const int64_t o = (int64_t)j * stride;
      double x = R[o];
      double p = kick64<KIND, DIA>(c.hk[j], c.hs[j], c.a[j], c.b[j], x, P[o], hu, hv);
      x = __fma_rn(c.dtm[j], p, x);
      d.a = __fma_rn(c.a[j], x, d.a);
      if (KIND == 1) d.b = __fma_rn(c.b[j], x, d.b);
      R[o] = x;
      // (the diabatic force does not wait for the decomposition: one pass)
      P[o] = DIA ? kick64<KIND, DIA>(c.hk[j], c.hs[j], c.a[j], c.b[j], x, p, hu, hv) : p;
    }
    decompose64<KIND, DIA>(d);
    if (!DIA) {
      const double hu2 = __dmul_rn(hsab, d.c2);
      const double hv2 = KIND == 1 ? __dmul_rn(hsab, d.s2) : 0.0;
      for (int j = 0; j < c.n; ++j) {
        const int64_t o = (int64_t)j * stride;
        const double p = kick64<KIND, DIA>(c.hk[j], c.hs[j], c.a[j], c.b[j], R[o], P[o], hu2, hv2);
        Av = __fma_rn(c.am[j], p, Av);
        if (KIND == 1) Bv = __fma_rn(c.bm[j], p, Bv);
        P[o] = p;
      }
    }
  }
  deg |= d.deg;
  // phase: hbar w_ab = e_a - e_b = (sig_a - sig_b) r; diabatic V_aa - V_bb =
  // -(sig_a - sig_b) a
  phi = __fma_rn(DIA ? -wab : wab, __dadd_rn(w0, DIA ? d.a : d.r), phi);
  // both events have |A_e| = |A|: A = dt g with the coupling contracted with P/M,
  // g = (a Bv - b Av) / (2 r^2), or c = V_01 dt / hbar (diabatic)
  double A;
  if (DIA) A = __dmul_rn(c.cg, d.b);
  else if (KIND == 1) A = __dmul_rn(__dmul_rn(c.cg, __fma_rn(d.a, Bv, -__dmul_rn(d.b, Av))), d.ir2);
  else A = __dmul_rn(__dmul_rn(c.cg, Av), d.ir2);
  // p = min(kappa |A|, p_max) quantised to T = floor(p 2^24); scaling two equal
  // thresholds down to a sum of at most Tmax in exact integers gives
  // min(T, floor(Tmax / 2)) (the conversion saturates, and takes 0 for NaN)
  const uint32_t T = min(__double2uint_rz(__dmul_rn(c.kamp, fabs(A))), c.tmax2);
  Step64 o;
  o.ev = y < T ? 1 : (y < 2u * T ? 2 : 0);
  o.dq = (DIA && o.ev) ? (o.ev == 1 ? 3 : 1) : 0;  // amplitudes -i c and +i c
  const uint32_t iden = o.ev ? T : 16777216u - 2u * T;
  // A_1 = -sig_a dt g, A_2 = -sig_b dt g (index 0 is sigma = -1)
  const bool neg = !DIA && (o.ev == 1 ? al : be);
  o.num = o.ev ? (neg ? -A : A) : 1.0;
  o.den = __dmul_rn(int_double(iden), 0x1p-24);
  return o;
}

// m num / den by a division: a stay (num = 1, most steps) rounds once.  (A factor
// from a reciprocal, rounded before it meets m, rounds twice: 3 to 5 % more error
// of the weight against 128-bit trajectories.)
__device__ __forceinline__ double weight64(double m, const Step64& o) {
  return __ddiv_rn(__dmul_rn(m, o.num), o.den);
}

// Loads a walker's modes (NP > 0) and evaluates the decomposition at its R,
// with the step's operations in its order.
template <int NP, int NC, int KIND, bool DIA>
__device__ __forceinline__ void walker_load_f64(const Coef64<NC>& c, const double* Rg,
                                                const double* Pg, int64_t stride, double* R,
                                                double* P, Dec64& d) {
  d.a = c.a0;
  d.b = c.b0;
  if constexpr (NP > 0) {
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      const bool on = j < c.n;
      R[j] = on ? Rg[(int64_t)j * stride] : 0.0;
      P[j] = on ? Pg[(int64_t)j * stride] : 0.0;
    }
#pragma unroll
    for (int j = 0; j < NP; ++j)
      if (NP <= 4 || j < c.n) {
        d.a = __fma_rn(c.a[j], R[j], d.a);
        if (KIND == 1) d.b = __fma_rn(c.b[j], R[j], d.b);
      }
  } else {
    for (int j = 0; j < c.n; ++j) {
      const double x = Rg[(int64_t)j * stride];
      d.a = __fma_rn(c.a[j], x, d.a);
      if (KIND == 1) d.b = __fma_rn(c.b[j], x, d.b);
    }
  }
  decompose64<KIND, DIA>(d);
}

template <int NP>
__device__ __forceinline__ void walker_store_f64(int n, const double* R, const double* P,
                                                 double* Rg, double* Pg, int64_t stride) {
#pragma unroll
  for (int j = 0; j < NP; ++j)
    if (j < n) {
      Rg[(int64_t)j * stride] = R[j];
      Pg[(int64_t)j * stride] = P[j];
    }
}

// Not finite, by the exponent bits.
__device__ __forceinline__ bool nonfinite64(double x) {
  return (__double2hiint(x) & 0x7ff00000) == 0x7ff00000;
}

// Calls f(NP, NC, KIND, DIA as integral constants) for a model: modes in
// registers up to 16, beyond in memory.
template <typename F>
inline void dispatch_f64(const DevModel& h, F&& f) {
  auto np = [&](auto NP) {
    constexpr int np_ = decltype(NP)::value;
    std::integral_constant<int, (np_ > 0 ? np_ : kMaxN)> NC;
    const std::integral_constant<int, 0> k0{};
    const std::integral_constant<int, 1> k1{};
    if (h.repr == QCL_REPR_DIABATIC)
      h.kind == 0 ? f(NP, NC, k0, std::true_type{}) : f(NP, NC, k1, std::true_type{});
    else
      h.kind == 0 ? f(NP, NC, k0, std::false_type{}) : f(NP, NC, k1, std::false_type{});
  };
  if (h.n <= 1) np(std::integral_constant<int, 1>{});
  else if (h.n <= 2) np(std::integral_constant<int, 2>{});
  else if (h.n <= 3) np(std::integral_constant<int, 3>{});
  else if (h.n <= 4) np(std::integral_constant<int, 4>{});
  else if (h.n <= 8) np(std::integral_constant<int, 8>{});
  else if (h.n <= 16) np(std::integral_constant<int, 16>{});
  else np(std::integral_constant<int, 0>{});
}

// The 16 observable contributions of one walker and their squares (v[16..31])
// from the decomposition at its R (of the adiabatic form): z = m exp(-i phi) i^q
// at the walker's own pair in its own representation, z U_ia U_jb (U symmetric) at
// every element of the other.  The eigenvector angle by the cancellation-free
// half-angle form: the larger of cos, sin theta is sqrt((1 + |cos 2theta|) / 2).
__device__ __forceinline__ void contrib_f64(const Dec64& d, double m, double phi, uint16_t ab,
                                            bool dia, double (&v)[32]) {
  double s2 = __dmul_rn(d.b, __dmul_rn(d.r, d.ir2));
  if (d.deg) s2 = d.r > 0.0 ? d.b / d.r : 0.0;
  const double t = __fma_rn(0.5, fabs(d.c2), 0.5);
  const double rt = rsqrt64(t);
  const double big = __dmul_rn(t, rt), small = __dmul_rn(__dmul_rn(0.5, fabs(s2)), rt);
  const bool cpos = d.c2 >= 0.0;
  const double c = cpos ? big : small;
  const double s = copysign(cpos ? small : big, s2);
  const int al = ab & 0xf, be = (ab >> 8) & 0xf, q = (ab >> 4) & 3;
  double sn, cs;
  sincos(phi, &sn, &cs);
  const double xr = __dmul_rn(m, cs), xi = -__dmul_rn(m, sn);
  const double zr = q == 0 ? xr : (q == 1 ? -xi : (q == 2 ? -xr : xi));
  const double zi = q == 0 ? xi : (q == 1 ? xr : (q == 2 ? -xi : -xr));
  const double r2 = __dmul_rn(zr, zr), i2 = __dmul_rn(zi, zi);
  const double ua[2] = {al ? c : -s, al ? s : c}, ub[2] = {be ? c : -s, be ? s : c};
  const int k0 = al * 2 + be;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double f = __dmul_rn(ua[k >> 1], ub[k & 1]);
    const double fr = __dmul_rn(zr, f), fi = __dmul_rn(zi, f);
    const double fr2 = __dmul_rn(fr, fr), fi2 = __dmul_rn(fi, fi);
    const bool hit = k == k0;
    const double hr = hit ? zr : 0.0, hi = hit ? zi : 0.0;
    const double hr2 = hit ? r2 : 0.0, hi2 = hit ? i2 : 0.0;
    // (the diabatic block first, the adiabatic one after it)
    v[2 * k] = dia ? hr : fr;
    v[2 * k + 1] = dia ? hi : fi;
    v[8 + 2 * k] = dia ? fr : hr;
    v[8 + 2 * k + 1] = dia ? fi : hi;
    v[16 + 2 * k] = dia ? hr2 : fr2;
    v[16 + 2 * k + 1] = dia ? hi2 : fi2;
    v[24 + 2 * k] = dia ? fr2 : hr2;
    v[24 + 2 * k + 1] = dia ? fi2 : hi2;
  }
}

}  // namespace qcl
