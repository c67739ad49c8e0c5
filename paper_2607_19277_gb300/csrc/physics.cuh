// Device physics traits for the finite-volume stage kernel (sm_103a).
//
// Each trait gives the conserved <-> primitive maps, the physical flux along one axis and
// the approximate Riemann flux at a face, evaluated per cell in registers (the paper's
// cell-local physics routines, Section 2.3):
//   HdPhys   : Eqs. 2-4 with e = p/(gamma-1) + rho v^2/2 (Eq. 6; Section 2.3.1; HD flux listing)
//   MhdPhys  : Eqs. 11-13 with GLM (Eq. 14), e = p/(gamma-1) + rho v^2/2 + B^2/2 (Section 2.3.3)
//   SrhdPhys : Eqs. 15-20 with the ideal-gas enthalpy of Eq. 21 (Section 2.3.4), and
//   SrhdSyngePhys with the approximate Synge-gas enthalpy (Eq. 22, Mathews' form); the
//              conserved-to-primitive recovery is a Newton root find in xi = Gamma^2 rho h,
//              in FP64, or (FP32 stencil, where its guards hold) finished in FP32 pairs.
// Riemann fluxes: HLL with Davis wave-speed estimates, or TVDLF (Rusanov) with the larger
// of the two sides' fastest speeds (paper Table 1 lists the solvers per module).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

namespace agile {

enum : int { LIM_MINMOD = 0, LIM_VANLEER = 1 };
enum : int { FLUX_TVDLF = 0, FLUX_HLL = 1, FLUX_HLLC = 2 };
enum : int { ST_ENOCONV = 1, ST_EUNPHYS = 2 };

// Equation parameters in the stencil precision R, formed on the host for a launch (the cleaning
// speed's per solve in the kernel; the FP64 copy of gamma serves the SRHD primitive recovery in FP64).
template <typename R>
struct PhysParamsT {
  double gamma_d, gm_d;    // gamma and (gamma - 1) / gamma in FP64 (SRHD primitive recovery)
  R gamma, g1, ig1, gg1;   // gamma, gamma - 1, 1 / (gamma - 1), gamma / (gamma - 1)
  R gmr;                   // (gamma - 1) / gamma in the stencil precision
  R gml;                   // its remainder: gmr + gml holds it to twice the precision (FP32 pairs)
  R ch, ich, ch2;          // GLM cleaning speed c_h = c_max of U^n (MHD), 1 / c_h, c_h^2
  __host__ __device__ void set(double gamma_, double ch_) {
    gamma_d = gamma_;
    gm_d = (gamma_ - 1.0) / gamma_;
    gamma = R(gamma_);
    g1 = R(gamma_ - 1.0);
    ig1 = R(1.0 / (gamma_ - 1.0));
    gg1 = R(gamma_ / (gamma_ - 1.0));
    gmr = R(gm_d);
    gml = R(gm_d - (double)gmr);
    set_ch(ch_);
  }
  __host__ __device__ void set_ch(double ch_) {
    ch = R(ch_);
    ich = ch_ > 0.0 ? R(1.0 / ch_) : R(0);
    ch2 = R(ch_ * ch_);
  }
};

__device__ __forceinline__ float rabs(float a) { return fabsf(a); }
__device__ __forceinline__ double rabs(double a) { return fabs(a); }
__device__ __forceinline__ float rmin(float a, float b) { return fminf(a, b); }
// FP64 comparisons, minima and maxima run on the bit patterns: GB300 has two FP64 lanes per SM,
// so one FP64 instruction, a comparison included, costs the issue slots of some 60 integer ones,
// of which the FP64 stencil leaves nine tenths idle. Same results as fmin / fmax / ">": of one
// NaN and a number the number, of two zeros -0 as the smaller. bits_key orders every value.
__device__ __forceinline__ long long bits_key(double a) {
  const long long i = __double_as_longlong(a);
  return i ^ ((i >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ bool bits_nan(double a) {
  return (__double_as_longlong(a) & 0x7fffffffffffffffLL) > 0x7ff0000000000000LL;
}
__device__ __forceinline__ bool rpos(float a) { return a > 0.0f; }
__device__ __forceinline__ bool rpos(double a) {   // a > 0
  return (unsigned long long)(__double_as_longlong(a) - 1) < 0x7ff0000000000000ULL;
}
__device__ __forceinline__ bool rneg(float a) { return !(a >= 0.0f); }
__device__ __forceinline__ bool rneg(double a) {   // not a >= 0: below zero, or a NaN
  const long long i = __double_as_longlong(a);
  return i < 0 ? (unsigned long long)i != 0x8000000000000000ULL : bits_nan(a);
}
__device__ __forceinline__ double rmin(double a, double b) {
  return bits_nan(a) || (bits_key(b) < bits_key(a) && !bits_nan(b)) ? b : a;
}
__device__ __forceinline__ float rmax(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ double rmax(double a, double b) {
  return bits_nan(a) || (bits_key(b) > bits_key(a) && !bits_nan(b)) ? b : a;
}
__device__ __forceinline__ float rsqrt_(float a) { return sqrtf(a); }
// FP64 square root: the hardware estimate y of a^-1/2 (PTX rsqrt.approx.ftz.f64), s = a y, and
// with e = 1 - s y the series s / sqrt(1 - e) = s + s e (1/2 + 3/8 e + ...), in which s e is formed
// as r y from the residual r = a - s^2: r is exact to a rounding of its own, so the rounding of s
// drops out and the last addition's is what remains. On 3 M arguments from 2^-450 to 2^450 at most
// 0.515 ulp off (the estimate is good to 9e-7, the terms left out are below 0.02 ulp), rms 0.289 as
// the correctly rounded root, 0.09% not the nearest; 6 FP64 operations (the library's root takes
// about twice as many; with s e from the rounded s, 5 operations, 0.76 ulp and rms 0.323, and stage
// launches of HD 210 blocks 790 us instead of 802, MHD 512 blocks 4127 and 4247, SRHD 512 blocks 3252
// and 3325, with the same in rsqrt_div and the range of the MHD face speed unchecked). Arguments
// below 2^-959, where r would lose bits, negative and non-finite ones take the library's.
constexpr unsigned ROOT64_LO = (1023u - 959u) << 20;    // high word of 2^-959
__device__ __forceinline__ bool root64_range(double a) {
  return (unsigned)__double2hiint(a) - ROOT64_LO < 0x7ff00000u - ROOT64_LO;
}
__device__ __forceinline__ double sqrt64(double a) {
  if (!root64_range(a)) return sqrt(a);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
  const double s = a * y;
  const double e = fma(-s, y, 1.0), r = fma(-s, s, a);
  return fma(r * y, fma(e, 0.375, 0.5), s);
}
__device__ __forceinline__ double rsqrt_(double a) { return sqrt64(a); }
__device__ __forceinline__ double rcp64(double s);
// sqrt(a / b) of positive a, b. FP64: with the estimate y of (a b)^-1/2 and s = a y, w = b s is
// sqrt(a b) and r = a - w s the residual of s^2 = a / b; the same series with e = 1 - w y. Only the
// rounding of w (halved) and the last one remain: at most 0.98 ulp off on the same arguments, rms
// 0.328, in 8 FP64 operations. (The reciprocal, the product and the root take 10; with the library's
// root they are 1.2 ulp and rms 0.364 off; e from a b y^2 takes 7, 1.8 ulp and rms 0.463.) Outside
// the range of normal products, or of arguments whose residual keeps its bits, the quotient's root.
__device__ __forceinline__ float rsqrt_div(float a, float b) { return sqrtf(a / b); }
__device__ __forceinline__ double rsqrt_div(double a, double b) {
  const double q = a * b;
  if ((unsigned)__double2hiint(q) - 0x00100000u >= 0x7fe00000u || !root64_range(a)) return sqrt64(a * rcp64(b));
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(q));
  const double s = a * y, w = b * s;
  const double e = fma(-w, y, 1.0), r = fma(-w, s, a);
  return fma(r * y, fma(e, 0.375, 0.5), s);
}
__device__ __forceinline__ float rsign(float a) { return copysignf(1.0f, a); }
// Reciprocal and quotient in the stencil precision. FP32: the build's fast single-precision
// divide. FP64: the hardware reciprocal estimate (PTX rcp.approx.ftz.f64) refined by one
// third-order Newton-Raphson step: with e = 1 - s r0, r1 = r0 (1 + e + e^2) is the series of
// r0 / (s r0) = r0 / (1 - e) truncated after e^2, so its relative error is e^3, far below
// 2^-53 for the estimate's error. The product a r1 lies within 1 ulp of the rounded quotient
// a / s (4 FP64 operations against about twice as many for the IEEE divide, which the FP64
// units of this GPU make the costly part of the stencil). Valid for normal, finite s with
// |s| < 2^1022; every divisor below is a density, a sum of two same-sign slopes, a signal-
// speed interval or a Newton derivative (a zero or non-finite one yields NaN, as the IEEE
// quotient's use would).
__device__ __forceinline__ double rcp64(double s) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(s));
  const double e = fma(-s, r, 1.0);
  return fma(r, fma(e, e, e), r);
}
__device__ __forceinline__ float rrcp(float s) { return 1.0f / s; }
__device__ __forceinline__ double rrcp(double s) { return rcp64(s); }
__device__ __forceinline__ float rdiv(float a, float s) { return a / s; }
__device__ __forceinline__ double rdiv(double a, double s) { return a * rcp64(s); }
template <typename R> __device__ __forceinline__ R rtiny();
template <> __device__ __forceinline__ float rtiny<float>() { return 1e-30f; }
template <> __device__ __forceinline__ double rtiny<double>() { return 1e-300; }

// Half of the limited slope, sigma / 2, from the two one-sided differences a and b, written
// without branches (the final choice is a select):
//   minmod: sigma = (sgn a + sgn b)/2 min(|a|, |b|)  (0 unless a and b share a sign);
//   van Leer (1974): sigma = 2ab / (a + b) when ab > 0, else 0. The quotient is formed for
//   every input and discarded when ab <= 0, where a + b may vanish.
// Halving is exact, so sigma / 2 equals half the limiter value bit for bit.
template <typename R, int LIM>
__device__ __forceinline__ R half_slope(R a, R b) {
  if (LIM == LIM_MINMOD) {
    if constexpr (sizeof(R) == 8) {
      // (sgn a + sgn b)/4 is +-1/2 or 0, and |a|, |b| order like their bit patterns (a NaN
      // above every number): one FP64 operation
      const long long ia = __double_as_longlong(a), ib = __double_as_longlong(b);
      const long long ma = ia & 0x7fffffffffffffffLL, mb = ib & 0x7fffffffffffffffLL;
      const long long sg = (ia ^ ib) < 0 ? 0 : 0x3fe0000000000000LL | (ia & (long long)0x8000000000000000ULL);
      return __longlong_as_double(sg) * __longlong_as_double(ma < mb ? ma : mb);
    } else {
      return (R(0.25) * (rsign(a) + rsign(b))) * rmin(rabs(a), rabs(b));
    }
  } else {
    const R ab = a * b;
    const R q = ab * rrcp(a + b);
    return rpos(ab) ? q : R(0);
  }
}

// ------------------------------------------------------------------------------ hydro
template <typename R>
struct HdPhys {
  static constexpr int NV = 5;   // rho, m, e
  static constexpr int NA = 0;
  static constexpr int BOFF = -1;  // no magnetic field
  static constexpr int IV = 1;     // first velocity / momentum component
  static constexpr int NREC = NV;  // reconstructed variables
  static constexpr int FROZEN = NV;  // variables from this index on are never updated
  static constexpr int QV = -1;      // a variable with no face flux (source-only), or -1
  static constexpr int IE = 4;     // energy in U, pressure in P
  static constexpr bool SOURCE = false;
  static constexpr bool GLM = false;

  __device__ static __forceinline__ void cons2prim(const R* u, R* p, R*, const PhysParamsT<R>& pp,
                                                   int& st) {
    const R g1 = pp.g1;
    const R rho = u[0];
    const R ir = rrcp(rho);
    const R vx = u[1] * ir, vy = u[2] * ir, vz = u[3] * ir;
    p[0] = rho;
    p[1] = vx;
    p[2] = vy;
    p[3] = vz;
    p[4] = g1 * (u[4] - R(0.5) * (u[1] * vx + u[2] * vy + u[3] * vz));
    st |= (!rpos(rho) | !rpos(p[4])) ? ST_EUNPHYS : 0;
  }

  __device__ static __forceinline__ void prim2cons(const R* p, R* u, const PhysParamsT<R>& pp) {
    const R ig1 = pp.ig1;
    u[0] = p[0];
    u[1] = p[0] * p[1];
    u[2] = p[0] * p[2];
    u[3] = p[0] * p[3];
    u[4] = p[4] * ig1 + R(0.5) * p[0] * (p[1] * p[1] + p[2] * p[2] + p[3] * p[3]);
  }

  // Conserved state, flux along D and the interval mid -+ half of the speeds of a face state.
  template <int D>
  __device__ static __forceinline__ void side(const R* p, R* u, R* f, R& mid, R& half, const PhysParamsT<R>& pp) {
    const R vd = p[1 + D];
    u[0] = p[0];
    u[1] = p[0] * p[1];
    u[2] = p[0] * p[2];
    u[3] = p[0] * p[3];
    u[4] = p[4] * pp.ig1 + R(0.5) * (u[1] * p[1] + u[2] * p[2] + u[3] * p[3]);
    f[0] = u[1 + D];
    f[1] = u[1] * vd;
    f[2] = u[2] * vd;
    f[3] = u[3] * vd;
    f[1 + D] = u[1 + D] * vd + p[4];
    f[4] = vd * (u[4] + p[4]);
    waves<D>(p, mid, half, pp);
  }

  template <int D>
  __device__ static __forceinline__ void waves(const R* p, R& mid, R& half, const PhysParamsT<R>& pp) {
    mid = p[1 + D];
    half = rsqrt_div(pp.gamma * p[4], p[0]);
  }

  template <int D>
  __device__ static __forceinline__ void interface(R*, R*, const PhysParamsT<R>&) {}
};

// ------------------------------------------------------------------------------ MHD + GLM
template <typename R>
struct MhdPhys {
  static constexpr int NV = 9;   // rho, m, e, B, psi
  static constexpr int NA = 0;
  static constexpr int BOFF = 5;   // B_x is variable 5
  static constexpr int IV = 1;
  static constexpr int NREC = NV;
  static constexpr int FROZEN = NV;
  static constexpr int QV = -1;
  static constexpr int IE = 4;
  static constexpr bool SOURCE = false;
  static constexpr bool GLM = true;

  __device__ static __forceinline__ void cons2prim(const R* u, R* p, R*, const PhysParamsT<R>& pp,
                                                   int& st) {
    const R g1 = pp.g1;
    const R rho = u[0];
    const R ir = rrcp(rho);
    const R vx = u[1] * ir, vy = u[2] * ir, vz = u[3] * ir;
    const R b2 = u[5] * u[5] + u[6] * u[6] + u[7] * u[7];
    p[0] = rho;
    p[1] = vx;
    p[2] = vy;
    p[3] = vz;
    if constexpr (sizeof(R) == 8) p[4] = g1 * (u[4] - R(0.5) * ((u[1] * vx + u[2] * vy + u[3] * vz) + b2));
    else p[4] = g1 * (u[4] - R(0.5) * rho * (vx * vx + vy * vy + vz * vz) - R(0.5) * b2);
    p[5] = u[5];
    p[6] = u[6];
    p[7] = u[7];
    p[8] = u[8];
    st |= (!rpos(rho) | !rpos(p[4])) ? ST_EUNPHYS : 0;
  }

  __device__ static __forceinline__ void prim2cons(const R* p, R* u, const PhysParamsT<R>& pp) {
    const R ig1 = pp.ig1;
    u[0] = p[0];
    u[1] = p[0] * p[1];
    u[2] = p[0] * p[2];
    u[3] = p[0] * p[3];
    u[4] = p[4] * ig1 + R(0.5) * p[0] * (p[1] * p[1] + p[2] * p[2] + p[3] * p[3]) +
           R(0.5) * (p[5] * p[5] + p[6] * p[6] + p[7] * p[7]);
    u[5] = p[5];
    u[6] = p[6];
    u[7] = p[7];
    u[8] = p[8];
  }

  // Conserved state, flux along D (without those of B_d and psi, which riemann sets from the
  // face values) and the interval of the speeds of a face state. FP64: the fast speed from
  // S = gamma p + B^2, cf^2 = (S + sqrt(S^2 - 4 gamma p B_d^2)) / (2 rho), which divides by the
  // density once, for S from 2^-480 (S^2 keeps its bits below its terms down to there) to below
  // 2^511 (S^2 does not overflow; the subtrahend is at most S^2); elsewhere, and in FP32, from
  // quantities divided by the density (waves), whose squares are near a^4.
  template <int D>
  __device__ static __forceinline__ void side(const R* p, R* u, R* f, R& mid, R& half, const PhysParamsT<R>& pp) {
    const R vd = p[1 + D], bd = p[5 + D];
    const R b2 = p[5] * p[5] + p[6] * p[6] + p[7] * p[7];
    const R vb = p[1] * p[5] + p[2] * p[6] + p[3] * p[7];
    const R ptot = p[4] + R(0.5) * b2;
    u[0] = p[0];
    u[1] = p[0] * p[1];
    u[2] = p[0] * p[2];
    u[3] = p[0] * p[3];
    u[4] = p[4] * pp.ig1 + R(0.5) * ((u[1] * p[1] + u[2] * p[2] + u[3] * p[3]) + b2);
    u[5] = p[5];
    u[6] = p[6];
    u[7] = p[7];
    u[8] = p[8];
    f[0] = u[1 + D];
    f[1] = u[1] * vd - p[5] * bd;
    f[2] = u[2] * vd - p[6] * bd;
    f[3] = u[3] * vd - p[7] * bd;
    f[1 + D] += ptot;
    f[4] = vd * (u[4] + ptot) - bd * vb;
    f[5] = vd * p[5] - bd * p[1];
    f[6] = vd * p[6] - bd * p[2];
    f[7] = vd * p[7] - bd * p[3];
    f[5 + D] = R(0);
    f[8] = R(0);
    if constexpr (sizeof(R) == 8) {
      constexpr unsigned LO = (1023u - 480u) << 20, HI = (1023u + 511u) << 20;   // high words
      const R gp = pp.gamma * p[4];
      const R s = gp + b2;
      if ((unsigned)__double2hiint(s) - LO >= HI - LO) {   // a negative or non-finite S as well
        waves<D>(p, mid, half, pp);
        return;
      }
      const R disc = rmax(s * s - (R(4) * gp) * (bd * bd), R(0));
      mid = vd;
      half = rsqrt_div(R(0.5) * (s + rsqrt_(disc)), p[0]);
    } else {
      waves<D>(p, mid, half, pp);
    }
  }

  template <int D>
  __device__ static __forceinline__ void waves(const R* p, R& mid, R& half, const PhysParamsT<R>& pp) {
    const R ir = rrcp(p[0]);
    const R a2 = pp.gamma * p[4] * ir;
    const R b2 = (p[5] * p[5] + p[6] * p[6] + p[7] * p[7]) * ir;
    const R bd2 = p[5 + D] * p[5 + D] * ir;
    const R s = a2 + b2;
    const R disc = rmax(s * s - R(4) * a2 * bd2, R(0));
    mid = p[1 + D];
    half = rsqrt_(R(0.5) * (s + rsqrt_(disc)));
  }

  // Exact solution of the linear (B_d, psi) subsystem at the face (Dedner et al. 2002):
  // both face states carry B_d* and psi*, so the face flux of B_d is psi* and of psi is
  // c_h^2 B_d*.
  template <int D>
  __device__ static __forceinline__ void interface(R* pl, R* pr, const PhysParamsT<R>& pp) {
    const R ch = pp.ch;
    const R bl = pl[5 + D], br = pr[5 + D], sl = pl[8], sr = pr[8];
    const R bs = R(0.5) * (bl + br) - R(0.5) * (sr - sl) * pp.ich;
    const R ss = R(0.5) * (sl + sr) - R(0.5) * ch * (br - bl);
    pl[5 + D] = bs;
    pr[5 + D] = bs;
    pl[8] = ss;
    pr[8] = ss;
  }
};

// Ideal MHD with uniform resistivity eta (Section 2.3.3: -curl(eta J) in the induction
// equation, div(B x eta J) in the energy equation): the MHD trait with the RES flag, for
// which the stage kernel adds eta lap B to the induction equation and eta (J.J + B.lap B)
// to the energy equation, from the stage state with the compact stencil over the six face
// neighbours (central differences for J = curl B, the 7-point Laplacian).
template <typename R>
struct MhdResPhys : MhdPhys<R> {
  static constexpr bool RES = true;
};

// Whether a trait carries the resistive terms.
template <class P, class = void>
struct res_of {
  static constexpr bool value = false;
};
template <class P>
struct res_of<P, std::void_t<decltype(P::RES)>> {
  static constexpr bool value = P::RES;
};

// Whether a trait's primitive recovery is costly enough (an iteration) to be done once per
// cell in a pass of its own before the stage kernel, which then reads primitives: the stage
// kernel would otherwise recover each stored cell 1.75 times (own z-halo planes, x/y halo
// cells of the neighbours).
template <class P, class = void>
struct prim_pass_of {
  static constexpr bool value = false;
};
template <class P>
struct prim_pass_of<P, std::void_t<decltype(P::PRIM_PASS)>> {
  static constexpr bool value = P::PRIM_PASS;
};

// ------------------------------------------------------------------------------ FP32 pairs
// A value as an unevaluated sum h + l of two FP32 numbers, |l| <= ulp(h): about 46 significant
// bits (Dekker 1971, "A floating-point technique for extending the available precision"; the
// error of a product by one fused multiply-add). Every operation is rounded on its own
// (intrinsics, so that the compiler contracts nothing).
struct ff {
  float h, l;
};
__device__ __forceinline__ ff ff_renorm(float h, float l) {      // |l| well below |h|
  const float s = __fadd_rn(h, l);
  return {s, __fsub_rn(l, __fsub_rn(s, h))};
}
__device__ __forceinline__ ff ff_sum(float a, float b) {         // a + b exactly
  const float s = __fadd_rn(a, b);
  const float t = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ ff ff_prod(float a, float b) {        // a b exactly
  const float p = __fmul_rn(a, b);
  return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ ff ff_mul(ff a, float b) {
  const ff p = ff_prod(a.h, b);
  return ff_renorm(p.h, __fmaf_rn(a.l, b, p.l));
}
__device__ __forceinline__ ff ff_mul(ff a, ff b) {
  const ff p = ff_prod(a.h, b.h);
  return ff_renorm(p.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, p.l)));
}
__device__ __forceinline__ ff ff_sub(ff a, ff b) {
  const ff s = ff_sum(a.h, -b.h);
  return ff_renorm(s.h, __fadd_rn(s.l, __fsub_rn(a.l, b.l)));
}
__device__ __forceinline__ ff ff_rcp(float x) {                  // 1 / x, one Newton step
  const float r = 1.0f / x;
  return {r, __fmul_rn(r, __fmaf_rn(-x, r, 1.0f))};
}
// Square root of a, y an FP32 estimate of a^-1/2: the FP32 root s and its residual.
__device__ __forceinline__ ff ff_sqrt(ff a, float y) {
  const float s = __fmul_rn(a.h, y);
  const ff q = ff_prod(s, s);
  const float d = __fadd_rn(__fsub_rn(__fsub_rn(a.h, q.h), q.l), a.l);
  return ff_renorm(s, __fmul_rn(d, __fmul_rn(0.5f, y)));
}

// ------------------------------------------------------------------------------ SRHD
enum : int { EOS_IDEAL = 0, EOS_SYNGE = 1 };

// Closure h(rho, p) of Section 2.3.4: the ideal gas h = 1 + gamma/(gamma-1) theta (Eq. 21)
// or the Synge gas (Eq. 22) in Mathews' approximation h = 5/2 theta + sqrt(9/4 theta^2 + 1),
// theta = p / rho, which tends to the ideal gas with gamma = 5/3 (cold) and 4/3 (hot).
template <typename R, int EOS>
struct SrhdEos {
  __device__ static __forceinline__ R enthalpy(R theta, const PhysParamsT<R>& pp) {
    if constexpr (EOS == EOS_SYNGE) return R(2.5) * theta + rsqrt_(R(2.25) * theta * theta + R(1));
    else return R(1) + pp.gg1 * theta;
  }
  // squared sound speed: gamma theta / h, or theta (5h - 8 theta) / (3h (h - theta)) for the
  // approximate Synge gas (the isentropic derivative of its enthalpy)
  __device__ static __forceinline__ R sound_speed2(R theta, R h, const PhysParamsT<R>& pp) {
    if constexpr (EOS == EOS_SYNGE) return rdiv(theta * (R(5) * h - R(8) * theta), R(3) * h * (h - theta));
    else return rdiv(pp.gamma * theta, h);
  }
};

template <typename R, int EOS>
struct SrhdPhysE {
  static constexpr int NV = 5;   // D, m, tau ; primitives rho, u = Gamma v, p
  static constexpr int NA = 2;   // xi = Gamma^2 rho h, Gamma
  static constexpr bool PRIM_PASS = true;   // the Newton recovery runs once per cell
  static constexpr int BOFF = -1;
  static constexpr int IV = 1;
  static constexpr int NREC = NV;
  static constexpr int FROZEN = NV;
  static constexpr int QV = -1;
  static constexpr int IE = 4;
  static constexpr bool SOURCE = false;
  static constexpr bool GLM = false;
  using Eos = SrhdEos<R, EOS>;

  // FP32 start x of the iteration from the stored xi, in the bracket [E, k E] formed in FP32 from the
  // FP32 inputs, and their m^2.
  __device__ static __forceinline__ void bracket(const float* u, float xi, const PhysParamsT<float>& pp, float& x,
                                                 float& lo, float& hi, float& s2) {
    lo = u[4] + u[0];
    hi = (EOS == EOS_SYNGE ? 4.0f / 3.0f : pp.gamma) * lo;
    x = xi > lo && xi < hi ? xi : 0.5f * (lo + hi);
    s2 = u[1] * u[1] + u[2] * u[2] + u[3] * u[3];
  }

  // The same Newton iteration in FP32, to |dxi| <= 1e-6 xi (at most 12 steps): in the FP32
  // stencil it moves the starting point close to the root, so that one more step in higher
  // precision (finish_pairs, or the FP64 iteration) reaches it.
  // Leaves x at the start when it does not converge; returns whether it did.
  __device__ static __forceinline__ bool seed_f32(float& x, float df_, float s2f, float ef, float l, float h,
                                                  const PhysParamsT<R>& pp) {
    const float gmf = (float)pp.gmr;
    const float idf = EOS == EOS_SYNGE ? 1.0f / df_ : 0.0f;
    const float x0 = x;
    for (int it = 0; it < 12; ++it) {
      const float ixi = 1.0f / x;
      const float w = s2f * ixi * ixi;
      const float ig2 = 1.0f - w;
      const float lor = rsqrtf(ig2);
      const float rho = df_ * (ig2 * lor);
      const float drho = df_ * lor * w * ixi;
      float pr, dp;
      if constexpr (EOS == EOS_SYNGE) {
        const float hh = x * (ig2 * lor) * idf;
        const float q = 9.0f * hh * hh + 16.0f;
        const float iq = rsqrtf(q);
        const float th = 0.125f * (5.0f * hh - q * iq);
        pr = rho * th;
        dp = th * drho + 0.125f * (5.0f - 9.0f * hh * iq);
      } else {
        pr = gmf * (x * ig2 - rho);
        dp = gmf * (1.0f + w - drho);
      }
      const float f = x - pr - ef;
      if (f < 0.0f) l = x; else h = x;
      float xn = x - f / (1.0f - dp);
      if (!(xn >= l && xn <= h)) xn = 0.5f * (l + h);
      const bool conv = fabsf(xn - x) <= 1e-6f * xn;
      x = xn;
      if (conv) return true;
    }
    x = x0;
    return false;
  }

  // The last Newton step and the primitives in FP32 pairs instead of FP64 (FP32 stencil): from
  // the converged FP32 start x the step dx = -f(x) / f'(x), f evaluated in pairs from the FP32
  // inputs (which are exact), and the first-order update of every quantity by dx, the formulas
  // of the FP64 iteration below. GB300 runs FP64 at 1/64 of the FP32 rate, and these about 45
  // FP64 operations are some 150 FP32 ones here. Pairs have 46 bits instead of 53: absolute errors
  // of a few 2^-46 of xi (of 1 in v^2); the guards keep what the subtractions 1 - v^2 and
  // xi / Gamma^2 - rho amplify of them below 2^-29 of the result, 1/32 of the FP32 rounding of the
  // outputs: Gamma^2 <= 2^13 and p >= 2^-14 xi, xi within 2^+-36 (no product's error is flushed to
  // zero). Returns false, with nothing written, outside them or when the step is not below 1e-6 xi
  // or leaves the bracket: the FP64 iteration takes the cell then. The first-order update leaves
  // out terms of some Gamma^4 (dxi / xi)^2, in FP64 and in pairs alike: at Gamma above 20 these, not
  // the arithmetic, are the largest errors (up to 113 units of 2^-24 in Gamma on 400,000 states to
  // Gamma = 88). Against the root in extended precision (400,000 random states per range, Gamma to
  // 60, p/rho from 1e-4 to 100, starts a few FP32 roundings off) the largest and the rms errors of
  // rho, u and p equal those of the FP64 step to three digits (rms 0.289 ulp at Gamma < 10).
  // Recovery pass over 1466 blocks: 883 -> 96 us.
  __device__ static __forceinline__ bool finish_pairs(const float* u, float x, float lo, float hi, float* p,
                                                      float* aux, const PhysParamsT<float>& pp) {
    const float D = u[0];
    const ff E = ff_sum(u[4], D);
    const ff mx = ff_prod(u[1], u[1]), my = ff_prod(u[2], u[2]), mz = ff_prod(u[3], u[3]);
    const ff sxy = ff_sum(mx.h, my.h), sxyz = ff_sum(sxy.h, mz.h);
    const ff s2 = ff_renorm(sxyz.h, __fadd_rn(__fadd_rn(sxy.l, sxyz.l), __fadd_rn(__fadd_rn(mx.l, my.l), mz.l)));
    const ff ixi = ff_rcp(x);
    const ff w = ff_mul(s2, ff_mul(ixi, ixi));                  // v^2
    const ff ig2 = ff_sub({1.0f, 0.0f}, w);                     // 1 / Gamma^2
    const float y = rsqrtf(ig2.h);
    const ff ig = ff_sqrt(ig2, y);                              // 1 / Gamma
    // Gamma = y + y (1 - y / Gamma), y the FP32 estimate
    const float lorl = __fmul_rn(y, __fmaf_rn(-y, ig.l, __fmaf_rn(-y, ig.h, 1.0f)));
    const ff rho = ff_mul(ig, D);
    const float drho = D * y * w.h * ixi.h;
    ff pr;
    float dp;
    if constexpr (EOS == EOS_SYNGE) {
      const ff hh = ff_mul(ff_mul(ig, x), ff_rcp(D));
      const ff h9 = ff_mul(ff_mul(hh, hh), 9.0f);
      const ff q0 = ff_sum(h9.h, 16.0f);
      const ff q = ff_renorm(q0.h, __fadd_rn(q0.l, h9.l));
      const float iq = rsqrtf(q.h);
      const ff d = ff_sub(ff_mul(hh, 5.0f), ff_sqrt(q, iq));
      const ff th = {0.125f * d.h, 0.125f * d.l};
      pr = ff_mul(rho, th);
      dp = th.h * drho + 0.125f * (5.0f - 9.0f * hh.h * iq);
    } else {
      const ff d = ff_sub(ff_mul(ig2, x), rho);
      const ff g = {pp.gmr, pp.gml};
      pr = ff_mul(d, g);
      dp = pp.gmr * (1.0f + w.h - drho);
    }
    const ff f1 = ff_sum(x, -E.h), f2 = ff_sum(f1.h, -pr.h);
    const float f = __fadd_rn(f2.h, __fadd_rn(__fadd_rn(f2.l, f1.l), -__fadd_rn(E.l, pr.l)));
    const float dx = -f / (1.0f - dp);
    const float xn = x + dx;
    const float pn = pr.h + fmaf(dp, dx, pr.l);
    const float rn = rho.h + fmaf(drho, dx, rho.l);
    const bool ok = (fabsf(dx) <= 1e-6f * x) & (x > 1.5e-11f) & (x < 6.8e10f) & (xn > lo) & (xn < hi) &
                    (ig2.h >= 1.220703125e-4f) & (pn >= 6.103515625e-5f * x) & (rn > 1e-30f);
    if (!ok) return false;
    const float dl = -(y * y * y) * (w.h * ixi.h) * dx;         // change of Gamma
    const ff sc = ff_prod(y, ixi.h);                            // Gamma / xi and its first-order parts
    const float scl = fmaf(dl, ixi.h, fmaf(-sc.h, ixi.h * dx, fmaf(y, ixi.l, fmaf(lorl, ixi.h, sc.l))));
    const float scr = sc.h + scl;
    p[0] = rn;
    p[1] = u[1] * scr;
    p[2] = u[2] * scr;
    p[3] = u[3] * scr;
    p[4] = pn;
    aux[0] = xn;
    aux[1] = y + (lorl + dl);
    return true;
  }

  // Newton root find for f(xi) = xi - p(xi) - (tau + D) = 0 inside the bracket [E, k E]
  // (k = gamma for the ideal gas, whose p <= (gamma-1)/gamma xi; k = 4/3 for the approximate
  // Synge gas, whose h >= 4 theta gives p <= xi/4); starts from the stored xi when it lies
  // strictly inside the bracket, else from the midpoint (in the FP32 stencil first refined by
  // seed_f32); a step leaving the closed bracket is replaced by bisection; stops when
  // |dxi| <= tol xi (below); at most 50 iterations. FP64.
  __device__ static __forceinline__ void cons2prim(const R* u, R* p, R* aux, const PhysParamsT<R>& pp,
                                                   int& st) {
    float xf = 0.0f;
    if constexpr (sizeof(R) == 4) {
      float ef, hif, s2f;
      bracket(u, aux[0], pp, xf, ef, hif, s2f);
      if (seed_f32(xf, u[0], s2f, ef, ef, hif, pp) && finish_pairs(u, xf, ef, hif, p, aux, pp)) return;
    }
    const double g = pp.gamma_d;
    const double gm = pp.gm_d;
    const double D = (double)u[0];
    const double mx = (double)u[1], my = (double)u[2], mz = (double)u[3];
    const double s2 = mx * mx + my * my + mz * mz;
    const double E = (double)u[4] + D;
    double lo = E, hi = (EOS == EOS_SYNGE ? 4.0 / 3.0 : g) * E;
    const double iD = EOS == EOS_SYNGE ? rcp64(D) : 0.0;
    double xi;
    if constexpr (sizeof(R) == 4) {
      xi = (double)xf;     // lands in the FP64 bracket or the FP64 midpoint is taken
    } else {
      xi = (double)aux[0];
    }
    if (!(xi > lo && xi < hi)) xi = 0.5 * (lo + hi);
    // FP64 stencil: |dxi| <= 1e-14 xi. FP32 stencil: |dxi| <= 1e-6 xi; Newton converges
    // quadratically, so the iterate after such a step is within about (1e-6)^2 relative
    // (times a factor that grows like Gamma^3), far below the FP32 rounding of the output.
    constexpr double tol = sizeof(R) == 4 ? 1e-6 : 1e-14;
    bool ok = false;
    // quantities of the last iteration, evaluated at its starting point xs
    double xs = xi, ixi = 1.0, w = 0.0, lor = 1.0, rho = 0.0, drho = 0.0, pr = 0.0, dp = 0.0;
    for (int it = 0; it < 50; ++it) {
      xs = xi;
      ixi = rcp64(xi);
      w = s2 * ixi * ixi;                       // v^2
      const double ig2 = 1.0 - w;               // 1 / Gamma^2
      lor = rsqrt(ig2);                         // Gamma
      rho = D * (ig2 * lor);                    // D / Gamma
      drho = D * lor * w * ixi;                 // d rho / d xi
      if constexpr (EOS == EOS_SYNGE) {
        // h = xi / (D Gamma), theta(h) = (5h - sqrt(9h^2 + 16)) / 8, dh/dxi = Gamma / D
        const double h = xi * (ig2 * lor) * iD;
        const double q = 9.0 * h * h + 16.0;
        const double iq = rsqrt(q);
        const double th = 0.125 * (5.0 * h - q * iq);
        pr = rho * th;
        dp = th * drho + 0.125 * (5.0 - 9.0 * h * iq);
      } else {
        pr = gm * (xi * ig2 - rho);
        dp = gm * (1.0 + w - drho);
      }
      const double f = xi - pr - E;
      const double df = 1.0 - dp;
      if (f < 0.0) lo = xi; else hi = xi;
      double xn = xi - f * rcp64(df);
      if (!(xn >= lo && xn <= hi)) xn = 0.5 * (lo + hi);
      const bool conv = fabs(xn - xi) <= tol * xn;
      xi = xn;
      if (conv) { ok = true; break; }
    }
    if (!ok) st |= ST_ENOCONV;
    // The primitives at the converged xi from those of the last iterate xs by first-order
    // Taylor steps (the derivatives are the iteration's own): |xi - xs| <= tol xi, so the
    // neglected second-order terms are of relative size tol^2 (1e-28 in the FP64 stencil,
    // 1e-12 in the FP32 one), far below the rounding of the result.
    const double dx = xi - xs;
    const double ixn = fma(-ixi * ixi, dx, ixi);                    // d(1/xi) = -dx / xi^2
    const double lorn = fma(-(lor * lor * lor) * (w * ixi), dx, lor);   // dGamma/dxi = -Gamma^3 v^2 / xi
    const double rhon = fma(drho, dx, rho);
    const double prn = fma(dp, dx, pr);
    const double sc = lorn * ixn;
    p[0] = (R)rhon;
    if constexpr (sizeof(R) == 4) {   // u = Gamma v = m Gamma / xi: one conversion of the factor
      const R scr = (R)sc;
      p[1] = u[1] * scr;
      p[2] = u[2] * scr;
      p[3] = u[3] * scr;
    } else {
      p[1] = (R)(mx * sc);
      p[2] = (R)(my * sc);
      p[3] = (R)(mz * sc);
    }
    pr = prn;
    rho = rhon;
    lor = lorn;
    p[4] = (R)pr;
    aux[0] = (R)xi;
    aux[1] = (R)lor;
    if (!(rho > 0.0) || !(pr > 0.0)) st |= ST_EUNPHYS;
  }

  __device__ static __forceinline__ void prim2cons(const R* p, R* u, const PhysParamsT<R>& pp) {
    const R lor = rsqrt_(R(1) + p[1] * p[1] + p[2] * p[2] + p[3] * p[3]);
    R h;
    if constexpr (EOS == EOS_SYNGE) h = Eos::enthalpy(rdiv(p[4], p[0]), pp);
    else h = R(1) + rdiv(pp.gg1 * p[4], p[0]);
    const R lr = lor * p[0];
    const R lrh = lr * h;
    u[0] = lr;
    u[1] = lrh * p[1];
    u[2] = lrh * p[2];
    u[3] = lrh * p[3];
    u[4] = lor * lrh - p[4] - lr;
  }

  // Conserved state, flux along D and the interval of the speeds of a face state: one root and one
  // quotient for Gamma, rho h = rho + gamma/(gamma-1) p without a quotient (ideal gas), the two
  // factors of the speeds' root under one root: three quotients and two roots where formulas
  // taken one by one need six and four. Quotients and roots are most of these kernels' work:
  // a 48x64x80 FP64 solve took 6.56 -> 5.45 ms, a batch of 12 FP32 solves 10.9 -> 10.2 ms.
  template <int D>
  __device__ static __forceinline__ void side(const R* p, R* u, R* f, R& mid, R& half, const PhysParamsT<R>& pp) {
    const R lor = rsqrt_(R(1) + p[1] * p[1] + p[2] * p[2] + p[3] * p[3]);
    const R il = rrcp(lor);
    const R vd = p[1 + D] * il;
    R w, cs2;
    closure(p, w, cs2, pp);
    const R lr = lor * p[0], lw = lor * w;
    u[0] = lr;
    u[1] = lw * p[1];
    u[2] = lw * p[2];
    u[3] = lw * p[3];
    u[4] = lor * lw - p[4] - lr;
    f[0] = u[0] * vd;
    f[1] = u[1] * vd;
    f[2] = u[2] * vd;
    f[3] = u[3] * vd;
    f[1 + D] += p[4];
    f[4] = u[1 + D] - f[0];
    speeds_of(vd, il, cs2, mid, half);
  }

  // rho h and the squared sound speed
  __device__ static __forceinline__ void closure(const R* p, R& w, R& cs2, const PhysParamsT<R>& pp) {
    if constexpr (EOS == EOS_SYNGE) {
      const R th = p[4] * rrcp(p[0]);
      const R h = Eos::enthalpy(th, pp);
      w = p[0] * h;
      cs2 = Eos::sound_speed2(th, h, pp);
    } else {
      w = p[0] + pp.gg1 * p[4];
      cs2 = (pp.gamma * p[4]) * rrcp(w);
    }
  }
  // Middle and half width of the interval of characteristic speeds along a direction with velocity
  // vd, il = 1 / Gamma.
  __device__ static __forceinline__ void speeds_of(R vd, R il, R cs2, R& mid, R& half) {
    const R il2 = il * il;                      // 1 - v^2
    const R den = R(1) - (R(1) - il2) * cs2, a = vd * (R(1) - cs2);
    const R iden = rrcp(den);
    mid = a * iden;
    half = rsqrt_(rmax((cs2 * il2) * (den - vd * a), R(0))) * iden;
  }

  template <int D>
  __device__ static __forceinline__ void waves(const R* p, R& mid, R& half, const PhysParamsT<R>& pp) {
    const R il = rrcp(rsqrt_(R(1) + p[1] * p[1] + p[2] * p[2] + p[3] * p[3]));
    R w, cs2;
    closure(p, w, cs2, pp);
    speeds_of(p[1 + D] * il, il, cs2, mid, half);
  }

  template <int D>
  __device__ static __forceinline__ void interface(R*, R*, const PhysParamsT<R>&) {}
};

template <typename R> using SrhdPhys = SrhdPhysE<R, EOS_IDEAL>;
template <typename R> using SrhdSyngePhys = SrhdPhysE<R, EOS_SYNGE>;

// ------------------------------------------------------------------------------ FFHD
// Frozen-field hydrodynamics (Section 2.3.2, Eqs. 7-9): U = (rho, m_par, e, b), P = (rho,
// v_par, p, b) with b the frozen unit field, never updated and not reconstructed (cell
// values; the face value of b_d is the mean of the two cells'). The flux along d is
// b_d (rho v, rho v^2 + p, (e + p) v) and b_d for the variable b_d (0 for the other two), so
// the flux divergence of the b variables is -div b of the same face values; the source
// p div b of the m_par equation is added from it. TVDLF only (paper Table 1).
// With hyperbolic thermal conduction (HTC, Eqs. 9-10): U = (rho, m_par, e, q_par, b); q_par
// is reconstructed, has no face flux of its own (no dissipation either) and enters the
// energy flux as -q_par b_d; its relaxation towards kappa0 T^(5/2) b.grad T over tau = 4 dt
// is the stage kernel's source term for it.
template <typename R, bool HTC>
struct FfhdPhysT {
  static constexpr int NV = HTC ? 7 : 6;
  static constexpr int NA = 0;
  static constexpr int BOFF = HTC ? 4 : 3;   // b: swapped with the x/y trick, b_n negated at walls
  static constexpr int IV = -1;              // no vector velocity
  static constexpr int NREC = HTC ? 4 : 3;
  static constexpr int FROZEN = BOFF;
  static constexpr int QV = HTC ? 3 : -1;
  static constexpr int IE = 2;
  static constexpr bool SOURCE = true;
  static constexpr bool GLM = false;

  __device__ static __forceinline__ void cons2prim(const R* u, R* p, R*, const PhysParamsT<R>& pp,
                                                   int& st) {
    const R rho = u[0];
    const R v = u[1] * rrcp(rho);
    p[0] = rho;
    p[1] = v;
    p[2] = pp.g1 * (u[2] - R(0.5) * rho * v * v);
#pragma unroll
    for (int i = 3; i < NV; ++i) p[i] = u[i];
    st |= (!rpos(rho) | !rpos(p[2])) ? ST_EUNPHYS : 0;
  }

  __device__ static __forceinline__ void prim2cons(const R* p, R* u, const PhysParamsT<R>& pp) {
    u[0] = p[0];
    u[1] = p[0] * p[1];
    u[2] = p[2] * pp.ig1 + R(0.5) * p[0] * p[1] * p[1];
#pragma unroll
    for (int i = 3; i < NV; ++i) u[i] = p[i];
  }

  // Conserved state, flux along D and the interval mid -+ half of the speeds of a face state.
  template <int D>
  __device__ static __forceinline__ void side(const R* p, R* u, R* f, R& mid, R& half, const PhysParamsT<R>& pp) {
    prim2cons(p, u, pp);
    waves<D>(p, mid, half, pp);
    const R b = p[BOFF + D];
    const R vb = p[1] * b;
    f[0] = u[0] * vb;
    f[1] = u[1] * vb + p[2] * b;
    if constexpr (HTC) f[2] = (u[2] + p[2]) * vb - p[3] * b;
    else f[2] = (u[2] + p[2]) * vb;
#pragma unroll
    for (int i = 3; i < NV; ++i) f[i] = R(0);
    f[BOFF + D] = b;
  }

  template <int D>
  __device__ static __forceinline__ void waves(const R* p, R& mid, R& half, const PhysParamsT<R>& pp) {
    const R c = rsqrt_(rdiv(pp.gamma * p[2], p[0]));
    const R b = p[BOFF + D];
    mid = p[1] * b;
    half = c * rabs(b);
  }

  template <int D>
  __device__ static __forceinline__ void interface(R* pl, R* pr, const PhysParamsT<R>&) {
    const R bf = R(0.5) * (pl[BOFF + D] + pr[BOFF + D]);
    pl[BOFF + D] = bf;
    pr[BOFF + D] = bf;
  }

  // L holds -div F of every variable: L[BOFF..BOFF+2] sum to -div b; adds p div b to m_par.
  __device__ static __forceinline__ void source(R* L, const R* pcell) {
    L[1] = L[1] - pcell[2] * ((L[BOFF] + L[BOFF + 1]) + L[BOFF + 2]);
  }
};
template <typename R> using FfhdPhys = FfhdPhysT<R, false>;
template <typename R> using FfhdHtcPhys = FfhdPhysT<R, true>;

// The scalar solver returns the TVDLF flux times two: (F_l + F_r) - c (U_r - U_l); the halving
// goes into the factor 1 / dx that multiplies every flux (a power of two: the same bits), which
// takes one operation per variable and face off the FP64 units.
template <int FLUX>
__host__ __device__ constexpr double flux_unit() {
  return FLUX == FLUX_TVDLF ? 0.5 : 1.0;
}

// Riemann flux at a face from reconstructed primitive states (modified in place), in units of
// flux_unit<FLUX>().
template <class P, typename R, int D, int FLUX>
__device__ __forceinline__ void riemann(R* pl, R* pr, R* f, const PhysParamsT<R>& pp) {
  constexpr int NV = P::NV;
  R vml, vhl, vmr, vhr;   // middle and half width of each side's speeds
  if constexpr (FLUX == FLUX_HLLC) {
    // HLLC (Toro, Spruce & Speares 1994) for hydrodynamics: the HLL fan with the contact restored.
    // The contact speed S* tells the side K whose flux F_K + S (U*_K - U_K) the face has, S the
    // outer speed of that side, or 0 where the whole fan lies beyond the face (then F_K); star
    // state U*_K = rho_K (S_K - u_K)/(S_K - S*) [1, S* e_d + v_t, E_K/rho_K + (S* - u_K)(S* +
    // p_K/(rho_K (S_K - u_K)))]. The side is chosen before its conserved state, flux and star
    // state are formed, so these are formed once (210 FP64 blocks 1206 -> 992 us a launch, 1728
    // FP32 blocks 256 -> 234, in packed pairs 224; with the later steps 908 and 215).
    P::template waves<D>(pl, vml, vhl, pp);
    P::template waves<D>(pr, vmr, vhr, pp);
    const R sl = rmin(vml - vhl, vmr - vhr), sr = rmax(vml + vhl, vmr + vhr);
    const R vl = pl[1 + D], vr = pr[1 + D];
    const R ml = pl[0] * (sl - vl), mr = pr[0] * (sr - vr);
    const R ss = rdiv(pr[4] - pl[4] + ml * vl - mr * vr, ml - mr);
    const bool left = !rneg(ss);
    R q[NV], u[NV], fk[NV], lo, hi;
#pragma unroll
    for (int v = 0; v < NV; ++v) q[v] = left ? pl[v] : pr[v];
    const R sk = left ? sl : sr, mk = left ? ml : mr;
    const R s = left ? rmin(sl, R(0)) : rmax(sr, R(0));
    P::template side<D>(q, u, fk, lo, hi, pp);   // (its speeds are not used)
    const R fac = rdiv(mk, sk - ss);
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const R us = v == 0 ? fac : (v == 1 + D ? fac * ss : fac * q[v]);
      f[v] = fk[v] + s * (us - u[v]);
    }
    const R us4 = fac * (rdiv(u[4], q[0]) + (ss - q[1 + D]) * (ss + rdiv(q[4], mk)));
    f[4] = fk[4] + s * (us4 - u[4]);
    return;
  }
  P::template interface<D>(pl, pr, pp);
  R ul[NV], ur[NV], fl[NV], fr[NV];
  P::template side<D>(pl, ul, fl, vml, vhl, pp);
  P::template side<D>(pr, ur, fr, vmr, vhr, pp);
  if constexpr (FLUX == FLUX_TVDLF) {
    const R c = rmax(rabs(vml) + vhl, rabs(vmr) + vhr);   // max |mid -+ half| = |mid| + half
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      if (v >= P::FROZEN) f[v] = fl[v] + fl[v];   // frozen variables: exact flux, no dissipation
      else if (v == P::QV) f[v] = R(0);           // no flux term at all
      else f[v] = (fl[v] + fr[v]) - c * (ur[v] - ul[v]);
    }
  } else {
    const R sl = rmin(rmin(vml - vhl, vmr - vhr), R(0));
    const R sr = rmax(rmax(vml + vhl, vmr + vhr), R(0));
    const R inv = rrcp(sr - sl);
    const R wl = sr * inv, wr = sl * inv, wd = sl * wl;
#pragma unroll
    for (int v = 0; v < NV; ++v) f[v] = wl * fl[v] - wr * fr[v] + wd * (ur[v] - ul[v]);
  }
  if constexpr (P::GLM) {   // both sides carry B_d* and psi*: their flux is theirs, no dissipation
    constexpr R unit = R(1.0 / flux_unit<FLUX>());
    f[P::BOFF + D] = unit * pl[NV - 1];
    f[NV - 1] = (unit * pp.ch2) * pl[P::BOFF + D];
  }
}

// PLM face states: pl = P_i + phi_i / 2, pr = P_{i+1} - phi_{i+1} / 2 from the four cells
// i-1, i, i+1, i+2 around face i+1/2.
template <int NV, typename R, int LIM, int NREC = NV>
__device__ __forceinline__ void plm(const R* a, const R* b, const R* c, const R* d, R* pl, R* pr) {
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    if (v < NREC) {
      const R d0 = b[v] - a[v], d1 = c[v] - b[v], d2 = d[v] - c[v];
      pl[v] = b[v] + half_slope<R, LIM>(d0, d1);
      pr[v] = c[v] - half_slope<R, LIM>(d1, d2);
    } else {                 // not reconstructed: the cell values
      pl[v] = b[v];
      pr[v] = c[v];
    }
  }
}

}  // namespace agile
