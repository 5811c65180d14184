// heston_step.cuh -- one time step of the Heston model in each working
// precision: Andersen's quadratic-exponential scheme (the paper's
// discretisation, Sec. 2.2.1) and full-truncation Euler, with the per-group
// scheme constants.  Shared by the forward pass (forward.cu) and the inner
// simulations of the dual upper bound (dual.cu).
#pragma once

#include <type_traits>

#include "device_common.cuh"
#include "df_math.cuh"
#include "dfloat.cuh"
#include "plan.h"

namespace lsmc {

// Bytes of a precision's tables, and their copy into shared memory (the
// caller synchronises the block).
template <typename Real> __host__ __device__ constexpr size_t tab_bytes() {
  return std::is_same<Real, float>::value ? 0 : sizeof(Tab<Real>);
}
template <typename Real> __device__ __forceinline__ void load_tables(Tab<Real>* t) {
  if constexpr (std::is_same<Real, df>::value) {
    load_df_tables(t);
  } else if constexpr (std::is_same<Real, double>::value) {
    static_assert(sizeof(F64Tables) % sizeof(double2) == 0, "copied by pairs");
    const double2* src = reinterpret_cast<const double2*>(&kF64Tables);
    for (int i = threadIdx.x; i < (int)(sizeof(F64Tables) / sizeof(double2)); i += blockDim.x)
      reinterpret_cast<double2*>(t)[i] = __ldg(&src[i]);
  }
}
// The kernels' shared memory above 48 KB (static and dynamic) needs an opt-in.
// It holds for the kernel in the whole process, so `bytes` is the largest size
// any launch of the kernel takes: with a size per launch, a thread could lower
// it between another thread's opt-in and launch.
template <auto Kernel> static cudaError_t allow_dynamic(size_t bytes) {
  if (bytes == 0) return cudaSuccess;
  return cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// The unit of a path's log price x: double keeps x in units of
// ln 2 / kExpN (float pairs ln 2 / kDfExpN), so that its exponential needs no argument reduction (k is x
// rounded to an integer, exactly); the constants that x is made of are
// converted once per group, with the unit as a pair.
template <typename Real> __device__ __forceinline__ double in_log_units(double c) {
  if (std::is_same<Real, double>::value) return fma(kExpUnit, c, kExpUnitLo * c);
  return std::is_same<Real, df>::value ? kDfExpUnit * c : c;
}

// exp(X ln 2 / kExpN) for a log price X in those units.  X is split by integer
// operations into k = rint(X) and f = X - k to 44 bits; 2^(f / kExpN) - 1
// (at most 1.7e-4, so float pairs carry it past the double's last bit) by a
// cubic with f in units of 2^-22, its first two terms in pairs; times
// 2^(k / kExpN) from the table and the exponent: 2 FP64 operations and about
// 50 integer and FP32 ones, against 10 FP64 of exp_f64.  Beyond |x| = 177
// CUDA's exp.
__device__ __forceinline__ double exp_log_price(double X, const F64Tables* tab) {
  const int hi = __double2hiint(X), mag = hi & 0x7fffffff;
  if (mag >= ((1023 + 19) << 20)) return exp(X * kExpUnitInv);
  const uint32_t lo = (uint32_t)__double2loint(X);
  // |X| 2^44: the mantissa shifted left by 11 and right by 1042 - exponent
  const uint32_t mh = ((uint32_t)mag & 0xfffffu) | 0x100000u;
  const unsigned long long m =
      ((unsigned long long)__funnelshift_l(lo, mh, 11) << 32) | (lo << 11);
  unsigned long long u;
  asm("shr.u64 %0, %1, %2;" : "=l"(u) : "l"(m), "r"(1042 - (mag >> 20)));
  const long long s = (long long)(hi >> 31);
  const long long R = ((long long)u ^ s) - s + (1ll << 43);
  const int k = (int)(R >> 32) >> 12;
  const float f = __uint_as_float(0x4b000000u | (__funnelshift_r((uint32_t)R, (uint32_t)(R >> 32),
                                                                 22) & 0x3fffffu)) -
                  (8388608.0f + 2097152.0f);
  const float fl = __uint_as_float(0x3f800000u | (((uint32_t)R & 0x3fffffu) << 1)) - 1.0f;
  df p = two_prod(f, kExpA1);
  float e = __fmaf_rn(fl, kExpA1, __fmaf_rn(f, kExpA1Lo, p.lo));
  const df f2 = two_prod(f, f);
  const float t2 = __fmul_rn(f2.hi, kExpA2);
  e = __fadd_rn(e, __fmaf_rn(f2.hi, kExpA2, -t2));
  e = __fmaf_rn(__fmaf_rn(f + f, fl, f2.lo), kExpA2, __fmaf_rn(f2.hi, kExpA2Lo, e));
  e = __fmaf_rn(__fmul_rn(f2.hi, f), kExpA3, e);
  p = quick_two_sum(p.hi, t2);
  const double T = tab->exp2[k & (kExpN - 1)];
  const double y = fma(T, widen_float(p.hi) + widen_float(__fadd_rn(p.lo, e)), T);
  return __hiloint2double(__double2hiint(y) + ((k >> kExpNLog2) << 20), __double2loint(y));
}

// Elementary functions per precision (t: the precision's tables).
template <typename Real> struct Fm;
template <> struct Fm<double> {
  __device__ static double exp_(double a, const F64Tables* t) { return exp_log_price(a, t); }
};
template <> struct Fm<float> {
  __device__ static float div(float a, float b) { return __fdividef(a, b); }
  __device__ static float sqrt_(float a) {
    float r;  // approximate square root (MUFU), exact at 0
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
  }
  __device__ static float log_(float a, const NoTables*) { return __logf(a); }
  __device__ static float exp_(float a, const NoTables*) { return __expf(a); }
};
template <> struct Fm<df> {
  __device__ static df div(df a, df b) { return a / b; }
  __device__ static df sqrt_(df a) { return sqrt_df(a); }
  __device__ static df log_(df a, const DfTables* t) { return log_df(a, t->exp2); }
  __device__ static df exp_(df a, const DfTables* t) { return exp_log_price_df(a, t->fwd); }
};

template <typename Real>
struct GroupConst {
  // QE: m = mA + mB v, s^2 = sA + sB v, x1 = x + c0 + K1 v + K2 v1 +
  // sqrt(K3 (v + v1)) Z.  In double and float pairs sA + sB v is half of s^2,
  // the state is x - K2 v, K1
  // holds K1 + K2 (x - K2 v moves by c0 + (K1 + K2) v + sqrt(...) Z: K1 and K2
  // are large and nearly cancel, and their rounding errors would grow with the
  // steps), and c0, K1, K2, K3, mudt, hdt,
  // rho and rhob carry the unit of x (in_log_units)
  Real mA, mB, sA, sB, c0, K1, K2, K3;
  // FT-Euler
  Real dt, kdt, theta, xi, rho, rhob, mudt, hdt;
  Real v0, out_scale;
  void* E;            // rows of the path store (element type: the launch's store format)
  void* V;
  Real* CX;
  Real* CV;
  uint64_t ld;
};

// Scheme constants of one path group, from the model (Andersen 2008 for QE
// with gamma1 = gamma2 = 1/2; the plain Euler coefficients for FT).
template <typename Real>
__device__ void make_group_const(const FwdGroup& g, GroupConst<Real>& c) {
  constexpr bool kWide = !std::is_same<Real, float>::value;  // double, float pairs
  auto u = [](double x) { return in_log_units<Real>(x); };
  const double dt = g.dt, k = g.kappa, th = g.theta, xi = g.xi, rho = g.rho;
  const double E = exp(-k * dt);
  const double omE = -expm1(-k * dt);  // 1 - E without cancellation
  c.mA = (Real)(th * omE);
  c.mB = (Real)E;
  if (xi > 0.0) {
    const double half = kWide ? 0.5 : 1.0;
    c.sB = (Real)(half * (xi * xi * E * omE / k));
    c.sA = (Real)(half * (th * xi * xi * omE * omE / (2.0 * k)));
    const double K0 = -rho * k * th * dt / xi;
    const double h = 0.5 * dt * (k * rho / xi - 0.5);
    c.K1 = (Real)(kWide ? u(2.0 * h) : u(h - rho / xi));
    c.K2 = (Real)u(h + rho / xi);
    c.c0 = (Real)u((g.r - g.q) * dt + K0);
  } else {
    c.sA = c.sB = c.K1 = c.K2 = c.c0 = (Real)0;
  }
  c.K3 = (Real)u(u(0.5 * dt * (1.0 - rho * rho)));
  c.dt = (Real)dt;
  c.kdt = (Real)(k * dt);
  c.theta = (Real)th;
  c.xi = (Real)xi;
  c.rho = (Real)u(rho);
  c.rhob = (Real)u(sqrt(1.0 - rho * rho));
  c.mudt = (Real)u((g.r - g.q) * dt);
  c.hdt = (Real)u(0.5 * dt);
  c.v0 = (Real)g.v0;
  c.out_scale = (Real)g.out_scale;
  c.E = g.E;
  c.V = g.V;
  c.CX = (Real*)g.CX;
  c.CV = (Real*)g.CV;
  c.ld = g.ld;
}

// Andersen QE step: variance by the quadratic branch (psi <= 1.5) or the
// exponential branch, then the log price from both variances.  With
// psi = s^2 / m^2 the branch quantities are written with one division
// each: 2 / psi = 2 m^2 / s^2, p = (psi - 1) / (psi + 1) = (s^2 - m^2) /
// (s^2 + m^2), 1 - p = 2 m^2 / (s^2 + m^2), 1 / beta = m / (1 - p); the
// point mass is taken when U_V <= p, i.e. 1 - U_V >= 1 - p.
template <typename Real>
__device__ __forceinline__ void qe_core(Real mA, Real mB, Real sA, Real sB, Real c0, Real K1,
                                        Real K2, Real K3, Real& x, Real& v, Real omu, Real zV,
                                        Real zX, const Tab<Real>* t) {
  using F = Fm<Real>;
  const Real m = fma(mB, v, mA);
  const Real s2 = fma(sB, v, sA);
  const Real m2 = m * m;
  Real v1;
  if (s2 <= (Real)1.5 * m2) {
    const Real inv = F::div(m2 + m2, s2);
    const Real tt = inv - (Real)1;
    const Real b2 = tt + F::sqrt_(inv * tt);
    const Real b = F::sqrt_(b2);
    const Real a = F::div(m, (Real)1 + b2);
    const Real q = b + zV;
    v1 = a * q * q;
  } else {
    const Real rden = F::div((Real)1, s2 + m2);
    const Real omp = (m2 + m2) * rden;
    v1 = (omu >= omp) ? (Real)0 : F::div(m, omp) * F::log_(F::div(omp, omu), t);
  }
  x = x + c0 + K1 * v + K2 * v1 + F::sqrt_(K3 * (v + v1)) * zX;
  v = v1;
}

// ---- double precision --------------------------------------------------------
// An FP64 instruction holds the pipe of an SM for 18 clocks a warp on GB300;
// CUDA's square root and division are eight of them each (142 clocks).  The
// special-function unit's seeds take 2 clocks, so square roots are formed from
// rsqrt_seed (its seed improved in FP32) and quotients from a seed y and one
// third-order correction (e ~ 2^-20), sharing what can be shared.

// max(v, 0) of a double, the sign read as an integer
__device__ __forceinline__ double positive_part(double v) {
  return __double2hiint(v) < 0 ? 0.0 : v;
}

__device__ __forceinline__ double rcp_f64(double a) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
  const double e = fma(-a, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
// a double of a known exponent range as a float, within 2^-20 relative
__device__ __forceinline__ float seed_float(int hi) {
  return __int_as_float((hi - (896 << 20)) << 3);
}

// the variance step of the scheme's definition, for means so small or large
// that the products below could leave the range of double
static __device__ __noinline__ double qe_variance_plain(double m, double h2, double omu, double zV) {
  const double s2 = h2 + h2, m2 = m * m;
  if (s2 <= 1.5 * m2) {
    const double inv = (m2 + m2) / s2;
    const double tt = inv - 1.0;
    const double b2 = tt + sqrt(inv * tt);
    const double q = sqrt(b2) + zV;
    return m / (1.0 + b2) * q * q;
  }
  const double omp = (m2 + m2) / (s2 + m2);
  return omu >= omp ? 0.0 : m / omp * log_f64(omp / omu);
}

// Andersen QE step in double.  With h2 = s^2 / 2 and d = sqrt(m^2 - h2) the
// quadratic branch's a and b are a = m - d = h2 / (m + d) and a b^2 = d, so
//   v1 = a (b + Z)^2 = d (1 + w)^2,  w = sqrt(a / d) Z,
//   sqrt(a / d) = h2 / sqrt(h2 (d m + d^2)),
// two reciprocal square roots in place of two square roots and two divisions.  Exponential branch: with A = m^2,
// B = A + 2 h2: 1 - p = 2 A / B and 1 / beta = B / (2 m), and one reciprocal
// of B U m (U = 1 - U_V) gives both quotients of v1 = B / (2 m) log(2 A / (B U)).
// 26 FP64 operations with the quadratic branch and the exponential against 70
// before (the
// FP64 forward pass of the 131,072 x 252 book 27.5 -> 14.3 ms with the table
// quantile and exponential, -> 11.5 with what can be in FP32 moved there).
template <>
__device__ __forceinline__ void qe_core<double>(double mA, double mB, double sA, double sB,
                                                double c0, double K1, double K2, double K3,
                                                double& x, double& v, double omu, double zV,
                                                double zX, const F64Tables*) {
  const double m = fma(mB, v, mA);
  const double h2 = fma(sB, v, sA);
  double v1;
  // 1e-60 < m < 1e60, tested on the exponent
  if ((unsigned)(__double2hiint(m) - ((1023 - 200) << 20)) < (400u << 20)) {
    const double D = fma(m, m, -h2);  // psi <= 3/2  <=>  3 D >= h2
    // decided in float from the high words, clamped to float's range; the
    // exact comparison (two FP64 operations) only next to the threshold
    const int hh = __double2hiint(h2);
    const float fD = seed_float(min(max(__double2hiint(D), 900 << 20), 1140 << 20));
    const float fh = seed_float(hh), fd = fmaf(3.0f, fD, -fh);
    bool quad;
    if ((unsigned)(hh - (900 << 20)) < (240u << 20) && fabsf(fd) > 1e-5f * fh) quad = fd > 0.0f;
    else quad = 3.0 * D >= h2;
    if (quad) {
      double y, g, ep;
      rsqrt_seed(D, y, g, ep);
      const double d = fma(g, ep, g);
      rsqrt_seed(h2 * fma(d, m, D), y, g, ep);
      const double hy = h2 * y;
      const double w = fma(hy, ep, hy) * zV, q = fma(d, w, d);
      v1 = positive_part(fma(q, w, q));
    } else {
      const double A = m * m, B = fma(2.0, h2, A), bu = B * omu;
      // 2 A and B / 2 by their exponents
      const double A2 = __hiloint2double(__double2hiint(A) + (1 << 20), __double2loint(A));
      if (__double_as_longlong(bu) >= __double_as_longlong(A2)) {
        v1 = 0.0;
      } else {
        const double R = rcp_f64(bu * m);
        const double Bh = __hiloint2double(__double2hiint(B) - (1 << 20), __double2loint(B));
        v1 = Bh * (R * bu) * log_f64(A2 * (R * m));
      }
    }
  } else {
    v1 = qe_variance_plain(m, h2, omu, zV);
  }
  double y, g, ep;
  rsqrt_seed(K3 * (v + v1), y, g, ep);
  x = x + fma(fma(g, ep, g), zX, fma(K1, v, c0));
  v = v1;
}

// ---- float pairs ----------------------------------------------------------------
// the variance step of the scheme's definition (means outside the range where
// the products below keep their low words)
static __device__ __noinline__ df qe_variance_plain(df m, df h2, df omu, df zV,
                                                    const DfTables* t) {
  const df s2 = twice_df(h2), m2 = m * m;
  if (s2 <= mul_f(m2, 1.5f)) {
    const df inv = twice_df(m2) / s2;
    const df tt = inv - df(1.0f, 0.0f);
    const df b2 = tt + sqrt_df(inv * tt);
    const df q = sqrt_df(b2) + zV;
    return m / (df(1.0f, 0.0f) + b2) * q * q;
  }
  const df omp = twice_df(m2) / (s2 + m2);
  return omu >= omp ? df(0.0f, 0.0f) : m / omp * log_df(omp / omu, t->exp2);
}

// The step in the form of qe_core<double>: about 190 FP32 operations with the
// quadratic branch where the direct form took 380 (a pair's division is 25, its
// full addition 20, a product with a sum that cannot cancel 15).
template <>
__device__ __forceinline__ void qe_core<df>(df mA, df mB, df sA, df sB, df c0, df K1, df K2, df K3,
                                            df& x, df& v, df omu, df zV, df zX,
                                            const DfTables* t) {
  const df m = madd_df(mB, v, mA);
  const df h2 = madd_df(sB, v, sA);
  df v1;
  if (m.hi > 1e-6f && m.hi < 1e6f) {
    const df A = mul_nr(m, m);
    const df D = add_sloppy(A, -h2);
    // psi <= 3/2  <=>  3 D >= h2
    if (__fadd_rn(__fmaf_rn(3.0f, D.hi, -h2.hi), __fmaf_rn(3.0f, D.lo, -h2.lo)) >= 0.0f) {
      float y, g, gl, ep;
      rsqrt_seed_df(D, y, g, gl, ep);
      const df d = quick_two_sum(g, __fmaf_rn(g, ep, gl));
      const df X = mul_nr(h2, madd_df(d, m, D));
      rsqrt_seed_df(quick_two_sum(X.hi, X.lo), y, g, gl, ep);
      df w = two_prod(h2.hi, y);  // h2 / sqrt(X)
      w.lo = __fmaf_rn(w.hi, ep, __fmaf_rn(h2.lo, y, w.lo));
      w = mul_nr(w, zV);
      const df q = madd_df(d, w, d);
      v1 = madd_df(q, w, q);
      if (v1.hi < 0.0f) v1 = df(0.0f, 0.0f);
    } else {
      const df B = add_sloppy(A, twice_df(h2)), A2 = twice_df(quick_two_sum(A.hi, A.lo));
      const df bu = B * omu;
      if (bu >= A2) {
        v1 = df(0.0f, 0.0f);
      } else {
        const df R = df(1.0f, 0.0f) / (bu * m);
        v1 = half_df(B) * (R * bu) * log_df(A2 * (R * m), t->exp2);
      }
    }
  } else {
    v1 = qe_variance_plain(m, h2, omu, zV, t);
  }
  const df w = mul_nr(K3, add_sloppy(v, v1));
  float y, g, gl, ep;
  rsqrt_seed_df(quick_two_sum(w.hi, w.lo), y, g, gl, ep);
  const df sq = quick_two_sum(g, __fmaf_rn(g, ep, gl));
  x = add_sloppy(x, add_sloppy(mul_nr(sq, zX), madd_df(K1, v, c0)));
  v = v1;
}

template <typename Real>
__device__ __forceinline__ void qe_step(const GroupConst<Real>& c, Real& x, Real& v,
                                        Real omu, Real zV, Real zX, const Tab<Real>* t) {
  qe_core<Real>(c.mA, c.mB, c.sA, c.sB, c.c0, c.K1, c.K2, c.K3, x, v, omu, zV, zX, t);
}

// The state of a path's log price at date 0, and the log price (in its unit)
// of a state x with variance v.
template <typename Real, int SCHEME>
__device__ __forceinline__ Real log_price_start(const GroupConst<Real>& c) {
  if constexpr (!std::is_same<Real, float>::value && SCHEME == kSchemeQE) return -(c.K2 * c.v0);
  else return (Real)0;
}
template <typename Real, int SCHEME>
__device__ __forceinline__ Real log_price(const GroupConst<Real>& c, Real x, Real v) {
  if constexpr (std::is_same<Real, double>::value && SCHEME == kSchemeQE) return fma(c.K2, v, x);
  else if constexpr (std::is_same<Real, df>::value && SCHEME == kSchemeQE)
    return madd_df(c.K2, v, x);
  else return x;
}

// Full-truncation Euler: v+ = max(v, 0) in drift and diffusion.
template <typename Real>
__device__ __forceinline__ void ft_step(const GroupConst<Real>& c, Real& x,
                                        Real& v, Real zV, Real zX) {
  using F = Fm<Real>;
  const Real vp = v > (Real)0 ? v : (Real)0;
  const Real sq = F::sqrt_(vp * c.dt);
  const Real v1 = v + c.kdt * (c.theta - vp) + c.xi * sq * zV;
  x = x + (c.mudt - (Real)0.5 * vp * c.dt) + sq * (c.rho * zV + c.rhob * zX);
  v = v1;
}

template <>
__device__ __forceinline__ void ft_step<double>(const GroupConst<double>& c, double& x, double& v,
                                                double zV, double zX) {
  const double vp = positive_part(v);
  double y, g, ep;
  rsqrt_seed(vp * c.dt, y, g, ep);
  const double sq = fma(g, ep, g);
  const double v1 = fma(c.xi, sq * zV, fma(c.kdt, c.theta - vp, v));
  x = x + fma(-c.hdt, vp, c.mudt) + sq * fma(c.rhob, zX, c.rho * zV);
  v = v1;
}

template <>
__device__ __forceinline__ void ft_step<df>(const GroupConst<df>& c, df& x, df& v, df zV, df zX) {
  const df vp = v.hi > 0.0f ? v : df(0.0f, 0.0f);
  float y, g, gl, ep;
  rsqrt_seed_df(vp * c.dt, y, g, gl, ep);
  const df sq = quick_two_sum(g, __fmaf_rn(g, ep, gl));
  const df v1 = (v + mul_nr(c.kdt, c.theta - vp)) + mul_nr(c.xi, sq * zV);
  const df shock = mul_nr(sq, madd_df(c.rhob, zX, mul_nr(c.rho, zV)));
  x = x + add_sloppy(shock, madd_df(-c.hdt, vp, c.mudt));
  v = v1;
}

}  // namespace lsmc
