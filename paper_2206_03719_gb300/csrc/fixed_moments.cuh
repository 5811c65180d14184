// fixed_moments.cuh -- the moment sums of a regression in fixed point, for
// double-precision paths.
//
// What bounds it: on GB300 an FP64 instruction holds an SM's pipe for 18
// clocks a warp, a 32 x 32 -> 64-bit integer multiply-add for 0.66.  The 21
// sums of an in-the-money path took 25 FP64 operations (425 clocks per 32
// paths), four fifths of the backward pass's FP64 work; here 2 FP64
// operations, 47 integer multiply-adds and about 110 other integer
// instructions do it, and the sums are exact, so their order does not matter.
// (The FP64 matrix instruction m8n8k4 runs at 3.6 times the FP64 rate, 36
// clocks, but an 8 x 8 tile holds the 21 sums once: 377 clocks for 32 paths.)
//
// Format.  A value q (x, w or the cash flow y, formed in double) is the
// integer round(q 2^F), |.| < 2^54, from its mantissa by shifts, split into
// limbs h 2^28 + l, |l| <= 2^27.  The squares and the product x w keep the
// format (round(X X 2^-54), ...).  A product of two values adds h h' to one
// 64-bit sum and h l' + l h' to another; l l' is below 2^-54 of the range and
// of mean zero.  256 paths a lane (the largest job) stay below 2^63.
//
// Range.  2^(54 - F) is at least 4 (x) or 8 (w) times the root mean square of
// the previous exercise date's paths, 16 times the mean for y (integers from
// the exponents of its sums, published with its coefficients); a path outside
// (any x, w or y, infinities and NaN among them) is summed in double by the
// whole warp, a monomial per lane.  In a model of this arithmetic (x normal
// with deviations 0.003 to 0.2, w gamma; 8 to 60,000 paths) the fitted values
// are within 3e-15 to 4e-17 of the exact regression's, against 4e-15 to 6e-16
// with double sums; 49 bits, which one fused multiply-add could produce, gave
// 9e-14 to 1e-15.
#pragma once

#include <cstdint>

#include "plan.h"

namespace lsmc {
namespace {

constexpr int kFixBits = 54;  // |integer| < 2^54
constexpr int kFixRangeMin = -40, kFixRangeMax = 40;  // exponents of the ranges

// F of each variable, as the shift from a double's exponent field
struct FixScale {
  int Fx, Fw, Fy;
};

__device__ __forceinline__ double exp2_int(int k) {  // 2^k, k in the normal range
  return __hiloint2double((1023 + k) << 20, 0);
}

// A value's integer round(q 2^F) = h 2^28 + l, |l| <= 2^27.
struct Limbs {
  int h, l;
  Limbs() = default;
  // the limbs of v
  __device__ __forceinline__ explicit Limbs(long long v) {
    const long long r = v + (1ll << 27);
    h = (int)__funnelshift_r((uint32_t)r, (uint32_t)(r >> 32), 28);
    l = ((int)r & 0xfffffff) - (1 << 27);
  }
};

// The limbs of |q| 2^F, from the mantissa m and the exponent field e of q
// (|q| = m 2^(e - 1075)); hi: the high word of |q|.  bad: |q| outside the
// range (then the limbs mean nothing).
__device__ __forceinline__ Limbs fix_magnitude(int hi, int lo, int F, bool& bad) {
  // m shifted left by 3 and right by n: twice the integer, the last bit rounding
  const int n = 1077 - F - (hi >> 20);
  bad = bad || n < 1;
  const uint32_t mh = ((uint32_t)hi & 0xfffffu) | 0x100000u;
  const unsigned long long m = ((unsigned long long)__funnelshift_l((uint32_t)lo, mh, 3) << 32) |
                               ((uint32_t)lo << 3);
  unsigned long long t;  // zero for shifts beyond 63 (small values, and the bad ones)
  asm("shr.u64 %0, %1, %2;" : "=l"(t) : "l"(m), "r"(n));
  t += 1ull + (1ull << 28);
  Limbs r;
  r.h = (int)__funnelshift_r((uint32_t)t, (uint32_t)(t >> 32), 29);
  r.l = (int)(((uint32_t)t & 0x1fffffffu) >> 1) - (1 << 27);
  return r;
}
// ... of q itself
__device__ __forceinline__ Limbs fix_signed(double q, int F, bool& bad) {
  const int hi = __double2hiint(q), s = hi >> 31;
  Limbs r = fix_magnitude(hi & 0x7fffffff, __double2loint(q), F, bad);
  r.h = (r.h ^ s) - s;
  r.l = (r.l ^ s) - s;
  return r;
}

// Exponent of the range of the next date from this date's sums: 2^e >= m
// times the root mean square (or, order 1, the mean) of `sum` over `count`;
// m2 = log2(m) * order; `keep` where nothing was summed.
__device__ __forceinline__ int fix_range(double sum, double count, int m2, int order, int keep) {
  const int es = (__double2hiint(sum) >> 20) & 0x7ff, en = (__double2hiint(count) >> 20) & 0x7ff;
  if (es == 0 || es == 0x7ff || en == 0 || en == 0x7ff) return keep;
  const int d = es - en + 1 + m2;  // sum / count < 2^(es - en + 1)
  const int e = order == 2 ? (d + 1) >> 1 : d;
  return min(max(e, kFixRangeMin), kFixRangeMax);
}

// The sums of a basis as units, in slot order without the count: a sum of
// products (hh 2^56 + hl 2^28) 2^-E or a plain sum of integers.  Packed per
// unit: powers of x, w, y (4 bits each), the number of operands that are
// themselves products (each drops 2^54), and whether it is a plain sum.
constexpr uint32_t fix_unit(int a, int b, int c, int prods, int plain) {
  return (uint32_t)(a | b << 4 | c << 8 | prods << 12 | plain << 16);
}
__device__ const uint32_t kFixUnitsSV2[20] = {
    fix_unit(1, 0, 0, 0, 1), fix_unit(2, 0, 0, 1, 1), fix_unit(3, 0, 0, 1, 0),
    fix_unit(4, 0, 0, 2, 0), fix_unit(0, 1, 0, 0, 1), fix_unit(1, 1, 0, 1, 1),
    fix_unit(2, 1, 0, 1, 0), fix_unit(3, 1, 0, 2, 0), fix_unit(0, 2, 0, 1, 1),
    fix_unit(1, 2, 0, 1, 0), fix_unit(2, 2, 0, 2, 0), fix_unit(0, 3, 0, 1, 0),
    fix_unit(1, 3, 0, 2, 0), fix_unit(0, 4, 0, 2, 0), fix_unit(0, 0, 1, 0, 1),
    fix_unit(1, 0, 1, 0, 0), fix_unit(2, 0, 1, 1, 0), fix_unit(0, 1, 1, 0, 0),
    fix_unit(1, 1, 1, 1, 0), fix_unit(0, 2, 1, 1, 0)};
__device__ const uint32_t kFixUnitsS2[7] = {
    fix_unit(1, 0, 0, 0, 1), fix_unit(2, 0, 0, 1, 1), fix_unit(3, 0, 0, 1, 0),
    fix_unit(4, 0, 0, 2, 0), fix_unit(0, 0, 1, 0, 1), fix_unit(1, 0, 1, 0, 0),
    fix_unit(2, 0, 1, 1, 0)};

// one monomial x^a w^b y^c of a packed unit, in double (the rare paths)
__device__ __noinline__ double fix_monomial(uint32_t unit, double x, double w, double y) {
  double p = (unit >> 8) & 15u ? y : 1.0;
  for (uint32_t k = unit & 15u; k > 0; --k) p *= x;
  for (uint32_t k = (unit >> 4) & 15u; k > 0; --k) p *= w;
  return p;
}

// a b + c as one instruction (written out: from 64-bit C expressions the
// compiler forms full 64-bit products: 394 instructions a path against 266)
__device__ __forceinline__ long long wide(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
// round(A B 2^-54)
__device__ __forceinline__ long long fix_product(const Limbs& a, const Limbs& b) {
  return wide(4 * a.h, b.h, wide(a.l, b.h, wide(a.h, b.l, 1ll << 25)) >> 26);
}
// the same for a square; l l, of mean 2^54 / 3, is not formed: its mean is
// added instead
__device__ __forceinline__ long long fix_square(const Limbs& a) {
  return wide(4 * a.h, a.h, wide(a.h + a.h, a.l, (1ll << 25) + (1ll << 26) / 3) >> 26);
}

// Sums of one warp: per unit and lane two 64-bit sums, of h h' and of
// h l' + l h' (one for the plain sums, in hh).  The x here is |S / K - 1|
// (in-the-money paths lie on one side of the strike); value() gives odd powers
// their sign.
template <int BASIS> struct FixedSums {
  static constexpr bool kV = BASIS == kBasisSV2;
  static constexpr int NU = kV ? 20 : 7;
  long long hh[NU], hl[NU];
  double spill;  // lane u < NU: unit u over the paths outside the range
  bool spilled;

  __device__ __forceinline__ static uint32_t unit(int u) {
    return kV ? kFixUnitsSV2[u] : kFixUnitsS2[u];
  }
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int i = 0; i < NU; ++i) hh[i] = hl[i] = 0;
    spill = 0.0;
    spilled = false;
  }
  __device__ __forceinline__ void plain(int i, const Limbs& a) {
    hh[i] = wide(a.h, 1 << 28, wide(a.l, 1, hh[i]));
  }
  __device__ __forceinline__ void product(int i, const Limbs& a, const Limbs& b) {
    hh[i] = wide(a.h, b.h, hh[i]);
    hl[i] = wide(a.l, b.h, wide(a.h, b.l, hl[i]));
  }
  __device__ __forceinline__ void square(int i, const Limbs& a) {
    hh[i] = wide(a.h, a.h, hh[i]);
    hl[i] = wide(a.h + a.h, a.l, hl[i]);
  }
  // one path per lane (valid lanes): row values e, v and cash flow z; called
  // by the whole warp
  __device__ __forceinline__ void add(const FixScale& f, double e, double v, double z, bool valid,
                                      double xK, double invTh) {
    const double xd = fma(e, xK, -1.0), wd = kV ? fma(v, invTh, -1.0) : 0.0;
    bool bad = false;
    Limbs x = fix_magnitude(__double2hiint(xd) & 0x7fffffff, __double2loint(xd), f.Fx, bad);
    Limbs y = fix_magnitude(__double2hiint(z) & 0x7fffffff, __double2loint(z), f.Fy, bad);
    Limbs w;
    if (kV) w = fix_signed(wd, f.Fw, bad);
    if (__any_sync(0xffffffffu, bad || !valid)) {
      unsigned m = __ballot_sync(0xffffffffu, bad && valid);
      spilled = spilled || m != 0;
      const int lane = threadIdx.x & 31;
      const uint32_t u = unit(lane < NU ? lane : 0);
#pragma unroll 1
      while (m) {
        const int src = __ffs(m) - 1;
        m &= m - 1;
        const double xs = __shfl_sync(0xffffffffu, xd, src);
        const double ws = __shfl_sync(0xffffffffu, wd, src);
        const double ys = __shfl_sync(0xffffffffu, z, src);
        spill += fix_monomial(u, xs, ws, ys);
      }
      if (bad || !valid) x.h = x.l = y.h = y.l = w.h = w.l = 0;
    }
    const Limbs x2(fix_square(x));
    plain(0, x);
    plain(1, x2);
    product(2, x2, x);
    square(3, x2);
    if (kV) {
      const Limbs xw(fix_product(x, w)), w2(fix_square(w));
      plain(4, w);
      plain(5, xw);
      product(6, x2, w);
      product(7, x2, xw);
      plain(8, w2);
      product(9, xw, w);
      product(10, x2, w2);
      product(11, w2, w);
      product(12, xw, w2);
      square(13, w2);
      plain(14, y);
      product(15, x, y);
      product(16, x2, y);
      product(17, w, y);
      product(18, xw, y);
      product(19, w2, y);
    } else {
      plain(4, y);
      product(5, x, y);
      product(6, x2, y);
    }
  }
  // the units in slot order, in two parts small enough to be added over 32
  // lanes: products as a 2^28 + b in units of 2^56, plain sums in units of 1
  __device__ __forceinline__ void units(long long (&a)[NU], long long (&b)[NU]) const {
    constexpr long long kMask = (1ll << 28) - 1;
#pragma unroll
    for (int i = 0; i < NU; ++i) {
      const bool is_plain = i == 0 || i == 1 || (kV ? i == 4 || i == 5 || i == 8 || i == 14 : i == 4);
      a[i] = hh[i] >> 28;
      b[i] = (hh[i] & kMask) + (is_plain ? 0 : (hl[i] + (1ll << 27)) >> 28);
    }
  }
  // neg: x is negative (puts)
  __device__ __forceinline__ static double value(int u, long long a, long long b,
                                                 const FixScale& f, bool neg) {
    const uint32_t t = unit(u);
    const int E = (int)(t & 15u) * f.Fx + (int)((t >> 4) & 15u) * f.Fw +
                  (int)((t >> 8) & 15u) * f.Fy - kFixBits * (int)((t >> 12) & 15u) +
                  56 * (int)(t >> 16);
    const double v = fma((double)a, 268435456.0, (double)b) * exp2_int(56 - E);
    return neg && (t & 1u) ? -v : v;
  }
};

// Reduce-scatter of C units over the warp by recursive halving over the lane
// bits O, ..., 1: at each level a lane and its partner split the units they
// hold (the lane with the bit clear keeps the lower half) and each adds the
// partner's copy of its half; in the end a lane holds at most one unit summed
// over the 32 lanes (idx, or -1).
template <int C, int O>
__device__ __forceinline__ void halving_units(const long long (&a)[C], const long long (&b)[C],
                                              int lane, int base, int real, long long& oa,
                                              long long& ob, int& idx) {
  constexpr int H = (C + 1) / 2;
  const bool upper = (lane & O) != 0;
  long long na[H], nb[H];
#pragma unroll
  for (int i = 0; i < H; ++i) {
    constexpr int kLast = C - 1;
    const bool have = H + i < C;
    const int j = have ? H + i : kLast;
    const long long ha = have ? a[j] : 0, hb = have ? b[j] : 0;
    na[i] = (upper ? ha : a[i]) + __shfl_xor_sync(0xffffffffu, upper ? a[i] : ha, O);
    nb[i] = (upper ? hb : b[i]) + __shfl_xor_sync(0xffffffffu, upper ? b[i] : hb, O);
  }
  const int nbase = upper ? base + H : base;
  const int nreal = upper ? (real > H ? real - H : 0) : (real < H ? real : H);
  if constexpr (O == 1) {
    static_assert(H == 1, "at most 32 units");
    oa = na[0];
    ob = nb[0];
    idx = nreal >= 1 ? nbase : -1;
  } else {
    halving_units<H, O / 2>(na, nb, lane, nbase, nreal, oa, ob, idx);
  }
}

}  // namespace
}  // namespace lsmc
