// fixed_moments.cuh -- the moment sums of a regression in fixed point, for
// double-precision paths.
//
// What bounds it: on GB300 an FP64 instruction holds an SM's pipe for 18
// clocks a warp, a 32 x 32 -> 64-bit integer multiply-add for 0.66.  The 21
// sums of an in-the-money path took 25 FP64 operations (425 clocks per 32
// paths), four fifths of the backward pass's FP64 work; here 2 FP64
// operations, 47 integer multiply-adds and about 110 other integer
// instructions do it.
// (The FP64 matrix instruction m8n8k4 runs at 3.6 times the FP64 rate, 36
// clocks, but an 8 x 8 tile holds the 21 sums once: 377 clocks for 32 paths.)
//
// Format.  A value q (x, w or the cash flow y, formed in double) is the
// integer round(q 2^F), |.| < 2^56, from its mantissa by shifts, split into
// limbs h 2^28 + l, |l| <= 2^27.  The squares and the product x w keep the
// format (round(X X 2^-56), ...).  A product of two values adds h h' to one
// 64-bit sum and h l' + l h' to another; l l' is below 2^-58 of the range's
// product and of mean zero, but for the squares of x^2 and w^2, which get its
// mean.  A lane sums 126 paths at most before its sums are taken out, added over
// the warp without a rounding and converted.  (With 54 bits, which 256 paths, a
// whole job, do not overflow, the part left out is 16 times larger and its mean
// put the sums of x^4 and w^4 1e-14 to 1e-13 too low; with the products of the
// low limbs summed as well the book of 131,072 x 252 x 55 took 41.3 ms, against
// 39.6 like this.)  Over maturities from a day to a year, volatilities of variance
// from 0.001 to 0.3 and 60 to 2,000 paths the sums are 0.61 to 0.96 times as far
// from the exact ones as sums in double, the fits 0.63 to 0.98 times
// (tests/test_fixed_moments_host.py runs this code on the host).
//
// Range.  2^(56 - F) is the smallest power of two above the largest |q| that
// the warp has summed in its job, for x, w and y each (for y, of which only
// first powers are summed, with two bits to spare while more paths may come).
// It is taken from the first list of paths; when a later path lies beyond it,
// the sums held are shifted to the larger range (hl keeps what hh drops).  So
// the scales follow the warp's own paths alone, whatever the maturity, the
// volatilities or the distance of v0 from theta, and depend on no earlier date
// and no other warp.  (With ranges fixed for the first date and taken from the
// date before for the others, narrow distributions lost their digits: at one
// day and xi = 0.005, 3,001 paths, the coefficients scaled by their functions'
// norms were off by 5e-2, where a fit in double may be off by 2e-10.)  Growing
// is outside the loop over the paths: inside it, its registers cost twice as
// much as its work (book of 131,072 x 252 x 55: fixed ranges 37.8 ms, grown in
// the loop 42.5, outside 39.4).  Values beyond 2^100 (x, w) or 2^400 (y),
// infinities and NaN are summed in double by the whole warp, a monomial per
// lane.
#pragma once

#include <cstdint>

#include "plan.h"

namespace lsmc {
namespace {

constexpr int kFixBits = 56;  // |integer| < 2^56
// Paths a lane may sum before its sums are taken out: h h', h l' + l h' and the
// values themselves are at most 2^56 each, so 126 of them, and what shifts and
// means add, stay below 2^63.
constexpr int kFixItems = 126;
// Largest ranges: x and w < 2^kFixTopXW, cash flows < 2^kFixTopY (values
// beyond, infinities and NaN are summed in double).  The scales start at ranges
// 2^-kFixTopXW and 2^-kFixTopY.  With these every scale of a sum is a normal
// double.
constexpr int kFixTopXW = 100, kFixTopY = 400;

// F of each variable: the integer of q is round(q 2^F)
struct FixScale {
  int x, w, y;
};

__device__ __forceinline__ double exp2_int(int k) {  // 2^k, k in the normal range
  return __hiloint2double((1023 + k) << 20, 0);
}

// v >> n, zero for any n (read unsigned) beyond 63
__device__ __forceinline__ unsigned long long shr_clamped(unsigned long long v, int n) {
#ifdef __CUDA_ARCH__
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
#else
  return (unsigned)n > 63u ? 0ull : v >> n;
#endif
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
// range, e > kFixTop - F (then the limbs mean nothing).
constexpr int kFixTop = 1022 + kFixBits;
__device__ __forceinline__ Limbs fix_magnitude(int hi, int lo, int F, bool& bad) {
  // m shifted left by 5 and right by n: twice the integer, the last bit rounding
  const int n = kFixTop + 1 - F - (hi >> 20);
  bad = bad || n < 1;
  const uint32_t mh = ((uint32_t)hi & 0xfffffu) | 0x100000u;
  const unsigned long long m = ((unsigned long long)__funnelshift_l((uint32_t)lo, mh, 5) << 32) |
                               ((uint32_t)lo << 5);
  // zero for shifts beyond 63 (small values, and the bad ones)
  const unsigned long long t = shr_clamped(m, n) + (1ull + (1ull << 28));
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

// The sums of a basis as units, in slot order without the count: a sum of
// products (hh 2^56 + hl 2^28) 2^-E or a plain sum of integers.  Packed per
// unit: powers of x, w, y (4 bits each), the number of operands that are
// themselves products (each drops 2^kFixBits), and whether it is a plain sum.
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
#ifdef __CUDA_ARCH__
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (long long)a * b + c;
#endif
}
// round(A B 2^-56)
__device__ __forceinline__ long long fix_product(const Limbs& a, const Limbs& b) {
  return wide(a.h, b.h, wide(a.l, b.h, wide(a.h, b.l, 1ll << 27)) >> 28);
}
// the same for a square; l l, of mean 2^54 / 3, is not formed: its mean is
// added instead
__device__ __forceinline__ long long fix_square(const Limbs& a) {
  return wide(a.h, a.h, wide(a.h + a.h, a.l, (1ll << 27) + (1ll << 26) / 3) >> 28);
}

// What a warp's lanes share, in shared memory: the scales of the sums, and the
// sums over the paths beyond the largest range.
struct FixWarp {
  FixScale scale;
  int spilled;       // whether spill holds anything
  double spill[20];
};

// Sums of one warp: per unit and lane two 64-bit sums, of h h' and of
// h l' + l h' (one for the plain sums, in hh).  The x here is |S / K - 1|
// (in-the-money paths lie on one side of the strike); value() gives odd powers
// their sign.
template <int BASIS> struct FixedSums {
  static constexpr bool kV = BASIS == kBasisSV2;
  static constexpr int NU = kV ? 20 : 7;
  long long hh[NU], hl[NU];

  __device__ __forceinline__ static constexpr bool is_plain(int u) {
    return u == 0 || u == 1 || (kV ? u == 4 || u == 5 || u == 8 || u == 14 : u == 4);
  }
  __device__ __forceinline__ static uint32_t unit(int u) {
    return kV ? kFixUnitsSV2[u] : kFixUnitsS2[u];
  }
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < NU; ++i) hh[i] = hl[i] = 0;
  }
  // called by the whole warp, once per job
  __device__ __forceinline__ void start(FixWarp& ws) {
    clear();
    const int lane = threadIdx.x & 31;
    if (lane < NU) ws.spill[lane] = 0.0;
    if (lane == 0) {
      ws.scale = FixScale{kFixBits + kFixTopXW, kFixBits + kFixTopXW, kFixBits + kFixTopY};
      ws.spilled = 0;
    }
    __syncwarp();
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
  // The sums from scales f to scales n <= f, in steps that divide no unit by
  // more than 2^28: a plain sum is rounded, of the others hl keeps what hh
  // drops (errors below a unit of hl, 2^-80 of the new range's product).
  __device__ __forceinline__ void rescale(const FixScale& f, const FixScale& n) {
    // beyond 2^98 nothing is left of a sum
    int dx = min(f.x - n.x, 98), dw = min(f.w - n.w, 98), dy = min(f.y - n.y, 98);
#pragma unroll 1
    while (dx > 0 || dw > 0 || dy > 0) {
      const int sx = min(dx, 7), sw = min(dw, 7), sy = min(dy, 14);
      dx -= sx;
      dw -= sw;
      dy -= sy;
#pragma unroll
      for (int i = 0; i < NU; ++i) {
        const uint32_t t = unit(i);
        const int s = (int)(t & 15u) * sx + (int)((t >> 4) & 15u) * sw + (int)((t >> 8) & 15u) * sy;
        if (is_plain(i)) {
          hh[i] = (hh[i] + (long long)((1u << s) >> 1)) >> s;
        } else {
          hl[i] = (hl[i] >> s) + (long long)(((uint32_t)hh[i] & ((1u << s) - 1u)) << (28 - s));
          hh[i] >>= s;
        }
      }
    }
  }
  // Adds one path per lane (valid lanes): row values e, v and cash flow z.
  // Called by the whole warp; false, and nothing added, where a path lies
  // beyond the range of the scales f.
  __device__ __forceinline__ bool add(const FixScale& f, double e, double v, double z, bool valid,
                                      double xK, double invTh) {
    const double xd = fma(e, xK, -1.0), wd = kV ? fma(v, invTh, -1.0) : 0.0;
    bool bad = false;
    Limbs x = fix_magnitude(__double2hiint(xd) & 0x7fffffff, __double2loint(xd), f.x, bad);
    Limbs y = fix_magnitude(__double2hiint(z) & 0x7fffffff, __double2loint(z), f.y, bad);
    Limbs w;
    if (kV) w = fix_signed(wd, f.w, bad);
    if (__any_sync(0xffffffffu, bad || !valid)) {
      if (__any_sync(0xffffffffu, bad && valid)) return false;
      if (!valid) x.h = x.l = y.h = y.l = w.h = w.l = 0;
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
    return true;
  }
  // Adds to the squares the mean of the l l left out of `items` of this lane's
  // paths, at the scales they were summed at.
  __device__ __forceinline__ void settle_mean(uint32_t items) {
    hl[3] += (long long)items * ((1 << 26) / 3);
    if (kV) hl[kV ? 13 : 0] += (long long)items * ((1 << 26) / 3);
  }
  // Takes the scales (and the sums, if there are any) to what covers every path
  // from j0 on of a list of `full`; or, where they do already and add() refused
  // paths [j0, j0 + 32), sums this chunk's paths beyond the largest range in
  // double, a monomial per lane, and returns true for their lanes.
  // item(j, e, v, z) gives a path's values.  more: other lists may follow; y,
  // of which only first powers are summed, then gets two bits above its
  // largest value.  After settle_mean of all paths added; called by the whole
  // warp.
  template <typename Item>
  __device__ __forceinline__ bool grow(FixWarp& ws, bool any, int j0, int full, bool more,
                                       const Item& item, double xK, double invTh) {
    const int lane = threadIdx.x & 31;
    const FixScale f = ws.scale;
    auto exponent = [](double q) { return (__double2hiint(q) >> 20) & 0x7ff; };
    // largest exponent fields, below the largest ranges'
    constexpr int kTopXW = 1023 + kFixTopXW, kTopY = 1023 + kFixTopY;
    int ex = 0, ew = 0, ey = 0;
#pragma unroll 1
    for (int j = j0 + lane; j < full; j += 32) {
      double e, v, z;
      item(j, e, v, z);
      const int tx = exponent(fma(e, xK, -1.0)), ty = exponent(z);
      const int tw = kV ? exponent(fma(v, invTh, -1.0)) : 0;
      ex = max(ex, tx < kTopXW ? tx : 0);
      ew = max(ew, tw < kTopXW ? tw : 0);
      ey = max(ey, ty < kTopY ? ty : 0);
    }
    ex = __reduce_max_sync(0xffffffffu, ex);
    if (kV) ew = __reduce_max_sync(0xffffffffu, ew);
    ey = __reduce_max_sync(0xffffffffu, ey);
    FixScale n = f;
    n.x = min(f.x, kFixTop - ex);
    if (kV) n.w = min(f.w, kFixTop - ew);
    n.y = ey > kFixTop - f.y ? kFixTop - ey - (more ? 2 : 0) : f.y;
    if (n.x != f.x || n.w != f.w || n.y != f.y) {
      if (any) rescale(f, n);
      __syncwarp();
      if (lane == 0) ws.scale = n;
      __syncwarp();
      return false;
    }
    double e, v, z;
    item(min(j0 + lane, full - 1), e, v, z);
    const double xd = fma(e, xK, -1.0), wd = kV ? fma(v, invTh, -1.0) : 0.0;
    const bool bad = j0 + lane < full && (exponent(xd) > kFixTop - f.x ||
                                          exponent(wd) > kFixTop - f.w ||
                                          exponent(z) > kFixTop - f.y);
    double p = 0.0;
    const uint32_t u = unit(lane < NU ? lane : 0);
    unsigned m = __ballot_sync(0xffffffffu, bad);
#pragma unroll 1
    while (m) {
      const int src = __ffs(m) - 1;
      m &= m - 1;
      const double xs = __shfl_sync(0xffffffffu, xd, src);
      const double wv = __shfl_sync(0xffffffffu, wd, src);
      const double ys = __shfl_sync(0xffffffffu, z, src);
      p += fix_monomial(u, xs, wv, ys);
    }
    if (lane < NU) ws.spill[lane] += p;
    if (lane == 0) ws.spilled = 1;
    __syncwarp();
    return bad;
  }
  // the units in slot order, in two parts small enough to be added over 32
  // lanes, a 2^56 + b: products in units of 2^28, plain sums of 2^-28
  __device__ __forceinline__ void units(long long (&a)[NU], long long (&b)[NU]) const {
    constexpr long long kMask = (1ll << 28) - 1;
#pragma unroll
    for (int i = 0; i < NU; ++i) {
      const long long h = is_plain(i) ? hh[i] : hh[i] + (hl[i] >> 28);
      a[i] = h >> 28;
      b[i] = (h & kMask) << 28 | (is_plain(i) ? 0 : hl[i] & kMask);
    }
  }
  // a unit added over the lanes; neg: x is negative (puts)
  __device__ __forceinline__ static double value(int u, long long a, long long b,
                                                 const FixScale& f, bool neg) {
    const uint32_t t = unit(u);
    const int E = (int)(t & 15u) * f.x + (int)((t >> 4) & 15u) * f.w +
                  (int)((t >> 8) & 15u) * f.y - kFixBits * (int)((t >> 12) & 15u) +
                  56 * (int)(t >> 16);
    const double v = fma((double)a, 0x1p56, (double)b) * exp2_int(28 - E);
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
