// Arithmetic that keeps off GB300's FP64 unit where it can, or asks little of it:
// conversions, reciprocals and roots, logarithms and the circle's functions, sums.
// Plain functions of numbers, apart from the kernels that use them.
#pragma once

#include <cstdint>

namespace hpic {

// ---------------------------------------------------------------- FP64 off the FP64 unit
// GB300 completes two FP64 operations per clock and SM, conversions from and
// to FP64 included, so a warp-wide one holds the SM's FP64 unit for 16 clocks
// where an integer instruction takes a fraction of one.  Conversions of
// positive numbers well inside FP32's range are therefore done on the bits.
// in_range: a double in [2^-40, 2^60); zero, negative, infinite and NaN
// values are not (callers take the plain expressions then).
__device__ __forceinline__ bool in_range(double x) {
  return (unsigned)(__double2hiint(x) - 0x3d700000) < 0x06400000u;
}
// (float)x of an in_range x: round to nearest, ties to even
__device__ __forceinline__ float narrow(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned m = __funnelshift_l(lo, hi, 3) - 0xc0000000u;  // 29 bits cut, exponent rebiased
  return __uint_as_float(m + (((lo << 3) | (m & 1u)) > 0x80000000u ? 1u : 0u));
}
// (double)x of a positive normal x
__device__ __forceinline__ double widen(float x) {
  const unsigned b = __float_as_uint(x);
  return __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
}
// the smaller of two positive numbers, by their bits
__device__ __forceinline__ double min_positive(double a, double b) {
  return __double_as_longlong(a) < __double_as_longlong(b) ? a : b;
}

// FP64 reciprocals, roots and quotients for the per-electron arithmetic, of positive
// normal numbers well inside FP32's range (others take the plain expressions): from
// the FP32 estimate by one step of the series in the residual e (about 1e-7), to e^2:
// three operations for 1/x, six for x^(-1/2), whose residual is exact but for one
// rounding as the square of 24 bits fits.  Roots and quotients end with a step on
// their own residual, so that all are rounded but for rare last places (at most
// 0.501 of one off), as the library's are.
__device__ __forceinline__ bool fp32_range(double x) {  // [2^-100, 2^100)
  return (unsigned)(__double2hiint(x) - 0x39b00000) < 0x0c800000u;
}
__device__ __forceinline__ double m_rcp(double x) {
  if (!fp32_range(x)) return 1.0 / x;
  const double y = widen(__fdividef(1.0f, narrow(x)));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ double m_rsqrt(double x) {
  if (!fp32_range(x)) return rsqrt(x);
  const double y = widen(rsqrtf(narrow(x)));
  const double e = fma(-x, y * y, 1.0);
  return fma(y, e * fma(0.375, e, 0.5), y);
}
// sqrt(x), inv its reciprocal; half of inv by its exponent
__device__ __forceinline__ double root_of(double x, double inv) {
  const double s = x * inv;
  const double h = __hiloint2double(__double2hiint(inv) - 0x00100000, __double2loint(inv));
  return fma(fma(-s, s, x), h, s);
}
__device__ __forceinline__ double m_sqrt_near(double x) { return root_of(x, m_rsqrt(x)); }
// n/d, inv the reciprocal of d
__device__ __forceinline__ double quotient_of(double n, double d, double inv) {
  const double q = n * inv;
  return fma(fma(-q, d, n), inv, q);
}
__device__ __forceinline__ double m_div_near(double n, double d) {
  return quotient_of(n, d, m_rcp(d));
}
// p = sqrt(x) and 1/p
__device__ __forceinline__ void m_sqrt_both(double x, double &p, double &inv) {
  inv = m_rsqrt(x);
  p = root_of(x, inv);
}

// ---- tables of the FP64 push
// Logarithms and the circle's functions cost 20 to 30 FP64 operations each in
// full generality.  By Tang's table-driven methods (ACM TOMS 15(2), 1989, and
// 16(4), 1990) the logarithm of a normal number takes fifteen, and sine and cosine
// of a 23-bit deviate of the circle, whose sector and rest are exact integers,
// seventeen.  The tables' rows lie so that where a result passes zero (ln 1, the
// axes of the circle) its row is exactly zero and the short series alone makes it,
// so that the errors are in proportion to the result, however small that is:
// in its last places the logarithm of a deviate is 0.50 off at most (the library's
// 0.53), of numbers near 1 0.70 (0.50), 0.25 on average like the library's; sine
// and cosine 1.41 (sincospi 1.43), 0.25 on average (0.30).  (The FP64 push of 1e6
// electrons takes 1150 us with them; with the library's logarithm and circle functions
// it took 1290 although its roots and quotients were rougher.)
//
// Pairs of doubles for the tables, worked out by the compiler: sums and products
// by Knuth's and Dekker's error-free forms (Dekker, "A floating-point technique
// for extending the available precision", Numer. Math. 18, 1971).
struct Double2 {
  double h, l;
};
constexpr Double2 pair_sum(double a, double b) {
  const double s = a + b, t = s - a;
  return Double2{s, (a - (s - t)) + (b - t)};
}
constexpr Double2 pair_product(double a, double b) {
  const double p = a * b, ca = 134217729.0 * a, cb = 134217729.0 * b;
  const double ah = ca - (ca - a), al = a - ah, bh = cb - (cb - b), bl = b - bh;
  return Double2{p, ((ah * bh - p) + ah * bl + al * bh) + al * bl};
}
constexpr Double2 add(Double2 a, Double2 b) {
  const Double2 s = pair_sum(a.h, b.h);
  return pair_sum(s.h, s.l + (a.l + b.l));
}
constexpr Double2 mul(Double2 a, Double2 b) {
  const Double2 p = pair_product(a.h, b.h);
  return pair_sum(p.h, p.l + (a.h * b.l + a.l * b.h));
}
constexpr Double2 over(Double2 a, double d) {
  const double q = a.h / d;
  const Double2 p = pair_product(q, d);
  return pair_sum(q, ((a.h - p.h) - p.l + a.l) / d);
}

// ln x of x in [1/2, 2] of 24 bits, 2 artanh((x - 1)/(x + 1)), as a multiple of
// 2^-42 (2^10 + 2^9 has its last place there) and the rest
constexpr Double2 ln_split(double x) {
  const Double2 y = over(Double2{x - 1.0, 0.0}, x + 1.0), y2 = mul(y, y);
  Double2 s{0.0, 0.0};
  for (int k = 67; k >= 1; k -= 2) s = add(mul(s, y2), over(Double2{1.0, 0.0}, (double)k));
  const Double2 v = mul(Double2{2.0 * y.h, 2.0 * y.l}, s);
  const double hi = (v.h + 1536.0) - 1536.0;
  return Double2{hi, (v.h - hi) + v.l};
}
constexpr Double2 kLn2 = ln_split(2.0);
constexpr double kLn2Hi = kLn2.h, kLn2Lo = kLn2.l;

struct Fp64Tables {
  // c: a 24-bit reciprocal of m = 1 + j/256 (1 for j = 0); hi + lo = -ln c, from
  // row kHalf on -ln(2 c), hi a multiple of 2^-42
  struct alignas(32) Log {
    double c, hi, lo, pad;
  } log[256];
  // cosine and sine of 2 pi j/256 in two parts
  struct alignas(32) Turn {
    double c, c_lo, s, s_lo;
  } turn[256];
  static constexpr int kHalf = 106;  // from here on m/2 lies nearer to 1 than m (m > sqrt 2)
  static constexpr Double2 sine(Double2 a) {  // |a| <= pi/4
    const Double2 t = mul(a, a);
    Double2 s{0.0, 0.0};
    for (int k = 25; k >= 1; k -= 2) {
      const Double2 q = over(mul(s, t), (double)((k + 1) * (k + 2)));
      s = add(Double2{1.0, 0.0}, Double2{-q.h, -q.l});
    }
    return mul(a, s);
  }
  static constexpr Double2 cosine(Double2 a) {
    const Double2 t = mul(a, a);
    Double2 s{0.0, 0.0};
    for (int k = 26; k >= 0; k -= 2) {
      const Double2 q = over(mul(s, t), (double)((k + 1) * (k + 2)));
      s = add(Double2{1.0, 0.0}, Double2{-q.h, -q.l});
    }
    return s;
  }
  constexpr Fp64Tables() : log(), turn() {
    constexpr Double2 pi{3.141592653589793116, 1.2246467991473532e-16};
    for (int j = 0; j < 256; ++j) {
      const double c = (double)(float)(256.0 / (256.0 + j));
      const Double2 l = ln_split((j < kHalf ? 1.0 : 2.0) * c);
      log[j] = Log{c, -l.h, -l.l, 0.0};
      const int q = j / 64, r = j % 64;  // quadrant, and 256ths of the circle in it
      const bool far = r > 32;           // beyond pi/4: by the complement
      const Double2 a = mul(pi, Double2{(far ? 64 - r : r) / 128.0, 0.0});
      const Double2 s = far ? cosine(a) : sine(a), o = far ? sine(a) : cosine(a);
      const double cs = q == 0 || q == 3 ? 1.0 : -1.0, ss = q < 2 ? 1.0 : -1.0;
      const Double2 x = q % 2 ? s : o, y = q % 2 ? o : s;
      turn[j] = Turn{cs * x.h, cs * x.l, ss * y.h, ss * y.l};
    }
  }
};
static __device__ const Fp64Tables kFp64 = Fp64Tables();

// x = 2^k m, m in [1 - 2^-10, 2 - 2^-9) in row j; r = m c - 1, |r| < 2^-9 + 2^-24;
// ln x = k ln 2 - ln c + ln(1 + r), with ln(1 + r) = r - r^2/2 + ... to r^6 (the
// next term below 2^-65), where rows from kHalf on count to k + 1
__device__ __forceinline__ double table_log(double x) {
  const int xh = __double2hiint(x);
  if ((unsigned)(xh - 0x00100000) >= 0x7fe00000u) return log(x);  // not positive and normal
  const int up = xh + 0x800;                                      // half a row on
  const int j = (up >> 12) & 255;
  const double m = __hiloint2double(xh - (up & 0x7ff00000) + 0x3ff00000, __double2loint(x));
  const int n = ((up + ((256 - Fp64Tables::kHalf) << 12)) >> 20) - 1023;
  const double k = __hiloint2double(0x43300000, n ^ (int)0x80000000) -
                   4503601774854144.0;  // by the bits of n + 2^52 + 2^31
  const double2 *row = reinterpret_cast<const double2 *>(kFp64.log + j);
  const double2 ch = __ldg(row);
  const double r = fma(m, ch.x, -1.0), r2 = r * r;
  double q = fma(r, -1.0 / 6.0, 0.2);
  q = fma(r, q, -0.25);
  q = fma(r, q, 1.0 / 3.0);
  q = fma(r, q, -0.5);
  const double base = fma(k, kLn2Hi, ch.y);  // exact
  const double rest = fma(k, kLn2Lo, __ldg(row + 1).x);
  const double sum = base + r, left = r - (sum - base);  // |r| < |base|, or base is 0
  return sum + (left + fma(r2, q, rest));
}
// The same of a positive normal x for results kept in FP32: ln x = base + rest within
// 2^-33, the short series and the last 29 bits of x in FP32 (two FP64 operations, and
// what the sum takes)
__device__ __forceinline__ void log_parts(double x, double &base, float &rest) {
  const int xh = __double2hiint(x), up = xh + 0x800, j = (up >> 12) & 255;
  const int mh = xh - (up & 0x7ff00000) + 0x3ff00000;  // of m
  const int n = ((up + ((256 - Fp64Tables::kHalf) << 12)) >> 20) - 1023;
  const double k = __hiloint2double(0x43300000, n ^ (int)0x80000000) - 4503601774854144.0;
  const double2 *row = reinterpret_cast<const double2 *>(kFp64.log + j);
  const double2 ch = __ldg(row);
  const unsigned lo = (unsigned)__double2loint(x);
  // m in 24 bits, cut, and what was cut; c, which has 24 bits, by its own bits
  const float a = __uint_as_float(__funnelshift_l(lo, (unsigned)mh, 3) - 0xc0000000u);
  const float b = (float)(lo & 0x1fffffffu) * (mh < 0x3ff00000 ? 0x1p-53f : 0x1p-52f);
  const float c = __uint_as_float(
      __funnelshift_l((unsigned)__double2loint(ch.x), (unsigned)__double2hiint(ch.x), 3) - 0xc0000000u);
  const float p = __fmul_rn(a, c), r = __fadd_rn(p, -1.0f);  // exact, p being near 1
  float q = fmaf(r, -0.25f, 1.0f / 3.0f);
  q = fmaf(r, q, -0.5f);
  const float s = fmaf(b, c, fmaf(a, c, -p));  // what r lacks: s/(1 + r) of the logarithm
  rest = __fadd_rn(r, fmaf(__fmul_rn(r, r), q, fmaf(-s, r, s)));
  base = fma(k, 0.693147180559945309417232, ch.y);  // (the rows' lo: below 2^-43)
}
// sine and cosine of 2 pi u, u = (n + 1/2) 2^-23 the deviate of x: 2 n + 1 2^-24ths
// of the circle, f of them from the axis of row j
__device__ __forceinline__ void table_turn(uint32_t x, double &s, double &c) {
  const uint32_t u = 2u * (x >> 9) + 1u, row = (u + 0x8000u) >> 16;
  const int j = (int)(row & 255u), f = (int)(u - (row << 16));
  const double a = (double)f * (3.14159265358979323846 / 8388608.0), t = a * a;
  const double sa = fma(a * t, fma(t, fma(t, -1.0 / 5040.0, 1.0 / 120.0), -1.0 / 6.0), a);
  const double ca = t * fma(t, fma(t, -1.0 / 720.0, 1.0 / 24.0), -0.5);  // cos a - 1
  const double2 *at = reinterpret_cast<const double2 *>(kFp64.turn + j);
  const double2 cj = __ldg(at), sj = __ldg(at + 1);
  c = cj.x + fma(cj.x, ca, fma(-sj.x, sa, cj.y));
  s = sj.x + fma(sj.x, ca, fma(cj.x, sa, sj.y));
}

// sine and cosine of a deflection: by their series up to |x| = 1/2 (to x^15 and
// x^16: below 1e-18), where nearly all are
__device__ __forceinline__ void m_sincos_small(double x, double *s, double *c) {
  if ((__double2hiint(x) & 0x7fffffff) < 0x3fe00000) {
    const double t = x * x;
    double p = fma(t, -1.0 / 1307674368000.0, 1.0 / 6227020800.0);
    p = fma(t, p, -1.0 / 39916800.0);
    p = fma(t, p, 1.0 / 362880.0);
    p = fma(t, p, -1.0 / 5040.0);
    p = fma(t, p, 1.0 / 120.0);
    p = fma(t, p, -1.0 / 6.0);
    *s = fma(x * t, p, x);
    double q = fma(t, 1.0 / 20922789888000.0, -1.0 / 87178291200.0);
    q = fma(t, q, 1.0 / 479001600.0);
    q = fma(t, q, -1.0 / 3628800.0);
    q = fma(t, q, 1.0 / 40320.0);
    q = fma(t, q, -1.0 / 720.0);
    q = fma(t, q, 1.0 / 24.0);
    q = fma(t, q, -0.5);
    *c = fma(t, q, 1.0);
  } else {
    sincos(x, s, c);
  }
}

// Rotate unit d by polar angle (cos ct, sin st) at azimuth (cp, sp) in the frame of
// Duff et al. (rotate() of common.cuh), with the sums over the frame's vectors carried
// out: with (qx, qy) = st (cp, sp), sg = +1 for dz >= 0 and else -1, V = sg dx qx + dy qy
// and T = -sg V/(1 + |dz|) the rotated direction is (dx (ct + T) + qx, dy (ct + T) +
// sg qy, dz ct - V).  The divisor lies in [1, 2] for both signs of dz, where the quick
// reciprocal serves every lane.
__device__ __forceinline__ void rotate_near(double &dx, double &dy, double &dz, double ct,
                                            double st, double cp, double sp) {
  const bool up = dz >= 0.0;
  const double qx = st * cp, qy = st * sp;
  const double V = (up ? dx : -dx) * qx + dy * qy;
  const double T = (up ? -V : V) * m_rcp(1.0 + fabs(dz));
  const double k = ct + T;
  dx = dx * k + qx;
  dy = dy * k + (up ? qy : -qy);
  dz = dz * ct - V;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// A sum of reals with the accuracy of an FP64 sum of them that keeps off the
// FP64 unit where it can.  GB300 completes two FP64 operations per clock and
// SM, so one warp-wide FP64 add holds that unit for 16 clocks: the tree sums
// at the end of a kernel cost microseconds there.  An FP32 sum is carried in
// three parts by Knuth's branch-free two-sum (TAOCP vol. 2, 4.2.2), 72 bits
// wide, on the FP32 units; what is rounded is the last part and, in value(),
// the result.
template <typename R>
struct WideSum;
template <>
struct WideSum<float> {
  float hi, mid, lo;  // all zero to begin with
  // a + x in a, and what that rounding left
  static __device__ __forceinline__ float into(float &a, float x) {
    const float s = __fadd_rn(a, x), t = __fadd_rn(s, -a);
    const float left = __fadd_rn(__fadd_rn(a, -__fadd_rn(s, -t)), __fadd_rn(x, -t));
    a = s;
    return left;
  }
  __device__ __forceinline__ void add(float x) {
    lo = __fadd_rn(lo, into(mid, into(hi, x)));
  }
  __device__ __forceinline__ void over_lanes(int first) {  // of 2 first lanes, in every lane
#pragma unroll
    for (int o = first; o > 0; o >>= 1) {
      const float h = __shfl_xor_sync(0xffffffffu, hi, o), m = __shfl_xor_sync(0xffffffffu, mid, o);
      const float l = __shfl_xor_sync(0xffffffffu, lo, o);
      add(h);
      lo = __fadd_rn(__fadd_rn(lo, l), into(mid, m));
    }
  }
  __device__ __forceinline__ void over_warp() { over_lanes(16); }  // the total, in every lane
  // (an infinite or NaN sum is hi's; the other parts are NaN then)
  __device__ __forceinline__ double value() const {
    return isfinite(hi) ? (double)hi + ((double)mid + (double)lo) : (double)hi;
  }
};
template <>
struct WideSum<double> {
  double v;
  __device__ __forceinline__ void add(double x) { v += x; }
  __device__ __forceinline__ void over_lanes(int first) {
#pragma unroll
    for (int o = first; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  }
  __device__ __forceinline__ void over_warp() { over_lanes(16); }
  __device__ __forceinline__ double value() const { return v; }
};

// The warp's sums of two values of each lane, of a in lanes 0 to 15 and of b in lanes
// 16 to 31: a half each, after each half has sent the other its share.
template <typename R>
__device__ __forceinline__ WideSum<R> warp_sums(R a, R b) {
  const bool upper = (threadIdx.x & 16) != 0;
  WideSum<R> s{};
  s.add(upper ? b : a);
  s.add(__shfl_xor_sync(0xffffffffu, upper ? a : b, 16));
  s.over_lanes(8);
  return s;
}

}  // namespace hpic
