// Device-side building blocks of the fast-electron step (arXiv 2107.01723).
//
// Units inside the kernels are normalised so that FP32 keeps its range:
//   length in cells (dx), time in steps (dt), momentum u = p/(m_e c),
//   energy in m_e c^2, electric field as the per-step momentum kick
//   E_n = -e E dt/(m_e c), magnetic field as the per-step rotation
//   parameter B_n = -e B dt/m_e, current as J = sum w (u/gamma) S(x)
//   (electrons x beta per cell).  Every SI coefficient of the paper is folded
//   into these units once, in double precision, on the host (see api.cu).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace hpic {

constexpr uint32_t kDead = 0xFFFFFFFFu;  // id of an absorbed/escaped slot

// tally slots (device array of doubles); energies in m_e c^2 x weight
enum Tally {
  T_E_INJ = 0, T_N_INJ, T_W_FIELD, T_E_DRAG, T_E_XRAY, T_E_XRAY_ABOVE,
  T_E_ESC, T_E_REFLUX, T_E_OHMIC, T_N_INJECTED, T_N_ESC, T_N_REFLUX,
  T_N_REFLUX_ABS, T_N_CUT, T_N_EMIT, T_PSTEPS, T_N_NONFINITE,
  T_E_LIVE, T_E_BFIELD, T_COUNT
};

// device-resident counters
struct Counters {
  long long n;        // particle slots in use (live + dead until the next sort)
  long long step;     // step counter (Philox counter word 0)
  long long next_id;  // id of the next injected electron
  long long inj_cnt;  // electrons injected by the current step's injection
  unsigned int flags; // bit 0: capacity exceeded during injection
};

// Constants of one target, folded on the host.  R is the particle/field
// precision; temperature, resistivity and tallies are always double.
struct Consts {
  int nx, ny, nz;
  long long nvec, ncell;
  int nti, ntj, ntk;       // 4x4x4 cell tiles per axis (sort order)
  long long nkeys;         // nti*ntj*ntk*64 sort keys (the dead bin is nkeys)
  double cdt_dx;           // c dt / dx: cells per step at v = c
  double w;                // macro-electron weight (real electrons)
  // per element of the solid (a compound has up to kMaxSolids):
  // drag, Eq. (5): d_eps = sum K_ion/beta * bracket, L_I = ln(m_e c^2 / I_ex);
  // scatter, Eq. (B4): sigma^2 = sum K_sc gamma/u^3 ln(K_lg u)
  int n_solids;
  double K_ion[4], L_I[4], K_sc[4], K_lg[4];
  // heating of a compound, Eq. (A7): 1/C averaged with the weights ne_frac
  // (n_e of each element over the total), T' = T Tp_fac_s
  double ne_frac[4], Tp_fac_s[4];
  // bremsstrahlung optical depth: d_tau = K_tau u/eps G(k_min/eps)
  double K_tau, k_min, boost, inv_boost;
  // cut and reflux (Sec. II.A)
  double E_cut, eps_esc, du_reflux, sigma_dtheta;
  // photon tally
  int n_E, n_th;
  double tE_min, tE_max, inv_dlogE;   // n_E / ln(tE_max/tE_min)
  double ce_thr;
  int max_history;
  // inverse-CDF table
  int t_rows, t_cols;
  double t_inv_dlog;                  // (rows-1)/ln(E_max/k_min)
  // fields, Eqs. (A2)-(A3)
  double F_curl, F_j;
  // heating, Eqs. (A4)-(A8), SI
  double F_ohm, F_H, dx3, heat_den;
  double eta_num, A_hot, B_cold, eta_max, lambda1;
  double eta_hot_T, eta_cold_T;  // eta's two limits at T = 1 K (cold: 0 without lambda1)
  double eta_Tlo, eta_Thi;            // eta(T) is at its cap for eta_Tlo < T < eta_Thi (K)
  // F_sigma (App. B) = 1 + fs_q (ln T_i / 2 + fs_c), T_i in K
  double fs_q, fs_c;
  // e-i equilibration (App. A): rate_e = ei_a / (T_e m_i + T_i m_e)^(3/2)
  // (masses in u), rate_i = Z* rate_e
  double ei_a, ei_mi, ei_me, Zstar;
  // injection, Eq. (B1)
  double T_hot, spot_r, spot_y, spot_z, omc_cone;  // omc_cone = 1 - cos(cone)
  long long n_macro, n_inj_steps;
  // RNG
  uint32_t key0, key1, target_index;
  int physics;
  // Gaussian injection envelope (App. B): per_cell electrons in each of the
  // n_inj_cells cells of inj_cells while g = exp(-g_c (s + 1/2 - t_pk)^2) >=
  // g_min (s in steps); weight inj_unit sqrt(f g), mean energy T_hot sqrt(f g)
  int weighted;   // electrons carry their own weight
  int moore;      // Moore-scaling cap on the cone half-angle
  long long per_cell, n_inj_cells;
  double g_c, t_pk, g_min, inj_unit;
  const void *inj_cells;
};

// one injecting face cell: indices and sqrt(f(r)) at its centre
struct InjCell {
  int j, k;
  double sf;
};

enum {
  P_DRAG = 1, P_SCATTER = 2, P_BREM = 4, P_FIELDS = 8, P_FARADAY = 16, P_HEATING = 32,
  P_UNBOUNDED = 64, P_FSIGMA = 128, P_EI = 256
};

// ---------------------------------------------------------------- Philox
// Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11): ten rounds, each two
// 32x32 multiplies whose high halves are mixed with the other counter words
// and a Weyl-sequence key.
struct U4 { uint32_t a, b, c, d; };

__device__ __forceinline__ U4 philox10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                       uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t lo0 = 0xD2511F53u * c0, hi0 = __umulhi(0xD2511F53u, c0);
    const uint32_t lo1 = 0xCD9E8D57u * c2, hi1 = __umulhi(0xCD9E8D57u, c2);
    const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
    c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
    k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
  }
  return U4{c0, c1, c2, c3};
}

// open-interval uniform from the top 23 bits; exact in float and double
template <typename R>
__device__ __forceinline__ R unif(uint32_t x);
template <>
__device__ __forceinline__ float unif<float>(uint32_t x) {
  return ((float)(x >> 9) + 0.5f) * (1.0f / 8388608.0f);
}
template <>
__device__ __forceinline__ double unif<double>(uint32_t x) {  // 1 + m 2^-23 by its bits
  const uint32_t m = x >> 9;
  return __hiloint2double((int)(0x3ff00000u | (m >> 3)), (int)(m << 29)) - (1.0 - 1.0 / 16777216.0);
}

// ---------------------------------------------------------------- math wrappers
__device__ __forceinline__ float m_log(float x) { return logf(x); }
__device__ __forceinline__ double m_log(double x) { return log(x); }
// hardware log (absolute error ~5e-7) for terms of order 1-10 whose error
// budget allows it; exact log in double precision
__device__ __forceinline__ float m_flog(float x) { return __logf(x); }
__device__ __forceinline__ double m_flog(double x) { return log(x); }
__device__ __forceinline__ float m_exp(float x) { return expf(x); }
__device__ __forceinline__ double m_exp(double x) { return exp(x); }
__device__ __forceinline__ float m_expm1(float x) { return expm1f(x); }
__device__ __forceinline__ double m_expm1(double x) { return expm1(x); }
__device__ __forceinline__ float m_sqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double m_sqrt(double x) { return sqrt(x); }
__device__ __forceinline__ float m_atan2(float y, float x) { return atan2f(y, x); }
__device__ __forceinline__ double m_atan2(double y, double x) { return atan2(y, x); }
__device__ __forceinline__ void m_sincos(float x, float *s, float *c) { sincosf(x, s, c); }
__device__ __forceinline__ void m_sincos(double x, double *s, double *c) { sincos(x, s, c); }
// sin/cos of 2 pi u without rounding 2 pi u first
__device__ __forceinline__ void m_sincos2pi(float u, float *s, float *c) { sincospif(2.0f * u, s, c); }
__device__ __forceinline__ void m_sincos2pi(double u, double *s, double *c) { sincospi(2.0 * u, s, c); }
// Round-to-nearest square root and division.  The FP32 particle kernels are
// compiled with approximate division and square root; these wrappers keep
// IEEE rounding where the push converts between an electron's energy and
// its momentum (kinetic, u_of_eps, the rescale after drag or a photon) and
// where it builds the frame of a rotation, so that no systematic rounding
// bias enters an energy change that no tally records.
__device__ __forceinline__ float m_sqrt_rn(float x) { return __fsqrt_rn(x); }
__device__ __forceinline__ double m_sqrt_rn(double x) { return sqrt(x); }
__device__ __forceinline__ float m_div_rn(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ double m_div_rn(double a, double b) { return a / b; }
__device__ __forceinline__ float m_rsqrt_rn(float x) { return __frsqrt_rn(x); }
__device__ __forceinline__ double m_rsqrt_rn(double x) { return 1.0 / sqrt(x); }
// cos(2 pi u) for u in (0, 1): in FP32 from the hardware unit on the angle
// 2 pi (u - 1) for u > 1/2 (exact shift, |angle| <= pi, absolute error
// about 5e-7); exact cospi in FP64
__device__ __forceinline__ float m_fcos2pi(float u) {
  return __cosf(6.28318530717958647692f * (u > 0.5f ? u - 1.0f : u));
}
__device__ __forceinline__ double m_fcos2pi(double u) { return cospi(2.0 * u); }
__device__ __forceinline__ float m_floor(float x) { return floorf(x); }
__device__ __forceinline__ double m_floor(double x) { return floor(x); }

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

// FP64 reciprocals and roots for the per-electron arithmetic, of positive normal
// numbers well inside FP32's range (others take the plain expressions): from the
// FP32 estimate by one step of the series in the residual e (about 1e-7), to e^2:
// three operations for 1/x, five for x^(-1/2), of a unit that completes two per
// clock and SM.
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
  const double e = fma(-x * y, y, 1.0);
  return fma(y, e * fma(0.375, e, 0.5), y);
}
__device__ __forceinline__ double m_rsqrt_near(double x) { return m_rsqrt(x); }
__device__ __forceinline__ double m_sqrt_near(double x) { return x * m_rsqrt(x); }
__device__ __forceinline__ double m_div_near(double n, double d) { return n * m_rcp(d); }
// p = sqrt(x) and 1/p
__device__ __forceinline__ void m_sqrt_both(double x, double &p, double &inv) {
  inv = m_rsqrt(x);
  p = x * inv;
}

// ---- tables of the FP64 push
// Logarithms and the circle's functions cost 20 to 30 FP64 operations each in
// full generality.  By Tang's table-driven methods (ACM TOMS 15(2), 1989, and
// 16(4), 1990) the logarithm of a normal number takes ten, and sine and cosine
// of a 23-bit deviate of the circle, whose sector and rest are exact integers,
// thirteen.  All errors are of a few 1e-16 of 1.  With them, small-angle series
// and deviates and range tests by the bits the FP64 push of 1e6 electrons went
// from 1290 to 1062 us.
struct Fp64Tables {
  double c[256], l[256];    // c: a 24-bit reciprocal of 1 + (j + 1/2)/256; l = -ln c
  double cs[256], sn[256];  // of the angle 2 pi (j + 1/2)/256
  static constexpr double ln(double x) {  // x in [1/2, 1]
    const double y = (x - 1.0) / (x + 1.0), y2 = y * y;
    double s = 0.0;
    for (int k = 41; k >= 1; k -= 2) s = s * y2 + 1.0 / k;
    return 2.0 * y * s;
  }
  static constexpr double sine(double a) {  // |a| <= pi/4
    double s = 0.0;
    for (int k = 19; k >= 1; k -= 2) s = 1.0 - s * a * a / ((k + 1) * (k + 2));
    return a * s;
  }
  static constexpr double cosine(double a) {
    double s = 0.0;
    for (int k = 20; k >= 0; k -= 2) s = 1.0 - s * a * a / ((k + 1) * (k + 2));
    return s;
  }
  constexpr Fp64Tables() : c(), l(), cs(), sn() {
    constexpr double pi = 3.14159265358979323846;
    for (int j = 0; j < 256; ++j) {
      c[j] = (double)(float)(512.0 / (512.0 + 2 * j + 1));
      l[j] = -ln(c[j]);
      const int q = j / 64, r = j % 64;  // quadrant, and 2 r + 1 512ths of the circle in it
      const bool far = r >= 32;          // beyond pi/4: by the complement
      const double a = (far ? 127 - 2 * r : 2 * r + 1) * pi / 256.0;
      const double s = far ? cosine(a) : sine(a), o = far ? sine(a) : cosine(a);
      cs[j] = q == 0 ? o : (q == 1 ? -s : (q == 2 ? -o : s));
      sn[j] = q == 0 ? s : (q == 1 ? o : (q == 2 ? -s : -o));
    }
  }
};
static __device__ const Fp64Tables kFp64 = Fp64Tables();

__device__ __forceinline__ double table_log(double x) {
  const int hi = __double2hiint(x);
  if ((unsigned)(hi - 0x00100000) >= 0x7fe00000u) return log(x);  // not positive and normal
  const int j = (hi >> 12) & 255;
  const double m = __hiloint2double((hi & 0x000fffff) | 0x3ff00000, __double2loint(x));
  const double k = __hiloint2double(0x43300000, ((hi >> 20) - 1023) ^ (int)0x80000000) -
                   4503601774854144.0;  // by the bits of k + 2^52 + 2^31
  const double r = fma(m, __ldg(kFp64.c + j), -1.0);  // |r| < 2^-9 + 2^-23
  double q = fma(r, -1.0 / 6.0, 0.2);
  q = fma(r, q, -0.25);
  q = fma(r, q, 1.0 / 3.0);
  q = fma(r, q, -0.5);
  q = fma(r, q, 1.0);
  return fma(r, q, fma(k, 0.693147180559945309417232, __ldg(kFp64.l + j)));
}
// cos (and sin) of 2 pi u, u = (m + 1/2) 2^-23 the deviate of x
__device__ __forceinline__ void table_turn(uint32_t x, double &s, double &c) {
  const uint32_t m = x >> 9;
  const int j = (int)(m >> 15), f = 2 * (int)(m & 0x7fffu) - 32767;  // 2^-24ths from the middle
  const double a = (double)f * (3.14159265358979323846 / 8388608.0), t = a * a;
  const double sa = fma(a * t, fma(t, 1.0 / 120.0, -1.0 / 6.0), a);
  const double ca = fma(t, fma(t, fma(t, -1.0 / 720.0, 1.0 / 24.0), -0.5), 1.0);
  const double cj = __ldg(kFp64.cs + j), sj = __ldg(kFp64.sn + j);
  c = fma(cj, ca, -(sj * sa));
  s = fma(sj, ca, cj * sa);
}

// the push's logarithms: of a deviate, and the quick one
__device__ __forceinline__ double p_log(double x) { return table_log(x); }
__device__ __forceinline__ float p_flog(float x) { return m_flog(x); }
__device__ __forceinline__ double p_flog(double x) { return table_log(x); }
// sine and cosine of the deviate x of the circle; its cosine for a normal deviate
__device__ __forceinline__ void p_turn(uint32_t x, double &s, double &c) { table_turn(x, s, c); }
__device__ __forceinline__ void p_cos_turn(uint32_t x, double &c) {
  double s;
  table_turn(x, s, c);
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

// Sort key of cell (i, j, k): 4x4x4 tiles in x-fastest tile order, cells
// x-fastest inside a tile, so consecutive electrons share a compact box.
__host__ __device__ __forceinline__ uint32_t tile_key(int i, int j, int k, int nti, int ntj) {
  const uint32_t t = (uint32_t)(((k >> 2) * ntj + (j >> 2)) * nti + (i >> 2));
  return t * 64u + (uint32_t)(((k & 3) << 4) | ((j & 3) << 2) | (i & 3));
}

// kinetic energy (m_e c^2) of momentum u, without the gamma - 1 cancellation
template <typename R>
__device__ __forceinline__ R kinetic(R ux, R uy, R uz) {
  const R u2 = ux * ux + uy * uy + uz * uz;
  return m_div_rn(u2, R(1) + m_sqrt_rn(R(1) + u2));
}

// the same of u^2, with gamma: near-rounded
template <typename R>
__device__ __forceinline__ R kinetic_near(R u2, R &gam) {
  gam = m_sqrt_near(R(1) + u2);
  return m_div_near(u2, R(1) + gam);
}

// momentum |u| of kinetic energy e (m_e c^2)
template <typename R>
__device__ __forceinline__ R u_of_eps(R e) { return m_sqrt_rn(e * (e + R(2))); }

// Rotate unit d by polar angle (cos ct, sin st) at azimuth (cp, sp) in the
// orthonormal frame of Duff et al., "Building an orthonormal basis,
// revisited", JCGT 6(1), 2017.
template <typename R>
__device__ __forceinline__ void rotate(R &dx, R &dy, R &dz, R ct, R st, R cp, R sp) {
  const R sg = dz >= R(0) ? R(1) : R(-1);
  const R a = m_div_rn(R(-1), sg + dz);
  const R b = dx * dy * a;
  const R e1x = R(1) + sg * dx * dx * a, e1y = sg * b, e1z = -sg * dx;
  const R e2x = b, e2y = sg + dy * dy * a, e2z = -dy;
  const R px = e1x * cp + e2x * sp, py = e1y * cp + e2y * sp, pz = e1z * cp + e2z * sp;
  const R ox = dx * ct + px * st, oy = dy * ct + py * st, oz = dz * ct + pz * st;
  dx = ox; dy = oy; dz = oz;
}

// The same rotation with the sums over the frame's vectors carried out: with
// (qx, qy) = st (cp, sp), V = sg dx qx + dy qy and T = a V the rotated
// direction is (dx (ct + T) + qx, dy (ct + T) + sg qy, dz ct - V).
template <typename R>
__device__ __forceinline__ void rotate_near(R &dx, R &dy, R &dz, R ct, R st, R cp, R sp) {
  const bool up = dz >= R(0);
  const R qx = st * cp, qy = st * sp;
  const R V = (up ? dx : -dx) * qx + dy * qy;
  const R T = m_div_near(V, (up ? R(-1) : R(1)) - dz);
  const R k = ct + T;
  dx = dx * k + qx;
  dy = dy * k + (up ? qy : -qy);
  dz = dz * ct - V;
}

// none of them infinite or NaN: zero times each is zero (in FP64 by the
// exponents, off the FP64 unit)
__device__ __forceinline__ bool all_finite(float a, float b, float c, float d, float e, float f,
                                           float g) {
  return 0.0f * a + 0.0f * b + 0.0f * c + 0.0f * d + 0.0f * e + 0.0f * f + 0.0f * g == 0.0f;
}
__device__ __forceinline__ bool all_finite(double a, double b, double c, double d, double e,
                                           double f, double g) {
  const int m = 0x7ff00000;
  int x = max(__double2hiint(a) & m, __double2hiint(b) & m);
  x = max(max(x, __double2hiint(c) & m), __double2hiint(d) & m);
  x = max(max(x, __double2hiint(e) & m), max(__double2hiint(f) & m, __double2hiint(g) & m));
  return x != m;
}

// ---------------------------------------------------------------- reductions
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// A sum of reals with the accuracy of an FP64 sum of them that keeps off the
// FP64 unit where it can.  GB300 completes two FP64 operations per clock and
// SM, so one warp-wide FP64 add holds that unit for 16 clocks: the tree sums
// at the end of a kernel cost microseconds there.  An FP32 sum is carried as
// a pair (hi, lo) by Knuth's branch-free two-sum (TAOCP vol. 2, 4.2.2), 48
// bits wide, on the FP32 units.
template <typename R>
struct WideSum;
template <>
struct WideSum<float> {
  float hi = 0.0f, lo = 0.0f;
  __device__ __forceinline__ void add(float x) {
    const float s = __fadd_rn(hi, x), t = __fadd_rn(s, -hi);
    lo = __fadd_rn(lo, __fadd_rn(__fadd_rn(hi, -__fadd_rn(s, -t)), __fadd_rn(x, -t)));
    hi = s;
  }
  __device__ __forceinline__ void over_warp() {  // the total, in every lane
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float h = __shfl_xor_sync(0xffffffffu, hi, o), l = __shfl_xor_sync(0xffffffffu, lo, o);
      add(h);
      lo = __fadd_rn(lo, l);
    }
  }
  // (an infinite or NaN sum is hi's; lo is NaN then)
  __device__ __forceinline__ double value() const {
    return isfinite(hi) ? (double)hi + (double)lo : (double)hi;
  }
};
template <>
struct WideSum<double> {
  double v = 0.0;
  __device__ __forceinline__ void add(double x) { v += x; }
  __device__ __forceinline__ void over_warp() { v = warp_sum(v); }
  __device__ __forceinline__ double value() const { return v; }
};

// warp-aggregated atomic increment: lanes with equal keys share one atomic
__device__ __forceinline__ uint32_t agg_inc(uint32_t *ctr, uint32_t key) {
  const unsigned mask = __activemask();
  const unsigned peers = __match_any_sync(mask, key);
  const int lane = threadIdx.x & 31;
  const int leader = __ffs(peers) - 1;
  const uint32_t rank = __popc(peers & ((1u << lane) - 1u));
  uint32_t base = 0;
  if (lane == leader) base = atomicAdd(ctr + key, (uint32_t)__popc(peers));
  base = __shfl_sync(peers, base, leader);
  return base + rank;
}

// Sum `nq` per-thread values over the block and add them to dst[slot[q]].
// smem must hold nq * 32 doubles.  All threads of the block must call it.
template <int NQ>
__device__ __forceinline__ void block_flush(const double (&v)[NQ], const int (&slot)[NQ],
                                            double *dst, double *smem) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const double s = warp_sum(v[q]);
    if (lane == 0) smem[q * 32 + warp] = s;
  }
  __syncthreads();
  if (threadIdx.x < NQ) {
    double s = 0.0;
    for (int w = 0; w < nwarps; ++w) s += smem[threadIdx.x * 32 + w];
    if (s != 0.0) atomicAdd(dst + slot[threadIdx.x], s);
  }
  __syncthreads();
}

}  // namespace hpic
