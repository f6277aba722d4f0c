// Per-node device code of the field solve and heating (arXiv 2107.01723,
// Eqs. (A2)-(A8)), shared by the single-target and the batched kernels.
#pragma once

#include "kernels.h"

namespace hpic {

// (i, j, k) of node q.  The two divisions by the row and plane lengths go
// through multiplications by rounded-up reciprocals (Granlund & Montgomery,
// "Division by invariant integers using multiplication", PLDI 1994): exact for
// the node counts here, below 2^29 (checked at creation).
template <typename R>
__device__ __forceinline__ void node_of(const FieldK<R> &K, unsigned q, int &i, int &j, int &k) {
  const unsigned kk = K.by_sz.quotient(q), r = q - kk * (unsigned)K.sz;
  const unsigned jj = K.by_sy.quotient(r);
  k = (int)kk;
  j = (int)jj;
  i = (int)(r - jj * (unsigned)K.sy);
}

// Element at a byte offset.  Grids stay below 2^32 bytes per array (at most
// 2^27 - 2 cells, so 3^3/2^3 as many nodes), and a 32-bit offset to a base that
// is the same for all lanes takes one instruction less per access than a
// 64-bit index: these kernels issue some thirty accesses per node.
template <typename T>
__device__ __forceinline__ T &at(T *p, unsigned off) {
  return *reinterpret_cast<T *>(reinterpret_cast<char *>(p) + off);
}
template <typename T>
__device__ __forceinline__ T at(const T *p, unsigned off) {
  return *reinterpret_cast<const T *>(reinterpret_cast<const char *>(p) + off);
}

// r^2 of a positive normal r, exactly, in integers (24 x 24 bits)
__device__ __forceinline__ double exact_square(float r) {
  const unsigned b = __float_as_uint(r), m = (b & 0x007fffffu) | 0x00800000u;
  const unsigned long long p = (unsigned long long)m * m;  // in [2^46, 2^48)
  const unsigned top = (unsigned)(p >> 47);
  const unsigned long long frac = p << (6 - top);  // leading one at bit 52
  const unsigned exp = 2u * (b >> 23) + 769u + top;
  return __longlong_as_double((long long)((frac & 0x000fffffffffffffull) |
                                          ((unsigned long long)exp << 52)));
}
// c x^(-3/2) of an in_range x: r, an FP32 estimate of x^(-1/2), then c r^3
// (1 + e)^(-3/2) with e = x r^2 - 1 (about 1e-7) to second order, the next term
// being below 1e-19: six FP64 operations, where rsqrt(x) cubed takes about
// fifteen
__device__ __forceinline__ double times_pow_m32(double c, double x) {
  const float r = rsqrtf(narrow(x));
  const double r2 = exact_square(r), e = fma(x, r2, -1.0);
  const double s = c * r2 * widen(r);
  return fma(s, e * fma(1.875, e, -1.5), s);
}

// ---------------------------------------------------------------- E, Eq. (A2)
// E on the three edges owned by node q (tangential E = 0 on the walls)
template <typename R>
__device__ __forceinline__ void efield_node(const FieldK<R> &K, const GView<R> &g, unsigned node) {
  constexpr unsigned Z = sizeof(R);
  const int nx = K.nx, ny = K.ny, nz = K.nz;
  const unsigned q = node * Z, sy = K.sy * Z, sz = K.sz * Z;
  const unsigned cy = nx * Z, cz = nx * ny * Z;
  const R Fc = K.F_curl, Fj = K.F_j;
  const R *Bx = g.B[0], *By = g.B[1], *Bz = g.B[2], *eta = g.eta_r;
  int i, j, k;
  node_of(K, node, i, j, k);
  R ex = 0, ey = 0, ez = 0;
  const unsigned c = (unsigned)(i + nx * (j + ny * k)) * Z;  // cell (i, j, k)
  const bool in_i = i >= 1 && i < nx, in_j = j >= 1 && j < ny, in_k = k >= 1 && k < nz;
  if (in_i && in_j && in_k) {
    // away from the walls all three edges share their loads, which are issued
    // together: the kernel lives on memory latency
    const R bx = at(Bx, q), bxy = at(Bx, q - sy), bxz = at(Bx, q - sz);
    const R by = at(By, q), byx = at(By, q - Z), byz = at(By, q - sz);
    const R bz = at(Bz, q), bzx = at(Bz, q - Z), bzy = at(Bz, q - sy);
    const R jx = at<const R>(g.J[0], q), jy = at<const R>(g.J[1], q), jz = at<const R>(g.J[2], q);
    const R e0 = at(eta, c), ei = at(eta, c - Z), ej = at(eta, c - cy), ek = at(eta, c - cz);
    const R eij = at(eta, c - Z - cy), eik = at(eta, c - Z - cz), ejk = at(eta, c - cy - cz);
    ex = R(0.25) * (ejk + ek + ej + e0) * (Fc * ((bz - bzy) - (by - byz)) - Fj * jx);
    ey = R(0.25) * (eik + ek + ei + e0) * (Fc * ((bx - bxz) - (bz - bzx)) - Fj * jy);
    ez = R(0.25) * (eij + ej + ei + e0) * (Fc * ((by - byx) - (bx - bxy)) - Fj * jz);
  } else {
    if (i < nx && in_j && in_k) {
      const R curl = (at(Bz, q) - at(Bz, q - sy)) - (at(By, q) - at(By, q - sz));
      const R e = R(0.25) * (at(eta, c - cy - cz) + at(eta, c - cz) + at(eta, c - cy) + at(eta, c));
      ex = e * (Fc * curl - Fj * at<const R>(g.J[0], q));
    }
    if (j < ny && in_i && in_k) {
      const R curl = (at(Bx, q) - at(Bx, q - sz)) - (at(Bz, q) - at(Bz, q - Z));
      const R e = R(0.25) * (at(eta, c - Z - cz) + at(eta, c - cz) + at(eta, c - Z) + at(eta, c));
      ey = e * (Fc * curl - Fj * at<const R>(g.J[1], q));
    }
    if (k < nz && in_i && in_j) {
      const R curl = (at(By, q) - at(By, q - Z)) - (at(Bx, q) - at(Bx, q - sy));
      const R e = R(0.25) * (at(eta, c - Z - cy) + at(eta, c - cy) + at(eta, c - Z) + at(eta, c));
      ez = e * (Fc * curl - Fj * at<const R>(g.J[2], q));
    }
  }
  at(g.E[0], q) = ex;
  at(g.E[1], q) = ey;
  at(g.E[2], q) = ez;
}

// rho / (Z n_i k_B C(T)) with the heat capacity of Eq. (A8),
// C = 0.3 + 1.2 T'(2.2 + T')/(1.1 + T')^2, T' = (k_B T/e) Z^(-4/3), brought
// over one denominator (one division per cell), in the field precision: in
// the FP32-mixed path the increment carries a relative error of ~1e-7 of
// itself; T itself accumulates in FP64
template <typename R>
__device__ __forceinline__ R heat_increment(const FieldK<R> &K, R T, R rho) {
  if (K.n_solids == 1) {
    const R tp = T * K.Tp_fac[0], D = R(1.1) + tp;
    const R D2 = D * D;
    return rho * D2 / (K.heat_den * (R(0.3) * D2 + R(1.2) * tp * (R(2.2) + tp)));
  }
  // a compound: heat_den = k_B sum Z n_i, 1/C averaged with the n_e weights
  R inv_c = R(0);
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    if (s >= K.n_solids) break;
    const R tp = T * K.Tp_fac[s], D = R(1.1) + tp;
    const R D2 = D * D;
    inv_c += K.ne_frac[s] * D2 / (R(0.3) * D2 + R(1.2) * tp * (R(2.2) + tp));
  }
  return rho * inv_c / K.heat_den;
}

// reduced Lee-More resistivity, Eqs. (A4)-(A6), capped; inside the band
// where the cap holds, the cap itself.  eta_num / max(tau_hot, tau_cold) is
// the smaller of eta_num/(A_hot (kT)^1.5) and eta_num sqrt(kT)/B_cold.
// In range, both come from T^(-3/2) (sqrt(T) = T^2 T^(-3/2)) without a division,
// a root or a compare on the FP64 unit (Tf = (float)T tells the band, whose
// float ends lie inside the exact one, where the formula gives the cap too).
// A heated cell took 29 FP64 instructions, the SM's FP64 unit a warp-wide one
// in 19 clocks: 128 us for 128^3 cells, now 8 to 9 and 51 us; a batch of 7.9e6
// cells (each target's constants in shared memory, its Ohmic sums made in the
// warp) 542 -> 133 us.
__device__ __forceinline__ double resistivity(const FieldCommon &K, double T, float Tf) {
  if (Tf > K.eta_Tlo && Tf < K.eta_Thi) return K.eta_max;
  double eta = times_pow_m32(K.eta_hot, T);
  if (K.cold) eta = min_positive(eta, times_pow_m32(K.eta_cold, T) * (T * T));
  return min_positive(eta, K.eta_max);
}
// the same for any T
inline __device__ __noinline__ double resistivity_any(double eta_hot, double eta_cold, double eta_max,
                                               double T) {
  const double r = rsqrt(T);
  double eta = eta_hot * (r * r * r);
  if (eta_cold > 0.0) {
    const double ec = eta_cold * (T * r);
    eta = ec < eta ? ec : eta;
  }
  return eta < eta_max ? eta : eta_max;
}

// F_sigma (App. B) of the ion temperature; for the FP32 push within 2^-33 (times fs_q,
// below 1/4) before it is rounded to FP32: the rounded value but for one in a thousand
template <typename R>
__device__ __forceinline__ R fsigma(const FieldCommon &K, double Ti) {
  double log_Ti;
  if (sizeof(R) == 4 && in_range(Ti)) {
    float rest;
    log_parts(Ti, log_Ti, rest);
    log_Ti += (double)rest;
  } else {
    log_Ti = table_log(Ti);
  }
  return R(fma(K.fs_q, fma(0.5, log_Ti, K.fs_c), 1.0));
}

// ---------------------------------------------------------------- B, Eq. (A3), and heating
// Faraday on the faces owned by node q, then heating of cell q; returns the cell's
// Ohmic energy density (J/m^3)
template <typename R>
__device__ __forceinline__ R bheat_node(const FieldK<R> &K, const GView<R> &g, unsigned node) {
  constexpr unsigned Z = sizeof(R), D = sizeof(double);
  const int nx = K.nx, ny = K.ny, nz = K.nz;
  const unsigned q = node * Z, sy = K.sy * Z, sz = K.sz * Z;
  const R cdt = K.cdt;
  const R *Ex = g.E[0], *Ey = g.E[1], *Ez = g.E[2];
  int i, j, k;
  node_of(K, node, i, j, k);
  const bool in_i = i < nx, in_j = j < ny, in_k = k < nz, cell = in_i && in_j && in_k;
  const unsigned c = (unsigned)(i + nx * (j + ny * k));
  const bool faraday = (K.physics & P_FARADAY) != 0, ohmic = (K.physics & P_FIELDS) != 0;
  // everything a node reads but T and eta, before its first store: one round
  // trip to memory, where loads between the stores of B made four
  double Hc = 0.0;
  R jx = 0, jy = 0, jz = 0;
  if (cell) {
    Hc = at<const double>(g.H, c * D);
    if (ohmic) {
      const R *Jx = g.J[0], *Jy = g.J[1], *Jz = g.J[2];
      jx = at(Jx, q) + at(Jx, q + sy) + at(Jx, q + sz) + at(Jx, q + sy + sz);
      jy = at(Jy, q) + at(Jy, q + Z) + at(Jy, q + sz) + at(Jy, q + Z + sz);
      jz = at(Jz, q) + at(Jz, q + Z) + at(Jz, q + sy) + at(Jz, q + Z + sy);
    }
  }
  if (faraday) {
    if (cell) {
      const R ex = at(Ex, q), exy = at(Ex, q + sy), exz = at(Ex, q + sz);
      const R ey = at(Ey, q), eyx = at(Ey, q + Z), eyz = at(Ey, q + sz);
      const R ez = at(Ez, q), ezx = at(Ez, q + Z), ezy = at(Ez, q + sy);
      const R bx = at<const R>(g.B[0], q), by = at<const R>(g.B[1], q), bz = at<const R>(g.B[2], q);
      at(g.B[0], q) = bx - cdt * ((ezy - ez) - (eyz - ey));
      at(g.B[1], q) = by - cdt * ((exz - ex) - (ezx - ez));
      at(g.B[2], q) = bz - cdt * ((eyx - ey) - (exy - ex));
    } else {
      if (in_j && in_k) at(g.B[0], q) -= cdt * ((at(Ez, q + sy) - at(Ez, q)) - (at(Ey, q + sz) - at(Ey, q)));
      if (in_i && in_k) at(g.B[1], q) -= cdt * ((at(Ex, q + sz) - at(Ex, q)) - (at(Ez, q + Z) - at(Ez, q)));
      if (in_i && in_j) at(g.B[2], q) -= cdt * ((at(Ey, q + Z) - at(Ey, q)) - (at(Ex, q + sy) - at(Ex, q)));
    }
  }
  if (cell) {
    // cell-centred mean of the edge current in the field precision
    jx *= R(0.25);
    jy *= R(0.25);
    jz *= R(0.25);
    const R jb2 = jx * jx + jy * jy + jz * jz;
    // a cell without drag heat or current keeps T and eta (and adds no
    // Ohmic energy) unless e-i equilibration moves it
    const bool no_heat = (__double_as_longlong(Hc) << 1) == 0;  // +0 or -0
    if (no_heat && jb2 == R(0) && !(K.physics & P_EI)) return R(0);
    double Te = at<const double>(g.T, c * D);
    bool changed = false;
    const R ro = at<const R>(g.eta_r, c * Z) * K.F_ohm * jb2;
    R rho = ro;
    if (!no_heat) {
      const double h = Hc * K.F_H;
      if constexpr (sizeof(R) == 4) rho += in_range(h) ? narrow(h) : (float)h;
      else rho += h;
    }
    if ((K.physics & P_HEATING) && rho != R(0)) {  // rho = 0 leaves T as it is
      if constexpr (sizeof(R) == 4) {
        const float Tf = in_range(Te) ? narrow(Te) : (float)Te;
        const float d = heat_increment<R>(K, Tf, rho);
        Te += d > 1e-30f && d < 1e30f ? widen(d) : (double)d;
      } else {
        Te += heat_increment<R>(K, Te, rho);
      }
      changed = true;
    }
    // e-i equilibration over the step (App. A): with a = rate_e dt and
    // b = rate_i dt frozen, the gap d = T_e - T_i decays by exp(-(a + b)) and
    // b T_e + a T_i is kept
    if (K.physics & P_EI) {
      double Ti = at<const double>(g.Ti, c * D);
      const double d = Te - Ti, X = Te * K.ei_mi + Ti * K.ei_me;
      // (1.4e5 aluminium cells with this and F_sigma: 60.7 -> 16.2 us by the
      // power, the series and fsigma() in place of pow, expm1, a division and log)
      const double a = in_range(X) ? times_pow_m32(K.ei_a, X) : K.ei_a / pow(X, 1.5);
      const double b = K.Zstar * a, s = a + b;
      if (d != 0.0 && s > 0.0) {
        // (e^{-s} - 1)/s: its series up to s = 1/64 (remainder below 1e-17)
        double f;
        if (s < 0.015625) {
          f = fma(s, -1.0 / 5040.0, 1.0 / 720.0);
          f = fma(s, f, -1.0 / 120.0);
          f = fma(s, f, 1.0 / 24.0);
          f = fma(s, f, -1.0 / 6.0);
          f = fma(s, f, 0.5);
          f = fma(s, f, -1.0);
        } else {
          f = expm1(-s) / s;
        }
        Te += a * d * f;
        Ti -= b * d * f;
        at(g.Ti, c * D) = Ti;
        if (K.physics & P_FSIGMA) at(g.Fsig, c * Z) = fsigma<R>(K, Ti);
        changed = true;
      }
    }
    if (changed) {  // eta(T) follows T_e
      double e;
      if (in_range(Te)) {
        e = resistivity(K, Te, narrow(Te));
      } else {
        e = resistivity_any(K.eta_hot, K.eta_cold, K.eta_max, Te);
      }
      at(g.T, c * D) = Te;
      at(g.eta, c * D) = e;
      if constexpr (sizeof(R) == 4) at(g.eta_r, c * Z) = in_range(e) ? narrow(e) : (float)e;
    }
    return ro;
  }
  return R(0);
}

}  // namespace hpic
