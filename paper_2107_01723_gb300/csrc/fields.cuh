// Per-node device code of the field solve and heating (arXiv 2107.01723,
// Eqs. (A2)-(A8)), shared by the single-target and the batched kernels.
#pragma once

#include "kernels.h"

namespace hpic {

// (i, j, k) of node q.  The two divisions by the row and plane lengths go
// through multiplications by rounded-up reciprocals (Granlund & Montgomery,
// "Division by invariant integers using multiplication", PLDI 1994): exact for
// the node counts here, below 2^31 (checked at creation).
template <typename R>
__device__ __forceinline__ void node_of(const FieldK<R> &K, long long q, int &i, int &j, int &k) {
  const unsigned uq = (unsigned)q;
  const unsigned kk = K.by_sz.quotient(uq), r = uq - kk * (unsigned)K.sz;
  const unsigned jj = K.by_sy.quotient(r);
  k = (int)kk;
  j = (int)jj;
  i = (int)(r - jj * (unsigned)K.sy);
}

// x^(-3/2) of an in_range x: an FP32 estimate y, then y (1 - e)^(-1/2) with
// e = 1 - x^3 y^2 (about 1e-6) to second order, the next term being below
// 1e-18: eight FP64 operations, where rsqrt(x) cubed takes about fourteen
__device__ __forceinline__ double pow_m32(double x) {
  const float r = rsqrtf(narrow(x));
  const double y = widen(r * r * r);
  const double e = fma(-(x * x * x), y * y, 1.0);
  return fma(y, e * fma(0.375, e, 0.5), y);
}

// ---------------------------------------------------------------- E, Eq. (A2)
// E on the three edges owned by node q (tangential E = 0 on the walls)
template <typename R>
__device__ __forceinline__ void efield_node(const FieldK<R> &K, const GView<R> &g, long long q) {
  const int nx = K.nx, ny = K.ny, nz = K.nz;
  const int sy = K.sy;
  const long long sz = K.sz;
  const long long cy = nx, cz = (long long)nx * ny;
  const R Fc = K.F_curl, Fj = K.F_j;
  const R *Bx = g.B[0], *By = g.B[1], *Bz = g.B[2];
  int i, j, k;
  node_of(K, q, i, j, k);
  R ex = 0, ey = 0, ez = 0;
  const long long c = i + cy * j + cz * k;  // cell (i, j, k)
  if (i < nx && j >= 1 && j <= ny - 1 && k >= 1 && k <= nz - 1) {
    const R curl = (Bz[q] - Bz[q - sy]) - (By[q] - By[q - sz]);
    const R eta = R(0.25) * (g.eta_r[c - cy - cz] + g.eta_r[c - cz] + g.eta_r[c - cy] + g.eta_r[c]);
    ex = eta * (Fc * curl - Fj * g.J[0][q]);
  }
  if (j < ny && i >= 1 && i <= nx - 1 && k >= 1 && k <= nz - 1) {
    const R curl = (Bx[q] - Bx[q - sz]) - (Bz[q] - Bz[q - 1]);
    const R eta = R(0.25) * (g.eta_r[c - 1 - cz] + g.eta_r[c - cz] + g.eta_r[c - 1] + g.eta_r[c]);
    ey = eta * (Fc * curl - Fj * g.J[1][q]);
  }
  if (k < nz && i >= 1 && i <= nx - 1 && j >= 1 && j <= ny - 1) {
    const R curl = (By[q] - By[q - 1]) - (Bx[q] - Bx[q - sy]);
    const R eta = R(0.25) * (g.eta_r[c - 1 - cy] + g.eta_r[c - cy] + g.eta_r[c - 1] + g.eta_r[c]);
    ez = eta * (Fc * curl - Fj * g.J[2][q]);
  }
  g.E[0][q] = ex;
  g.E[1][q] = ey;
  g.E[2][q] = ez;
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
// In range, both come from p = T^(-3/2) (sqrt(T) = T^2 p) without a division,
// a root or a compare on the FP64 unit (Tf = (float)T tells the band, whose
// float ends lie inside the exact one, where the formula gives the cap too):
// this and the conversions took the heating of 128^3 cells from 128 to 71 us,
// and of a 16-target batch of 7.9e6 cells (each with its constants in shared
// memory and its Ohmic sums made in the warp) from 542 to 199 us.
__device__ __forceinline__ double resistivity(const FieldCommon &K, double T, float Tf) {
  if (Tf > K.eta_Tlo && Tf < K.eta_Thi) return K.eta_max;
  const double p = pow_m32(T);
  double eta = K.eta_hot * p;
  if (K.eta_cold > 0.0) eta = min_positive(eta, K.eta_cold * (T * T * p));
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

// ---------------------------------------------------------------- B, Eq. (A3), and heating
// Faraday on the faces owned by node q, then heating of cell q; the cell's
// Ohmic energy density (J/m^3) goes to `ohm`
template <typename R>
__device__ __forceinline__ void bheat_node(const FieldK<R> &K, const GView<R> &g, long long q,
                                           WideSum<R> &ohm) {
  const int nx = K.nx, ny = K.ny, nz = K.nz;
  const int sy = K.sy;
  const long long sz = K.sz;
  const R cdt = K.cdt;
  const R *Ex = g.E[0], *Ey = g.E[1], *Ez = g.E[2];
  int i, j, k;
  node_of(K, q, i, j, k);
  if (K.physics & P_FARADAY) {
    if (j < ny && k < nz) g.B[0][q] -= cdt * ((Ez[q + sy] - Ez[q]) - (Ey[q + sz] - Ey[q]));
    if (i < nx && k < nz) g.B[1][q] -= cdt * ((Ex[q + sz] - Ex[q]) - (Ez[q + 1] - Ez[q]));
    if (i < nx && j < ny) g.B[2][q] -= cdt * ((Ey[q + 1] - Ey[q]) - (Ex[q + sy] - Ex[q]));
  }
  if (i < nx && j < ny && k < nz) {
    const long long c = i + (long long)nx * (j + (long long)ny * k);
    const double Hc = g.H[c];
    R jb2 = R(0);
    if (K.physics & P_FIELDS) {
      const R *Jx = g.J[0], *Jy = g.J[1], *Jz = g.J[2];
      // cell-centred mean of the edge current in the field precision
      const R jbx = R(0.25) * (Jx[q] + Jx[q + sy] + Jx[q + sz] + Jx[q + sy + sz]);
      const R jby = R(0.25) * (Jy[q] + Jy[q + 1] + Jy[q + sz] + Jy[q + 1 + sz]);
      const R jbz = R(0.25) * (Jz[q] + Jz[q + 1] + Jz[q + sy] + Jz[q + 1 + sy]);
      jb2 = jbx * jbx + jby * jby + jbz * jbz;
    }
    // a cell without drag heat or current keeps T and eta (and adds no
    // Ohmic energy) unless e-i equilibration moves it
    const bool no_heat = (__double_as_longlong(Hc) << 1) == 0;  // +0 or -0
    if (no_heat && jb2 == R(0) && !(K.physics & P_EI)) return;
    double Te = g.T[c];
    bool changed = false;
    const R ro = g.eta_r[c] * K.F_ohm * jb2;
    ohm.add(ro);
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
      double Ti = g.Ti[c];
      const double d = Te - Ti;
      const double a = K.ei_a / pow(Te * K.ei_mi + Ti * K.ei_me, 1.5), b = K.Zstar * a;
      if (d != 0.0 && a + b > 0.0) {
        const double f = expm1(-(a + b)) / (a + b);
        Te += a * d * f;
        Ti -= b * d * f;
        g.Ti[c] = Ti;
        if (K.physics & P_FSIGMA) g.Fsig[c] = R(1.0 + K.fs_q * (0.5 * log(Ti) + K.fs_c));
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
      g.T[c] = Te;
      g.eta[c] = e;
      if constexpr (sizeof(R) == 4) g.eta_r[c] = in_range(e) ? narrow(e) : (float)e;
    }
  }
}

}  // namespace hpic
