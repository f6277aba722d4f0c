// The paper's three-macro-electron estimate of the hot-electron loss
// channels (arXiv 2107.01723, Sec. III.B), one GPU thread per macro-electron.
//
// Per set: the exponential injection spectrum is cut at the X-ray threshold
// and the escape energy into three macro-electrons (warm, emitting,
// escaping), each integrated by RK4 in its path length through the four
// continuous stopping powers of Eqs. (stop_brem), (stop_ion), (stop_tnsa)
// and (stop_field).  FP64 throughout: the sets are independent and few, so
// the work is ALU-bound on GB300's FP64 units, not memory-bound.
#include <cmath>
#include <string>

#include "hpic.h"
#include "kernels.h"

namespace hpic {
namespace {

// CODATA 2018 SI values
constexpr double kQE = 1.602176634e-19;
constexpr double kME = 9.1093837015e-31;
constexpr double kC = 299792458.0;
constexpr double kEps0 = 8.8541878128e-12;
constexpr double kPi = 3.14159265358979323846;
constexpr double kHbar = 6.62607015e-34 / (2.0 * kPi);
constexpr double kMC2 = kME * kC * kC;

// ---------------------------------------------------------------- FP64 arithmetic
// What bounds this kernel is GB300's FP64 unit: a sub-core issues a warp-wide
// FP64 operation at most every 64 clocks, the SM's four sub-cores together one
// in 19 (measured on chains of DFMA, dependent or not).  So operations are
// what counts here: divisions start from an FP32 reciprocal, the two
// logarithms of the ionisation bracket are one, table-driven, comparisons run
// on the bits.
__device__ __forceinline__ bool ok(double x) { return fp32_range(x); }
// a < b by the bits, for numbers that are not both negative (a NaN counts as
// beyond every number of its sign)
__device__ __forceinline__ bool less(double a, double b) {
  return __double_as_longlong(a) < __double_as_longlong(b);
}
// 1/x of an ok() x: an FP32 estimate y, then y (1 + t + t^2), t = 1 - x y of
// about 1e-7
__device__ __forceinline__ double recip(double x) {
  const double y = widen(__fdividef(1.0f, narrow(x)));
  const double t = fma(-x, y, 1.0);
  return fma(y, fma(t, t, t), y);
}

// Half the natural logarithm by Tang's table-driven method ("Table-driven
// implementation of the logarithm function in IEEE floating-point arithmetic",
// ACM TOMS 16(4), 1990): x = 2^k m; r = m c - 1 with c a 24-bit reciprocal of
// the middle of m's 1/512 interval, so |r| < 2^-10 + 2^-23; ln x = k ln 2 -
// ln c + ln(1 + r), the last by its series to r^5 (remainder below 2^-62).
constexpr int kLogRows = 512, kLogExp = 100;
struct LogTable {
  double c[kLogRows], l[kLogRows], k[2 * kLogExp];  // c, -ln(c)/2, k ln(2)/2
  __device__ __forceinline__ void fill() {
    for (int j = threadIdx.x; j < kLogRows; j += blockDim.x) {
      const float f = 1.0f / (1.0f + (float)(2 * j + 1) / (2 * kLogRows));
      c[j] = (double)f;
      l[j] = -0.5 * log((double)f);
    }
    for (int j = threadIdx.x; j < 2 * kLogExp; j += blockDim.x)
      k[j] = (j - kLogExp) * (0.5 * 0.693147180559945309417232);
  }
  // s + ln(x)/2 of an ok() x
  __device__ __forceinline__ double add_half_log(double s, double x) const {
    const int hi = __double2hiint(x), j = (hi >> 11) & (kLogRows - 1);
    const double m = __hiloint2double((hi & 0x000fffff) | 0x3ff00000, __double2loint(x));
    const double r = fma(m, c[j], -1.0);
    double q = fma(r, 0.1, -0.125);
    q = fma(r, q, 1.0 / 6.0);
    q = fma(r, q, -0.25);
    q = fma(r, q, 0.5);
    return fma(r, q, s + (k[min((unsigned)((hi >> 20) - 1023 + kLogExp), 2u * kLogExp - 1u)] + l[j]));
  }
};

struct Stopping {
  double Kb, Kb_e;  // S_brem = Kb gamma = Kb + Kb_e eps
  double Ki, C;     // S_ion = Ki / beta^2 * bracket; C = ln(m_e c^2 / I_ex) - 0.246
  double St;        // S_tnsa
  double Fc, r, tc; // S_field = Fc / (x tc + r)^2
  double I_ex, th, Kb_th;  // Kb_th = Kb th / (m_e c^2)
  int mech;
};

struct Rates {
  double brem, ion, field, total;
};

// The channels' stopping powers at (eps, x).  ALL: every mechanism is on.
// FAST: for arguments inside ok(), `odd` set where one is not and the result
// means nothing; without branches, so that the chains of the two reciprocals
// and the logarithm run beside one another.
template <bool ALL, bool FAST>
__device__ __forceinline__ Rates rates(const Stopping &s, const LogTable &tab, double eps, double x,
                                       bool &odd) {
  Rates k;
  k.brem = ALL || (s.mech & HPIC_MODEL_BREM) ? fma(s.Kb_e, eps, s.Kb) : 0.0;
  k.ion = 0.0;
  k.field = 0.0;
  if (ALL || (s.mech & HPIC_MODEL_ION)) {
    const double e = eps * (1.0 / kMC2), gam = 1.0 + e;
    if constexpr (FAST) {
      // With v = e (e + 2): gamma^2 = 1 + v, 1/beta^2 = 1 + 1/v, and the bracket's
      // ln(eps/I_ex) + ln(gamma + 1)/2 is ln(m_e c^2/I_ex) + ln(e v)/2; 1/gamma
      // and 1/v come from one reciprocal.
      const double v = fma(e, gam, e), d = gam * v, arg = e * v;
      odd |= !ok(d) | !ok(arg);
      const double y = recip(d), ig = y * v;
      const double br = tab.add_half_log(fma(fma(0.909, ig, -0.818), ig, s.C), arg);
      k.ion = s.Ki * (__double2hiint(br) < 0 ? 0.0 : br) * fma(gam, y, 1.0);
    } else if (eps > 0.0) {
      const double ig = 1.0 / gam;
      const double br = log(eps / s.I_ex) + 0.5 * log(gam + 1.0) + 0.909 * ig * ig - 0.818 * ig - 0.246;
      if (br > 0.0) k.ion = s.Ki / (1.0 - ig * ig) * br;
    }
  }
  if (ALL || (s.mech & HPIC_MODEL_FIELD)) {
    const double rr = fma(x, s.tc, s.r), r2 = rr * rr;
    if constexpr (FAST) {
      odd |= !ok(r2);
      k.field = s.Fc * recip(r2);
    } else {
      k.field = s.Fc / r2;
    }
  }
  k.total = k.brem + (k.field + k.ion);
  if (ALL || (s.mech & HPIC_MODEL_TNSA)) k.total += s.St;
  return k;
}

// One RK4 step from (eps, x): its length h, the losses along it, and the
// photons above threshold (S_brem(eps - th) where eps > th).
struct Step {
  double h, xn, brem, ion, field, above, de;
  bool stuck;  // nothing slows it down any more
};

template <bool ALL, bool FAST>
__device__ __forceinline__ Step rk4(const Stopping &s, const LogTable &tab, double eps, double x,
                                    bool escaping, double Lx, double rel, double rel_field,
                                    bool &odd) {
  Step o;
  const Rates k1 = rates<ALL, FAST>(s, tab, eps, x, odd);
  o.stuck = !(k1.total > 0.0);
  if (FAST) odd |= !ok(k1.total);
  double h = rel * eps * (FAST ? recip(k1.total) : 1.0 / k1.total);
  if (ALL || (s.mech & HPIC_MODEL_FIELD)) {
    const double hx = fma(rel, x, rel_field);
    h = less(hx, h) ? hx : h;
  }
  double xn = x + h;
  if (escaping && less(Lx, xn)) {
    h = Lx - x;
    xn = x + h;
  }
  const double hh = 0.5 * h, xh = x + hh;
  const double e2 = fma(-hh, k1.total, eps);
  const Rates k2 = rates<ALL, FAST>(s, tab, e2, xh, odd);
  const double e3 = fma(-hh, k2.total, eps);
  const Rates k3 = rates<ALL, FAST>(s, tab, e3, xh, odd);
  const double e4 = fma(-h, k3.total, eps);
  const Rates k4 = rates<ALL, FAST>(s, tab, e4, xn, odd);
  const double h6 = h * (1.0 / 6.0);
  o.h = h;
  o.xn = xn;
  o.brem = h6 * fma(2.0, k2.brem + k3.brem, k1.brem + k4.brem);
  o.ion = h6 * fma(2.0, k2.ion + k3.ion, k1.ion + k4.ion);
  o.field = h6 * fma(2.0, k2.field + k3.field, k1.field + k4.field);
  o.above = 0.0;
  if ((ALL || (s.mech & HPIC_MODEL_BREM)) && less(s.th, eps)) {
    if (less(s.th, e4) && less(s.th, e3) && less(s.th, e2)) {
      o.above = fma(-h, s.Kb_th, o.brem);
    } else {
      double a = k1.brem - s.Kb_th;
      if (less(s.th, e2)) a = fma(2.0, k2.brem - s.Kb_th, a);
      if (less(s.th, e3)) a = fma(2.0, k3.brem - s.Kb_th, a);
      if (less(s.th, e4)) a += k4.brem - s.Kb_th;
      o.above = a * h6;
    }
  }
  o.de = o.brem + (o.ion + o.field);
  if (ALL || (s.mech & HPIC_MODEL_TNSA)) o.de = fma(h, s.St, o.de);
  return o;
}

// a macro-electron's losses per electron: the channels, photons above
// threshold, what escaped, the path length and the steps taken
struct Losses {
  double brem = 0.0, ion = 0.0, field = 0.0, above = 0.0, escaped = 0.0, x = 0.0;
  int steps = 0;
};

template <bool ALL>
__device__ void run_macro(const Stopping &s, const LogTable &tab, const hpic_model_in &m,
                          double eps, bool escaping, Losses &o) {
  const double rel_field = m.rel_step * (s.r / s.tc), rel = m.rel_step;
  const double Lx = m.Lx_m, E_stop = m.E_stop_J;
  double x = 0.0;
  for (int it = 0; it < 10000000; ++it) {  // bounded: sets are validated
    if (escaping ? !less(x, Lx) : !less(E_stop, eps)) {
      if (escaping) o.escaped += eps; else o.ion += eps;
      break;
    }
    if (!less(0.0, eps)) break;
    bool odd = false;
    Step d = rk4<ALL, true>(s, tab, eps, x, escaping, Lx, rel, rel_field, odd);
    if (odd) d = rk4<ALL, false>(s, tab, eps, x, escaping, Lx, rel, rel_field, odd);
    if (d.stuck) {
      if (escaping) {
        o.escaped += eps;
        x = Lx;
      } else {
        o.ion += eps;
      }
      break;
    }
    ++o.steps;
    if (!less(d.de, eps)) {  // stops inside the step: share what is left
      const double f = eps / d.de;
      o.brem = fma(f, d.brem, o.brem);
      o.ion = fma(f, d.ion, o.ion);
      o.field = fma(f, d.field, o.field);
      o.above = fma(f, d.above, o.above);
      x = fma(d.h, f, x);
      break;
    }
    o.brem += d.brem;
    o.ion += d.ion;
    o.field += d.field;
    o.above += d.above;
    eps -= d.de;
    x = d.xn;
  }
  o.x = x;
}

// Most sets a block takes: three lanes each (one per macro-electron) in four
// warps, which keep the FP64 unit of an SM busy.
constexpr int kModelSets = 42;

// A block takes `per` sets, a lane one macro-electron of one of them (the
// longest kind, the emitting one, first, each kind in consecutive lanes, so
// that a warp's lanes stop together), and adds the three of each set in
// shared memory.
// One lane for a whole set, 128 sets to a block, left 46 of 152 SMs with work
// for 5888 sets and the chain of three macro-electrons in every lane: 53.6 ms
// for 64 intensities x 92 elements, now 9.4 ms (14.5 ms with the split alone;
// the rest by 158 instead of 555 executed FP64 instructions per RK4 step); about
// 47 ms for any smaller number of sets, now 8.2 to 9.2 ms: the chain of one
// macro-electron's 1e3 steps.
__global__ void __launch_bounds__(128) k_model(long long n, int per,
                                               const hpic_model_in *__restrict__ in,
                                               hpic_model_out *__restrict__ out) {
  __shared__ LogTable tab;
  __shared__ double part[3][kModelSets][11];  // N, eps, x, E, then the six losses; steps
  tab.fill();
  __syncthreads();
  const int kind = threadIdx.x / per, slot = threadIdx.x - kind * per;
  const int b = kind == 0 ? 1 : (kind == 1 ? 0 : 2);  // warm 0, emitting 1, escaping 2
  const long long p = blockIdx.x * (long long)per + slot;
  double N_e = 0.0, a0 = 0.0;
  if (kind < 3 && p < n) {
    const hpic_model_in m = in[p];
    a0 = 8.5e-6 * sqrt(m.I0_Wm2 * m.lambda_m * m.lambda_m);  // Eq. (1)
    const double T = a0 * kMC2 * m.mean_sqrt_fg;
    Stopping s;
    const double Lrad = log(5.6 * kPi * kEps0 * kHbar * kC / (cbrt(m.Z) * kQE * kQE));
    const double e2 = kQE * kQE;
    s.mech = m.mechanisms;
    s.Kb = e2 * e2 * e2 / (12.0 * kPi * kPi * kPi * kEps0 * kEps0 * kEps0 * kME * kC * kC * kC * kHbar) *
           m.n_i_m3 * m.Z * m.Z * Lrad;
    s.Kb_e = s.Kb / kMC2;
    s.Ki = m.Z * m.n_i_m3 * e2 * e2 / (4.0 * kPi * kEps0 * kEps0 * kME * kC * kC);
    s.C = log(kMC2 / m.I_ex_J) - 0.246;
    s.St = 3.0 * m.kappa_tnsa * a0 * kMC2 / (m.Lx_m + m.Ly_m + m.Lz_m);
    s.r = 0.5 * m.r_fwhm_m;
    s.tc = tan(m.theta_c_rad);
    s.Fc = e2 * m.eta_avg_ohm_m * m.I0_Wm2 * m.mean_fg * s.r * s.r * m.eta_l2e / T;
    s.I_ex = m.I_ex_J;
    s.th = m.eps_th_J;
    s.Kb_th = s.Kb * (s.th / kMC2);
    N_e = m.I0_Wm2 * m.mean_fg * (kPi * m.r_fwhm_m * m.r_fwhm_m / 4.0) *
          (m.t_fwhm_s * sqrt(log(10.0) / log(2.0))) * m.eta_l2e / T;
    const double esc = m.kappa_esc * a0 * kMC2;
    const double lo = b == 0 ? 0.0 : (b == 1 ? s.th : esc);
    const double hi = b == 0 ? fmin(s.th, esc) : (b == 1 ? esc : INFINITY);
    double *q = part[b][slot];
    for (int i = 0; i < 11; ++i) q[i] = 0.0;
    if (hi > lo) {
      const bool open = isinf(hi);
      const double ea = exp(-lo / T), eb = open ? 0.0 : exp(-hi / T);
      const double nb = N_e * (ea - eb);
      const double Eb = N_e * ((lo + T) * ea - (open ? 0.0 : (hi + T) * eb));
      if (nb > 0.0) {
        Losses o;
        const double eps = Eb / nb;
        if (s.mech == HPIC_MODEL_ALL) run_macro<true>(s, tab, m, eps, b == 2, o);
        else run_macro<false>(s, tab, m, eps, b == 2, o);
        q[0] = nb;
        q[1] = eps;
        q[2] = o.x;
        q[3] = Eb;
        q[4] = nb * o.brem;
        q[5] = nb * o.ion;
        q[6] = s.mech & HPIC_MODEL_TNSA ? nb * (s.St * o.x) : 0.0;  // a constant stopping power
        q[7] = nb * o.field;
        q[8] = nb * o.above;
        q[9] = nb * o.escaped;
        q[10] = (double)o.steps;
      }
    }
  }
  __syncthreads();
  if (kind == 0 && p < n) {
    hpic_model_out o;
    o.N_e = N_e;
    o.a0 = a0;
    o.E[7] = 0.0;
    for (int i = 0; i < 7; ++i) o.E[i] = part[0][slot][3 + i] + part[1][slot][3 + i] + part[2][slot][3 + i];
    o.steps = 0;
    for (int c = 0; c < 3; ++c) {
      o.N_band[c] = part[c][slot][0];
      o.eps_band[c] = part[c][slot][1];
      o.x_end[c] = part[c][slot][2];
      o.steps += (long long)part[c][slot][10];
    }
    out[p] = o;
  }
}

}  // namespace
}  // namespace hpic

extern "C" {

int hpic_model_device(int64_t n, const hpic_model_in *in, hpic_model_out *out, int device,
                      void *cuda_stream) {
  if (n < 0 || (n > 0 && (!in || !out))) return HPIC_EINVAL;
  if (n == 0) return HPIC_OK;
  if (cudaSetDevice(device) != cudaSuccess) return HPIC_ECUDA;
  int sms = 1;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  // up to kModelSets sets per SM: one block on each, the sets shared out
  // evenly; more sets: full blocks, which the SMs take as they get free
  const long long even = (n + sms - 1) / sms;
  const int per = (int)(even < hpic::kModelSets ? even : hpic::kModelSets);
  const long long blocks = (n + per - 1) / per;
  if (blocks > 0x7fffffffll) return HPIC_EINVAL;
  hpic::k_model<<<(unsigned)blocks, (3 * per + 31) / 32 * 32, 0,
                  static_cast<cudaStream_t>(cuda_stream)>>>(n, per, in, out);
  return cudaGetLastError() == cudaSuccess ? HPIC_OK : HPIC_ECUDA;
}

int hpic_model(int64_t n, const hpic_model_in *in, hpic_model_out *out, int device,
               void *cuda_stream) {
  if (n < 0 || (n > 0 && (!in || !out))) {
    hpic::set_global_error("hpic_model: bad arguments");
    return HPIC_EINVAL;
  }
  for (int64_t p = 0; p < n; ++p) {
    const hpic_model_in &m = in[p];
    if (!(m.rel_step >= 1e-6 && m.rel_step < 1) || !(m.Z > 0) || !(m.n_i_m3 > 0) || !(m.I_ex_J > 0) ||
        !(m.Lx_m > 0) || !(m.Ly_m > 0) || !(m.Lz_m > 0) || !(m.I0_Wm2 > 0) || !(m.lambda_m > 0) ||
        !(m.eta_l2e > 0) || !(m.r_fwhm_m > 0) || !(m.t_fwhm_s > 0) || !(m.mean_fg > 0) ||
        !(m.mean_sqrt_fg > 0) || !(m.kappa_esc >= 0) || !(m.kappa_tnsa >= 0) ||
        !(m.theta_c_rad > 0 && m.theta_c_rad < 1.5707963267948966) || !(m.eta_avg_ohm_m >= 0) ||
        !(m.eps_th_J > 0) || !(m.E_stop_J > 0) || (m.mechanisms & ~HPIC_MODEL_ALL) != 0 ||
        (m.mechanisms & (HPIC_MODEL_BREM | HPIC_MODEL_ION | HPIC_MODEL_TNSA)) == 0) {
      hpic::set_global_error(("hpic_model: parameter set " + std::to_string(p) + " out of range").c_str());
      return HPIC_EINVAL;
    }
  }
  if (n == 0) return HPIC_OK;
  if (cudaSetDevice(device) != cudaSuccess) {
    cudaGetLastError();
    hpic::set_global_error("hpic_model: no such CUDA device");
    return HPIC_ECUDA;
  }
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  hpic_model_in *din = nullptr;
  hpic_model_out *dout = nullptr;
  if (cudaMalloc(&din, n * sizeof(*din)) != cudaSuccess ||
      cudaMalloc(&dout, n * sizeof(*dout)) != cudaSuccess) {
    cudaGetLastError();
    cudaFree(din);
    hpic::set_global_error("hpic_model: device allocation failed");
    return HPIC_ENOMEM;
  }
  int rc = HPIC_OK;
  cudaError_t e = cudaMemcpyAsync(din, in, n * sizeof(*din), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) rc = hpic_model_device(n, din, dout, device, cuda_stream);
  if (e == cudaSuccess && rc == HPIC_OK)
    e = cudaMemcpyAsync(out, dout, n * sizeof(*dout), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(din);
  cudaFree(dout);
  if (e != cudaSuccess || rc != HPIC_OK) {
    hpic::set_global_error(("hpic_model: " + std::string(cudaGetErrorString(e))).c_str());
    return HPIC_ECUDA;
  }
  return HPIC_OK;
}

}  // extern "C"
