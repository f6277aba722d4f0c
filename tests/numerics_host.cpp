// Host build of csrc/numerics.cuh for test_numerics_host.py: the intrinsics it uses,
// in plain C++, and one entry per function over arrays.
#include <cmath>
#include <cstdint>
#include <cstring>

#define __device__
#define __forceinline__ inline

namespace {
template <typename T, typename F>
T bits(F f) {
  static_assert(sizeof(T) == sizeof(F), "same size");
  T t;
  std::memcpy(&t, &f, sizeof(t));
  return t;
}
// The hardware's quick estimates, as far off as the documentation allows: the
// rounded result moved by `off` of its last places.
struct double2 {
  double x, y;
};
int off = 0;
float moved(double exact) { return bits<float>(bits<int32_t>((float)exact) + off); }

inline int __double2hiint(double x) { return (int)(bits<uint64_t>(x) >> 32); }
inline int __double2loint(double x) { return (int)(uint32_t)bits<uint64_t>(x); }
inline double __hiloint2double(int h, int l) {
  return bits<double>((uint64_t)(uint32_t)h << 32 | (uint32_t)l);
}
inline unsigned __float_as_uint(float x) { return bits<uint32_t>(x); }
inline float __uint_as_float(unsigned x) { return bits<float>(x); }
inline long long __double_as_longlong(double x) { return bits<int64_t>(x); }
inline unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) {
  return (unsigned)(((uint64_t)hi << 32 | lo) << s >> 32);
}
inline float __fdividef(float a, float b) { return moved((double)a / b); }
inline float rsqrtf(float x) { return moved(1.0 / std::sqrt((double)x)); }
inline double rsqrt(double x) { return 1.0 / std::sqrt(x); }
template <typename T>
T __ldg(const T *p) { return *p; }
inline float __fadd_rn(float a, float b) { return a + b; }
// a warp's exchange, of one lane: the lanes' values are handed over in `other`
const float *other = nullptr;
inline float __shfl_xor_sync(unsigned, float, int) { return *other++; }
inline double __shfl_xor_sync(unsigned, double v, int) { return v; }
using std::fma;
using std::isfinite;
}  // namespace

#include "numerics.cuh"

using namespace hpic;

extern "C" {
void set_off(int n) { off = n; }
void run_log(const double *x, double *y, long n) { for (long i = 0; i < n; ++i) y[i] = table_log(x[i]); }
void run_turn(const uint32_t *x, double *s, double *c, long n) {
  for (long i = 0; i < n; ++i) table_turn(x[i], s[i], c[i]);
}
void run_sincos(const double *x, double *s, double *c, long n) {
  for (long i = 0; i < n; ++i) m_sincos_small(x[i], s + i, c + i);
}
void run_rcp(const double *x, double *y, long n) { for (long i = 0; i < n; ++i) y[i] = m_rcp(x[i]); }
void run_rsqrt(const double *x, double *y, long n) { for (long i = 0; i < n; ++i) y[i] = m_rsqrt(x[i]); }
void run_sqrt(const double *x, double *y, long n) { for (long i = 0; i < n; ++i) y[i] = m_sqrt_near(x[i]); }
void run_div(const double *a, const double *b, double *y, long n) {
  for (long i = 0; i < n; ++i) y[i] = m_div_near(a[i], b[i]);
}
}
