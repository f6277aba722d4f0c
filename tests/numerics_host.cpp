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
inline float __fmul_rn(float a, float b) { return a * b; }
// a warp's exchange as one lane sees it: over_warp() runs all its rounds, and only
// that of `round` finds another lane's parts, the rest zeros
const float *other = nullptr;
int round_of = 0;
inline float __shfl_xor_sync(unsigned, float, int o) { return o == round_of ? *other++ : 0.0f; }
inline double __shfl_xor_sync(unsigned, double v, int) { return v; }
struct {
  unsigned x;
} threadIdx;
using std::fma;
using std::fabs;
using std::isfinite;
}  // namespace

#include "numerics.cuh"

using namespace hpic;

namespace {
template <int parts>
void exchange(WideSum<float> &mine, const WideSum<float> &theirs, int o) {
  float v[parts];
  std::memcpy(v, &theirs, sizeof(v));
  other = v;
  round_of = o;
  mine.over_warp();
}
}  // namespace

extern "C" {
void set_off(int n) { off = n; }
void run_log(const double *x, double *y, long n) { for (long i = 0; i < n; ++i) y[i] = table_log(x[i]); }
void run_log_parts(const double *x, double *base, double *rest, long n) {
  for (long i = 0; i < n; ++i) {
    float r;
    log_parts(x[i], base[i], r);
    rest[i] = r;
  }
}
void run_turn(const uint32_t *x, double *s, double *c, long n) {
  for (long i = 0; i < n; ++i) table_turn(x[i], s[i], c[i]);
}
void run_sincos(const double *x, double *s, double *c, long n) {
  for (long i = 0; i < n; ++i) m_sincos_small(x[i], s + i, c + i);
}
void run_rotate(double *d, const double *ct, const double *st, const double *cp, const double *sp, long n) {
  for (long i = 0; i < n; ++i) rotate_near(d[3 * i], d[3 * i + 1], d[3 * i + 2], ct[i], st[i], cp[i], sp[i]);
}
void run_rcp(const double *x, double *y, long n) { for (long i = 0; i < n; ++i) y[i] = m_rcp(x[i]); }
void run_rsqrt(const double *x, double *y, long n) { for (long i = 0; i < n; ++i) y[i] = m_rsqrt(x[i]); }
void run_sqrt(const double *x, double *y, long n) { for (long i = 0; i < n; ++i) y[i] = m_sqrt_near(x[i]); }
void run_div(const double *a, const double *b, double *y, long n) {
  for (long i = 0; i < n; ++i) y[i] = m_div_near(a[i], b[i]);
}
// `steps` values of each of 32 lanes, x[step][lane], then the sum over the warp by
// exchanges: lane 0's total
double warp_total(const float *x, long steps) {
  WideSum<float> lane[32] = {};
  for (long i = 0; i < steps; ++i)
    for (int l = 0; l < 32; ++l) lane[l].add(x[32 * i + l]);
  constexpr int parts = sizeof(WideSum<float>) / sizeof(float);
  for (int o = 16; o > 0; o >>= 1) {
    WideSum<float> before[32];
    std::memcpy(before, lane, sizeof(lane));
    for (int l = 0; l < 32; ++l) exchange<parts>(lane[l], before[l ^ o], o);
  }
  return lane[0].value();
}
}
