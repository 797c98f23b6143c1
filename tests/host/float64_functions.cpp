// The float64 functions of sidp_laws.cuh compiled for the host, so that a CPU test can compare them with longer
// arithmetic.  The fast float32 functions that they start from are modelled at their documented error bounds
// (CUDA C++ Programming Guide, mathematical functions: __fdividef and rsqrtf 2 ulp; __log2f 2 ulp, 2^-22 absolute
// in [0.5, 2]; __powf(x, y) = exp2f(y * __log2f(x)), its last step 2 ulp): `tilt` in [-1, 1] says how much of the
// bound they are off and in which direction.
#include <cmath>
#include <cstring>
#include <algorithm>
#include <cuda_runtime.h>
#undef __device__
#undef __forceinline__
#undef __noinline__
#define __device__
#define __forceinline__ inline
#define __noinline__
using std::fma;
using std::max;
using std::min;

static double tilt = 0.0;
static double tilt_log = 0.0;
static float off(double exact, double ulps) { return (float)(exact * (1.0 + tilt * ulps * 0x1p-23)); }

static inline long long __double_as_longlong(double x) { long long r; std::memcpy(&r, &x, 8); return r; }
static inline double __longlong_as_double(long long x) { double r; std::memcpy(&r, &x, 8); return r; }
static inline int __double2hiint(double x) { return (int)(__double_as_longlong(x) >> 32); }
static inline int __double2loint(double x) { return (int)__double_as_longlong(x); }
static inline double __hiloint2double(int hi, int lo) { return __longlong_as_double(((long long)hi << 32) | (unsigned)lo); }
static inline unsigned __float_as_uint(float x) { unsigned r; std::memcpy(&r, &x, 4); return r; }
static inline float __uint_as_float(unsigned x) { float r; std::memcpy(&r, &x, 4); return r; }
static inline unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) {
  s &= 31;
  return s ? (hi << s) | (lo >> (32 - s)) : hi;
}
static inline float __fdividef(float a, float b) { return off((double)a / b, 2); }
static inline float fast_rsqrt(float x) { return off(1.0 / std::sqrt((double)x), 2); }
static inline float fast_log2(float x) {
  const double l = std::log2((double)x);
  return (float)(x >= 0.5f && x <= 2.0f ? l + tilt_log * 0x1p-22 : l * (1.0 + (l > 0 ? 1 : -1) * tilt_log * 2 * 0x1p-23));
}
static inline float fast_pow(float x, float y) {
  const float e = y * fast_log2(x);
  return off(std::exp2((double)e), 2);
}
#define rsqrtf fast_rsqrt
#define __log2f fast_log2
#define __powf fast_pow
static inline float2 __ffma2_rn(float2 a, float2 b, float2 c) { return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y)); }
static inline float2 __fadd2_rn(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
static inline float2 __fmul2_rn(float2 a, float2 b) { return make_float2(a.x * b.x, a.y * b.y); }

#include "sidp_laws.cuh"

using namespace sidp;
using EulerD = LawEuler<double>;

extern "C" {
// value: the fast functions' last steps; log: __log2f (its error enters a power multiplied by the exponent)
void set_tilt(double value, double log) { tilt = value; tilt_log = log; }

void compare_ops(int n, const double* a, const double* b, double* out) {  // out: [5][n]
  for (int i = 0; i < n; ++i) {
    out[i] = tmax(a[i], b[i]);
    out[n + i] = tmin(a[i], b[i]);
    out[2 * n + i] = tpos(a[i]);
    out[3 * n + i] = tneg(a[i]);
    out[4 * n + i] = is_pos(a[i]) ? 1.0 : 0.0;
  }
}
void compare_ops_nonneg(int n, const double* a, const double* b, double* out) {  // out: [2][n]
  for (int i = 0; i < n; ++i) {
    out[i] = pmax(a[i], b[i]);
    out[n + i] = pmin(a[i], b[i]);
  }
}
void quotients(int n, const double* a, const double* b, double* out) {  // out: [3][n]: a / b, 1 / b, sqrt b
  for (int i = 0; i < n; ++i) {
    out[i] = sidp::fdiv(a[i], b[i]);
    out[n + i] = sidp::frcp(b[i]);
    out[2 * n + i] = sidp::psqrt(b[i]);
  }
}
void powers(int n, double gamma, const double* x, double* out) {  // out: [4][n]: x^-e, x^-gamma, x^gamma, x^(1/e)
  const double zero[2] = {0.0, 0.0};
  const LawParamsT<double> lp = make_law_params<double>(gamma, zero, zero);
  for (int i = 0; i < n; ++i) {
    out[i] = pow_neg_e(x[i], lp);
    out[n + i] = pow_neg_gamma(x[i], lp);
    out[2 * n + i] = pow_gamma(x[i], lp);
    out[3 * n + i] = pstar_pow(x[i], lp);
  }
}
// The screen of one candidate u + tcap sc w (given as +xp; the other three are zero): 1 when it is left undecided.
void screen(int n, double gamma, const double* u, const double* K, const double* w, double sc, double tcap, int* out) {
  const double zero[4] = {0.0, 0.0, 0.0, 0.0};
  const LawParamsT<double> lp = make_law_params<double>(gamma, zero, zero);
  for (int i = 0; i < n; ++i)
    out[i] = (int)(EulerD::psi_screen(u + 4 * i, K[i], w + 4 * i, zero, zero, zero, sc, tcap, lp) & 1u);
}
void certainly_above(int n, double gamma, const double* u, const double* K, int* out) {
  const double zero[2] = {0.0, 0.0};
  const LawParamsT<double> lp = make_law_params<double>(gamma, zero, zero);
  for (int i = 0; i < n; ++i) out[i] = EulerD::sigma_certainly_above(u + 4 * i, K[i], lp) ? 1 : 0;
}
}
