// Host build of the integer conversions (fdlb_cvt.cuh) for CPU unit tests.
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __forceinline__ inline
#define __restrict__
static inline long long __double_as_longlong(double x) { long long b; std::memcpy(&b, &x, 8); return b; }
static inline double __longlong_as_double(long long b) { double x; std::memcpy(&x, &b, 8); return x; }
using std::fma;
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
#include "../../paper_1909_08390_gb300/csrc/fdlb_cvt.cuh"
extern "C" void widen_all(const float* x, double* y, long n) { for (long i = 0; i < n; ++i) y[i] = fdlb::widen(x[i]); }
extern "C" void narrow_all(const double* x, float* y, long n) { for (long i = 0; i < n; ++i) y[i] = fdlb::narrow(x[i]); }
