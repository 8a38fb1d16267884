// Host build of the fixed-point MP-9 march (fdlb_mp9i.cuh) for CPU unit tests.
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __forceinline__ inline
#define __noinline__
#define __restrict__
static inline long long __double_as_longlong(double x) { long long b; std::memcpy(&b, &x, 8); return b; }
static inline double __longlong_as_double(long long b) { double x; std::memcpy(&x, &b, 8); return x; }
using std::fma;
using std::fabs;
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
#include "../../paper_1909_08390_gb300/csrc/fdlb_mp9i.cuh"

// Flux differences of n cells of a line with 5 ghosts per side (ext[0..n+9]),
// marched for velocity sign sgn in segments of nc cells (2, 4, 8 or 16) whose
// scale is the largest exponent of ext[0..n+9]; out[c], cell c, carries the
// march's sign, converted to binary64.  Returns the largest biased exponent.
template <int NC>
static void march(const int64_t* ext, int n, int sgn, int64_t* out) {
  for (int c0 = 0; c0 < n; c0 += NC) {
    const int first = sgn > 0 ? c0 : c0 + NC - 1;
    const int up = (sgn > 0 ? first - 1 : first + 1) + 5;
    fdlb::mp9_march_delta_int<NC>(ext + up, sgn, out + first, sgn);
  }
}
extern "C" int mp9i_line(const double* ext, int n, int sgn, int nc, double* out) {
  int m = 0;
  for (int i = 0; i < n + 10; ++i) m = m > fdlb::mag_word(ext[i]) ? m : fdlb::mag_word(ext[i]);
  const int emax = m >> 20;
  int64_t e[80], q[64];
  for (int i = 0; i < n + 10; ++i) e[i] = fdlb::q_of(ext[i], emax);
  if (nc == 2) march<2>(e, n, sgn, q);
  else if (nc == 4) march<4>(e, n, sgn, q);
  else if (nc == 8) march<8>(e, n, sgn, q);
  else march<16>(e, n, sgn, q);
  for (int i = 0; i < n; ++i) out[i] = fdlb::q_to_double(q[i], emax);
  return emax;
}
// |cx| dx + |cy| dy of flux differences given in units of 2^(emax - 1081)
extern "C" double adv_term(double cx, double cy, int64_t dx, int64_t dy, int emax) {
  int ex;
  const fdlb::AdvCoef c = fdlb::advection_coef(cx, cy, ex);
  return fdlb::q_to_double(fdlb::advection_int(c, dx, dy), emax + ex);
}
extern "C" void mp9_delta64(const double* ext, int n, int sgn, double* out) {
  const int first = sgn > 0 ? 0 : n - 1;
  const int up = (sgn > 0 ? first - 1 : first + 1) + 5;
  fdlb::mp9_march_delta_fp64(ext + up, sgn, reinterpret_cast<int64_t*>(out) + first, sgn, n);
}
