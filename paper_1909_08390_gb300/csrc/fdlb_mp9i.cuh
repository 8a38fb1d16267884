// fdlb_mp9i.cuh -- the MP-9 march of fdlb_mp9.cuh (Sec. IV) in 64-bit
// fixed point, for the 2-D binary64 stage kernels.
//
// GB300 runs 2 binary64 operations per clock and SM, but 64 integer
// operations (shifts, logic, compares, 32 x 32 -> 64 multiply-adds) and about
// 128 integer additions.  The march is a fixed sequence of differences, one
// stencil with integer coefficients and a limiter made of comparisons, so it
// needs no exponents as long as its values are of similar size: the 17 values
// that a marching thread reads for the 8 cells of its half line are scaled to
// integers
//   q = F 2^(59 - E),  2^E > max |F| of those values,
// truncated at one unit.  A unit is 2^-59 of the largest value's power of two;
// differences, curvatures and flux differences are then exact, the stencil and
// the limiter's bounds lose at most two units each, and the flux difference of
// a cell goes back to binary64 with one rounding.  Sizes: |q| < 2^59,
// differences < 2^60, curvatures < 2^61, 4 m - M <= 3 m < 2^62.6, bounds <
// 2^62: all inside 63 bits.
//
// So the error is relative to the largest of these values, where the binary64
// march rounds every interface value to 2^-53 of itself: the smaller a cell
// beside the largest, the less the fixed-point march is worth.  Root mean
// square error of a flux difference over its cell's own value, smooth lines |
// rough ones (uniform within 50 %), for cells r times below the largest,
// against 7e-17 | 4.5e-17 in binary64:
//   r = 1 2e-18 | 6e-18,  4 5e-18 | 1.2e-17,  16 2e-17 | 4.4e-17,
//   32 4e-17 | 8e-17,  64 1e-16 | 1.6e-16.
// Hence the rule (takes_fixed_point): a half line whose own cells lie no more
// than a factor of 16 below the largest value read, so that no cell's error is
// larger than in binary64 (root mean square).  The others, lines with a zero
// among nonzero cells, and those whose largest exponent leaves no room for the
// scaling (an infinity or NaN among the values, beyond 2^1007 or below 2^-823),
// march in binary64 (mp9_march_delta_fp64), with the other lines of their warp.
//
// One scale for a population's whole tile needs a conversion per cell instead
// of two, but sends whole tiles to the binary64 march where a smooth field
// varies by more than 16 over 26 cells.  512 x 512 x 128 populations, a step,
// tile's scale -> line's: smooth field 3.05 -> 3.36 ms, four quadrants 3.89 ->
// 3.87; 400 x 400 quadrants 3.23 -> 2.95; 96 x 70, smooth 0.405 -> 0.324,
// quadrants 0.824 -> 0.760.
//
// The scales belong to half lines and the choice to warps, so the last bits of
// a result depend on where the tiles lie: a periodic field shifted by other than
// whole tiles, or run on a device with another number of SMs (which sets the
// tile height of small grids), differs by roundings, and an interface on the
// edge of a half line, computed once on either side, cancels to rounding only.
//
// The flux differences stay integers until the update of a cell: the
// advection term dt p . grad F is their sum times 61-bit fixed-point
// coefficients (advection_int), converted to binary64 once.
//
// Negative magnitudes are taken as one's complements (x ^ mask), one unit
// away from the negation.
#pragma once

#include <cstdint>

#include "fdlb_mp9.cuh"

namespace fdlb {

constexpr int kQBits = 59;  // |q| < 2^kQBits
// biased exponents of the cells' largest magnitude that the march takes
constexpr int kQExpMin = 200, kQExpMax = 2030;
// and the distance of its magnitude word from the smallest one's: 2^4
constexpr int kQRange = 4 << 20;

// x >> n for any n >= 0 (zero from 64 on)
__device__ __forceinline__ uint64_t shr64(uint64_t x, int n) {
#ifdef __CUDA_ARCH__
  uint64_t r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));  // clamps n
  return r;
#else
  return n > 63 ? 0 : x >> n;
#endif
}
// x >> n (arithmetic) for any n >= 0
__device__ __forceinline__ int64_t sar64(int64_t x, int n) {
#ifdef __CUDA_ARCH__
  int64_t r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));  // clamps n
  return r;
#else
  return x >> (n > 63 ? 63 : n);
#endif
}
__device__ __forceinline__ int clz64(uint64_t x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return x ? __builtin_clzll(x) : 64;
#endif
}

// high word of |x|: its biased exponent is bits 20..30; ordered like |x|
__device__ __forceinline__ int mag_word(double x) { return (int)(dbits(x) >> 32) & 0x7fffffff; }
// Whether the fixed-point march takes cells whose largest magnitude word is mx
// and whose flux differences are wanted down to magnitude word mn (see the head
// of this file).
__device__ __forceinline__ bool takes_fixed_point(int mx, int mn) {
  const int e = mx >> 20;
  return e >= kQExpMin && e <= kQExpMax && mx - mn <= kQRange;
}

// x as a fixed-point integer of the scale whose largest biased exponent is emax
__device__ __forceinline__ int64_t q_of(double x, int emax) {
  const long long b = dbits(x);
  const int hi = (int)(b >> 32);
  const int n = emax - ((hi >> 20) & 0x7ff);
  const uint64_t m = ((uint64_t)b & 0xfffffffffffffULL) | 0x10000000000000ULL;
  const int64_t s = (int64_t)(hi >> 31);  // sign mask
  return (int64_t)shr64(m << (kQBits - 53), n) ^ s;
}

// u 2^(ex - kQScale) as binary64, rounded to nearest (ties away from zero; ex
// well inside the exponent range)
constexpr int kQScale = 1022 + kQBits;
__device__ __forceinline__ double q_to_double(int64_t u, int ex) {
  const int64_t s = u >> 63;
  const uint64_t a = (uint64_t)((u ^ s) - s);
  const int lz = clz64(a);
  const uint64_t t = a << (lz & 63);
  const uint64_t m = (t >> 11) + ((uint32_t)t >> 10 & 1u);  // leading bit at 52 (or a carry to 53)
  // m carries the leading bit, so the field takes the biased exponent - 1
  const int e = ex + (63 - kQBits) - lz;
  const uint32_t hi = (uint32_t)(m >> 32) + ((uint32_t)e << 20);
  const uint64_t r = ((uint64_t)hi << 32) | (uint32_t)m;
  const long long bits = a == 0 ? 0 : (long long)(r | ((uint64_t)s & (uint64_t)kSign));
  return dfrom(bits);
}

// |cx|, |cy| (dt |p| / ds, at most 1) as 64-bit fractions of a common power
// of two: |c| = (h 2^32 + l) 2^-64 2^ex, the larger one in [1/8, 1/4).
struct AdvCoef {
  int32_t xh, xl, yh, yl;
};
__device__ __forceinline__ void split_coef(uint64_t c, int32_t& h, int32_t& l) {
  l = (int32_t)(uint32_t)c;
  h = (int32_t)((c - (uint64_t)(int64_t)l) >> 32);
}
__device__ __forceinline__ AdvCoef advection_coef(double cx, double cy, int& ex) {
  const long long bx = dbits(cx) & kMag, by = dbits(cy) & kMag;
  const int ix = (int)(bx >> 52), iy = (int)(by >> 52);
  int e = ix > iy ? ix : iy;
  e = e < 900 ? 900 : e;  // coefficients below 2^-123 lose their last bits
  const uint64_t mx = ((uint64_t)bx & 0xfffffffffffffULL) | 0x10000000000000ULL;
  const uint64_t my = ((uint64_t)by & 0xfffffffffffffULL) | 0x10000000000000ULL;
  AdvCoef c;
  split_coef(ix == 0 ? 0 : shr64(mx << 9, e - ix), c.xh, c.xl);
  split_coef(iy == 0 ? 0 : shr64(my << 9, e - iy), c.yh, c.yl);
  ex = e - 1020;
  return c;
}
// (|cx| dx + |cy| dy) 2^-ex in units, to 3 units
__device__ __forceinline__ int64_t advection_int(const AdvCoef& c, int64_t dx, int64_t dy) {
  const int32_t xh = (int32_t)(dx >> 32), yh = (int32_t)(dy >> 32);
  const uint64_t tx = (uint64_t)(uint32_t)dx * (uint32_t)c.xh;
  const uint64_t ty = (uint64_t)(uint32_t)dy * (uint32_t)c.yh;
  const int64_t low = (int64_t)xh * c.xl + (int64_t)yh * c.yl;
  return (int64_t)xh * c.xh + (int64_t)yh * c.yh + (int64_t)(tx >> 32) + (int64_t)(ty >> 32) + (low >> 32);
}

// Sliding state of one line.  The differences d_-4..d_3 of interface t sit in
// d[(t + k) % 8], k = 0..7, so that a march unrolled by 8 moves no registers.
struct Mp9Int {
  int64_t d[8];
  int64_t v;     // the newest value F_{s+4}
  int64_t c0;    // magnitude of the curvature C_s
  int32_t s0;    // and its sign mask
  int64_t dmm;   // magnitude of DM- (the previous interface's DM+)
  int32_t smm;   // and its sign mask
};

__device__ __forceinline__ int64_t wide(int32_t s) {
  return (int64_t)(((uint64_t)(uint32_t)s << 32) | (uint32_t)s);
}

// DM = minmod4(4a - b, 4b - a, a, b) of curvatures given as magnitudes and
// sign masks: 0 unless the signs agree, else min(m, 4m - M) if positive (m
// the smaller magnitude, M the larger).  Returns its magnitude; its sign is
// that of either.
__device__ __forceinline__ int64_t dm_int(int64_t ma, int32_t sa, int64_t mb, int32_t sb) {
  const bool a_small = ma < mb;
  const int64_t m = a_small ? ma : mb, M = a_small ? mb : ma;
  const int64_t u = (int64_t)(4 * (uint64_t)m - (uint64_t)M);
  const int64_t r = u < m ? u : m;
  const int32_t off = ((int32_t)(u >> 32) | (sa ^ sb)) >> 31;  // -1: zero
  return r & ~wide(off);
}

// The offset of the interface value from the upwind value, limited:
// Fhat - F_s of interface t (J = t % 8); c1, s1 and dmp are C_{s+1} and DM+
// for the next interface.
template <int J>
__device__ __forceinline__ int64_t mp9_offset_int(const Mp9Int& L, int64_t& c1, int32_t& s1,
                                                  int64_t& dmp) {
#define FDLB_D(k) L.d[(J + (k)) & 7]
  const int64_t d0 = FDLB_D(4), dm1 = FDLB_D(3);
  // 2520 (F^L - F_s) = sum c_k d_k, |c| = 4 37 162 479 1120 255 50 5: the
  // high words exactly, the low words of each sign apart, then >> 10 and
  // times 1024/2520 as a 64-bit fraction
  int64_t ah = 0;
  uint64_t lp = 0, ln = 0;
#define FDLB_T(k, c)                                                                \
  {                                                                                 \
    ah += (int64_t)(c) * (int32_t)(FDLB_D(k) >> 32);                                \
    if ((c) > 0) lp += (uint64_t)(uint32_t)((c) > 0 ? (c) : 0) * (uint32_t)FDLB_D(k); \
    else ln += (uint64_t)(uint32_t)((c) > 0 ? 0 : -(c)) * (uint32_t)FDLB_D(k);      \
  }
  FDLB_T(0, -4) FDLB_T(1, 37) FDLB_T(2, -162) FDLB_T(3, 479)
  FDLB_T(4, 1120) FDLB_T(5, -255) FDLB_T(6, 50) FDLB_T(7, -5)
#undef FDLB_T
  const int64_t t = (int64_t)((uint64_t)ah << 22) + ((int64_t)(lp - ln) >> 10);
  constexpr int32_t kh = 0x68068068, kl = 0x06806806;  // 1024/2520 * 2^64
  const int32_t th = (int32_t)(t >> 32);
  const int64_t mid = (int64_t)th * kl + (int64_t)((uint64_t)(uint32_t)t * (uint32_t)kh);
  const int64_t a = (int64_t)th * kh + (mid >> 32);
  // curvature C_{s+1} and DM+
  const int64_t c = FDLB_D(5) - d0;
  s1 = (int32_t)(c >> 63);
  c1 = c ^ wide(s1);
  dmp = dm_int(L.c0, L.s0, c1, s1);
  // Both intervals [min(0, .., ..), max(0, .., ..)] of the limiter hold 0, so
  // only the bounds on a's side count: with every quantity reflected to a's
  // sign, Fhat - F_s = max(0, min(a, max(d_0, md), max(ul, lc))).
  const int32_t sg = (int32_t)(a >> 63);
  const int64_t w = wide(sg);
  const int64_t e0 = d0 ^ w, em = dm1 ^ w;
  const int64_t ep = dmp ^ wide(L.s0 ^ sg), en = L.dmm ^ wide(L.smm ^ sg);
  const int64_t md = (e0 - ep) >> 1;
  const int64_t ul = (int64_t)((uint64_t)em << 2);
  // lc = em/2 + (4/3) DM-; x/3 = x * 0x5555555555555555 / 2^64
  constexpr int32_t k3 = 0x55555555;
  const int64_t p3 = (int64_t)(int32_t)(en >> 32) * k3;
  const int64_t q3 = p3 + (int64_t)((uint64_t)(uint32_t)en * (uint32_t)k3);
  const int64_t lc = (em >> 1) + en + p3 + (q3 >> 32);
  const int64_t b1 = e0 < md ? md : e0, b2 = ul < lc ? lc : ul;
  int64_t r = a ^ w;
  r = r < b1 ? r : b1;
  r = r < b2 ? r : b2;
  return (r & ~wide((int32_t)(r >> 63))) ^ w;
#undef FDLB_D
}

// The cells of a line as integers: stored so, or binary64 values scaled as
// they're read.
struct IntCells {
  const int64_t* p;
  __device__ __forceinline__ int64_t operator[](int i) const { return p[i]; }
};
struct ScaledCells {
  const double* p;
  int emax;
  __device__ __forceinline__ int64_t operator[](int i) const { return q_of(p[i], emax); }
};

// The window of the first interface: F_{s-4}..F_{s+4} at p[(j - 4) ss].
template <typename Cells>
__device__ __forceinline__ void mp9_start_int(Mp9Int& L, const Cells& p, int ss) {
  int64_t v = p[-4 * ss];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int64_t x = p[(k - 3) * ss];
    L.d[k] = x - v;
    v = x;
  }
  L.v = v;
  const int64_t cm = L.d[3] - L.d[2], c = L.d[4] - L.d[3];
  const int32_t sm = (int32_t)(cm >> 63);
  L.s0 = (int32_t)(c >> 63);
  L.c0 = c ^ wide(L.s0);
  L.dmm = dm_int(cm ^ wide(sm), sm, L.c0, L.s0);
  L.smm = sm;
}

// One step of the march: interface J (mod 8), then the window moves on.
template <int J>
__device__ __forceinline__ int64_t mp9_step_int(Mp9Int& L, int64_t vnew, bool more) {
  int64_t c1, dmp;
  int32_t s1;
  const int64_t r = mp9_offset_int<J>(L, c1, s1, dmp);
  if (more) {
    L.d[J & 7] = vnew - L.v;
    L.v = vnew;
    L.dmm = dmp;
    L.smm = L.s0;
    L.c0 = c1;
    L.s0 = s1;
  }
  return r;
}

// March the NC + 1 interfaces around NC cells (NC a multiple of 8, or less
// than 8) upwind to downwind and write each cell's flux difference
// sgn (Fhat_right - Fhat_left) = d_-1 + a_cur - a_prev, in units of the scale,
// at out[t * ostep] (|.| < 2^62.4: two offsets below 2^61 and a difference); `p`
// points at the upwind cell of the first interface, ss is the signed element
// stride.
template <int NC, typename Cells>
__device__ __forceinline__ void mp9_march_delta(Cells p, int ss, int64_t* __restrict__ out, int ostep) {
  constexpr int NB = NC >= 8 ? NC / 8 : 1;   // blocks of NU interfaces
  constexpr int NU = NC >= 8 ? 8 : NC;
  static_assert(NB * NU == NC, "whole blocks");
  Mp9Int L;
  mp9_start_int(L, p, ss);
  int64_t dprev = L.d[4];  // d_-1 of the next interface
  int64_t aprev = mp9_step_int<0>(L, p[5 * ss], true);
#define FDLB_STEP(j)                                                               \
  if constexpr ((j) < NU) {                                                        \
    const bool more = NB > 1 || (j) + 1 < NU;                                      \
    const int64_t dm1 = dprev;                                                     \
    dprev = L.d[((j) + 1 + 4) & 7];                                                \
    const int64_t vn = more ? p[(6 + (j)) * ss] : 0;                               \
    const int64_t a = mp9_step_int<((j) + 1) & 7>(L, vn, more);                    \
    out[(j) * ostep] = dm1 + a - aprev;                                            \
    aprev = a;                                                                     \
  }
#pragma unroll 1
  for (int b = 0; b < NB; ++b) {
    FDLB_STEP(0) FDLB_STEP(1) FDLB_STEP(2) FDLB_STEP(3)
    FDLB_STEP(4) FDLB_STEP(5) FDLB_STEP(6) FDLB_STEP(7)
    p.p += 8 * ss;
    out += 8 * ostep;
  }
#undef FDLB_STEP
}
template <int NC>
__device__ __forceinline__ void mp9_march_delta_int(const int64_t* p, int ss, int64_t* out, int ostep) {
  mp9_march_delta<NC>(IntCells{p}, ss, out, ostep);
}

// The scale (largest biased exponent) of the values that march reads for NC
// cells, and whether fixed point takes the line.
template <int NC>
__device__ __forceinline__ bool scale_of_line(const double* p, int ss, int& emax) {
  int mx = 0, mn = 0x7fffffff;
#pragma unroll
  for (int k = -4; k <= NC + 4; ++k) {
    const int m = mag_word(p[k * ss]);
    mx = mx < m ? m : mx;
    if (k >= 1 && k <= NC) mn = m < mn ? m : mn;
  }
  emax = mx >> 20;
  return takes_fixed_point(mx, mn);
}

// The same flux differences in binary64 (their bits), for tiles the
// fixed-point march does not take.  The window slides (15 binary64 operations
// an interface) in a loop that isn't unrolled (kept small).
__device__ __noinline__ void mp9_march_delta_fp64(const double* p, int ss, int64_t* out, int ostep,
                                                  int nc) {
  Mp9Line L;
  double v = p[-4 * ss];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const double x = p[(k - 3) * ss];
    L.d[k] = x - v;
    v = x;
  }
  L.c0 = L.d[4] - L.d[3];
  L.dmm = dm_bits(L.d[3] - L.d[2], L.c0);
  double prev = 0.0;
#pragma unroll 1
  for (int t = 0; t <= nc; ++t) {
    double c1;
    long long dmp;
    L.fs[0] = p[t * ss];
    const double f = mp9_face_fp64(L, c1, dmp);
    if (t > 0) out[(t - 1) * ostep] = dbits(f - prev);
    prev = f;
    if (t < nc) {
      const double x = p[(t + 5) * ss];
#pragma unroll
      for (int k = 0; k < 7; ++k) L.d[k] = L.d[k + 1];
      L.d[7] = x - v;
      v = x;
      L.c0 = c1;
      L.dmm = dmp;
    }
  }
}

// |cx| dx + |cy| dy of flux differences of which one or both are binary64 bits
// (exponent 0).  A call, so that the compiler does not run its binary64
// operations beside the fixed-point ones and select.
__device__ __noinline__ double advection_fp64(double cx, double cy, int64_t dx, int ex, int64_t dy, int ey) {
  const double x = ex ? q_to_double(dx, ex) : dfrom(dx), y = ey ? q_to_double(dy, ey) : dfrom(dy);
  return fma(fabs(cy), y, fabs(cx) * x);
}

}  // namespace fdlb
