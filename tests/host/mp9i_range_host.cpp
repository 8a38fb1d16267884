// Host build of the choice between the fixed-point and the binary64 MP-9 march
// (fdlb_mp9i.cuh) for CPU unit tests.
#include "mp9i_host.cpp"

extern "C" double q_value(int64_t u, int ex) { return fdlb::q_to_double(u, ex); }

// Flux differences of the 16 own cells of a line with 5 ghosts per side, marched
// as its two half lines of 8 cells: each on its own scale where fixed point
// takes it, else in binary64.  Returns which were scaled (bit 0: cells 0-7).
extern "C" int mp9i_choice(const double* ext, int sgn, double* out) {
  int scaled = 0;
  for (int h = 0; h < 2; ++h) {
    const int first = 8 * h + (sgn > 0 ? 0 : 7);
    const double* up = ext + 5 + first - sgn;
    int64_t q[16];
    int emax;
    const bool fixed = fdlb::scale_of_line<8>(up, sgn, emax);
    if (fixed) fdlb::mp9_march_delta<8>(fdlb::ScaledCells{up, emax}, sgn, q + first, sgn);
    else fdlb::mp9_march_delta_fp64(up, sgn, q + first, sgn, 8);
    for (int i = 8 * h; i < 8 * h + 8; ++i) out[i] = fixed ? fdlb::q_to_double(q[i], emax) : fdlb::dfrom(q[i]);
    scaled |= (int)fixed << h;
  }
  return scaled;
}

// |cx| dx + |cy| dy in units of the larger of two scales
extern "C" double adv_two_scales(double cx, double cy, int64_t dx, int ex, int64_t dy, int ey) {
  int ec;
  const fdlb::AdvCoef c = fdlb::advection_coef(cx, cy, ec);
  const int e = ex > ey ? ex : ey;
  return fdlb::q_to_double(fdlb::advection_int(c, fdlb::sar64(dx, e - ex), fdlb::sar64(dy, e - ey)), e + ec);
}
extern "C" double adv_fp64(double cx, double cy, int64_t dx, int ex, int64_t dy, int ey) {
  return fdlb::advection_fp64(cx, cy, dx, ex, dy, ey);
}
