// Host build of the choice between the fixed-point and the binary64 MP-9 march
// (fdlb_mp9i.cuh) for CPU unit tests.
#include "mp9i_host.cpp"

// Flux differences of the 16 own cells of a line with 5 ghosts per side, taken
// as a tile: scaled by the largest magnitude of all 26 values if the own cells
// lie close enough to it, else marched in binary64.  Returns whether scaled.
extern "C" int mp9i_choice(const double* ext, int sgn, double* out) {
  int mx = 0, mn = 0x7fffffff;
  for (int i = 0; i < 26; ++i) {
    const int w = fdlb::mag_word(ext[i]);
    mx = w > mx ? w : mx;
    if (i >= 5 && i < 21) mn = w < mn ? w : mn;
  }
  const bool fixed = fdlb::takes_fixed_point(mx, mn);
  if (fixed) mp9i_line(ext, 16, sgn, 8, out);
  else mp9_delta64(ext, 16, sgn, out);
  return fixed;
}
