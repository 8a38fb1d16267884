// Host check of the chunked landing (chunk_offset, chunk_slot) on arrays whose
// rows are padded to whole 16-cell tiles, and the rule that pads them.
#include "tile_index_host.cpp"

// Every tile of an nx x ny grid in a padded array: chunks aligned and inside
// the array, and every staged position reading a copied slot that holds the
// cell it needs, never the padding.
extern "C" int check_padded_chunks(int nx, int ny, int bc) {
  bad = 0;
  const int TX = 16, TY = 16, H = kGhost;
  const int pitch = (nx + 15) / 16 * 16, rows = (ny + 15) / 16 * 16;
  const int NCHK = chunk_count(TX, TY), NSC = staged_count(2, TX, TY);
  for (int y0 = 0; y0 < ny; y0 += TY)
    for (int x0 = 0; x0 < nx; x0 += TX) {
      std::vector<long> land(4 * NCHK, -1);  // array offset held by each slot
      for (int q = 0; q < NCHK; ++q) {
        const int o = chunk_offset(q, TX, TY, x0, y0, nx, ny, bc, pitch);
        if (o < 0) {
          CHECK(bc == 0, "periodic chunks are always copied");
          continue;
        }
        CHECK(o % 4 == 0 && o + 3 < pitch * rows, "chunk q=%d offset %d", q, o);
        CHECK(o / pitch < ny && o % pitch < nx && o % pitch + 3 < pitch, "chunk q=%d within its row", q);
        for (int k = 0; k < 4; ++k) land[4 * q + k] = o + k;
      }
      for (int e = 0; e < NSC; ++e) {
        int r, c;
        staged_pos(e, 2, TX, TY, r, c);
        // (what lies right of a ragged tile's halo feeds no cell of the grid)
        const int s = chunk_slot(r, c, TX, TY, x0, nx, bc);
        CHECK(s >= 0 && s < 4 * NCHK, "slot e=%d s=%d", e, s);
        if (!(s >= 0 && s < 4 * NCHK)) continue;
        const long want = (long)wrap_or_clamp(y0 - H + r, ny, bc) * pitch + wrap_or_clamp(x0 - H + c, nx, bc);
        CHECK(land[s] == want, "tile (%d,%d) e=%d reads %ld, needs %ld", x0, y0, e, land[s], want);
      }
    }
  return bad;
}

extern "C" int pads(long long nx, long long ny) { return pads_to_tiles(nx, ny); }
