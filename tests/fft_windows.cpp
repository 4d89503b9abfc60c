// Restates, for every tile that the planner makes of a map, which FFTs of each bin meet it, row by row
// from the fixed-point tables, and counts the FFTs that the kernel's window leaves out or takes for a
// cover of the tile where they are none.  Cases on stdin, one per line:
//   n df bin_lo bin_hi n_fft t_first n_k k_min_rows dk_cols rows cols
// (dk_cols: x0 columns that the last FFT moves per k row; rows = 0: planned tiles, two blocks on each
// of 152 SMs; rows = -1: those of a plan that is executed once.)  Prints per case: tiles, FFTs that meet a tile, missed ones, false covers, covers.
#include "../paper_1810_09784_gb300/csrc/gfh_host.cpp"

#include <cstdio>

static int64_t floor_shift(int64_t v) { return v >> GFH_FRAC_BITS; }

int main() {
  gfh_grid g{};
  double k_min_rows, dk_cols;
  int rows, cols;
  while (std::scanf("%lf %lf %d %d %d %lf %d %lf %lf %d %d", &g.n, &g.df, &g.bin_lo, &g.bin_hi, &g.n_fft,
                    &g.t_first, &g.n_k, &k_min_rows, &dk_cols, &rows, &cols) == 11) {
    g.t_hop = 1.0;
    g.f_max = (double)g.bin_hi * g.df;
    const double m = slope_of(&g), t_last = g.t_first + (g.n_fft - 1) * g.t_hop;
    g.t_obs = t_last + g.t_hop;
    g.dk = dk_cols * m * g.df / std::pow(g.f_max, g.n) / (m * t_last);
    g.k_min = k_min_rows * g.dk;
    g.ana_lo = g.bin_lo * g.df;
    g.ana_hi = g.bin_hi * g.df;
    g.band_hz = g.ana_hi - g.ana_lo;
    if (gfh_grid_make(&g) != GFH_OK) { std::printf("bad grid\n"); return 1; }
    std::vector<HostMap> hms(1);
    HostMap& hm = hms[0];
    if (gfh_host_tables(&g, hm.U, hm.B, hm.S) || gfh_host_columns(&g, hm.band, hm.f0, hm.f0n)) return 1;
    find_analysis_columns(hm);
    std::vector<TileDev> tiles;
    hm.one = sparse_map(g, hm, false);
    if (rows < 0) {
      sampled_tiles(g, hm, 0, kRoom[2], 304, tiles);
    } else if (rows > 0) {
      cut_tiles(g, hm, 0, 0, g.n_k, 0, g.ld_x0, rows, cols, tiles);
    } else {
      map_tiles(g, hm, 0, kRoom[2], 0, g.n_k, 0, g.ld_x0, tiles);
      std::vector<double> work;
      for (const TileDev& t : tiles) work.push_back(tile_work(g, hm, t));
      balance_tiles({g}, hms, 304, tiles, work);
    }
    const ShiftLine sl = shift_line(hm);
    long long meet = 0, missed = 0, covers = 0, wrong = 0;
    for (const TileDev& t : tiles) {
      const int ub = std::min<int64_t>(t.ncols - 1, g.n_x0 - 1 - t.col0);
      const TileLine line = tile_line(sl, t.row0, (int64_t)t.row0 + t.nrows - 1);
      // the tile's bins, and the next on either side, of which no FFT may meet it
      const bool none = t.bin_a > t.bin_b;
      for (int j = none ? g.bin_lo : std::max(g.bin_lo, t.bin_a - 1); j <= (none ? g.bin_hi : std::min(g.bin_hi, t.bin_b + 1)); ++j) {
        const bool read = j >= t.bin_a && j <= t.bin_b;
        const int64_t left = hm.U[j - g.bin_lo + 1], right = hm.U[j - g.bin_lo] - 1;
        const BinFfts w = bin_ffts(line, left, right, t.col0, ub, ub == t.ncols - 1, g.n_fft);
        for (int i = 0; i < g.n_fft; ++i) {
          const int64_t first = hm.B[i] + t.row0 * hm.S[i] + (t.col0 << GFH_FRAC_BITS);
          const int64_t last = first + (t.nrows - 1) * hm.S[i];
          const bool in = floor_shift(right - first) >= 0 && floor_shift(left - last) <= ub;
          const bool cover = floor_shift(left - first) <= 0 && floor_shift(right - last) >= ub;
          const bool counted = i >= w.lo && i <= w.hi && i > w.c_lo && i < w.c_hi;
          meet += in;
          missed += in && (!read || i < w.lo || i > w.hi);
          covers += counted;
          wrong += counted && !cover;
        }
      }
    }
    std::printf("%zu %lld %lld %lld %lld\n", tiles.size(), meet, missed, wrong, covers);
  }
  return 0;
}
