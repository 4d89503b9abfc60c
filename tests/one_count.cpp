// Whether maps are drawn with one count per cell: n bin_lo nb n_fft n_k k_min_rows dk_cols on stdin, a grid
// of half-Hz bins, an FFT a second; prints 0 or 1, and 1 or 0 where the map takes the x-direction form.
#include "../paper_1810_09784_gb300/csrc/gfh_host.cpp"

#include <cstdio>

int main() {
  gfh_grid g{};
  int nb;
  double k_min_rows, dk_cols;
  while (std::scanf("%lf %d %d %d %d %lf %lf", &g.n, &g.bin_lo, &nb, &g.n_fft, &g.n_k, &k_min_rows, &dk_cols) == 7) {
    g.df = 0.5;
    g.bin_hi = g.bin_lo + nb - 1;
    g.t_first = g.t_hop = 1.0;
    g.t_obs = g.n_fft + 1.0;
    g.f_max = g.bin_hi * g.df;
    const double m = slope_of(&g);
    g.dk = dk_cols * m * g.df / std::pow(g.f_max, g.n) / (m * g.t_obs);
    g.k_min = k_min_rows * g.dk;
    g.ana_lo = g.bin_lo * g.df;
    g.ana_hi = (g.bin_hi + 1) * g.df;
    g.band_hz = 1.0;
    HostMap hm;
    if (gfh_grid_make(&g) || gfh_host_tables(&g, hm.U, hm.B, hm.S)) return 1;
    const bool xd = hm.S.back() > (int64_t(2) << GFH_FRAC_BITS);
    std::printf("%d %d\n", (int)sparse_map(g, hm, xd), (int)xd);
  }
  return 0;
}
