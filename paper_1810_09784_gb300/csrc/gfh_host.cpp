// Host side of libgfh: grid derivation (Sec. VI), fixed-point tables, column tables, contexts and
// plans.  Compiled with -ffp-contract=off so that every double expression rounds exactly as
// written (no fused multiply-add), which the bit-exact tables rely on.
#include <algorithm>
#include <functional>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <numeric>
#include <string>

#include "gfh_internal.h"

namespace {

int64_t fixed_floor(double v) { return (int64_t)std::floor(std::ldexp(v, GFH_FRAC_BITS)); }

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// n = 0 selects the original FrequencyHough (Sec. III Eq. fdotslope): x = -f, x0 = -f0 and
// x0 = x - k t with k = -fdot, the orientation and slope convention of Eq. transform's
// x0 = x - (n-1) k t with (n-1) replaced by 1.  Only this form accepts k < 0 (spin-up).
bool original_fh(const gfh_grid* g) { return g->n == 0.0; }

double slope_of(const gfh_grid* g) { return original_fh(g) ? 1.0 : g->n - 1.0; }

// x of frequency f: Eq. transform (n > 1) or -f (n = 0).
double x_of_f(const gfh_grid* g, double f) {
  return original_fh(g) ? -f : std::pow(f, 1.0 - g->n);
}

bool grid_request_ok(const gfh_grid* g) {
  return g && (g->n > 1.0 || g->n == 0.0) && g->df > 0.0 && g->bin_lo >= 1 &&
         g->bin_hi >= g->bin_lo && g->n_fft >= 1 && g->n_k >= 1 && g->t_first >= 0.0 &&
         g->t_hop >= 0.0 && g->t_obs > 0.0 && (g->k_min >= 0.0 || g->n == 0.0) &&
         std::isfinite(g->k_min) && g->ana_hi > g->ana_lo && g->band_hz > 0.0 &&
         std::isfinite(g->n) && std::isfinite(g->df);
}

bool grid_made(const gfh_grid* g) {
  return grid_request_ok(g) && g->dx0 > 0.0 && g->dk > 0.0 && g->n_x0 > 0 &&
         g->ld_x0 >= g->n_x0 && g->n_bands > 0;
}

}  // namespace

extern "C" const char* gfh_strerror(int code) {
  switch (code) {
    case GFH_OK: return "ok";
    case GFH_ERR_ARG: return "invalid argument";
    case GFH_ERR_SIZE: return "size out of range or capacity too small";
    case GFH_ERR_CUDA: return "CUDA or cuFFT call failed";
    case GFH_ERR_INPUT: return "device-side input check failed (unsorted peaks or index out of range)";
    case GFH_ERR_TIMEOUT: return "bounded device-side wait ran out";
    case GFH_ERR_NOMEM: return "allocation failed";
    default: return "unknown error";
  }
}

// ---- Sec. VI grids ----------------------------------------------------------------------------

extern "C" int gfh_grid_make(gfh_grid* g) {
  if (!grid_request_ok(g)) return GFH_ERR_ARG;
  const double n = g->n;
  const double m = slope_of(g);
  if (!(g->f_max > 0.0)) g->f_max = (double)g->bin_hi * g->df;
  g->dx0 = m * g->df / std::pow(g->f_max, n);                        // Sec. VI.C (df for n = 0)
  if (!(g->dk > 0.0)) g->dk = g->dx0 / (m * g->t_obs);
  const double k_max = g->k_min + (double)(g->n_k - 1) * g->dk;
  const double t_max = g->t_first + (double)(g->n_fft - 1) * g->t_hop;
  const double x_top = x_of_f(g, ((double)g->bin_hi + 0.5) * g->df);  // Eq. transform
  const double x_bot = x_of_f(g, ((double)g->bin_lo - 0.5) * g->df);
  // lowest x0 of any line: x_top moved by the largest positive k; highest: x_bot moved by the most
  // negative k (none for k_min >= 0)
  g->x0_min = x_top - m * (k_max > 0.0 ? k_max : 0.0) * t_max - g->dx0;
  const double x0_hi = g->k_min < 0.0 ? x_bot - m * g->k_min * t_max : x_bot;
  const double w = std::ceil((x0_hi - g->x0_min) / g->dx0);
  if (!(g->dx0 > 0.0) || !std::isfinite(w) || w < 0.0 || w > 2.0e9) return GFH_ERR_SIZE;
  g->n_x0 = (int64_t)w + 1;
  g->ld_x0 = (g->n_x0 + 31) / 32 * 32;
  const double nb = std::ceil((g->ana_hi - g->ana_lo) / g->band_hz);
  if (!(nb >= 1.0) || nb > 1.0e8) return GFH_ERR_ARG;
  g->n_bands = (int32_t)nb;
  return GFH_OK;
}

int gfh_host_tables(const gfh_grid* g, std::vector<int64_t>& U, std::vector<int64_t>& B,
                    std::vector<int64_t>& S) {
  if (!grid_made(g)) return GFH_ERR_ARG;
  const int J = g->bin_hi - g->bin_lo + 1;
  U.resize((size_t)J + 1);
  for (int e = 0; e <= J; ++e) {
    const double f = ((double)(g->bin_lo + e) - 0.5) * g->df;
    const double x = x_of_f(g, f);
    U[e] = fixed_floor((x - g->x0_min) / g->dx0);
  }
  B.resize(g->n_fft);
  S.resize(g->n_fft);
  const double m = slope_of(g);
  for (int i = 0; i < g->n_fft; ++i) {
    const double t = g->t_first + (double)i * g->t_hop;
    B[i] = fixed_floor(m * g->k_min * t / g->dx0);
    S[i] = fixed_floor(m * g->dk * t / g->dx0);
  }
  return GFH_OK;
}

int gfh_host_columns(const gfh_grid* g, std::vector<int32_t>& band, std::vector<double>& f0,
                     std::vector<double>& f0n) {
  if (!grid_made(g)) return GFH_ERR_ARG;
  const int64_t W = g->n_x0;
  band.assign((size_t)g->ld_x0, -1);
  f0.assign((size_t)W, 0.0);
  f0n.assign((size_t)W, 0.0);
  const double e = -1.0 / (g->n - 1.0);
  for (int64_t m = 0; m < W; ++m) {
    const double x0c = g->x0_min + ((double)m + 0.5) * g->dx0;
    const double f = original_fh(g) ? -x0c : (x0c > 0.0 ? std::pow(x0c, e) : 0.0);
    if (!(f > 0.0)) continue;
    f0[m] = f;
    f0n[m] = std::pow(f, g->n);
    if (g->ana_lo <= f && f < g->ana_hi) {
      int32_t b = (int32_t)std::floor((f - g->ana_lo) / g->band_hz);
      if (b > g->n_bands - 1) b = g->n_bands - 1;
      band[m] = b;
    }
  }
  return GFH_OK;
}

extern "C" int gfh_grid_tables(const gfh_grid* g, int64_t* h_U, int64_t* h_B, int64_t* h_S) {
  std::vector<int64_t> U, B, S;
  int rc = gfh_host_tables(g, U, B, S);
  if (rc) return rc;
  if (h_U) std::memcpy(h_U, U.data(), U.size() * sizeof(int64_t));
  if (h_B) std::memcpy(h_B, B.data(), B.size() * sizeof(int64_t));
  if (h_S) std::memcpy(h_S, S.data(), S.size() * sizeof(int64_t));
  return GFH_OK;
}

extern "C" int gfh_grid_columns(const gfh_grid* g, int32_t* h_band, double* h_f0, double* h_f0n) {
  std::vector<int32_t> band;
  std::vector<double> f0, f0n;
  int rc = gfh_host_columns(g, band, f0, f0n);
  if (rc) return rc;
  if (h_band) std::memcpy(h_band, band.data(), (size_t)g->n_x0 * sizeof(int32_t));
  if (h_f0) std::memcpy(h_f0, f0.data(), f0.size() * sizeof(double));
  if (h_f0n) std::memcpy(h_f0n, f0n.data(), f0n.size() * sizeof(double));
  return GFH_OK;
}

// ---- contexts -----------------------------------------------------------------------------------

extern "C" int gfh_create(gfh_ctx** out, int device, void* stream) {
  if (!out) return GFH_ERR_ARG;
  *out = nullptr;
  int count = 0;
  if (cudaGetDeviceCount(&count) != cudaSuccess || device < 0 || device >= count)
    return GFH_ERR_CUDA;
  GFH_CUDA_TRY(cudaSetDevice(device));
  gfh_ctx* c = new (std::nothrow) gfh_ctx();
  if (!c) return GFH_ERR_NOMEM;
  c->device = device;
  c->stream = (cudaStream_t)stream;
  if (cudaDeviceGetAttribute(&c->num_sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
      cudaMalloc(&c->d_flag, sizeof(unsigned int)) != cudaSuccess ||
      cudaMemset(c->d_flag, 0, sizeof(unsigned int)) != cudaSuccess ||
      cudaMallocHost(&c->h_pinned, 64) != cudaSuccess) {
    gfh_destroy(c);
    return GFH_ERR_CUDA;
  }
  // image channel 0 for small peak counts: bf16 (round to nearest even) of float(log1p(count))
  std::vector<uint16_t> tab(kLogTable);
  for (int i = 0; i < kLogTable; ++i) {
    const float f = (float)std::log1p((double)i);
    uint32_t u;
    std::memcpy(&u, &f, 4);
    tab[i] = (uint16_t)((u + 0x7fffu + ((u >> 16) & 1u)) >> 16);
  }
  if (cudaMalloc(&c->d_log1p, kLogTable * sizeof(uint16_t)) != cudaSuccess ||
      cudaMemcpy(c->d_log1p, tab.data(), kLogTable * sizeof(uint16_t), cudaMemcpyHostToDevice) !=
          cudaSuccess) {
    gfh_destroy(c);
    return GFH_ERR_CUDA;
  }
  *out = c;
  return GFH_OK;
}

extern "C" int gfh_destroy(gfh_ctx* c) {
  if (!c) return GFH_OK;
  cudaSetDevice(c->device);
  if (c->stream) cudaStreamSynchronize(c->stream);
  for (auto& f : c->fft)
    if (f.valid) cufftDestroy(f.h);
  if (c->pm_buf) cudaFree(c->pm_buf);
  if (c->d_flag) cudaFree(c->d_flag);
  if (c->h_pinned) cudaFreeHost(c->h_pinned);
  if (c->d_log1p) cudaFree(c->d_log1p);
  delete c;
  return GFH_OK;
}

extern "C" int gfh_set_stream(gfh_ctx* c, void* stream) {
  if (!c) return GFH_ERR_ARG;
  c->stream = (cudaStream_t)stream;
  for (auto& f : c->fft)
    if (f.valid && cufftSetStream(f.h, c->stream) != CUFFT_SUCCESS) return GFH_ERR_CUDA;
  return GFH_OK;
}

extern "C" int gfh_check(gfh_ctx* c) {
  if (!c) return GFH_ERR_ARG;
  GFH_CUDA_TRY(cudaSetDevice(c->device));
  unsigned int flag = 0;
  GFH_CUDA_TRY(cudaMemcpyAsync(&flag, c->d_flag, sizeof(flag), cudaMemcpyDeviceToHost, c->stream));
  GFH_CUDA_TRY(cudaStreamSynchronize(c->stream));
  if (flag) {
    GFH_CUDA_TRY(cudaMemsetAsync(c->d_flag, 0, sizeof(unsigned int), c->stream));
    GFH_CUDA_TRY(cudaStreamSynchronize(c->stream));
    if (flag & GFH_FLAG_TIMEOUT) return GFH_ERR_TIMEOUT;
    return (flag & (GFH_FLAG_UNSORTED | GFH_FLAG_FFT_RANGE)) ? GFH_ERR_INPUT : GFH_ERR_SIZE;
  }
  return GFH_OK;
}

// ---- grids on n and k (Sec. VI) -------------------------------------------------------------------

namespace {

// f(t) / f0 of Eq. powlaws at u = |fdot0| t / f0.
double powlaw_ratio(double n, double u) { return std::exp(-std::log1p((n - 1.0) * u) / (n - 1.0)); }

// Largest |f_{n2} - f_{n1}| over the f0 and u lattice of gfh_n_grid.
double dn_max_df(double n1, double n2, double f_min, double f_max, double fdot_hi, double t_obs) {
  constexpr int kF = 64, kU = 256;
  double best = 0.0;
  for (int a = 0; a < kF; ++a) {
    const double f0 = f_min * std::pow(f_max / f_min, (double)a / (kF - 1));
    const double umax = fdot_hi * t_obs / f0;
    for (int b = 0; b < kU; ++b) {
      const double u = umax * b / (kU - 1);
      const double d = f0 * std::fabs(powlaw_ratio(n2, u) - powlaw_ratio(n1, u));
      if (d > best) best = d;
    }
  }
  return best;
}

}  // namespace

extern "C" int gfh_n_grid(double n_lo, double n_hi, double df, double f_min, double f_max,
                          double fdot_hi, double t_obs, int32_t cap, double* h_n, int32_t* n_out) {
  if (!h_n || !n_out || cap < 1 || !(n_lo > 1.0) || !(n_hi >= n_lo) || !(df > 0.0) ||
      !(f_min > 0.0) || !(f_max >= f_min) || !(fdot_hi >= 0.0) || !(t_obs > 0.0))
    return GFH_ERR_ARG;
  int32_t cnt = 0;
  h_n[cnt++] = n_lo;
  double n = n_lo;
  while (n < n_hi) {
    if (cnt >= cap) { *n_out = cnt; return GFH_ERR_SIZE; }
    const double span = n_hi - n;
    if (dn_max_df(n, n + span, f_min, f_max, fdot_hi, t_obs) <= df) {
      h_n[cnt++] = n_hi;
      break;
    }
    double lo = 0.0, hi = span;
    while (hi - lo > 1e-9 * hi) {
      const double mid = 0.5 * (lo + hi);
      if (dn_max_df(n, n + mid, f_min, f_max, fdot_hi, t_obs) <= df) lo = mid;
      else hi = mid;
    }
    if (lo <= 0.0) { *n_out = cnt; return GFH_ERR_ARG; }
    n = n + lo;
    h_n[cnt++] = n;
  }
  *n_out = cnt;
  return GFH_OK;
}

extern "C" int gfh_k_segments(double n, double df, double f_min, double f_max, double fdot_lo,
                              double fdot_hi, double growth, int32_t max_rows, int32_t cap,
                              gfh_k_segment* h_out, int32_t* n_out) {
  if (!h_out || !n_out || cap < 1 || !(n > 1.0) || !(df > 0.0) || !(f_min > 0.0) ||
      !(f_max >= f_min) || !(fdot_lo > 0.0) || !(fdot_hi >= fdot_lo) || !(growth >= 1.0) ||
      max_rows < 1)
    return GFH_ERR_ARG;
  const double c = 1.0 - std::pow(1.0 + df / f_max, -n);
  const double k_lo = fdot_lo / std::pow(f_max, n), k_hi = fdot_hi / std::pow(f_min, n);
  const double full = std::floor((growth - 1.0) / c) + 1.0;
  const int32_t rows_full = full > (double)max_rows ? max_rows : (int32_t)full;
  int32_t cnt = 0;
  double k = k_lo;
  for (;;) {
    if (cnt >= cap) { *n_out = cnt; return GFH_ERR_SIZE; }
    const double dk = k * c;
    int32_t rows = rows_full;
    if (k < k_hi) {
      const double need = std::ceil((k_hi - k) / dk) + 1.0;
      if (need < (double)rows) rows = (int32_t)need;
    } else {
      rows = 1;
    }
    if (rows < 1) rows = 1;
    h_out[cnt].k_min = k;
    h_out[cnt].dk = dk;
    h_out[cnt].n_k = rows;
    h_out[cnt].reserved = 0;
    ++cnt;
    if (k + (rows - 1) * dk >= k_hi) break;
    k = k + rows * dk;
  }
  *n_out = cnt;
  return GFH_OK;
}

// ---- Sec. VI.D: longer FFTs for later times ---------------------------------------------------

namespace {

// First time at which the largest |fdot(t)| over the power laws of braking index n with
// f0 <= f_hi and |fdot0| <= fdot_hi falls to fdot.  A member's |fdot(t)| = fdot0 (1 + u)^(-n/(n-1)),
// u = (n-1) fdot0 t / f0, peaks over fdot0 at u = n-1: the bound is the fastest member's while
// t fdot_hi < f_hi and f_hi n^(-n/(n-1)) / t after that.
double time_of_spindown(double fdot, double n, double f_hi, double fdot_hi) {
  if (fdot_hi <= fdot) return 0.0;
  const double t1 = (std::pow(fdot_hi / fdot, (n - 1.0) / n) - 1.0) * f_hi / ((n - 1.0) * fdot_hi);
  if (t1 * fdot_hi < f_hi) return t1;
  return f_hi * std::pow(n, -n / (n - 1.0)) / fdot;
}

}  // namespace

extern "C" int gfh_tfft_portions(double n, double f_hi, double fdot_hi, double t_fft0,
                                 double t_obs, int32_t max_levels, int32_t cap,
                                 gfh_portion* h_out, int32_t* n_out) {
  if (!h_out || !n_out || cap < 1 || !(n > 1.0) || !std::isfinite(n) || !(f_hi > 0.0) ||
      !(fdot_hi > 0.0) || !(t_fft0 > 0.0) || !(t_obs > 0.0) || max_levels < 1 || max_levels > 30)
    return GFH_ERR_ARG;
  int32_t cnt = 0;
  for (int L = 0; L < max_levels; ++L) {
    const double T = t_fft0 * std::ldexp(1.0, L);                    // Eq. dot_tfft: fdot <= 1/T^2
    double a = time_of_spindown(1.0 / (T * T), n, f_hi, fdot_hi);
    if (a > t_obs) a = t_obs;
    double b = t_obs;
    if (L + 1 < max_levels) {
      b = time_of_spindown(1.0 / ((2.0 * T) * (2.0 * T)), n, f_hi, fdot_hi);
      if (b > t_obs) b = t_obs;
    }
    if (b - a >= T) {
      if (cnt >= cap) { *n_out = cnt; return GFH_ERR_SIZE; }
      h_out[cnt].level = L;
      h_out[cnt].reserved = 0;
      h_out[cnt].t_begin = a;
      h_out[cnt].t_end = b;
      h_out[cnt].t_fft = T;
      ++cnt;
    }
  }
  *n_out = cnt;
  return GFH_OK;
}

// ---- plans --------------------------------------------------------------------------------------

namespace {

// ceil(2^89 / s) (FftRow::D) for a shift per row s > 2^25, else 0.
uint64_t rows_per_column(int64_t s) {
  if (s <= (int64_t(1) << 25)) return 0;
  const unsigned __int128 one = 1;
  return (uint64_t)(((one << 89) + (uint64_t)s - 1) / (uint64_t)s);
}

struct HostMap {
  std::vector<int64_t> U, B, S;
  std::vector<int32_t> band;
  std::vector<double> f0, f0n;
  int64_t cells = 0;
  bool one = false;                  // sparse: one count per cell
  int64_t ana_lo = 0, ana_hi = -1;   // first and last analysis column (contiguous: f0 falls with the column)
};

// max |v_i - line| over a table, in whole units rounded up, of the line through its ends.
float line_error(const std::vector<int64_t>& v) {
  const int64_t n = (int64_t)v.size() - 1;
  if (n < 1) return 0.f;
  const __int128 d = (__int128)v[n] - v[0];
  __int128 most = 0;
  for (int64_t i = 1; i < n; ++i) {
    const __int128 e = ((__int128)v[i] - v[0]) * n - d * i;
    most = std::max(most, e < 0 ? -e : e);
  }
  const int64_t up = (int64_t)((most + n - 1) / n);
  const float f = (float)up;
  return (int64_t)f < up ? std::nextafter(f, INFINITY) : f;
}

ShiftLine shift_line(const HostMap& hm) {
  return ShiftLine{hm.B[0], hm.S[0], hm.B.back() - hm.B[0], hm.S.back() - hm.S[0],
                   line_error(hm.B), line_error(hm.S), (int32_t)hm.B.size()};
}

void find_analysis_columns(HostMap& hm) {
  const int64_t n = (int64_t)hm.band.size();
  int64_t a = 0, b = n - 1;
  while (a < n && hm.band[a] < 0) ++a;
  while (b >= a && hm.band[b] < 0) --b;
  hm.ana_lo = a;
  hm.ana_hi = b;
}

// Peaks per (FFT, bin) of noise (threshold 2.5, local maxima).
constexpr double kNoisePeaks = 0.0755;

// Whether a map is drawn with one count per cell (+1 and -1) and not with two (+1 each).  Two halve a
// tile, one makes lanes that leave the same column wait for each other.  With few peaks per x0 column a
// tile costs what its cells and chains of loads cost, and fewer, larger ones are faster: 51 half-hour
// maps (0.85 peaks per column) 7.00 -> 4.73 ms, 11 braking indices (0.15 to 12.7) 5.78 -> 4.04 ms, one
// half-hour map (1.6) 138 -> 102 us.  The line lies at two peaks per column where neighbouring peaks of a
// bin, on the map's middle row, lie two columns apart (at 2.9 to 3.1 peaks 0.81 to 0.92 of the speed, at
// 50 half of it), and falls to one where they share a column (at 1.1 to 1.6 peaks 0.85 of the speed, at
// 0.6 to 0.75 1.44 of it).
// The x-direction form counts a left column on every row, so there the line lies at one: half-hour map
// at 3 and 12 columns per row (1.6) 238 -> 176 and 202 -> 186 us with two counts, 11 braking indices at 4
// columns 2.90 -> 2.55 ms with one for the maps below one.
bool sparse_map(const gfh_grid& g, const HostMap& hm, bool xd) {
  const double per_column = kNoisePeaks * g.n_fft * (double)(g.bin_hi - g.bin_lo + 1) / (double)g.n_x0;
  if (xd) return per_column < 1.0;
  const double shift = (double)(hm.B.back() - hm.B[0]) + 0.5 * g.n_k * (double)(hm.S.back() - hm.S[0]);
  const double apart = std::fabs(shift) / 4294967296.0 / std::max(1, g.n_fft - 1) / kNoisePeaks;
  return per_column < 1.0 + std::min(1.0, 0.5 * apart);
}

// Bin range [ja, jb] of the peaks that can touch columns [c0, c1) on rows [r0, r1) (tile planning).
// For bin j (local jl) and shift s in [s_min, s_max]: lo >= (U[jl+1]-s_max)>>32 and
// hi <= (U[jl]-s_min-1)>>32; U decreases with jl, so both conditions select a contiguous range.
void tile_bins(const gfh_grid& g, const HostMap& hm, int64_t s_min, int64_t s_max, int64_t c0,
               int64_t c1, int32_t* ja, int32_t* jb) {
  const int J = g.bin_hi - g.bin_lo + 1;
  if (c0 > g.n_x0 - 1) { *ja = 1; *jb = 0; return; }
  // (selected and not branched to: a plan makes thousands of tiles, and half the branches of a bisection
  // are mispredicted)
  const int64_t right = c1 << GFH_FRAC_BITS, left = c0 << GFH_FRAC_BITS;
  int a = 0, b = 0;                      // first bins with U[jl+1] - s_max < right, U[jl] - s_min <= left
  for (int n = J; n > 0;) {
    const int half = n / 2;
    const bool more = hm.U[a + half + 1] - s_max >= right;
    a = more ? a + half + 1 : a;
    n = more ? n - half - 1 : half;
  }
  for (int n = J; n > 0;) {
    const int half = n / 2;
    const bool more = hm.U[b + half] - s_min - 1 >= left;
    b = more ? b + half + 1 : b;
    n = more ? n - half - 1 : half;
  }
  *ja = g.bin_lo + a;
  *jb = g.bin_lo + b - 1;
}

// Candidate bands of columns [c0, c1) (bands follow the columns): lo > hi when there is none.
void column_bands(const HostMap& hm, int64_t c0, int64_t c1, int32_t* lo, int32_t* hi) {
  const int64_t a = std::max(c0, hm.ana_lo), b = std::min(c1 - 1, hm.ana_hi);
  *lo = 0;
  *hi = -1;
  if (a > b) return;
  *lo = std::min(hm.band[a], hm.band[b]);
  *hi = std::max(hm.band[a], hm.band[b]);
}

TileDev make_tile(const gfh_grid& g, const HostMap& hm, int m, int r0, int nr, int64_t c0, int nc) {
  // With k_min >= 0, B and S are non-decreasing in i (dk > 0, t_i non-decreasing), so the smallest
  // shift of the rows is at (i = 0, r0) and the largest at (last i, last row).  With k_min < 0
  // (n = 0 only) the shift of FFT i on row r is (k_min + r dk) t_i up to its rounding: its extremes
  // are at the first and last FFT and row, one lattice unit per row aside.
  const int last = g.n_fft - 1, r1 = r0 + nr - 1;
  int64_t s_min = hm.B[0] + (int64_t)r0 * hm.S[0], s_max = hm.B[last] + (int64_t)r1 * hm.S[last];
  if (g.k_min < 0.0) {
    for (int i : {0, last})
      for (int r : {r0, r1}) {
        const int64_t v = hm.B[i] + (int64_t)r * hm.S[i];
        s_min = std::min(s_min, v - 2 - r1);
        s_max = std::max(s_max, v + 2 + r1);
      }
  }
  TileDev t{};
  t.map = m;
  t.row0 = r0;
  t.nrows = nr;
  t.col0 = c0;
  t.ncols = nc;
  tile_bins(g, hm, s_min, s_max, c0, c0 + nc, &t.bin_a, &t.bin_b);
  column_bands(hm, c0, c0 + nc, &t.band_lo, &t.band_hi);
  t.one = hm.one;
  return t;
}

// Work of a tile, in warp instructions: measured costs of the kernel's parts (an empty tile, one
// with edges, its cells, a run of 32 peaks and its two events per column moved), with the peaks that
// have an edge in it estimated from up to 8 of its bins along the line that the shifts follow, at
// the density of noise peaks.
double tile_work(const gfh_grid& g, const HostMap& hm, const TileDev& t) {
  const double cells = (double)t.nrows * t.ncols;
  const int nb = t.bin_b - t.bin_a + 1;
  const double fill = 2500.0 + cells / 128.0 * 3.0;
  if (nb <= 0) return fill;
  const int n = g.n_fft;
  const double one = 1.0 / 4294967296.0;
  const int64_t r0 = t.row0, r1 = r0 + t.nrows - 1;
  const double b0 = (double)(hm.B[0] + r0 * hm.S[0]) * one, b1 = (double)(hm.B[0] + r1 * hm.S[0]) * one;
  const double e0 = (double)(hm.B[n - 1] + r0 * hm.S[n - 1]) * one,
               e1 = (double)(hm.B[n - 1] + r1 * hm.S[n - 1]) * one;
  const double s0 = n > 1 ? (e0 - b0) / (n - 1) : 0.0, s1 = n > 1 ? (e1 - b1) / (n - 1) : 0.0;
  const double inv0 = s0 != 0.0 ? 1.0 / s0 : 0.0, inv1 = s1 != 0.0 ? 1.0 / s1 : 0.0;
  const int samples = std::min(nb, 8);
  const double apart = samples > 1 ? (double)(nb - 1) / (samples - 1) : 0.0;
  double ffts = 0.0, moved = 0.0;
  for (int q = 0; q < samples; ++q) {
    const int jl = t.bin_a - g.bin_lo + (int)(q * apart);
    const double hi_x = (double)hm.U[jl] * one - (double)t.col0;              // right edge
    const double lo_x = (double)hm.U[jl + 1] * one - (double)t.col0;          // left edge
    double lo = 0.0, hi = n;
    auto at_most = [&](double x, double b, double inv) {                      // b + i / inv <= x
      if (inv > 0.0) hi = std::min(hi, (x - b) * inv);
      else if (inv < 0.0) lo = std::max(lo, (x - b) * inv);
      else if (b > x) hi = lo;
    };
    at_most(hi_x, b0, inv0);                                                  // reaches the first column
    at_most(-(lo_x - t.ncols), -b1, -inv1);                                   // not past the last
    double len = std::max(0.0, hi - lo);
    const double mid = 0.5 * (lo + hi);
    if (hi_x - lo_x > t.ncols && len > 0.0) {                                 // FFTs that cover the tile
      lo = 0.0;
      hi = n;
      at_most(-(lo_x - 1.0), -b0, -inv0);
      at_most(hi_x - t.ncols, b1, inv1);
      len = std::max(0.0, len - std::max(0.0, hi - lo));
    }
    const double i = std::min(std::max(mid, 0.0), (double)(n - 1));
    ffts += len;
    moved += len * ((b1 - b0) + i * (s1 - s0));
  }
  const double runs = kNoisePeaks / 32.0 * nb / samples;
  if (ffts <= 0.0) return fill;
  return 8000.0 + cells / 128.0 * 50.0 + 8.0 * nb + runs * (190.0 * ffts + 16.0 * moved);
}

// Words of one count of a tile; its columns for given rows and words of one count.
int64_t tile_words(int rows, int cols) { return (int64_t)rows * (cols + kHoughPad); }
int cols_for(int rows, int64_t words) {
  return (int)std::min<int64_t>(4096, std::max<int64_t>(64, (words / rows - kHoughPad) / 64 * 64));
}

// Uniform tiles of map m over rows [r0, r1) x columns [c_lo, c_hi) (both multiples of 4).
void cut_tiles(const gfh_grid& g, const HostMap& hm, int m, int r0, int r1, int64_t c_lo, int64_t c_hi,
               int rows, int cols, std::vector<TileDev>& out) {
  for (int r = r0; r < r1; r += rows)
    for (int64_t x = c_lo; x < c_hi; x += cols)
      out.push_back(make_tile(g, hm, m, r, std::min(rows, r1 - r), x, (int)std::min<int64_t>(cols, c_hi - x)));
}

// Tiles of map m over rows [r0, r1) x columns [c_lo, c_hi) (both multiples of 4), of at most `room`
// words: per region of kTall rows by the columns of the flattest shape, the shape of least work.
// Tall, narrow tiles halve the peaks' fixed work with every doubling of the rows, flat wide ones suit
// regions with few edges, whose cost is the cells'.
void map_tiles(const gfh_grid& g, const HostMap& hm, int m, int64_t room, int r0, int r1,
               int64_t c_lo, int64_t c_hi, std::vector<TileDev>& tiles) {
  const int64_t words = hm.one ? room : room / 2;
  constexpr int kTall = 128, kFlat = 8;
  const int wide = cols_for(kFlat, words);
  std::vector<TileDev> best, cand;
  for (int a = r0; a < r1; a += kTall) {
    const int b = std::min(r1, a + kTall);
    for (int64_t c = c_lo; c < c_hi; c += wide) {
      const int64_t d = std::min(c_hi, c + wide);
      double best_work = -1.0;
      for (int rows = kFlat; rows <= kTall; rows *= 2) {
        cand.clear();
        cut_tiles(g, hm, m, a, b, c, d, rows, cols_for(rows, words), cand);
        double work = 0.0;
        for (const TileDev& t : cand) work += tile_work(g, hm, t);
        if (best_work < 0.0 || work < best_work) { best_work = work; best.swap(cand); }
        if (rows >= b - a) break;
      }
      tiles.insert(tiles.end(), best.begin(), best.end());
    }
  }
}

// One shape for all of map m, by the estimated time of a few sampled tiles of each: for a plan that is
// executed once (map_tiles and balance_tiles take a few hundred us, more than they save one search).
void sampled_tiles(const gfh_grid& g, const HostMap& hm, int m, int64_t room, int blocks,
                   std::vector<TileDev>& tiles) {
  const int64_t words = hm.one ? room : room / 2;
  const int K = g.n_k;
  int best_rows = 0, best_cols = 0;
  double best = 0.0;
  for (int rows = 8; rows <= 128; rows *= 2) {
    const int nr = std::min(rows, K), most = cols_for(rows, words);
    for (int cols = most; cols >= std::max(32, most / 4); cols = cols / 2 & ~3) {
      const int64_t W = g.ld_x0, down = (K + nr - 1) / nr, across = (W + cols - 1) / cols;
      double sum = 0.0, longest = 0.0;
      int n = 0;
      for (int64_t i = 0; i < std::min<int64_t>(down, 4); ++i)
        for (int64_t j = 0; j < std::min<int64_t>(across, 4); ++j, ++n) {
          const int64_t r = down > 1 ? i * (down - 1) / (std::min<int64_t>(down, 4) - 1) * nr : 0;
          const int64_t c = across > 1 ? j * (across - 1) / (std::min<int64_t>(across, 4) - 1) * cols : 0;
          const double w = tile_work(g, hm, make_tile(g, hm, m, (int)r, (int)std::min<int64_t>(nr, K - r), c,
                                                      (int)std::min<int64_t>(cols, W - c)));
          sum += w;
          longest = std::max(longest, w);
        }
      const double time = sum / n * (double)(down * across) / blocks + 0.5 * longest;
      if (best_rows == 0 || time < best) { best = time; best_rows = nr; best_cols = cols; }
    }
    if (rows >= K) break;
  }
  cut_tiles(g, hm, m, 0, K, 0, g.ld_x0, best_rows, best_cols, tiles);
}

// Halves the tiles that hold more than `most` work, across columns or rows as makes the least of it.
void split_tiles(const std::vector<gfh_grid>& grids, const std::vector<HostMap>& hms, double most,
                 std::vector<TileDev>& tiles, std::vector<double>& work) {
  for (size_t q = 0; q < tiles.size(); ++q) {
    while (work[q] > most) {
      const TileDev t = tiles[q];
      const gfh_grid& g = grids[t.map];
      const HostMap& hm = hms[t.map];
      TileDev a{}, b{};
      double wa = 0.0, wb = 0.0;
      bool found = false;
      auto offer = [&](const TileDev& x, const TileDev& y) {
        const double u = tile_work(g, hm, x), v = tile_work(g, hm, y);
        if (!found || std::max(u, v) + 0.5 * (u + v) < std::max(wa, wb) + 0.5 * (wa + wb)) {
          a = x; b = y; wa = u; wb = v;
          found = true;
        }
      };
      if (t.ncols >= 16) {
        const int h = (t.ncols / 2 + 3) & ~3;
        offer(make_tile(g, hm, t.map, t.row0, t.nrows, t.col0, h),
              make_tile(g, hm, t.map, t.row0, t.nrows, t.col0 + h, t.ncols - h));
      }
      if (t.nrows >= 2) {
        const int h = (t.nrows + 1) / 2;
        offer(make_tile(g, hm, t.map, t.row0, h, t.col0, t.ncols),
              make_tile(g, hm, t.map, t.row0 + h, t.nrows - h, t.col0, t.ncols));
      }
      if (!found || std::max(wa, wb) > 0.9 * work[q]) break;
      tiles[q] = a;
      work[q] = wa;
      tiles.push_back(b);
      work.push_back(wb);
    }
  }
}

// Splits the tiles (in place, with their work) so that `blocks` blocks that run at a time finish
// together: in steps down to a sixth of a block's share of the whole, and to no less than
// what a tile with edges costs at all, keeping the step whose estimated time is least.  A split
// repeats a tile's fixed work and the peaks that cross it, which on maps of few, steep lines soon
// outgrows what it evens out: split to the end whatever it made, 1672 rows x 2494 columns of 383 FFTs
// went from 340 to 5544 tiles of 5.7 times the work.
void balance_tiles(const std::vector<gfh_grid>& grids, const std::vector<HostMap>& hms, int blocks,
                   std::vector<TileDev>& tiles, std::vector<double>& work) {
  if (tiles.empty()) return;
  // work per block, and half of the longest tile for the last wave
  double all, longest;
  auto time = [&]() {
    all = std::accumulate(work.begin(), work.end(), 0.0);
    longest = *std::max_element(work.begin(), work.end());
    return all / blocks + 0.5 * longest;
  };
  double best = time();
  const double least = std::max(all / (3.0 * blocks), 12000.0);
  std::vector<TileDev> best_tiles = tiles;
  std::vector<double> best_work = work;
  // (a split only adds work: done once no longest tile could make up for what the splits so far added)
  int worse = 0;
  for (double most = longest; most > least && worse < 2 && all / blocks + 0.5 * least < best;) {
    most = std::max(0.7 * most, least);
    split_tiles(grids, hms, most, tiles, work);
    const double now = time();
    ++worse;
    if (now < best) {
      best = now;
      best_tiles = tiles;
      best_work = work;
      worse = 0;
    } else if (now > 1.05 * best) {
      break;
    }
  }
  tiles.swap(best_tiles);
  work.swap(best_work);
}

// Most work first (ties by map, so that a block's consecutive tiles are often of one map).
void sort_tiles(std::vector<TileDev>& tiles, const std::vector<double>& work) {
  std::vector<int32_t> at(tiles.size());
  std::iota(at.begin(), at.end(), 0);
  std::stable_sort(at.begin(), at.end(), [&](int32_t x, int32_t y) { return work[x] > work[y]; });
  std::vector<TileDev> out(tiles.size());
  for (size_t q = 0; q < at.size(); ++q) out[q] = tiles[at[q]];
  tiles.swap(out);
}

// Shared-memory bytes of the largest tile's counts (rows_x: tiles of the x-direction form, all of that
// many rows), and the most bands in a tile.
size_t tile_bytes(const std::vector<TileDev>& tiles, int rows_x, int* bands) {
  int64_t words = 0;
  for (const TileDev& t : tiles) {
    words = std::max(words, tile_words(rows_x > 0 ? rows_x : t.nrows, t.ncols) * (t.one ? 1 : 2));
    *bands = std::max(*bands, t.band_hi - t.band_lo + 1);
  }
  return (size_t)words * 4;
}

constexpr gfh_tile_config kDefaultShape{16, 3072, 512, 0};

bool same_shape(const gfh_tile_config& a, const gfh_tile_config& b) {
  return a.rows == b.rows && a.cols == b.cols && a.threads == b.threads;
}

// The shape a plan takes for the requested one (null or zero fields: the default's).  form selects
// nothing and is not kept, so that it tells no two shapes apart.
int tile_config(const gfh_tile_config* cfg, gfh_tile_config* tc) {
  *tc = kDefaultShape;
  if (cfg) {
    if (cfg->rows) tc->rows = cfg->rows;
    if (cfg->cols) tc->cols = cfg->cols;
    if (cfg->threads) tc->threads = cfg->threads;
    if (!(cfg->form == 0 || cfg->form == 1)) return GFH_ERR_ARG;
  }
  if (!(tc->rows == 4 || tc->rows == 8 || tc->rows == 16 || tc->rows == 32) || tc->cols < 128 || tc->cols % 128 ||
      tc->cols > 4096 || !(tc->threads == 256 || tc->threads == 512 || (tc->threads == 1024 && tc->rows >= 16)))
    return GFH_ERR_ARG;
  const int nwarps = tc->threads / 32;
  if ((tc->cols / 128 + nwarps - 1) / nwarps > 4) return GFH_ERR_ARG;  // <= 4 chunks per warp
  return GFH_OK;
}

// The threads and blocks per SM of a plan, and the words that each block has for a tile.
struct SmShare {
  int threads, blocks;
  int64_t room;
};

// A shape decides how many blocks share an SM, by its shared memory and its threads; tiles of any rows
// and columns are then planned in a block's share.  (Taken as it is, a shape was up to 1.6 times as
// slow: 51 half-hour maps at 8 x 3072 8.3 -> 4.7 ms.)  1024 threads are two blocks of 512: one block
// has nothing to run while it waits at a tile's chain of loads and barriers (the same maps at
// 16 x 3072 5.7 -> 4.7 ms).
SmShare sm_share(const gfh_tile_config& tc) {
  if (tc.threads == 1024 || same_shape(tc, kDefaultShape)) return SmShare{512, 2, kRoom[2]};
  const size_t bytes = (size_t)tc.rows * (tc.cols + 2) * 4;
  const int blocks = (int)std::max<size_t>(1, std::min<size_t>(kSmemPerSm / (bytes + 1024), tc.threads == 256 ? 3 : 2));
  return SmShare{tc.threads, blocks, kRoom[blocks]};
}

// Whether two shapes make the same plan.  (The default's coarse tiles have a share of their own.)
bool same_share(const gfh_tile_config& a, const gfh_tile_config& b) {
  const SmShare x = sm_share(a), y = sm_share(b);
  return x.threads == y.threads && x.blocks == y.blocks;
}

}  // namespace

extern "C" int gfh_plan_destroy(gfh_plan* p) {
  if (!p) return GFH_OK;
  if (p->ctx) {
    cudaSetDevice(p->ctx->device);
    if (p->ctx->stream) cudaStreamSynchronize(p->ctx->stream);
  }
  if (p->d_buf) cudaFree(p->d_buf);
  if (p->d_coarse_buf) cudaFree(p->d_coarse_buf);
  delete p;
  return GFH_OK;
}

extern "C" int gfh_plan_create(gfh_ctx* ctx, int32_t n_maps, const gfh_grid* grids,
                               int32_t* const* h_maps, gfh_candidate* const* h_cands,
                               gfh_map_stats* d_stats, const gfh_tile_config* cfg,
                               gfh_plan** out) {
  return gfh_make_plan(ctx, n_maps, grids, h_maps, h_cands, d_stats, cfg, false, out);
}

int gfh_make_plan(gfh_ctx* ctx, int32_t n_maps, const gfh_grid* grids, int32_t* const* h_maps,
                  gfh_candidate* const* h_cands, gfh_map_stats* d_stats, const gfh_tile_config* cfg,
                  bool once, gfh_plan** out) {
  if (!ctx || !out || n_maps < 1 || !grids || !h_maps) return GFH_ERR_ARG;
  *out = nullptr;
  gfh_tile_config tc;
  if (tile_config(cfg, &tc) != GFH_OK) return GFH_ERR_ARG;
  const SmShare share = sm_share(tc);

  std::vector<HostMap> hms(n_maps);
  std::vector<TileDev> tiles, tiles_x;
  std::vector<char> map_xd(n_maps, 0);
  double cells_k = 0.0, cells_xd = 0.0;
  int max_tile_bands = 1, cfg_bands = 1;
  for (int m = 0; m < n_maps; ++m) {
    const gfh_grid& g = grids[m];
    if (!grid_made(&g) || !h_maps[m]) return GFH_ERR_ARG;
    if ((double)g.n_k * (double)g.n_x0 >= 4294967295.0) return GFH_ERR_SIZE;
    if (h_cands && !h_cands[m]) return GFH_ERR_ARG;
    HostMap& hm = hms[m];
    int rc = gfh_host_tables(&g, hm.U, hm.B, hm.S);
    if (rc) return rc;
    rc = gfh_host_columns(&g, hm.band, hm.f0, hm.f0n);
    if (rc) return rc;
    int64_t ana_cols = 0;
    for (int64_t c = 0; c < g.n_x0; ++c) ana_cols += hm.band[c] >= 0;
    hm.cells = ana_cols * g.n_k;
    if (((uintptr_t)h_maps[m]) % 16) return GFH_ERR_ARG;  // 16-byte vector stores
    // A line moving more than two columns per k row (coarse k steps, e.g. Eq. dkeqn's) costs
    // fewer events differenced along x0 on every row (2 per row) than along k (the columns it
    // crosses): such maps use the x-direction form.
    map_xd[m] = hm.S[g.n_fft - 1] > (int64_t(2) << GFH_FRAC_BITS);
    hm.one = sparse_map(g, hm, map_xd[m]);
    (map_xd[m] ? cells_xd : cells_k) += (double)g.n_k * (double)g.ld_x0;
    find_analysis_columns(hm);
    for (int64_t c = 0; c < g.ld_x0; c += tc.cols) {
      int32_t lo, hi;
      column_bands(hm, c, std::min<int64_t>(c + tc.cols, g.ld_x0), &lo, &hi);
      cfg_bands = std::max(cfg_bands, hi - lo + 1);
    }
  }
  // Twice the cells per tile are of no use where two counts make no more tiles than one and a half for
  // each block (2 to 7 Mcells: 0.90 to 1.19 of the speed with one).
  const bool few = cells_k < 1.5 * 0.5 * (double)share.room * share.blocks * ctx->num_sms;
  for (int m = 0; m < n_maps; ++m) {
    if (map_xd[m]) continue;
    HostMap& hm = hms[m];
    hm.one = hm.one && !few;
    if (once) sampled_tiles(grids[m], hm, m, share.room, share.blocks * ctx->num_sms, tiles);
    else map_tiles(grids[m], hm, m, share.room, 0, grids[m].n_k, 0, grids[m].ld_x0, tiles);
  }
  // x-direction tiles: uniform strips of 8 rows, four and more to each block of three per SM as far as
  // 256 columns allow.  (Tiles of 16 rows keep 16 carries in registers and fill an SM with one block,
  // which spilt or stood at barriers: half-hour map at 3 columns per row 242 us with 16 x 3072, 149 us so;
  // 11 braking indices at 4 columns 2.25 against 1.97 ms.)
  for (int m = 0; m < n_maps; ++m) {
    if (!map_xd[m]) continue;
    const int cols = std::max(256, (int)std::min(4096.0, cells_xd / (12.0 * ctx->num_sms * kRowsX)) / 64 * 64);
    cut_tiles(grids[m], hms[m], m, 0, grids[m].n_k, 0, grids[m].ld_x0, kRowsX,
              std::min(cols, cols_for(kRowsX, hms[m].one ? kRoom[3] : kRoom[3] / 2)), tiles_x);
  }
  // The given tile must fit in shared memory (one count per cell, chunk sums, band keys).
  const bool select = h_cands != nullptr || d_stats != nullptr;
  const size_t smem = (size_t)tc.rows * (tc.cols + 2) * 4 + 32 * 4 * (tiles_x.empty() ? 1 : tc.rows) +
                      (select ? (size_t)cfg_bands * 8 : 0);
  if (smem > kHoughSmemLimit) return GFH_ERR_SIZE;
  // Most work first; the x-direction tiles form a second list after the others.
  std::vector<double> work(tiles.size()), work_x(tiles_x.size());
  for (size_t q = 0; q < tiles.size(); ++q) work[q] = tile_work(grids[tiles[q].map], hms[tiles[q].map], tiles[q]);
  for (size_t q = 0; q < tiles_x.size(); ++q)
    work_x[q] = (double)std::max(0, tiles_x[q].bin_b - tiles_x[q].bin_a + 1) * tiles_x[q].nrows;
  if (!once) balance_tiles(std::vector<gfh_grid>(grids, grids + n_maps), hms, share.blocks * ctx->num_sms, tiles, work);
  sort_tiles(tiles, work);
  sort_tiles(tiles_x, work_x);
  const size_t cells = tile_bytes(tiles, 0, &max_tile_bands);
  const size_t cells_x = tile_bytes(tiles_x, kRowsX, &max_tile_bands);
  const int n_tiles_k = (int)tiles.size();
  tiles.insert(tiles.end(), tiles_x.begin(), tiles_x.end());

  // The index: per list the runs of bins that its maps cover, overlapping or adjacent maps in one run.
  std::vector<int> order(n_maps), run_of(n_maps);
  std::iota(order.begin(), order.end(), 0);
  std::sort(order.begin(), order.end(), [&](int a, int b) {
    return std::make_pair(grids[a].list, grids[a].bin_lo) < std::make_pair(grids[b].list, grids[b].bin_lo);
  });
  std::vector<ListDev> lists;
  std::vector<int> ffts;
  for (int m : order) {
    const gfh_grid& g = grids[m];
    const bool joins = !lists.empty() && lists.back().list == g.list &&
                       g.bin_lo - lists.back().bin_lo <= lists.back().n_bins;
    if (!joins) {
      lists.push_back(ListDev{nullptr, nullptr, g.list, g.bin_lo, 0, 0, 0, 0, nullptr, 0});
      ffts.push_back(0);
    }
    ListDev& ld = lists.back();
    ld.n_bins = std::max(ld.n_bins, g.bin_hi - ld.bin_lo + 1);
    ffts.back() = std::max(ffts.back(), g.n_fft);
    run_of[m] = (int)lists.size() - 1;
  }
  int64_t csr_entries = 0, copy_words = 0;
  for (size_t l = 0; l < lists.size(); ++l) {
    ListDev& ld = lists[l];
    // FFT blocks of 16 to 64, as fine as one per lane of the warp that looks a bin's up allows (a
    // window's ends are read by whole blocks: 2118 rows x 2540 columns of 652 FFTs 75 -> 71 us); longer
    // ones only so that a bin has at most 256.
    ld.shift = 4;
    while (((ffts[l] - 1) >> ld.shift) + 1 > (ld.shift < 6 ? 32 : kMaxFftBlocks)) ++ld.shift;
    ld.nb1 = ((ffts[l] - 1) >> ld.shift) + 2;
    if (csr_entries + ld.n_bins > INT32_MAX) return GFH_ERR_SIZE;
    ld.entry0 = (int32_t)csr_entries;
    csr_entries += ld.n_bins;
    // room to order a list out of FFT order: an eighth of its (FFT, bin) pairs, noise peaks and more
    ld.cap = (int64_t)ld.n_bins * ffts[l] / 8 + 1024;
    copy_words += ld.cap;
  }

  // One device buffer: map descriptors | tiles | lists | index list of each bin | keys | per-map tables.
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes, 256); return o; };
  const size_t o_maps = take(sizeof(MapDev) * n_maps);
  const size_t o_tiles = take(sizeof(TileDev) * tiles.size());
  const size_t o_lists = take(sizeof(ListDev) * lists.size());
  const size_t o_csrmap = take(sizeof(int32_t) * csr_entries);
  std::vector<size_t> o_csr(lists.size()), o_blk(lists.size());
  for (size_t l = 0; l < lists.size(); ++l) {
    o_csr[l] = take(sizeof(int64_t) * ((size_t)lists[l].n_bins + 1));
    o_blk[l] = take(sizeof(int32_t) * (size_t)lists[l].n_bins * lists[l].nb1);
  }
  size_t key_words = 0;
  for (int m = 0; m < n_maps; ++m) key_words += grids[m].n_bands + 2;
  // (an execution takes at most 65535 lists)
  int n_lists = 1;
  for (int m = 0; m < n_maps; ++m) n_lists = std::max(n_lists, std::min(grids[m].list, 65535) + 1);
  const size_t zeroed = sizeof(unsigned long long) * key_words + sizeof(int) * ((size_t)n_lists + 4);
  const size_t o_keys = take(zeroed);
  std::vector<size_t> o_U(n_maps), o_SD(n_maps), o_B(n_maps), o_band(n_maps), o_f0(n_maps),
      o_f0n(n_maps);
  for (int m = 0; m < n_maps; ++m) {
    o_U[m] = take(2 * sizeof(int64_t) * (hms[m].U.size() - 1));
    o_SD[m] = take(sizeof(FftRow) * hms[m].S.size());
    o_B[m] = grids[m].k_min != 0.0 ? take(sizeof(int64_t) * hms[m].B.size()) : 0;
    o_band[m] = take(sizeof(int32_t) * hms[m].band.size());
    o_f0[m] = take(sizeof(double) * hms[m].f0.size());
    o_f0n[m] = take(sizeof(double) * hms[m].f0n.size());
  }
  const size_t o_single = take(sizeof(int64_t) * 2);
  const size_t total = off;

  gfh_plan* p = new (std::nothrow) gfh_plan();
  if (!p) return GFH_ERR_NOMEM;
  p->ctx = ctx;
  p->n_maps = n_maps;
  p->grids.assign(grids, grids + n_maps);
  p->cfg = tc;
  p->threads = share.threads;
  // coarse tiles are small: the default's take three blocks of 256 threads
  p->list_threads = same_shape(tc, kDefaultShape) ? 256 : share.threads;
  p->list_room = same_shape(tc, kDefaultShape) ? kRoom[3] : share.room;
  p->cells = cells;
  p->cells_x = cells_x;
  if (cudaSetDevice(ctx->device) != cudaSuccess) { delete p; return GFH_ERR_CUDA; }
  // the room to order lists follows what is filled here; without it they are walked whole
  if (cudaMalloc(&p->d_buf, total + (size_t)copy_words * sizeof(uint32_t)) != cudaSuccess) {
    cudaGetLastError();
    for (ListDev& ld : lists) ld.cap = 0;
    if (cudaMalloc(&p->d_buf, total) != cudaSuccess) { delete p; return GFH_ERR_NOMEM; }
  }
  char* base = (char*)p->d_buf;
  std::vector<char> h(total, 0);
  std::vector<MapDev> mds(n_maps);
  std::vector<int32_t> csr_list;
  csr_list.reserve(csr_entries);
  uint32_t* copy = (uint32_t*)(base + total);
  for (size_t l = 0; l < lists.size(); ++l) {
    lists[l].copy = copy;
    copy += lists[l].cap;
    lists[l].csr = (int64_t*)(base + o_csr[l]);
    lists[l].blk = (int32_t*)(base + o_blk[l]);
    csr_list.insert(csr_list.end(), lists[l].n_bins, (int32_t)l);
  }
  size_t key_off = 0;
  for (int m = 0; m < n_maps; ++m) {
    const gfh_grid& g = grids[m];
    HostMap& hm = hms[m];
    MapDev& md = mds[m];
    md.out = h_maps[m];
    md.UP = (const longlong2*)(base + o_U[m]);
    md.SD = (const FftRow*)(base + o_SD[m]);
    md.B = g.k_min != 0.0 ? (const int64_t*)(base + o_B[m]) : nullptr;
    md.line = shift_line(hm);
    md.col_band = (const int32_t*)(base + o_band[m]);
    md.f0c = (const double*)(base + o_f0[m]);
    md.f0n = (const double*)(base + o_f0n[m]);
    const ListDev& ld = lists[run_of[m]];
    md.csr = ld.csr + (g.bin_lo - ld.bin_lo);
    md.blk = ld.blk + (size_t)(g.bin_lo - ld.bin_lo) * ld.nb1;
    md.csr_list = ld.csr;
    md.copy = ld.copy;
    md.nb1 = ld.nb1;
    md.shift = ld.shift;
    md.keys = (unsigned long long*)(base + o_keys) + key_off;
    md.sums = md.keys + g.n_bands;
    key_off += g.n_bands + 2;
    md.cands = h_cands ? h_cands[m] : nullptr;
    md.stats = d_stats ? d_stats + m : nullptr;
    md.W = g.n_x0;
    md.ld = g.ld_x0;
    md.cells = hm.cells;
    md.x0_min = g.x0_min;
    md.dx0 = g.dx0;
    md.k_min = g.k_min;
    md.dk = g.dk;
    md.K = g.n_k;
    md.bin_lo = g.bin_lo;
    md.bin_hi = g.bin_hi;
    md.n_fft = g.n_fft;
    md.list = g.list;
    md.n_bands = g.n_bands;
    // paired tables: one 16-byte load per bin and one per FFT in the kernel
    int64_t* up = (int64_t*)(h.data() + o_U[m]);
    for (size_t j = 0; j + 1 < hm.U.size(); ++j) { up[2 * j] = hm.U[j + 1]; up[2 * j + 1] = hm.U[j] - 1; }
    FftRow* sd = (FftRow*)(h.data() + o_SD[m]);
    for (size_t i = 0; i < hm.S.size(); ++i) sd[i] = FftRow{hm.S[i], rows_per_column(hm.S[i])};
    if (md.B) std::memcpy(h.data() + o_B[m], hm.B.data(), sizeof(int64_t) * hm.B.size());
    std::memcpy(h.data() + o_band[m], hm.band.data(), sizeof(int32_t) * hm.band.size());
    std::memcpy(h.data() + o_f0[m], hm.f0.data(), sizeof(double) * hm.f0.size());
    std::memcpy(h.data() + o_f0n[m], hm.f0n.data(), sizeof(double) * hm.f0n.size());
  }
  std::memcpy(h.data() + o_maps, mds.data(), sizeof(MapDev) * n_maps);
  if (!tiles.empty()) std::memcpy(h.data() + o_tiles, tiles.data(), sizeof(TileDev) * tiles.size());
  std::memcpy(h.data() + o_lists, lists.data(), sizeof(ListDev) * lists.size());
  std::memcpy(h.data() + o_csrmap, csr_list.data(), sizeof(int32_t) * csr_list.size());
  if (cudaMemcpy(p->d_buf, h.data(), total, cudaMemcpyHostToDevice) != cudaSuccess) {
    gfh_plan_destroy(p);
    return GFH_ERR_CUDA;
  }
  p->d_maps = (MapDev*)(base + o_maps);
  p->d_tiles = (TileDev*)(base + o_tiles);
  p->n_tiles = n_tiles_k;
  p->n_tiles_x = (int)tiles.size() - n_tiles_k;
  p->map_xd = map_xd;
  for (const HostMap& hm : hms) p->map_one.push_back(hm.one);
  p->max_tile_bands = max_tile_bands;
  p->d_zeroed = base + o_keys;
  p->zeroed_bytes = zeroed;
  p->d_keys = (unsigned long long*)(base + o_keys);
  p->d_list_state = (int*)(p->d_keys + key_words);
  p->n_list_states = n_lists;
  p->d_next = p->d_list_state + n_lists;
  p->d_sel_count = p->d_next + 2;
  p->csr_entries = (int32_t)csr_entries;
  p->d_lists = (ListDev*)(base + o_lists);
  p->d_csr_list = (int32_t*)(base + o_csrmap);
  p->select = h_cands != nullptr || d_stats != nullptr;
  p->d_offsets_single = (int64_t*)(base + o_single);
  p->h_maps.assign(h_maps, h_maps + n_maps);
  if (h_cands) p->h_cands.assign(h_cands, h_cands + n_maps);
  p->d_stats = d_stats;
  const int prc = gfh_prepare_plan(p);
  if (prc) {
    gfh_plan_destroy(p);
    return prc;
  }
  *out = p;
  return GFH_OK;
}

extern "C" int gfh_plan_execute(gfh_plan* p, const gfh_peaks* peaks) {
  if (!p || !peaks || !peaks->fft_idx || !peaks->bin || !peaks->offsets || peaks->n_lists < 1)
    return GFH_ERR_ARG;
  for (const gfh_grid& g : p->grids)
    if (g.list < 0 || g.list >= peaks->n_lists) return GFH_ERR_ARG;
  return gfh_launch_plan(p, peaks);
}

// ---- coarse tiles --------------------------------------------------------------------------------

extern "C" int gfh_plan_set_coarse(gfh_plan* p, int32_t coarse_k, int32_t coarse_x,
                                   int32_t max_sel) {
  if (!p || coarse_k < 1 || coarse_x < 1 || coarse_k > 4096 || coarse_x > 4096 || max_sel < 1 ||
      (int64_t)max_sel > (int64_t)coarse_k * coarse_x)
    return GFH_ERR_ARG;
  if (p->n_tiles_x > 0) return GFH_ERR_ARG;     // coarse tiles need lines moving <= 2 columns per row
  const int nct = coarse_k * coarse_x;
  std::vector<TileDev> fine;
  std::vector<int32_t> first;
  first.reserve((size_t)p->n_maps * (nct + 1) + 1);
  int max_bands = p->max_tile_bands;
  size_t worst = 0;                        // longest gathered list: every map at its largest
  for (int m = 0; m < p->n_maps; ++m) {
    const gfh_grid& g = p->grids[m];
    HostMap hm;
    int rc = gfh_host_tables(&g, hm.U, hm.B, hm.S);
    if (rc) return rc;
    rc = gfh_host_columns(&g, hm.band, hm.f0, hm.f0n);
    if (rc) return rc;
    hm.one = p->map_one[m];
    find_analysis_columns(hm);
    // columns of each f0 tile: analysis columns only; f0 falls with the column, so each range is
    // contiguous
    std::vector<int64_t> cmin(coarse_x, INT64_MAX), cmax(coarse_x, -1);
    const double span = g.ana_hi - g.ana_lo;
    for (int64_t c = 0; c < g.n_x0; ++c) {
      if (hm.band[c] < 0) continue;
      int xt = (int)std::floor((hm.f0[c] - g.ana_lo) / span * coarse_x);
      xt = std::min(std::max(xt, 0), coarse_x - 1);
      cmin[xt] = std::min(cmin[xt], c);
      cmax[xt] = std::max(cmax[xt], c);
    }
    std::vector<int> sizes;
    for (int kt = 0; kt < coarse_k; ++kt) {
      // rows r with floor(r coarse_k / K) = kt
      const int r0 = (int)(((int64_t)kt * g.n_k + coarse_k - 1) / coarse_k);
      const int r1 = (int)(((int64_t)(kt + 1) * g.n_k + coarse_k - 1) / coarse_k);
      for (int xt = 0; xt < coarse_x; ++xt) {
        first.push_back((int32_t)fine.size());
        const size_t before = fine.size();
        if (r1 > r0 && cmax[xt] >= 0) {
          // 16-byte aligned column range (vector stores): neighbouring tiles may share <= 3 columns
          const int64_t c_lo = cmin[xt] & ~int64_t(3);
          const int64_t c_hi = std::min<int64_t>(g.ld_x0, (cmax[xt] + 4) & ~int64_t(3));
          map_tiles(g, hm, m, p->list_room, r0, r1, c_lo, c_hi, fine);
        }
        const int cnt = (int)(fine.size() - before);
        sizes.push_back(cnt);
      }
    }
    // group nct: the whole map, as gfh_plan_execute tiles it
    first.push_back((int32_t)fine.size());
    const size_t before = fine.size();
    map_tiles(g, hm, m, p->list_room, 0, g.n_k, 0, g.ld_x0, fine);
    const size_t whole = fine.size() - before;
    std::sort(sizes.begin(), sizes.end(), std::greater<int>());
    size_t top = 0;
    for (int i = 0; i < max_sel && i < (int)sizes.size(); ++i) top += sizes[i];
    worst += std::max(whole, top);
  }
  first.push_back((int32_t)fine.size());
  if (fine.size() > (size_t)INT32_MAX || worst > (size_t)INT32_MAX) return GFH_ERR_SIZE;
  const size_t cells_list = tile_bytes(fine, 0, &max_bands);
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes, 256); return o; };
  const size_t o_fine = take(sizeof(TileDev) * std::max<size_t>(fine.size(), 1));
  const size_t o_first = take(sizeof(int32_t) * first.size());
  const size_t o_sel = take(sizeof(TileDev) * std::max<size_t>(worst, 1));
  GFH_CUDA_TRY(cudaSetDevice(p->ctx->device));
  if (p->ctx->stream) GFH_CUDA_TRY(cudaStreamSynchronize(p->ctx->stream));
  void* buf = nullptr;
  if (cudaMalloc(&buf, off) != cudaSuccess) return GFH_ERR_NOMEM;
  char* base = (char*)buf;
  cudaError_t e = cudaSuccess;
  if (!fine.empty())
    e = cudaMemcpy(base + o_fine, fine.data(), sizeof(TileDev) * fine.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMemcpy(base + o_first, first.data(), sizeof(int32_t) * first.size(), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) { cudaFree(buf); return GFH_ERR_CUDA; }
  if (p->d_coarse_buf) cudaFree(p->d_coarse_buf);
  p->d_coarse_buf = buf;
  p->d_fine = (TileDev*)(base + o_fine);
  p->d_coarse_first = (int32_t*)(base + o_first);
  p->d_sel_tiles = (TileDev*)(base + o_sel);
  p->sel_cap = (int)std::max<size_t>(worst, 1);
  p->coarse_k = coarse_k;
  p->coarse_x = coarse_x;
  p->max_sel = max_sel;
  p->max_tile_bands = max_bands;
  p->cells_list = cells_list;
  return GFH_OK;
}

extern "C" int gfh_plan_execute_tiles(gfh_plan* p, const gfh_peaks* peaks, const int32_t* d_coarse,
                                      int32_t n_sel, const int32_t* d_full) {
  if (!p || !peaks || !peaks->fft_idx || !peaks->bin || !peaks->offsets || peaks->n_lists < 1 ||
      p->coarse_k < 1 || n_sel < 0 || n_sel > p->max_sel || (n_sel > 0 && !d_coarse))
    return GFH_ERR_ARG;
  for (const gfh_grid& g : p->grids)
    if (g.list < 0 || g.list >= peaks->n_lists) return GFH_ERR_ARG;
  return gfh_launch_plan_tiles(p, peaks, d_coarse, n_sel, d_full);
}

// ---- autotuner ----------------------------------------------------------------------------------

namespace {

// Shapes the autotuner chose, by plan signature (plan_signature), for this process.
std::mutex g_tune_mu;
std::map<std::string, gfh_tile_config> g_tune_cache;

// Signature of a plan and its peak lists for the autotuner's cache: the device (compute capability,
// SMs), whether candidates are selected, and per map its k rows, x0 columns, bins, FFTs, line form
// (along k or along x0) and peak-density class: log2 of its list's peaks per (FFT, bin) of its
// band, in quarter steps (the list offsets are read back; the autotuner synchronises anyway).
int plan_signature(const gfh_plan* p, const gfh_peaks* peaks, std::string* key) {
  std::vector<int64_t> off((size_t)peaks->n_lists + 1);
  if (p->ctx->stream) GFH_CUDA_TRY(cudaStreamSynchronize(p->ctx->stream));
  GFH_CUDA_TRY(cudaMemcpy(off.data(), peaks->offsets, off.size() * sizeof(int64_t),
                          cudaMemcpyDeviceToHost));
  cudaDeviceProp prop{};
  GFH_CUDA_TRY(cudaGetDeviceProperties(&prop, p->ctx->device));
  std::string k = "cc" + std::to_string(prop.major) + "." + std::to_string(prop.minor) + " sm" +
                  std::to_string(prop.multiProcessorCount) + (p->select ? " sel" : " nosel");
  for (int m = 0; m < p->n_maps; ++m) {
    const gfh_grid& g = p->grids[m];
    if (g.list < 0 || g.list >= peaks->n_lists) return GFH_ERR_ARG;
    const double cells = (double)g.n_fft * (double)(g.bin_hi - g.bin_lo + 1);
    const double n = (double)(off[g.list + 1] - off[g.list]);
    const int cls = n > 0.0 ? (int)std::floor(4.0 * std::log2(n / cells)) : -1000;
    k += " " + std::to_string(g.n_k) + "x" + std::to_string(g.n_x0) + "b" +
         std::to_string(g.bin_hi - g.bin_lo + 1) + "f" + std::to_string(g.n_fft) +
         (p->map_xd[m] ? "x" : "k") + "d" + std::to_string(cls);
  }
  *key = k;
  return GFH_OK;
}

// Mean time of `reps` executions of plan q on its stream (after one untimed run), in ms.
int time_plan(gfh_plan* q, const gfh_peaks* peaks, int reps, float* ms) {
  cudaStream_t st = q->ctx->stream;
  cudaEvent_t a = nullptr, b = nullptr;
  if (cudaEventCreate(&a) != cudaSuccess || cudaEventCreate(&b) != cudaSuccess) {
    if (a) cudaEventDestroy(a);
    return GFH_ERR_CUDA;
  }
  int rc = gfh_plan_execute(q, peaks);
  if (!rc && cudaEventRecord(a, st) != cudaSuccess) rc = GFH_ERR_CUDA;
  for (int i = 0; i < reps && !rc; ++i) rc = gfh_plan_execute(q, peaks);
  if (!rc && cudaEventRecord(b, st) != cudaSuccess) rc = GFH_ERR_CUDA;
  if (!rc && cudaEventSynchronize(b) != cudaSuccess) rc = GFH_ERR_CUDA;
  if (!rc && cudaEventElapsedTime(ms, a, b) != cudaSuccess) rc = GFH_ERR_CUDA;
  if (!rc) *ms /= (float)reps;
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  return rc;
}

// Rebuilds plan p with tile shape `shape` (same grids and outputs; coarse tiles follow the shape).
int reshape_plan(gfh_plan* p, const gfh_tile_config& shape) {
  if (same_share(shape, p->cfg)) return GFH_OK;
  gfh_plan* q = nullptr;
  gfh_tile_config cfg = shape;
  int rc = gfh_plan_create(p->ctx, p->n_maps, p->grids.data(), p->h_maps.data(),
                           p->h_cands.empty() ? nullptr : p->h_cands.data(), p->d_stats, &cfg, &q);
  if (rc) return rc;
  if (p->ctx->stream) cudaStreamSynchronize(p->ctx->stream);
  const int ck = p->coarse_k, cx = p->coarse_x, ms = p->max_sel;
  std::swap(*p, *q);      // p takes the new tables; q holds the old ones and is freed
  gfh_plan_destroy(q);
  if (ck > 0) return gfh_plan_set_coarse(p, ck, cx, ms);
  return GFH_OK;
}

}  // namespace

extern "C" int gfh_plan_autotune(gfh_plan* p, const gfh_peaks* peaks, int32_t reps,
                                 gfh_tile_config* h_best, float* h_best_ms) {
  if (!p || !peaks || !peaks->offsets || peaks->n_lists < 1 || reps < 1) return GFH_ERR_ARG;
  static const int kRowsList[] = {4, 8, 16};
  static const int kColsList[] = {1024, 2048, 3072, 4096};
  static const int kThreadsList[] = {256, 512, 1024};
  std::string key;
  int rc = plan_signature(p, peaks, &key);
  if (rc) return rc;
  bool cached = false;
  gfh_tile_config best = p->cfg;
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    auto it = g_tune_cache.find(key);
    if (it != g_tune_cache.end()) { best = it->second; cached = true; }
  }
  float best_ms = 0.f;
  if (cached) {                 // tuned before: take that shape and time it alone
    rc = reshape_plan(p, best);
    if (!rc) rc = time_plan(p, peaks, reps, &best_ms);
    if (rc) return rc;
    if (h_best) *h_best = best;
    if (h_best_ms) *h_best_ms = best_ms;
    return GFH_OK;
  }
  rc = time_plan(p, peaks, reps, &best_ms);
  if (rc) return rc;
  std::vector<gfh_tile_config> tried{p->cfg};
  bool best_is_own = true;
  auto try_shape = [&](const gfh_tile_config& cfg) -> int {
    for (const gfh_tile_config& c : tried)
      if (same_share(c, cfg)) return GFH_OK;
    gfh_plan* q = nullptr;
    gfh_tile_config c = cfg;
    const int crc = gfh_plan_create(p->ctx, p->n_maps, p->grids.data(), p->h_maps.data(),
                                    p->h_cands.empty() ? nullptr : p->h_cands.data(), p->d_stats,
                                    &c, &q);
    if (crc == GFH_ERR_SIZE || crc == GFH_ERR_ARG) return GFH_OK;   // shape does not fit
    if (crc) return crc;
    tried.push_back(cfg);
    float ms = 0.f;
    const int trc = time_plan(q, peaks, reps, &ms);
    gfh_plan_destroy(q);
    if (trc) return trc;
    // (a shape is kept for less than 2 %: repeated runs differ by half of that, and every later plan of
    // this signature would be made twice, once at its own shape)
    if (ms < (best_is_own ? 0.98f : 1.f) * best_ms) { best_ms = ms; best = cfg; best_is_own = false; }
    return GFH_OK;
  };
  for (int r : kRowsList)
    for (int c : kColsList)
      for (int t : kThreadsList) {
        if (t == 1024 && r < 16) continue;     // 1024 threads only for 16-row tiles
        rc = try_shape(gfh_tile_config{r, c, t, 0});
        if (rc) return rc;
      }
  rc = reshape_plan(p, best);
  if (rc) return rc;
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tune_cache[key] = best;
  }
  if (h_best) *h_best = best;
  if (h_best_ms) *h_best_ms = best_ms;
  return GFH_OK;
}

extern "C" int gfh_autotune_cache_size(void) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  return (int)g_tune_cache.size();
}

extern "C" void gfh_autotune_cache_clear(void) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  g_tune_cache.clear();
}
