// Internal types shared by the translation units of libgfh (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <cufft.h>
#include <cmath>
#include <cstdint>
#include <cstddef>
#include <vector>

#include "gfh.h"

#define GFH_FRAC_BITS 32

// Largest dynamic shared memory a block may use on sm_103a (227 KB).
constexpr size_t kMaxSmemBytes = 227 * 1024;
constexpr size_t kSmemPerSm = 228 * 1024;   // shared memory of one SM
// dynamic shared memory a Hough tile may take: the kernels keep a few static bytes (tile counter)
constexpr size_t kHoughSmemLimit = kMaxSmemBytes - 64;

// Shared memory of a Hough tile: words between its rows' ends and starts (rows stay 16-byte aligned,
// and 4 words from row to row spread a line's cells over the banks).
constexpr int kHoughPad = 4;
// Room of a tile (words) with one, two or three blocks per SM; about 43, 15 and 10 KB of a block's shared
// memory are left for its chunk sums, band keys and windows.
constexpr int kRowsX = 8;   // k rows of a tile in the x-direction form
constexpr int64_t kRoom[4] = {0, 47104, 25088, 16448};

// Counter-based generator of the statistical peakmap model: the splitmix64 finaliser (Steele, Lea
// and Flood, "Fast splittable pseudorandom number generators", OOPSLA 2014) applied to a key built
// from (seed, sample, stream, FFT i, bin j); the top 24 bits are the cell's uniform.
__host__ __device__ __forceinline__ uint64_t gfh_mix64(uint64_t z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__host__ __device__ __forceinline__ uint32_t gfh_cell_u24(uint64_t seed, uint64_t sample,
                                                         uint32_t stream, uint32_t i, uint32_t j) {
  const uint64_t s = gfh_mix64(seed ^ (sample * 0xD1B54A32D192ED03ull) ^ ((uint64_t)stream << 56));
  return (uint32_t)(gfh_mix64(s ^ (((uint64_t)i << 32) | j)) >> 40);
}

// (FFT i, bin j) is a peak of the sample: a noise peak (stream 0 below p_noise24), or the cell of
// the injected track in FFT i and a track hit (stream 1 below p_track24).
__host__ __device__ __forceinline__ bool gfh_synth_peak(uint64_t seed, uint64_t sample, uint32_t i,
                                                       uint32_t j, uint32_t p_noise24,
                                                       int track_bin, uint32_t p_track24) {
  if (gfh_cell_u24(seed, sample, 0, i, j) < p_noise24) return true;
  return (int)j == track_bin && gfh_cell_u24(seed, sample, 1, i, j) < p_track24;
}

// Device-side error flag bits (gfh_check).
#define GFH_FLAG_UNSORTED 1u
#define GFH_FLAG_FFT_RANGE 2u
#define GFH_FLAG_CAPACITY 4u
#define GFH_FLAG_TIMEOUT 8u

#define GFH_CUDA_TRY(expr)                                \
  do {                                                    \
    cudaError_t e_ = (expr);                              \
    if (e_ != cudaSuccess) return GFH_ERR_CUDA;           \
  } while (0)

struct gfh_ctx {
  int device = 0;
  cudaStream_t stream = nullptr;
  int num_sms = 0;
  unsigned int* d_flag = nullptr;  // input-check flag
  // peakmap scratch (library-owned, grows on demand)
  void* pm_buf = nullptr;
  size_t pm_bytes = 0;
  // cuFFT plans of the interlaced frames (R2C for series, C2C for heterodyned series), kept for
  // the last few shapes so that searches alternating FFT lengths (Sec. VI.D portions) plan once
  struct FftPlan {
    cufftHandle h = 0;
    bool valid = false;
    bool c2c = false;
    int n = 0, batch = 0;
    unsigned long long used = 0;
  };
  static constexpr int kFftPlans = 4;
  FftPlan fft[kFftPlans];
  unsigned long long fft_clock = 0;
  // pinned host word for returning counts
  long long* h_pinned = nullptr;
  // bf16 bits of float(log(1 + c)) for c < kLogTable (image channel 0), built on the host
  uint16_t* d_log1p = nullptr;
};

constexpr int kLogTable = 4096;

// One FFT of a map's shift table: its lines move left by S per k row (2^-32 columns).
// D = ceil(2^89 / S): rows of 2^-57 per column, for S > 2^25 (0 otherwise).
struct alignas(16) FftRow {
  int64_t S;
  uint64_t D;
};

// A map's shifts B_i + r S_i against the FFT i: the line through the tables' ends, in whole lattice
// units, and the largest distance of the tables from it.
struct ShiftLine {
  int64_t b0, s0;           // B_0, S_0
  int64_t db, ds;           // B_last - B_0, S_last - S_0
  float eb, es;             // max |B_i - line|, max |S_i - line|, rounded up
  int32_t n_fft;
};

// The line on a tile's first and last row: FFT i is shifted by base + i / inv, within `slack` FFTs
// (the tables' distance from the line, and float32's rounding of what bin_ffts computes).
// inv = 0 where the line is level: every FFT may then meet the tile and none is known to cover it.
struct TileLine {
  int64_t base0, base1;
  float inv0, inv1, slack0, slack1;
};

// The slope is the difference of the ends on that row, formed in whole units: where db and r ds have
// opposite signs (k < 0) it can be a few units out of 2^40, and as a sum of two float32 slopes was
// rounding alone.  With a level line's few units the slack is all FFTs.
__host__ __device__ __forceinline__ TileLine tile_line(const ShiftLine& l, int64_t row0, int64_t row1) {
  const int64_t d0 = l.db + row0 * l.ds, d1 = l.db + row1 * l.ds;
  const float ffts = (float)l.n_fft, last = (float)(l.n_fft - 1);
  TileLine t;
  t.base0 = l.b0 + row0 * l.s0;
  t.base1 = l.b0 + row1 * l.s0;
  t.inv0 = d0 != 0 ? last / (float)d0 : 0.f;
  t.inv1 = d1 != 0 ? last / (float)d1 : 0.f;
  t.slack0 = 2.f + (l.eb + (float)row0 * l.es) * fabsf(t.inv0) + ffts * 0x1p-20f;
  t.slack1 = 2.f + (l.eb + (float)row1 * l.es) * fabsf(t.inv1) + ffts * 0x1p-20f;
  return t;
}

// The FFTs of one bin at a tile: those outside lo .. hi have no edge in it on any row and do not
// cover it; those strictly between c_lo and c_hi cover it on every row.  All in -1 .. n_fft.
struct BinFfts {
  int lo, hi, c_lo, c_hi;
};

// left, right: the bin's first and last position; c0, ub: the tile's first column and its last one
// inside the map, counted from c0; wide: the tile has no column past the map.
__host__ __device__ __forceinline__ BinFfts bin_ffts(const TileLine& t, int64_t left, int64_t right,
                                                     int64_t c0, int ub, bool wide, int n_fft) {
  const float ffts = (float)n_fft;
  auto clamp = [&](float x) { return (int)fminf(fmaxf(x, -1.f), ffts); };
  BinFfts b;
  // right edge on the first row reaches the tile (shift0 <= x); left edge on the last row is not
  // past it (shift1 >= y)
  const float x = (float)(right - (c0 << GFH_FRAC_BITS) - t.base0) * t.inv0;
  const float y = (float)(left - ((c0 + ub + 1) << GFH_FRAC_BITS) - t.base1) * t.inv1;
  float lo = -1.f, hi = ffts;
  if (t.inv0 > 0.f) hi = x + t.slack0;
  if (t.inv0 < 0.f) lo = x - t.slack0;
  if (t.inv1 > 0.f) lo = fmaxf(lo, y - t.slack1);
  if (t.inv1 < 0.f) hi = fminf(hi, y + t.slack1);
  b.lo = clamp(lo);
  b.hi = clamp(hi);
  // a bin wider than the tile: left edge at or before its first column on the first row, right edge
  // at or past its last on the last
  b.c_lo = (int)ffts;
  b.c_hi = -1;
  if (wide && ((right - left) >> GFH_FRAC_BITS) >= ub && t.inv0 != 0.f && t.inv1 != 0.f) {
    const float cx = (float)(left - ((c0 + 1) << GFH_FRAC_BITS) - t.base0) * t.inv0;
    const float cy = (float)(right - ((c0 + ub) << GFH_FRAC_BITS) - t.base1) * t.inv1;
    b.c_lo = clamp(fmaxf(t.inv0 > 0.f ? cx + t.slack0 : -1.f, t.inv1 < 0.f ? cy + t.slack1 : -1.f));
    b.c_hi = clamp(fminf(t.inv1 > 0.f ? cy - t.slack1 : ffts, t.inv0 < 0.f ? cx - t.slack0 : ffts));
  }
  return b;
}

// One map as the kernels see it.
struct MapDev {
  int32_t* out;             // [K][ld]
  const longlong2* UP;      // J: {U[j+1], U[j] - 1}: first and last position of bin j
  const FftRow* SD;         // n_fft
  const int64_t* B;         // n_fft: shift on row 0 (null: all 0, the default k_min = 0)
  const int32_t* col_band;  // ld entries, -1 outside the analysis band / beyond n_x0
  const double* f0c;        // n_x0
  const double* f0n;        // n_x0
  const int64_t* csr;       // J + 1 entries: first peak (absolute index) of bins bin_lo .. bin_hi+1
  const int32_t* blk;       // [J][nb1]: offset in a bin's peaks of its first of FFT >= 2^shift b
  int32_t nb1, shift;
  const int64_t* csr_list;  // first peak of the run's first bin
  const uint32_t* copy;     // the list's FFT indices from there, by blocks (lists out of FFT order)
  unsigned long long* keys; // n_bands
  unsigned long long* sums; // 2: sum, sum of squares
  gfh_candidate* cands;     // n_bands (may be null)
  gfh_map_stats* stats;     // 1 (may be null)
  int64_t W;                // n_x0
  int64_t ld;               // ld_x0
  int64_t cells;            // analysis cells
  double x0_min, dx0, k_min, dk;
  int32_t K;
  int32_t bin_lo, bin_hi;
  int32_t n_fft;
  int32_t list;
  int32_t n_bands;
  ShiftLine line;           // a bin's windows of FFTs
};

// FFT blocks of a bin, at most.
constexpr int kMaxFftBlocks = 256;

// The index of a peak list over a run of bins that maps read (built per execute, k_index).
struct ListDev {
  int64_t* csr;             // n_bins + 1
  int32_t* blk;             // [n_bins][nb1]
  int32_t list, bin_lo, n_bins, nb1, shift;
  int32_t entry0;           // its first bin in the plan-wide numbering
  uint32_t* copy;           // room for the FFT indices of `cap` peaks
  int64_t cap;
};

// One tile of the accumulation kernel: k rows [row0, row0+nrows) x columns [col0, col0+ncols).
struct TileDev {
  int32_t map;
  int32_t row0;
  int32_t nrows;
  int32_t ncols;
  int64_t col0;
  int32_t bin_a;      // peaks with bins in [bin_a, bin_b] may touch the tile (bin_a > bin_b: none)
  int32_t bin_b;
  int32_t band_lo;    // candidate bands present in the tile's columns (band_hi < 0: none)
  int32_t band_hi;
  int32_t one;        // drawn with one count per cell, not two
};

struct gfh_plan {
  gfh_ctx* ctx = nullptr;
  int n_maps = 0;
  std::vector<gfh_grid> grids;
  gfh_tile_config cfg{};
  int threads = 0, list_threads = 0;   // of a block: full search, coarse tiles
  int64_t list_room = 0;       // words of a coarse tile's tiles
  size_t cells = 0, cells_x = 0, cells_list = 0;   // shared memory of the largest tile's counts: full
                                                   // search's two lists, coarse tiles
  void* d_buf = nullptr;       // tables, map descriptors, tiles
  MapDev* d_maps = nullptr;
  TileDev* d_tiles = nullptr;          // tiles of x-direction maps follow the others
  int n_tiles = 0;                     // tiles differenced along k (rows > 0)
  int n_tiles_x = 0;                   // tiles of maps moving > 2 columns per k row: along x0
  std::vector<char> map_xd, map_one;   // per map: drawn in the x-direction form, with one count per cell
  int max_tile_bands = 0;
  // zeroed per execute, in one piece: all maps' keys and sums, the lists' order states, the tile
  // counters (full search's two launches; coarse-tile list length and next tile)
  void* d_zeroed = nullptr;
  size_t zeroed_bytes = 0;
  unsigned long long* d_keys = nullptr;
  int* d_list_state = nullptr;            // per peak list a map reads: order bits (k_check_sorted)
  int n_list_states = 0;                  // largest list index + 1
  int* d_next = nullptr;
  int* d_sel_count = nullptr;
  ListDev* d_lists = nullptr;             // the runs of bins that maps read
  int32_t csr_entries = 0;                // their bins in all
  int32_t* d_csr_list = nullptr;          // per bin: its entry of d_lists
  bool select = false;
  int64_t* d_offsets_single = nullptr;    // scratch offsets for gfh_hough
  // the bound outputs, kept so that the autotuner can rebuild the plan with another tile shape
  std::vector<int32_t*> h_maps;
  std::vector<gfh_candidate*> h_cands;
  gfh_map_stats* d_stats = nullptr;
  // coarse tiles (gfh_plan_set_coarse): per (map, coarse tile) the fine tiles that cover it
  // (group coarse_k * coarse_x of a map = all of the map's tiles, for a full search)
  int coarse_k = 0, coarse_x = 0, max_sel = 0;
  void* d_coarse_buf = nullptr;
  TileDev* d_fine = nullptr;           // fine tiles, grouped by (map, coarse tile)
  int32_t* d_coarse_first = nullptr;   // n_maps * (coarse_k * coarse_x + 1) + 1 group offsets
  TileDev* d_sel_tiles = nullptr;      // the gathered tile list (worst case: every map in full)
  int sel_cap = 0;                     // capacity of d_sel_tiles
};

// Host-side planning (gfh_host.cpp).
int gfh_host_tables(const gfh_grid* g, std::vector<int64_t>& U, std::vector<int64_t>& B,
                    std::vector<int64_t>& S);
int gfh_host_columns(const gfh_grid* g, std::vector<int32_t>& band, std::vector<double>& f0,
                     std::vector<double>& f0n);

// gfh_plan_create; once: for a single execution, planned in less time.
int gfh_make_plan(gfh_ctx* ctx, int32_t n_maps, const gfh_grid* grids, int32_t* const* h_maps,
                  gfh_candidate* const* h_cands, gfh_map_stats* d_stats, const gfh_tile_config* cfg,
                  bool once, gfh_plan** out);

// The context's scratch buffer (gfh_peakmap.cu), grown on demand.
int ensure_scratch(gfh_ctx* c, size_t bytes);
// Equaliser + peak test + compaction on band spectra d_x [n_fft][ld] holding bins j0 .. j0+ld-1
// (float2), with `extra` bytes at the front of the context scratch kept for the caller; the
// scratch that needs, to be ensured up front so that the caller's part is never reallocated.
int gfh_band_peaks(gfh_ctx* c, const float2* d_x, int64_t ld, int32_t j0, int32_t n_fft,
                   int32_t bin_lo, int32_t bin_hi, double theta, uint32_t* d_fft_idx,
                   uint32_t* d_bin, int64_t cap, int64_t* h_n_peaks, size_t extra);
size_t gfh_peaks_scratch(int32_t n_fft, int32_t bin_lo, int32_t bin_hi, size_t extra);
// A cuFFT plan of `batch` interlaced frames of N samples (hop N/2) on the context's stream.
int gfh_fft_plan(gfh_ctx* c, int N, int batch, bool c2c, cufftHandle* out);

// Launchers (gfh_hough.cu).
int gfh_launch_plan(gfh_plan* plan, const gfh_peaks* peaks);
int gfh_launch_plan_tiles(gfh_plan* plan, const gfh_peaks* peaks, const int32_t* d_coarse,
                          int n_sel, const int32_t* d_full);
int gfh_prepare_plan(gfh_plan* plan);   // one-time kernel attributes (outside any capture)
