// Generalized FrequencyHough accumulation (Sec. IV) on sm_103a.
//
// Each peak (FFT i, bin j) is the set of lines x0 = x - (n-1) k t_i for x across its bin
// (Eq. transform, Sec. IV).  On k row r it covers the x0 columns that the half-open fixed-point
// interval [U[j+1] - B_i - r S_i, U[j] - B_i - r S_i) overlaps.  The map is built per tile of
// k rows x x0 columns in shared memory by differential counting: +1 at the first covered column,
// -1 after the last on the tile's first row, then one event for every column an edge moves
// (shared-memory increments; intervals that start left of the tile go to a per-thread register carry
// instead of contending on column 0), then running sums and one vectorised streaming store of every
// map cell.  Candidate selection (Sec. IV: highest count
// per f0 band, critical ratio from the map's mean and deviation) is fused into the store pass.
#include <algorithm>
#include <type_traits>

#include "gfh_internal.h"

namespace {

constexpr int kLane = 32;
// Bits of a peak list's order state: bins not ascending, some bin's peaks not in FFT order, and no copy
// of its FFT indices by blocks of FFTs.
constexpr int kListUnsorted = 1, kListFftUnsorted = 2, kListNoCopy = 4;
constexpr int kIndexWarps = 8;   // bins per block of k_index
constexpr int kFewBands = 4;     // a tile of at most this many bands looks for its best cells only if they can win
template <int NT> constexpr int kSumBytes = NT / kLane * 16;   // two sums per warp
constexpr int kRowBits = 57;     // fraction bits of an event's row
constexpr int kEventUnroll = 4;  // events of each edge per turn of the drawing loop
constexpr int kSpareRows = kEventUnroll + 2;   // words for events that are not drawn, in rows of 32

__device__ __forceinline__ int warp_sum(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ long long warp_sum64(long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ int warp_incl_scan(int v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += u;
  }
  return v;
}

// Candidate key: count in the high word, inverted row-major cell index in the low word, so the
// maximum key is the highest count with ties to the lowest (row, column).
__device__ __forceinline__ unsigned long long cand_key(int count, uint32_t lin) {
  return ((unsigned long long)(uint32_t)count << 32) | (unsigned long long)(0xffffffffu - lin);
}

// ---- per-execute preparation --------------------------------------------------------------------

// Order of each peak list (state[l], l < n_states, zeroed before): kListUnsorted when its bins are not ascending
// (also flagged; such a list is not drawn), kListFftUnsorted when some bin's peaks are not in FFT
// order (k_index then copies them by blocks of FFTs).
//
// The blocks share out the peaks of all lists evenly, whatever the lists' lengths.  Bound by its 8 bytes
// per peak; with 8 blocks for each of 256 lists of 18 thousand to 18 million peaks it took 8 ms, the
// longest list's, where the bytes take 0.6.
__global__ void __launch_bounds__(256) k_check_sorted(const uint32_t* __restrict__ bins, const uint32_t* __restrict__ fft,
                               const int64_t* __restrict__ off, int n_lists, float per_block,
                               unsigned int* flag, int* __restrict__ state, int n_states) {
  const int64_t begin = off[0], end = off[n_lists];
  // an equal part, a little more for float32's rounding, of at least a pair per thread
  const int64_t part = max((int64_t)((float)(end - begin) * per_block) + 32, (int64_t)256) & ~(int64_t)31;
  const int64_t c0 = begin + blockIdx.x * part, c1 = min(c0 + part, end);
  if (c0 >= c1) return;
  int l = 0;                                       // last list that begins at or before c0
  for (int hi = n_lists - 1; l < hi;) {
    const int mid = (l + hi + 1) / 2;
    if (off[mid] <= c0) l = mid; else hi = mid - 1;
  }
  for (int64_t first = n_lists == 1 ? begin : off[l]; first < c1;) {
    const int64_t next = n_lists == 1 ? end : off[l + 1];
    const int64_t b = max(first + 1, c0), e = min(next, c1);
    int bad = 0;
    // four independent pairs per turn
    for (int64_t p0 = b + threadIdx.x; p0 < e; p0 += 4 * 256) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int64_t p = p0 + q * 256;
        if (p >= e) continue;
        const uint32_t j1 = bins[p], j0 = bins[p - 1], f1 = fft[p], f0 = fft[p - 1];
        if (j1 < j0) bad |= kListUnsorted;
        else if (j1 == j0 && f1 < f0) bad |= kListFftUnsorted;
      }
    }
    // one lane per warp, and only what is not known yet
    bad = (int)__reduce_or_sync(0xffffffffu, (unsigned)bad);
    if (bad && threadIdx.x % kLane == 0) {
      if (bad & kListUnsorted) atomicOr(flag, GFH_FLAG_UNSORTED);
      if (l < n_states && (bad & ~*reinterpret_cast<volatile int*>(&state[l]))) atomicOr(&state[l], bad);
    }
    if (++l >= n_lists) break;
    first = next;
  }
}

// First of the list's peaks [lo, hi) with bin >= key, by the whole warp (a 32-way search, five bits a
// step).
__device__ __forceinline__ int64_t first_of_bin(const uint32_t* __restrict__ bins, int64_t lo, int64_t hi,
                                                uint32_t key, int lane) {
  while (lo < hi) {
    const int64_t step = (hi - lo) / kLane + 1;    // probes lo + step (lane + 1) - 1
    const int64_t at = lo + step * (lane + 1) - 1;
    const bool less = at < hi && bins[at] < key;
    const int64_t l = lo + step * __popc(__ballot_sync(0xffffffffu, less));
    hi = min(hi, l + step - 1);
    lo = l;
  }
  return lo;
}

// A bin's n FFT indices f out of order: copied to dst by blocks of 2^shift FFTs, in any order inside one
// (the tiles read whole blocks), the largest last; begin[b], b < nb1: first of block b.  h: nb1 + 1
// words of the warp's.
__device__ __forceinline__ void order_bin(const uint32_t* __restrict__ f, int n, int nb1, int shift,
                                          int32_t* __restrict__ begin, uint32_t* __restrict__ dst, int* h,
                                          int lane) {
  for (int b = lane; b <= nb1; b += kLane) h[b] = 0;
  __syncwarp();
  uint32_t top = 0;
  for (int i = lane; i < n; i += kLane) {
    const uint32_t v = f[i];
    top = max(top, v);
    atomicAdd(&h[min(v >> shift, (uint32_t)(nb1 - 1))], 1);
  }
  top = __reduce_max_sync(0xffffffffu, top);
  __syncwarp();
  int before = 0;
  for (int b0 = 0; b0 < nb1; b0 += kLane) {
    const int b = b0 + lane, c = b < nb1 ? h[b] : 0, incl = warp_incl_scan(c, lane);
    if (b < nb1) {
      h[b] = before + incl - c;
      begin[b] = b + 1 < nb1 ? before + incl - c : n;
    }
    before += __shfl_sync(0xffffffffu, incl, kLane - 1);
  }
  __syncwarp();
  for (int i = lane; i < n; i += kLane) {
    const uint32_t v = f[i];
    const bool last = v == top && atomicExch(&h[nb1], 1) == 0;
    dst[last ? n - 1 : atomicAdd(&h[min(v >> shift, (uint32_t)(nb1 - 1))], 1)] = v;
  }
}

// Index of the peak lists, one warp per (list, bin): csr = the bin's first peak, and per block of
// 2^shift FFTs the offset inside the bin of its first peak with FFT index in that block or later.  The
// bins of a list out of FFT order are also copied by blocks, so that its tiles have their windows too:
// walked whole by the tiles planned for windows, such lists took up to 4.4 times as long (paper-shaped
// maps 20.3 ms for 4.64 in order, now 4.69; one half-hour map 186 us for 102, now 105).  A list of more
// peaks than the copy holds keeps none; its bins are walked whole.
__global__ void __launch_bounds__(kIndexWarps * kLane)
k_index(const ListDev* __restrict__ lists, const int32_t* __restrict__ entry_list, int n_entries,
        const uint32_t* __restrict__ bins, const uint32_t* __restrict__ fft, const int64_t* __restrict__ off,
        int* __restrict__ state) {
  __shared__ int s_h[kIndexWarps][kMaxFftBlocks + 2];
  const int e = blockIdx.x * kIndexWarps + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (e >= n_entries) return;
  const ListDev& ld = lists[entry_list[e]];
  const int jl = e - ld.entry0;
  const int st = state[ld.list];
  // first peaks with bin >= key and >= key + 1
  int64_t lo[2], hi[2];
#pragma unroll
  for (int w = 0; w < 2; ++w) { lo[w] = off[ld.list]; hi[w] = off[ld.list + 1]; }
  while (lo[0] < hi[0] || lo[1] < hi[1]) {
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      const int64_t n = hi[w] - lo[w];
      if (n <= 0) continue;
      const uint32_t key = (uint32_t)(ld.bin_lo + jl + w);
      const int64_t step = n / kLane + 1;          // probes lo + step (lane + 1) - 1
      const int64_t at = lo[w] + step * (lane + 1) - 1;
      const bool less = at < hi[w] && bins[at] < key;
      const int c = __popc(__ballot_sync(0xffffffffu, less));
      const int64_t l = lo[w] + step * c;
      hi[w] = min(hi[w], l + step - 1);
      lo[w] = l;
    }
  }
  if (lane == 0) {
    ld.csr[jl] = lo[0];
    if (jl == ld.n_bins - 1) ld.csr[jl + 1] = lo[1];
  }
  const int n = (int)(lo[1] - lo[0]);
  int32_t* const begin = ld.blk + (int64_t)jl * ld.nb1;
  if ((st & kListFftUnsorted) && !(st & kListUnsorted)) {
    const int64_t at = lo[0] - first_of_bin(bins, off[ld.list], off[ld.list + 1], (uint32_t)ld.bin_lo, lane);
    if (at + n <= ld.cap)
      order_bin(fft + lo[0], n, ld.nb1, ld.shift, begin, ld.copy + at, s_h[threadIdx.x >> 5], lane);
    else if (lane == 0)
      atomicOr(&state[ld.list], kListNoCopy);
    return;
  }
  for (int b = lane; b < ld.nb1; b += kLane) {
    const uint32_t key = (uint32_t)b << ld.shift;
    int l = 0, h = b + 1 < ld.nb1 ? n : 0;
    while (l < h) {
      const int mid = (l + h) >> 1;
      if (__ldg(fft + lo[0] + mid) < key) l = mid + 1; else h = mid;
    }
    begin[b] = b + 1 < ld.nb1 ? l : n;
  }
}

__global__ void k_set_offsets(int64_t* off, int64_t n) {
  if (threadIdx.x == 0) { off[0] = 0; off[1] = n; }
}

// (f D) / 2^32 rounded up: the time, in rows of 2^-kRowBits, at which an edge whose position has the
// fraction f (2^-32 columns) above a column boundary reaches that boundary.
__device__ __forceinline__ uint64_t first_crossing(uint32_t f, uint64_t D) {
  const uint64_t lo = (uint64_t)f * (uint32_t)D + 0xffffffffull;
  return (uint64_t)f * (uint32_t)(D >> 32) + (lo >> 32);
}

// Adds 1 to the shared word at byte address p.  A conditional increment with no upper bound: the
// hardware counts the lanes of a warp that hit one word at the full rate, as for atomicAdd(p, 1),
// while an atomicAdd(p, -1) serialises them (33 cycles a warp instruction with all lanes on one
// word, against 1.1).
__device__ __forceinline__ void inc_shared(uint32_t p) {
  asm volatile("red.shared.inc.u32 [%0], 0xffffffff;" ::"r"(p) : "memory");
}

// Counts a column that is left: 1 in the second count, or (TAKE) -1 in the only one.
template <bool TAKE>
__device__ __forceinline__ void leave_shared(uint32_t p) {
  if (TAKE) asm volatile("red.shared.add.u32 [%0], 0xffffffff;" ::"r"(p) : "memory");
  else inc_shared(p);
}

// One event: adds 1 (TAKE: -1) at row v / 2^kRowBits of the column Q before the one p points at; with
// LIMIT only if n > Q, else to one of the warp's spare words.  (A predicated increment compiles to a branch
// around it, with its reconvergence three instructions more per event; lanes that share the spare
// word cost nothing where 1 is added; -1 is added to a word of the lane's own: on one word for all it
// took 6.6 instead of 3.8 ms on 11 braking indices.)
template <int Q, bool LIMIT, bool TAKE>
__device__ __forceinline__ void event(uint64_t v, uint32_t p, int n, uint32_t row_bytes,
                                      uint32_t spare) {
  uint32_t at = (uint32_t)(v >> kRowBits) * row_bytes + p;
  if (LIMIT) at = n > Q ? at : spare;
  if (TAKE) asm volatile("red.shared.add.u32 [%0 + %1], 0xffffffff;" ::"r"(at), "n"(-4 * Q) : "memory");
  else asm volatile("red.shared.inc.u32 [%0 + %1], 0xffffffff;" ::"r"(at), "n"(-4 * Q) : "memory");
}

// kEventUnroll events of the left and of the right edge.
template <int Q, bool LIMIT, bool ONE>
__device__ __forceinline__ void events(uint64_t& v1, uint64_t& v2, uint64_t D, uint32_t p1,
                                       uint32_t p2, int n1, int n2, uint32_t row_bytes,
                                       uint32_t spare, uint32_t own) {
  if constexpr (Q < kEventUnroll) {
    event<Q, LIMIT, false>(v1, p1, n1, row_bytes, spare);
    event<Q, LIMIT, ONE>(v2, p2, n2, row_bytes, ONE ? own : spare);
    v1 += D;
    v2 += D;
    events<Q + 1, LIMIT, ONE>(v1, v2, D, p1, p2, n1, n2, row_bytes, spare, own);
  }
}

// Draws one peak of each lane on the nr rows of a tile (layout described at hough_tile below); all
// 32 lanes call it together, `ok` where the lane has a peak.  On row 0 the peak's interval is
// [a, b1 + 1) in 2^-32 columns from the tile's first column, and it moves left by s >= 0 per row
// (t_first >= 0 and dk > 0 make every S_i non-negative).  ge, gl: shared addresses of the entered
// and the left columns' counts.
//
// The rows after the first are drawn edge event by edge event and not row by row.  An edge at
// position p on row 0, f = frac(p), crosses its (e+1)-th column boundary (e = 0, 1, ...) at the
// first row r with r s > f + e 2^32, so r = floor(x_e) + 1 with x_e = (f + e 2^32) / s.  x_e is kept
// in rows of 2^-57 and stepped by D = ceil(2^89 / s), the rows per column (a table entry per FFT):
// every rounding is upwards and below 256 units of 2^-57 in all (at most 254 steps: two columns on each
// of 127 rows), while an x_e that is no integer lies at least 1/s >= 2^-33 below the next one, so
// floor() is exact.  The left edge enters a
// column at its event (one lower each event), the right edge leaves one.
// Lanes of a warp hold neighbouring FFTs of one bin, whose s, and so whose event counts, are nearly
// alike: the loop runs to the warp's largest count.
// D = 0 marks s <= 2^25 (D would not fit): at most one crossing in the tile's rows (at most 128),
// placed by an integer division.
template <bool ONE>
__device__ __forceinline__ void draw_peaks(uint32_t ge, uint32_t gl, uint32_t row_bytes,
                                           uint32_t spare, uint32_t own, int nr, int C, int ub, bool ok, int64_t a, int64_t b1, int64_t s,
                                           uint64_t D, int& carry) {
  const int64_t sr = (int64_t)((uint64_t)(uint32_t)(nr - 1) * (uint64_t)s);
  int lo = (int)(a >> GFH_FRAC_BITS), hr = (int)(b1 >> GFH_FRAC_BITS);
  const int lo_n = (int)((a - sr) >> GFH_FRAC_BITS), hr_n = (int)((b1 - sr) >> GFH_FRAC_BITS);
  // The interval meets the tile on some row: its right edge is highest on the first row, its left
  // edge lowest on the last.
  ok = ok && hr >= 0 && lo_n <= ub;
  if (!__any_sync(0xffffffffu, ok)) return;
  // row 0 along x0: clamped to the map's last column and to the tile; an interval that starts left
  // of the tile is a carry into its first column
  const int o1 = max(lo, 0), o2 = min(hr, ub);
  const bool on = ok && o1 <= o2;
  carry += on && lo < 0;
  inc_shared(on && lo >= 0 ? ge + 4u * (uint32_t)lo : spare);
  leave_shared<ONE>(on && o2 < C - 1 ? gl + 4u * (uint32_t)(o2 + 1) : (ONE ? own : spare));
  // events of the left and the right edge: columns entered, lo - 1 down to lo_n, and left, hr down to
  // hr_n + 1; those below 0 are not drawn
  int n1 = ok ? lo - max(lo_n, 0) : 0;
  int n2 = ok ? hr - max(hr_n, -1) : 0;
  if (__any_sync(0xffffffffu, max(n1, n2) > 0) == 0) return;
  uint64_t v1 = first_crossing((uint32_t)a, D), v2 = first_crossing((uint32_t)b1, D);
  if (D == 0 && ok) {
    const uint32_t d = max((uint32_t)s, 1u);
    v1 = (uint64_t)((uint32_t)a / d) << kRowBits;
    v2 = (uint64_t)((uint32_t)b1 / d) << kRowBits;
  }
  // columns right of the tile come first: skip their events
  if (__any_sync(0xffffffffu, ok && hr >= C)) {
    const int e1 = max(lo - C, 0), e2 = max(hr - (C - 1), 0);
    v1 += (uint64_t)(uint32_t)e1 * D;
    v2 += (uint64_t)(uint32_t)e2 * D;
    lo -= e1;
    n1 -= e1;
    hr -= e2;
    n2 -= e2;
  }
  uint32_t p1 = ge + row_bytes + 4u * (uint32_t)(lo - 1);
  uint32_t p2 = gl + row_bytes + 4u * (uint32_t)hr;
  // first the turns in which every lane has all its events, then the rest
  const int most = __reduce_max_sync(0xffffffffu, max(n1, n2));
  const int least = __reduce_min_sync(0xffffffffu, min(n1, n2));
  int e = 0;
  for (; e + kEventUnroll <= least; e += kEventUnroll) {
    events<0, false, ONE>(v1, v2, D, p1, p2, n1, n2, row_bytes, spare, own);
    p1 -= 4 * kEventUnroll;
    p2 -= 4 * kEventUnroll;
  }
  for (; e < most; e += kEventUnroll) {
    events<0, true, ONE>(v1, v2, D, p1, p2, n1 - e, n2 - e, row_bytes, spare, own);
    p1 -= 4 * kEventUnroll;
    p2 -= 4 * kEventUnroll;
  }
}

// Events of one peak on the R rows of a tile in the x-direction form: every row differenced along
// x0 (entered at its first column, left after its last), so a row costs two events whatever the
// shift per row; an interval entering from the left of the tile counts in that row's carry.
template <int R, bool ONE>
__device__ __forceinline__ void draw_peak_x(uint32_t ge, uint32_t gl, uint32_t row_bytes, int64_t a,
                                            int64_t b1, int64_t s, int C, int ub, int (&carry)[R]) {
#pragma unroll
  for (int rr = 0; rr < R; ++rr) {
    const int lo = (int)(a >> GFH_FRAC_BITS);
    const int hi = min((int)(b1 >> GFH_FRAC_BITS), ub);
    const int o1 = max(lo, 0);
    if (o1 <= hi) {
      if (lo < 0) carry[rr] += 1;
      else inc_shared(ge + rr * row_bytes + 4u * (uint32_t)o1);
      if (hi < C - 1) leave_shared<ONE>(gl + rr * row_bytes + 4u * (uint32_t)(hi + 1));
    }
    a -= s;
    b1 -= s;
  }
}

// ---- the accumulation + running sums + select kernel --------------------------------------------

// A tile that no edge meets: every cell holds the number of intervals that cover the tile.  mine: a
// warp's share of it (the same in all its lanes).
template <int NT, bool SELECT>
__device__ __forceinline__ void fill_tile(const MapDev& md, const TileDev& t, int mine, int* wsum,
                                          int nb_tile, uint64_t* s_sums) {
  constexpr int NW = NT / kLane;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __syncthreads();                               // wsum is free
  if (lane == 0) wsum[warp] = mine;
  __syncthreads();
  const int c = warp_sum(lane < NW ? wsum[lane] : 0);
  const int C = t.ncols, quads = C / 4;
  int32_t* const out = md.out + (int64_t)t.row0 * md.ld + t.col0;
  const int real = (int)min((int64_t)C, md.W - t.col0);          // the padding stays 0
  for (int rr = warp; rr < t.nrows; rr += NW)
    for (int q = lane; q < quads; q += kLane) {
      const int m = 4 * q;
      __stcs(reinterpret_cast<int4*>(out + rr * md.ld + m),
             make_int4(m < real ? c : 0, m + 1 < real ? c : 0, m + 2 < real ? c : 0, m + 3 < real ? c : 0));
    }
  if (!SELECT || nb_tile == 0) return;
  // each band's lowest cell is its first column on the tile's first row
  int n = 0;
  for (int m = tid; m < real; m += NT) {
    const int b = __ldg(md.col_band + t.col0 + m);
    if (b < 0) continue;
    ++n;
    if (m > 0 && __ldg(md.col_band + t.col0 + m - 1) == b) continue;
    const unsigned long long now = *reinterpret_cast<volatile unsigned long long*>(&md.keys[b]);
    if (now == 0 || c >= (int)(now >> 32))
      atomicMax(&md.keys[b], cand_key(c, (uint32_t)t.row0 * (uint32_t)md.W + (uint32_t)(t.col0 + m)));
  }
  n = warp_sum(n);
  if (lane == 0) {
    const uint64_t cells = (uint64_t)n * (uint32_t)t.nrows;
    s_sums[2 * warp] += cells * (uint32_t)c;
    s_sums[2 * warp + 1] += cells * (uint32_t)c * (uint32_t)c;
  }
}

// A tile is some k rows x C columns; each lane draws peaks of its own on all its rows.
//
// Shared memory holds two counts per cell, G[rows][C + pad] of the columns entered and, after it, of
// the columns left; their difference is a mixed differential of the tile:
//   row 0:     along x0 - +1 at the first column an interval covers, -1 after its last, so that
//              M[0][m] = sum_{m' <= m} G[0][m'];
//   row r > 0: along k - +1 at each column the interval newly covers on row r, -1 at each column it
//              covered on row r-1 but no longer does, so that M[r][m] = M[r-1][m] + G[r][m].
// (Two counts and not one signed one: see inc_shared.)  Tiles of sparse maps (TileDev::one) keep one
// signed count and have twice the cells in the same memory.
// Along k a peak's interval shifts left by S_i < 1 column per row with the default k step, so on
// most rows it enters no column and leaves none: rows after the first cost about one event per
// (peak, row) instead of two.  An interval entering from the left of the tile on row 0 is a
// per-thread carry into the first column.
//
// Peaks.  The tile reads the bins that some FFT can bring into it on some row.  Over tall maps the
// FFTs' shifts spread far wider than a bin, so of each bin only the FFTs of one window have an edge
// in the tile: the window comes from the line that the shifts follow, its peaks from the list's
// index (k_index), and only those are walked (whole blocks of FFTs, so a few beside them too).
// Peak lists that are not in FFT order inside a bin read their copy by blocks of FFTs, or whole bins
// where the list has none.  The windows of up to `batch`
// bins at a time are laid end to end, two pieces per bin: ent[] = {end of the piece in that order,
// where its peaks lie in the list less its begin}.  Each warp walks one contiguous part, 32 peaks at
// a time whatever bins they are of.  A tile that no edge meets holds one number and needs no sums.
//
// What bounds it: on dense maps (20 sub-band maps of 2000 rows, 226M cells, 9.0e9 peak rows) the
// events' integer instructions (0.48 warp instructions per peak row in all, about 70 % of the issue slots) and
// the increments' bank conflicts (2.43 wavefronts each): 4.64 ms against 7.56 ms for the row-by-row form
// on flat 16 x 3072 tiles.  On sparse maps (11 braking indices, 1.76e9 cells, 1.3 peak rows per cell)
// the tiles' chain of dependent loads and barriers (44 % of the issue slots): with one count per cell
// 4.04 against 5.67 ms, five maps of 228-1858 rows x 85,654-164,343 columns 1.10 against 1.46 ms.  Small
// maps gain from the planned tiles (whole calls): 500 rows x 51,695 columns 102 against 234 us, the 32
// rows of a followed-up candidate 41 against 86 us, 12 uneven peakmaps 0.48 against 1.42 ms.  Tall maps of
// a few hundred FFTs can be the slower ones, by up to a fifth below 75 us a call (2118 rows x 2540
// columns of 652 FFTs 73 against 65 us): their windows are a few peaks of many bins.
//
// Shared memory: tot[32] row-0 chunk sums | spare words | skey[bands] candidate keys | sums per warp
// | ent[2 batch] | G.
// XD (maps whose line moves more than two x0 columns per k row): every row differenced along x0
// and scanned on its own; chunk sums tot[R][32].
template <int R, int NT, bool SELECT, bool XD>
__device__ __forceinline__ void hough_tile(const MapDev* __restrict__ maps, const TileDev t,
                                           const uint32_t* __restrict__ fft_idx,
                                           const int* __restrict__ list_state,
                                           unsigned int* __restrict__ flag, unsigned char* smem,
                                           uint64_t* s_sums, int2* ent, int batch, int* G) {
  __shared__ int s_best[kFewBands], s_seek[kFewBands];
  constexpr int NW = NT / kLane;
  const MapDev& md = maps[t.map];
  const int C = t.ncols;
  const int lds = C + kHoughPad;                 // row stride
  const int words = (XD ? R : t.nrows) * lds;
  const bool one = t.one;
  const int gap = one ? 0 : words;               // from the columns entered to the columns left
  int* tot = reinterpret_cast<int*>(smem);
  int* wsum = tot;                               // the warps' sums while windows are laid out
  unsigned long long* skey = reinterpret_cast<unsigned long long*>(tot + ((XD ? R : 1) + kSpareRows) * kLane);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nb_tile = t.band_hi >= t.band_lo ? t.band_hi - t.band_lo + 1 : 0;
  const int c0 = (int)t.col0;
  const int ub = min(C - 1, (int)(md.W - 1 - t.col0));   // last column inside the map
  const uint32_t ge = (uint32_t)__cvta_generic_to_shared(G), gl = ge + 4u * (uint32_t)gap;
  const uint32_t row_bytes = 4u * (uint32_t)lds;
  // spare words: kEventUnroll per warp, then as many below the lanes' own (an event's offset reaches
  // them), which the warps share
  const uint32_t spares = (uint32_t)__cvta_generic_to_shared(tot + (XD ? R : 1) * kLane);
  const uint32_t spare = spares + 4u * (uint32_t)(kEventUnroll * (warp + 1) - 1);
  const uint32_t own = spares + 4u * (uint32_t)(kEventUnroll * kLane + kEventUnroll + lane);
  if (SELECT) {
    for (int i = tid; i < nb_tile; i += NT) skey[i] = 0ull;
    if (tid < kFewBands) s_best[tid] = 0;
  }
  int carry = 0;
  int carry_x[XD ? R : 1] = {};
  bool drawn = false;                            // some peak has an edge in the tile

  // ---- accumulate
  const int state = list_state[md.list];
  if (t.bin_a <= t.bin_b && !(state & kListUnsorted)) {
    const int bin0 = t.bin_a - md.bin_lo, nbw = t.bin_b - t.bin_a + 1;
    const int64_t pb = md.csr[bin0];
    // this tile's peaks with 32-bit offsets (a range beyond 2^31 - 2^20 peaks raises the capacity
    // flag and is not drawn)
    const bool fits = md.csr[bin0 + nbw] - pb <= (int64_t)0x7fffffff - (1 << 20);
    if (!fits && tid == 0) atomicOr(flag, GFH_FLAG_CAPACITY);
    const bool copied = (state & (kListFftUnsorted | kListNoCopy)) == kListFftUnsorted;
    const uint32_t* const fl = copied ? md.copy + (pb - *md.csr_list) : fft_idx + pb;
    const uint32_t nfft = (uint32_t)md.n_fft;
    const FftRow* const SD = md.SD;
    const int64_t* const Bt = md.B;
    const longlong2* const UP = md.UP + bin0;
    const bool window = copied || !(state & kListFftUnsorted);
    for (int q0 = 0; q0 < (fits ? nbw : 0); q0 += batch) {
      const int nq = min(batch, nbw - q0);
      // per bin (one thread each): its peaks that have an edge in the tile, in one or two pieces
      int st1 = 0, cnt1 = 0, st2 = 0, cnt2 = 0;
      if (tid < nq) {
        const int q = q0 + tid;
        const int64_t s = md.csr[bin0 + q];
        st1 = (int)(s - pb);
        cnt1 = (int)(md.csr[bin0 + q + 1] - s);
        if (window && cnt1 > 0) {
          const longlong2 up = __ldg(UP + q);
          const int32_t* const blk = md.blk + (int64_t)(bin0 + q) * md.nb1;
          const int n = cnt1;
          // indices past the table are flagged and drawn nowhere; the last is the largest
          const bool past = __ldg(fl + st1 + n - 1) >= nfft;
          if (past) atomicOr(flag, GFH_FLAG_FFT_RANGE);
          // first peaks of the FFT block that holds FFT i, and of the first block that starts there
          // or later (i <= 0: 0; i >= n_fft: all)
          auto from = [&](int i) { return i <= 0 ? 0 : (i >= md.n_fft ? n : __ldg(blk + (i >> md.shift))); };
          auto to = [&](int i) {
            return i <= 0 ? 0 : (i >= md.n_fft ? n : __ldg(blk + ((i - 1) >> md.shift) + 1));
          };
          const TileLine line = tile_line(md.line, t.row0, (int64_t)t.row0 + t.nrows - 1);
          const BinFfts w = bin_ffts(line, up.x, up.y, c0, ub, ub == C - 1, md.n_fft);
          const int o0 = from(w.lo), o1 = max(to(w.hi + 1), o0);
          st1 += o0;
          cnt1 = o1 - o0;
          // the FFTs that cover the tile on every row are counted without a walk
          if (!XD && w.c_lo < w.c_hi && cnt1 > 0) {
            const int m1 = max(to(w.c_lo + 1), o0);
            const int m2 = min(from(past ? min(w.c_hi, md.n_fft - 1) : w.c_hi), o1);
            if (m1 < m2) {
              carry += m2 - m1;
              cnt1 = m1 - o0;
              st2 = st1 - o0 + m2;
              cnt2 = o1 - m2;
            }
          }
        }
      }
      const int cnt = cnt1 + cnt2;
      const int incl = warp_incl_scan(cnt, lane);
      __syncthreads();                           // the previous batch is drawn
      if (lane == kLane - 1) wsum[warp] = incl;
      __syncthreads();
      const int ws = lane < NW ? wsum[lane] : 0;
      const int before = warp_sum(lane < warp ? ws : 0), total = warp_sum(ws);
      if (total == 0) continue;
      if (!drawn)
        for (int i = tid; i < (words + gap) / 4; i += NT) reinterpret_cast<int4*>(G)[i] = make_int4(0, 0, 0, 0);
      drawn = true;
      if (tid < nq) {
        const int e0 = before + incl - cnt;
        ent[2 * tid] = make_int2(e0 + cnt1, st1 - e0);
        ent[2 * tid + 1] = make_int2(e0 + cnt, st2 - (e0 + cnt1));
      }
      __syncthreads();
      // this warp's part: `units` runs of 32 peaks, split as evenly as they go
      const int units = (total + kLane - 1) / kLane;
      const int per = units / NW, rem = units % NW;
      const int u0 = warp * per + min(warp, rem);
      int v = u0 * kLane + lane;
      const int vend = min((u0 + per + (warp < rem ? 1 : 0)) * kLane, total);
      // the lane's place: piece q ends at q_end, peak v is fl[v + q_off]
      int q = 0, q_end = 0, q_off = 0;
      if (v < vend) {
        int hi = 2 * nq - 1;
        while (q < hi) {
          const int mid = (q + hi) >> 1;
          if (ent[mid].x > v) hi = mid; else q = mid + 1;
        }
        q_end = ent[q].x;
        q_off = ent[q].y;
      }
      auto fetch = [&](int x, uint32_t& f, int& j) {
        while (x >= q_end) {
          const int2 e = ent[++q];
          q_end = e.x;
          q_off = e.y;
        }
        f = __ldg(fl + x + q_off);
        j = q0 + (q >> 1);
      };
      // table rows of a peak; false (and the input flagged) for an out-of-range FFT index
      auto rows = [&](uint32_t f, int j, FftRow& sd, int64_t& B, longlong2& up) -> bool {
        if (f >= nfft) { atomicOr(flag, GFH_FLAG_FFT_RANGE); return false; }
        const longlong2 w = __ldg(reinterpret_cast<const longlong2*>(SD + f));
        sd.S = w.x;
        sd.D = (uint64_t)w.y;
        B = Bt ? __ldg(Bt + f) : 0;
        up = __ldg(UP + j);
        return true;
      };
      // Software pipeline: the FFT indices are loaded two runs of peaks ahead and the table rows one
      // run ahead of the peaks being drawn; the next peak's interval is formed from its rows after
      // the current one is drawn, so those loads have the whole drawing to arrive.  The lanes of a
      // warp stay together, also past the last peak.
      bool has_nx = false;                       // indices of peak v + 32
      uint32_t f_nx = 0;
      int j_nx = 0;
      int64_t a = 0, b1 = 0, s = 0;              // interval and shift of peak v
      uint64_t d = 0;
      bool ok = false;
      auto interval = [&](const FftRow& sd, int64_t B, const longlong2& up) {
        const int64_t base = B + (int64_t)((uint64_t)(uint32_t)t.row0 * (uint64_t)sd.S) +
                             ((int64_t)c0 << GFH_FRAC_BITS);
        a = up.x - base;                         // columns from the tile's first: [a, b1 + 1)
        b1 = up.y - base;
        s = sd.S;
        d = sd.D;
      };
      if (v < vend) {
        uint32_t f;
        int j;
        fetch(v, f, j);
        FftRow sd{};
        int64_t B = 0;
        longlong2 up = make_longlong2(0, 0);
        ok = rows(f, j, sd, B, up);
        interval(sd, B, up);
      }
      if (v + kLane < vend) { fetch(v + kLane, f_nx, j_nx); has_nx = true; }
      for (; v - lane < vend; v += kLane) {
        FftRow sd{};
        int64_t B = 0;
        longlong2 up = make_longlong2(0, 0);
        const bool ok_nx = has_nx && rows(f_nx, j_nx, sd, B, up);
        has_nx = v + 2 * kLane < vend;
        if (has_nx) fetch(v + 2 * kLane, f_nx, j_nx);
        if constexpr (XD) {
          // the interval meets the tile on some row (see draw_peaks)
          if (ok && (b1 >> GFH_FRAC_BITS) >= 0 && ((a - (R - 1) * s) >> GFH_FRAC_BITS) <= ub) {
            if (one) draw_peak_x<R, true>(ge, gl, row_bytes, a, b1, s, C, ub, carry_x);
            else draw_peak_x<R, false>(ge, gl, row_bytes, a, b1, s, C, ub, carry_x);
          }
        } else {
          if (one) draw_peaks<true>(ge, gl, row_bytes, spare, own, t.nrows, C, ub, ok, a, b1, s, d, carry);
          else draw_peaks<false>(ge, gl, row_bytes, spare, own, t.nrows, C, ub, ok, a, b1, s, d, carry);
        }
        interval(sd, B, up);
        ok = ok_nx;
      }
    }
  }
  if (!drawn) {
    fill_tile<NT, SELECT>(md, t, warp_sum(carry), wsum, nb_tile, s_sums);
    return;
  }
  if constexpr (XD) {
#pragma unroll
    for (int rr = 0; rr < R; ++rr) {
      const int v = warp_sum(carry_x[rr]);
      if (lane == 0 && v) atomicAdd(G + rr * lds, v);
    }
  } else {
    const int v = warp_sum(carry);
    if (lane == 0 && v) atomicAdd(G, v);
  }
  __syncthreads();

  // ---- running sums along x0: of row 0 in place, of every row (XD) as it is stored.  A chunk is 128
  // columns (32 lanes x 4).
  const int nch = (C + 127) / 128;
  const int nsum = XD ? t.nrows * nch : nch;
  auto load4 = [&](const int* g) {               // entered - left
    const int4 e = *reinterpret_cast<const int4*>(g);
    if (one) return e;
    const int4 l = *reinterpret_cast<const int4*>(g + gap);
    return make_int4(e.x - l.x, e.y - l.y, e.z - l.z, e.w - l.w);
  };
  for (int idx = warp; idx < nsum; idx += NW) {
    const int rr = idx / nch, ch = idx - rr * nch;
    const int col = ch * 128 + lane * 4;
    int s = 0;
    if (col < C) {
      const int4 g = load4(&G[rr * lds + col]);
      s = g.x + g.y + g.z + g.w;
    }
    s = warp_sum(s);
    if (lane == 0) tot[rr * kLane + ch] = s;
  }
  __syncthreads();
  if (!XD) {
    for (int ch = warp; ch < nch; ch += NW) {
      const int col = ch * 128 + lane * 4;
      const int before = warp_sum((lane < ch) ? tot[lane] : 0);
      int4 g = make_int4(0, 0, 0, 0);
      if (col < C) g = load4(&G[col]);
      g.y += g.x; g.z += g.y; g.w += g.z;
      const int add = before + warp_incl_scan(g.w, lane) - g.w;
      if (col < C) {
        *reinterpret_cast<int4*>(&G[col]) = make_int4(g.x + add, g.y + add, g.z + add, g.w + add);
        if (!one) *reinterpret_cast<int4*>(&G[col + gap]) = make_int4(0, 0, 0, 0);
      }
    }
    __syncthreads();
  }

  // ---- running sums along k; store; candidates.  A tile of few chunks is split into segments of
  // rows so that every warp has a share: first the column sums of all segments but the last (kept
  // where the windows were), then each (chunk, segment) from the sums before it.
  const int nseg = XD ? min(max(NW / nch, 1), t.nrows)
                      : max(1, min(min(NW / nch, t.nrows / 4), 1 + (int)(batch * 16) / (4 * C)));
  const int seg_rows = (t.nrows + nseg - 1) / nseg;
  int* const seg_sum = reinterpret_cast<int*>(ent);
  if (!XD && nseg > 1) {
    for (int u = warp; u < nch * (nseg - 1); u += NW) {
      const int sg = u / nch, col = (u - sg * nch) * 128 + lane * 4;
      if (col < C) {
        int4 v = make_int4(0, 0, 0, 0);
        for (int rr = sg * seg_rows; rr < min((sg + 1) * seg_rows, t.nrows); ++rr) {
          const int4 g = load4(&G[rr * lds + col]);
          v.x += g.x; v.y += g.y; v.z += g.z; v.w += g.w;
        }
        *reinterpret_cast<int4*>(seg_sum + sg * C + col) = v;
      }
    }
    __syncthreads();
  }
  // Candidates.  A tile with columns of at most kFewBands bands (wide bins) first takes each band's
  // largest count only, and looks for its cell in a second walk over the sums if it can win over the
  // map's best so far; with many bands every column tracks its best cell in the one walk.
  const bool few = !XD && nb_tile <= kFewBands;
  uint64_t s1 = 0, s2 = 0;
  const uint32_t W32 = (uint32_t)md.W;
  // map fields of the store pass read once (a global store could otherwise force a reload)
  int32_t* const out = md.out + t.col0;
  const int64_t ld_out = md.ld;
  const int32_t* const col_band = md.col_band + t.col0;
  for (int pass = 0; pass < 2; ++pass) {
    for (int u = warp; u < nch * nseg; u += NW) {
      const int sg = u / nch, col = (u - sg * nch) * 128 + lane * 4;
      const bool in = col < C;
      int band[4] = {-1, -1, -1, -1};
      if (SELECT && nb_tile > 0 && in) {
        const int4 bv = __ldg(reinterpret_cast<const int4*>(col_band + col));
        band[0] = bv.x; band[1] = bv.y; band[2] = bv.z; band[3] = bv.w;
      }
      bool any = SELECT && (band[0] & band[1] & band[2] & band[3]) != -1;
      if (XD) any = __any_sync(0xffffffffu, any);  // the warp stays together: it scans every row
      const bool all = SELECT && (band[0] | band[1] | band[2] | band[3]) >= 0;
      int4 v = make_int4(0, 0, 0, 0);
      if (!XD && in)
        for (int q = 0; q < sg; ++q) {
          const int4 g = *reinterpret_cast<const int4*>(seg_sum + q * C + col);
          v.x += g.x; v.y += g.y; v.z += g.z; v.w += g.w;
        }
      const int rb = sg * seg_rows, re = XD || in ? min(rb + seg_rows, t.nrows) : rb;
      const int* g0 = G + rb * lds + col;
      const int* tot0 = tot + rb * kLane;
      auto next = [&]() {
        if (!XD) {
          const int4 g = load4(g0);
          v.x += g.x; v.y += g.y; v.z += g.z; v.w += g.w;
        } else {
          int4 g = make_int4(0, 0, 0, 0);
          if (in) g = load4(g0);
          const int before = warp_sum(lane < u - sg * nch ? tot0[lane] : 0);
          tot0 += kLane;
          g.y += g.x; g.z += g.y; g.w += g.z;
          const int add = before + warp_incl_scan(g.w, lane) - g.w;
          v = make_int4(g.x + add, g.y + add, g.z + add, g.w + add);
        }
        g0 += lds;
      };
      if (pass == 1) {                             // the cells that hold a sought band's best count
        int want[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          want[q] = band[q] >= 0 && s_seek[band[q] - t.band_lo] ? s_best[band[q] - t.band_lo] : -1;
        const bool none = (want[0] & want[1] & want[2] & want[3]) == -1;
        if (XD ? __all_sync(0xffffffffu, none) : none) continue;
        for (int rr = rb; rr < re; ++rr) {
          next();
          const int vals[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (vals[q] == want[q])
              atomicMax(&skey[band[q] - t.band_lo],
                        cand_key(vals[q], (uint32_t)(t.row0 + rr) * W32 + (uint32_t)(t.col0 + col + q)));
        }
        continue;
      }
      int32_t* o = out + (int64_t)(t.row0 + rb) * ld_out + col;
      auto sums = [&]() {                          // of the analysis columns
        if (all) {
          s1 += (uint64_t)((uint32_t)v.x + (uint32_t)v.y) + (uint64_t)((uint32_t)v.z + (uint32_t)v.w);
          s2 += (uint64_t)(uint32_t)v.x * (uint32_t)v.x;
          s2 += (uint64_t)(uint32_t)v.y * (uint32_t)v.y;
          s2 += (uint64_t)(uint32_t)v.z * (uint32_t)v.z;
          s2 += (uint64_t)(uint32_t)v.w * (uint32_t)v.w;
        } else {
          const int vals[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (band[q] >= 0) {
              s1 += (uint32_t)vals[q];
              s2 += (uint64_t)(uint32_t)vals[q] * (uint32_t)vals[q];
            }
        }
      };
      if (!any) {
        for (int rr = rb; rr < re; ++rr) {
          next();
          if (!XD || in) __stcs(reinterpret_cast<int4*>(o), v);
          o += ld_out;
        }
      } else if (few) {
        int best[4] = {0, 0, 0, 0};
        for (int rr = rb; rr < re; ++rr) {
          next();
          if (!XD || in) __stcs(reinterpret_cast<int4*>(o), v);
          o += ld_out;
          sums();
          best[0] = max(best[0], v.x); best[1] = max(best[1], v.y);
          best[2] = max(best[2], v.z); best[3] = max(best[3], v.w);
        }
        if (all && band[0] == band[3]) {           // bands follow the columns
          atomicMax(&s_best[band[0] - t.band_lo], max(max(best[0], best[1]), max(best[2], best[3])));
        } else {
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (band[q] >= 0) atomicMax(&s_best[band[q] - t.band_lo], best[q]);
        }
      } else {
        // per column: best count over the rows so far and its row (strictly greater, so the first
        // row reaching the best count wins: the lowest cell index)
        int bc[4] = {-1, -1, -1, -1}, br[4] = {0, 0, 0, 0};
        for (int rr = rb; rr < re; ++rr) {
          next();
          if (!XD || in) __stcs(reinterpret_cast<int4*>(o), v);
          o += ld_out;
          sums();
          const int vals[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (vals[q] > bc[q]) { bc[q] = vals[q]; br[q] = rr; }
        }
        unsigned long long best[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          best[q] = bc[q] < 0 ? 0ull : cand_key(bc[q], (uint32_t)(t.row0 + br[q]) * W32 + (uint32_t)(t.col0 + col + q));
        // merge equal-band neighbours among the lane's 4 columns, then one shared atomic per run
        // (at the run's last column; every index static, so the arrays stay in registers)
        unsigned long long run = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          run = (q > 0 && band[q] == band[q - 1]) ? (best[q] > run ? best[q] : run) : best[q];
          const bool last = q == 3 || band[q < 3 ? q + 1 : q] != band[q];
          if (band[q] >= 0 && last) atomicMax(&skey[band[q] - t.band_lo], run);
        }
      }
    }
    if (!SELECT || nb_tile == 0) return;
    if (pass == 0) {
      // the block's sums so far, per warp (flushed to the map's when the block leaves the map)
      s1 = (uint64_t)warp_sum64((long long)s1);
      s2 = (uint64_t)warp_sum64((long long)s2);
      if (lane == 0) { s_sums[2 * warp] += s1; s_sums[2 * warp + 1] += s2; }
    }
    __syncthreads();
    if (!few || pass == 1) break;
    if (tid < nb_tile) {
      const unsigned long long now = *reinterpret_cast<volatile unsigned long long*>(&md.keys[t.band_lo + tid]);
      s_seek[tid] = now == 0 || s_best[tid] >= (int)(now >> 32);
    }
    if (!__syncthreads_or(tid < nb_tile && s_seek[tid])) return;
  }
  for (int i = tid; i < nb_tile; i += NT)
    if (skey[i]) atomicMax(&md.keys[t.band_lo + i], skey[i]);
}

// Persistent blocks over a list of tiles (every map of the plan in one launch): each block takes the
// next tile from the counter `next` (zeroed before the launch) until none is left.  The list holds
// n_tiles tiles, or min(*count, n_tiles) where count is given (the coarse-tile search's list, whose
// length is known on the device only).  A plan lists its tiles longest first, so the blocks finish
// together.  The index of a block's next tile is claimed when it starts a tile and read when it has
// finished it, so the atomic's round trip is hidden behind the tile.
template <int R, int NT, bool SELECT, bool XD>
__global__ void __launch_bounds__(NT, NT == 512 ? 2 : 3)
k_hough(const MapDev* __restrict__ maps, const TileDev* __restrict__ tiles, int n_tiles,
        const int* __restrict__ count, int* __restrict__ next, const uint32_t* __restrict__ fft_idx,
        const int* __restrict__ list_state, unsigned int* __restrict__ flag, int sum_off, int batch) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_next;
  uint64_t* const s_sums = reinterpret_cast<uint64_t*>(smem + sum_off);
  int2* const ent = reinterpret_cast<int2*>(smem + sum_off + kSumBytes<NT>);
  int* const G = reinterpret_cast<int*>(ent + 2 * batch);
  const int n = count ? min(*count, n_tiles) : n_tiles;
  if (threadIdx.x == 0) s_next = atomicAdd(next, 1);
  if (threadIdx.x < 2 * NT / kLane) s_sums[threadIdx.x] = 0;
  __syncthreads();
  int ti = s_next, map = -1;
  // adds the block's sums over the tiles of one map to the map's, and clears them
  auto flush = [&]() {
    if (!SELECT || map < 0 || threadIdx.x >= kLane) return;
    const int l = threadIdx.x;
    const bool on = l < NT / kLane;
    const long long a = warp_sum64(on ? (long long)s_sums[2 * l] : 0);
    const long long b = warp_sum64(on ? (long long)s_sums[2 * l + 1] : 0);
    if (on) s_sums[2 * l] = s_sums[2 * l + 1] = 0;
    if (l == 0 && (a | b)) {
      atomicAdd(&maps[map].sums[0], (unsigned long long)a);
      atomicAdd(&maps[map].sums[1], (unsigned long long)b);
    }
    __syncwarp();
  };
  while (ti < n) {
    __syncthreads();                                  // every thread has read s_next
    int claimed = 0;
    if (threadIdx.x == 0) claimed = atomicAdd(next, 1);
    const TileDev t = tiles[ti];
    if (t.map != map) { flush(); map = t.map; }
    if (t.nrows > 0)
      hough_tile<R, NT, SELECT, XD>(maps, t, fft_idx, list_state, flag, smem, s_sums, ent, batch, G);
    if (threadIdx.x == 0) s_next = claimed;
    __syncthreads();
    ti = s_next;
  }
  flush();
}

// ---- candidate records ----------------------------------------------------------------------------

// One thread per (map, band).  Every floating-point step uses an explicitly rounded intrinsic so
// no multiply-add is contracted: the records equal a plain IEEE double evaluation.
__global__ void k_finalize(const MapDev* __restrict__ maps) {
  const MapDev& md = maps[blockIdx.y];
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= md.n_bands) return;
  const unsigned long long s1u = md.sums[0], s2u = md.sums[1];
  const double cells = (double)md.cells;
  double mu = 0.0, sigma = 0.0;
  if (md.cells > 0) {
    mu = __ddiv_rn((double)(long long)s1u, cells);
    const double var = __dsub_rn(__ddiv_rn((double)(long long)s2u, cells), __dmul_rn(mu, mu));
    sigma = var > 0.0 ? __dsqrt_rn(var) : 0.0;
  }
  if (b == 0 && md.stats) {
    md.stats->sum = (int64_t)s1u;
    md.stats->sum_sq = (int64_t)s2u;
    md.stats->cells = md.cells;
  }
  if (!md.cands) return;
  gfh_candidate c;
  c.band = b;
  c.reserved = 0;
  const unsigned long long key = md.keys[b];
  if (key == 0ull) {
    c.row = -1; c.col = -1; c.count = -1;
    c.cr = 0.0; c.x0 = 0.0; c.k = 0.0; c.f0 = 0.0; c.fdot0 = 0.0;
  } else {
    const int count = (int)(key >> 32);
    const uint32_t lin = 0xffffffffu - (uint32_t)(key & 0xffffffffull);
    const int row = (int)(lin / (uint32_t)md.W);
    const int64_t col = (int64_t)(lin % (uint32_t)md.W);
    c.row = row;
    c.col = col;
    c.count = count;
    c.cr = sigma > 0.0 ? __ddiv_rn(__dsub_rn((double)count, mu), sigma) : 0.0;
    c.x0 = __dadd_rn(md.x0_min, __dmul_rn(__dadd_rn((double)col, 0.5), md.dx0));
    c.k = __dadd_rn(md.k_min, __dmul_rn((double)row, md.dk));
    c.f0 = md.f0c[col];
    c.fdot0 = -__dmul_rn(c.k, md.f0n[col]);
  }
  md.cands[b] = c;
}

// Selection alone on an existing map: one thread per column walks all rows.
__global__ void k_select_cols(const int32_t* __restrict__ map, const MapDev* __restrict__ mdp) {
  const MapDev& md = *mdp;
  const int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  long long s1 = 0, s2 = 0;
  if (m < md.W) {
    const int band = md.col_band[m];
    if (band >= 0) {
      unsigned long long best = 0ull;
      for (int r = 0; r < md.K; ++r) {
        const int v = map[(int64_t)r * md.ld + m];
        s1 += v;
        s2 += (long long)v * v;
        const unsigned long long k = cand_key(v, (uint32_t)r * (uint32_t)md.W + (uint32_t)m);
        best = k > best ? k : best;
      }
      atomicMax(&md.keys[band], best);
    }
  }
  s1 = warp_sum64(s1);
  s2 = warp_sum64(s2);
  if ((threadIdx.x & 31) == 0 && (s1 | s2)) {
    atomicAdd(&md.sums[0], (unsigned long long)s1);
    atomicAdd(&md.sums[1], (unsigned long long)s2);
  }
}

// Sets the shared-memory attribute of the kernels that a plan launches.  Doing so at plan creation
// keeps gfh_plan_execute to stream operations only (capturable).  The attribute belongs to the
// kernel, not to a plan, so it is set to the largest size any plan may request: each launch still
// asks only for its own size (which alone decides occupancy).
template <int R, int NT, bool XD>
int prepare_hough() {
  for (const void* f : {(const void*)k_hough<R, NT, false, XD>, (const void*)k_hough<R, NT, true, XD>}) {
    cudaFuncAttributes fa{};
    GFH_CUDA_TRY(cudaFuncGetAttributes(&fa, f));
    GFH_CUDA_TRY(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)(kMaxSmemBytes - fa.sharedSizeBytes)));
  }
  return GFH_OK;
}

enum { kFull, kFullX, kList };   // full search's two tile lists (XD: the second), coarse tiles

template <int R, int NT, bool XD>
int launch_hough_t(gfh_plan* p, const gfh_peaks* peaks, int which) {
  auto fn = p->select ? k_hough<R, NT, true, XD> : k_hough<R, NT, false, XD>;
  const bool list = which == kList;
  const int n_tiles = XD ? p->n_tiles_x : p->n_tiles;
  if (!list && n_tiles == 0) return GFH_OK;
  const TileDev* const tiles = list ? p->d_sel_tiles : p->d_tiles + (XD ? p->n_tiles : 0);
  const size_t cells = list ? p->cells_list : XD ? p->cells_x : p->cells;
  const size_t head = (size_t)kLane * 4 * (kSpareRows + (XD ? R : 1)) +
                      (p->select ? (size_t)p->max_tile_bands * 8 : 0);
  // head (chunk sums, spare words, band keys), sums, the windows of as many bins as there are
  // threads, or as fit beside the tile without lowering the blocks per SM, the tile
  constexpr size_t kOwn = 1024 + 64;             // reserved per block, and the kernel's static bytes
  const size_t sum_off = (head + 15) / 16 * 16;
  const size_t fixed = sum_off + kSumBytes<NT> + cells;
  const size_t blocks = std::max<size_t>(1, std::min<size_t>(kSmemPerSm / (fixed + 16 + kOwn), 2048 / NT));
  const size_t room = std::min(kSmemPerSm / blocks - kOwn, kMaxSmemBytes - 64);
  if (fixed + 16 > room) return GFH_ERR_SIZE;
  const int batch = (int)std::min<size_t>(NT, (room - fixed) / 16);
  const size_t bytes = fixed + (size_t)batch * 16;
  int per_sm = 0;
  GFH_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, NT, bytes));
  int grid = p->ctx->num_sms * (per_sm > 0 ? per_sm : 1);
  if (!list) grid = std::min(grid, n_tiles);
  fn<<<grid, NT, bytes, p->ctx->stream>>>(
      p->d_maps, tiles, list ? p->sel_cap : n_tiles, list ? p->d_sel_count : nullptr,
      list ? p->d_sel_count + 1 : p->d_next + (XD ? 1 : 0), peaks->fft_idx, p->d_list_state,
      p->ctx->d_flag, (int)sum_off, batch);
  GFH_CUDA_TRY(cudaGetLastError());
  return GFH_OK;
}

// The kernels of a plan: f(rows, threads, XD) as compile-time constants.
template <class F>
int with_kernel(const gfh_plan* p, int which, F f) {
  const std::integral_constant<int, 256> t256{};
  const std::integral_constant<int, 1> any{};
  if (which == kFullX) return f(std::integral_constant<int, kRowsX>{}, t256, std::true_type{});
  if ((which == kList ? p->list_threads : p->threads) == 256) return f(any, t256, std::false_type{});
  return f(any, std::integral_constant<int, 512>{}, std::false_type{});
}

int launch_hough(gfh_plan* p, const gfh_peaks* peaks, int which) {
  return with_kernel(p, which, [&](auto r, auto nt, auto xd) {
    return launch_hough_t<decltype(r)::value, decltype(nt)::value, decltype(xd)::value>(p, peaks, which);
  });
}

// Appends to one compact list the fine tiles of each map's selected coarse tiles, or, for a map
// flagged for a full search, all tiles of the map (group nct of the map).  count[0] = list length.
// The list holds at most cap tiles (enough unless a map lists a coarse tile twice): slots are
// claimed in contiguous ranges, every claimed slot below cap is written, and an overflow sets the
// capacity flag (the list kernel reads min(count, cap) tiles).
__global__ void k_gather_tiles(const TileDev* __restrict__ fine, const int32_t* __restrict__ first,
                               const int32_t* __restrict__ coarse, const int32_t* __restrict__ full,
                               int n_sel, int nct, TileDev* __restrict__ out, int* count, int cap,
                               unsigned int* flag) {
  const int m = blockIdx.y, s = blockIdx.x;
  const bool whole = full && full[m] != 0;
  int id;
  if (whole) id = s == 0 ? nct : -1;                // one block copies the whole map
  else if (s < n_sel) id = coarse[(int64_t)m * n_sel + s];
  else return;
  if (id < 0 || id > nct || (id == nct && !whole)) return;
  const int b = first[(int64_t)m * (nct + 1) + id];
  const int e = first[(int64_t)m * (nct + 1) + id + 1];
  if (e <= b) return;
  __shared__ int base;
  if (threadIdx.x == 0) {
    base = atomicAdd(count, e - b);
    if (base + (e - b) > cap) atomicOr(flag, GFH_FLAG_CAPACITY);
  }
  __syncthreads();
  for (int q = threadIdx.x; q < e - b && base + q < cap; q += blockDim.x) out[base + q] = fine[b + q];
}

}  // namespace

int gfh_prepare_plan(gfh_plan* p) {
  for (int which : {kFull, kFullX, kList}) {
    if (which == kFullX && p->n_tiles_x == 0) continue;
    const int rc = with_kernel(p, which, [&](auto r, auto nt, auto xd) {
      return prepare_hough<decltype(r)::value, decltype(nt)::value, decltype(xd)::value>();
    });
    if (rc) return rc;
  }
  return GFH_OK;
}

// Per-execute preparation shared by the full and the coarse-tile forms: input check, per-map CSR
// over bins, zeroed candidate keys.
static int launch_prologue(gfh_plan* p, const gfh_peaks* peaks) {
  gfh_ctx* ctx = p->ctx;
  cudaStream_t st = ctx->stream;
  if (peaks->n_lists > 65535) return GFH_ERR_CUDA;   // (the lists' states, and other launches, stop there)
  GFH_CUDA_TRY(cudaMemsetAsync(p->d_zeroed, 0, p->zeroed_bytes, st));
  const int check_blocks = 4 * ctx->num_sms;
  k_check_sorted<<<check_blocks, 256, 0, st>>>(peaks->bin, peaks->fft_idx, peaks->offsets, peaks->n_lists,
                                               (1.f + 0x1p-20f) / check_blocks, ctx->d_flag, p->d_list_state,
                                               p->n_list_states);
  GFH_CUDA_TRY(cudaGetLastError());
  k_index<<<(p->csr_entries + kIndexWarps - 1) / kIndexWarps, kIndexWarps * kLane, 0, st>>>(
      p->d_lists, p->d_csr_list, p->csr_entries, peaks->bin, peaks->fft_idx, peaks->offsets, p->d_list_state);
  GFH_CUDA_TRY(cudaGetLastError());
  return GFH_OK;
}

static int launch_epilogue(gfh_plan* p) {
  if (p->select) {
    int maxb = 1;
    for (const gfh_grid& g : p->grids) maxb = g.n_bands > maxb ? g.n_bands : maxb;
    dim3 grid((maxb + 127) / 128, p->n_maps);
    k_finalize<<<grid, 128, 0, p->ctx->stream>>>(p->d_maps);
    GFH_CUDA_TRY(cudaGetLastError());
  }
  return GFH_OK;
}

int gfh_launch_plan(gfh_plan* p, const gfh_peaks* peaks) {
  GFH_CUDA_TRY(cudaSetDevice(p->ctx->device));
  int rc = launch_prologue(p, peaks);
  if (rc) return rc;
  rc = launch_hough(p, peaks, kFull);
  if (!rc && p->n_tiles_x > 0) rc = launch_hough(p, peaks, kFullX);
  if (rc) return rc;
  return launch_epilogue(p);
}

int gfh_launch_plan_tiles(gfh_plan* p, const gfh_peaks* peaks, const int32_t* d_coarse, int n_sel,
                          const int32_t* d_full) {
  GFH_CUDA_TRY(cudaSetDevice(p->ctx->device));
  int rc = launch_prologue(p, peaks);
  if (rc) return rc;
  const int nct = p->coarse_k * p->coarse_x;
  cudaStream_t st = p->ctx->stream;
  const int gx = n_sel > 0 ? n_sel : 1;
  if (n_sel > 0 || d_full) {
    k_gather_tiles<<<dim3(gx, p->n_maps), 128, 0, st>>>(p->d_fine, p->d_coarse_first, d_coarse,
                                                       d_full, n_sel, nct, p->d_sel_tiles,
                                                       p->d_sel_count, p->sel_cap, p->ctx->d_flag);
    GFH_CUDA_TRY(cudaGetLastError());
    rc = launch_hough(p, peaks, kList);
    if (rc) return rc;
  }
  return launch_epilogue(p);
}

extern "C" int gfh_hough(gfh_ctx* ctx, const uint32_t* d_fft_idx, const uint32_t* d_bin,
                         int64_t n_peaks, const gfh_grid* g, int32_t* d_map,
                         gfh_candidate* d_cands, gfh_map_stats* d_stats) {
  if (!ctx || !g || !d_map || n_peaks < 0 || (n_peaks > 0 && (!d_fft_idx || !d_bin)))
    return GFH_ERR_ARG;
  gfh_grid g1 = *g;
  g1.list = 0;
  gfh_plan* p = nullptr;
  int32_t* maps[1] = {d_map};
  gfh_candidate* cands[1] = {d_cands};
  int rc = gfh_make_plan(ctx, 1, &g1, maps, d_cands ? cands : nullptr, d_stats, nullptr, true, &p);
  if (rc) return rc;
  k_set_offsets<<<1, 32, 0, ctx->stream>>>(p->d_offsets_single, n_peaks);
  rc = cudaGetLastError() == cudaSuccess ? GFH_OK : GFH_ERR_CUDA;
  if (!rc) {
    // An empty list still needs valid pointers for the kernels' (never executed) loads.
    gfh_peaks pk{d_fft_idx ? d_fft_idx : (const uint32_t*)p->d_offsets_single,
                 d_bin ? d_bin : (const uint32_t*)p->d_offsets_single, p->d_offsets_single, 1};
    rc = gfh_launch_plan(p, &pk);
  }
  const int rc2 = gfh_plan_destroy(p);
  return rc ? rc : rc2;
}

extern "C" int gfh_select(gfh_ctx* ctx, const int32_t* d_map, const gfh_grid* g,
                          gfh_candidate* d_cands, gfh_map_stats* d_stats) {
  if (!ctx || !d_map || !g) return GFH_ERR_ARG;
  std::vector<int32_t> band;
  std::vector<double> f0, f0n;
  int rc = gfh_host_columns(g, band, f0, f0n);
  if (rc) return rc;
  if ((double)g->n_k * (double)g->n_x0 >= 4294967295.0) return GFH_ERR_SIZE;
  int64_t ana = 0;
  for (int64_t c = 0; c < g->n_x0; ++c) ana += band[c] >= 0;
  GFH_CUDA_TRY(cudaSetDevice(ctx->device));
  const size_t nb = (size_t)g->n_bands;
  const size_t bytes = sizeof(MapDev) + 256 + (nb + 2) * 8 + band.size() * 4 + f0.size() * 16 + 1024;
  char* buf = nullptr;
  if (cudaMalloc(&buf, bytes) != cudaSuccess) return GFH_ERR_NOMEM;
  size_t off = 0;
  auto take = [&](size_t b) { size_t o = off; off = (off + b + 255) / 256 * 256; return o; };
  const size_t o_md = take(sizeof(MapDev)), o_keys = take((nb + 2) * 8),
               o_band = take(band.size() * 4), o_f0 = take(f0.size() * 8),
               o_f0n = take(f0n.size() * 8);
  MapDev md{};
  md.out = nullptr;
  md.col_band = (const int32_t*)(buf + o_band);
  md.f0c = (const double*)(buf + o_f0);
  md.f0n = (const double*)(buf + o_f0n);
  md.keys = (unsigned long long*)(buf + o_keys);
  md.sums = md.keys + nb;
  md.cands = d_cands;
  md.stats = d_stats;
  md.W = g->n_x0;
  md.ld = g->ld_x0;
  md.cells = ana * g->n_k;
  md.x0_min = g->x0_min;
  md.dx0 = g->dx0;
  md.k_min = g->k_min;
  md.dk = g->dk;
  md.K = g->n_k;
  md.n_bands = g->n_bands;
  cudaStream_t st = ctx->stream;
  cudaError_t e = cudaMemcpyAsync(buf + o_md, &md, sizeof(md), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(buf + o_band, band.data(), band.size() * 4, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(buf + o_f0, f0.data(), f0.size() * 8, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(buf + o_f0n, f0n.data(), f0n.size() * 8, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(buf + o_keys, 0, (nb + 2) * 8, st);
  if (e == cudaSuccess) {
    k_select_cols<<<(unsigned)((g->n_x0 + 255) / 256), 256, 0, st>>>(d_map, (const MapDev*)(buf + o_md));
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) {
    dim3 grid((unsigned)((nb + 127) / 128), 1);
    k_finalize<<<grid, 128, 0, st>>>((const MapDev*)(buf + o_md));
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);  // host vectors must outlive the copies
  cudaFree(buf);
  return e == cudaSuccess ? GFH_OK : GFH_ERR_CUDA;
}

// ---- shared-memory atomic throughput (the denominator of the accumulator's roofline) ------------
//
// Every thread adds 1 with atomicAdd to 32-bit shared words, `iters` times, cycling over four words
// of its own (so consecutive atomics of a thread do not wait on one word).  Mode 0: lane l of warp w
// uses words w * 32 + l + 1024 q (one word per bank per warp: conflict-free); mode 1: all lanes of
// a warp use the same word (same-address); mode 2: pseudo-random words of a 32 KB array.  The
// block's elapsed SM cycles go to cycles[block]; the array's sum goes to sink[block] (kept live).
namespace {

template <int MODE>
__global__ void __launch_bounds__(1024) k_smem_atomics(int iters, long long* __restrict__ cycles,
                                                       int* __restrict__ sink) {
  __shared__ int buf[8192];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < 8192; i += blockDim.x) buf[i] = 0;
  __syncthreads();
  int a[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (MODE == 0) a[q] = ((warp * 32 + lane) & 1023) + 1024 * q;
    else if (MODE == 1) a[q] = (warp & 255) * 32 + 1024 * q;
    else a[q] = (int)(gfh_mix64((uint64_t)(blockIdx.x * 1024 + tid) * 4 + q) & 8191u);
  }
  const long long t0 = clock64();
  for (int i = 0; i < iters; i += 4) {
#pragma unroll
    for (int q = 0; q < 4; ++q) atomicAdd(&buf[a[q]], 1);
  }
  __syncthreads();
  const long long t1 = clock64();
  int s = 0;
  for (int i = tid; i < 8192; i += blockDim.x) s += buf[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) atomicAdd(&sink[blockIdx.x], s);
  if (tid == 0) cycles[blockIdx.x] = t1 - t0;
}

}  // namespace

extern "C" int gfh_probe_smem_atomics(gfh_ctx* ctx, int32_t mode, int32_t blocks, int32_t threads,
                                      int32_t iters, long long* d_cycles, int32_t* d_sink) {
  if (!ctx || mode < 0 || mode > 2 || blocks < 1 || threads < 32 || threads > 1024 ||
      threads % 32 || iters < 4 || iters % 4 || !d_cycles || !d_sink)
    return GFH_ERR_ARG;
  GFH_CUDA_TRY(cudaSetDevice(ctx->device));
  if (mode == 0) k_smem_atomics<0><<<blocks, threads, 0, ctx->stream>>>(iters, d_cycles, d_sink);
  if (mode == 1) k_smem_atomics<1><<<blocks, threads, 0, ctx->stream>>>(iters, d_cycles, d_sink);
  if (mode == 2) k_smem_atomics<2><<<blocks, threads, 0, ctx->stream>>>(iters, d_cycles, d_sink);
  GFH_CUDA_TRY(cudaGetLastError());
  return GFH_OK;
}

extern "C" int gfh_device_sms(gfh_ctx* ctx, int32_t* h_sms) {
  if (!ctx || !h_sms) return GFH_ERR_ARG;
  *h_sms = ctx->num_sms;
  return GFH_OK;
}
