// tcw_step.cuh -- shared declarations of the step-function search kernel
// (tcw_step.cu): the exhaustive search of one or many events.
//
// Over the skies of a chunk, sorted by their Doppler factor, the bin of one
// (template, segment, detector) lookup is a step function: it changes only
// where the threshold between two bins (tcw_internal.cuh) falls between two
// neighbouring skies, one or two places for the whole sky at 500-3000 Hz.  So
// a lookup is the first sky's bin plus one difference per step, added to a
// per-template difference array over the sorted positions; a prefix sum at the
// end gives every sky's weighted power.  All sums are fixed-point integers
// (48 bits, two 32-bit words), so they are exact and do not depend on the order
// of the additions or on how the sky and the bank are cut into work items.
#pragma once

#include <cmath>

#include "tcw_internal.cuh"

namespace tcw {

constexpr int kStepBlock = 8;          // sorted skies per block of a Doppler row
constexpr int kStepMaxChunk = 1024;    // sorted skies per chunk
constexpr int kStepCells = 16384;      // difference cells of a CTA: chunk x templates

// One event.  Its segments and detectors are worked through in passes: a pass
// is a run of pass_seg segments of one detector (dets_per_pass = 1) or of all
// of them, over which the skies of a chunk keep one order, so that the rows'
// Doppler factors stay (almost) sorted.  Doppler rows: one per (chunk, segment,
// detector), cpad skies in the order of their pass (a multiple of kStepBlock;
// the last sky repeated):
//   q     [cpad]  floor(v.nhat/c / q-grid step)
//   head  {qmin, qmax, buckets per grid unit (32 fraction bits), w (float bits)}: the
//         smallest and largest q; {dt hi, dt lo, dt^2 hi, dt^2 lo}: t_j - t_a from
//         the tile's anchor time and its square as fp32 pairs (dt hi NaN before T0)
//   wfix  {W1 word, W2 word}: w and w^2 in fixed point (int64 each)
//   tab   per bucket of thresholds {first position not below all of them, first
//         position from which on every sky reaches all of them}, 11 bits each:
//         only the skies between the two are compared with a threshold
//   fast  the same in one load: {first position, a flag for windows of more than 3
//         skies or out of order, place of the first sky; places of the second and
//         third}, places in 2^-14 buckets from the start of the bucket before on
// Track constants of one (template, tile), the position x = (f - f_min)/df of
// the unshifted track (Eq. 1) around the anchor time t_a: x = base + frac +
// A dt + Q dt^2 + X (cubic and higher terms in dt s).
struct __align__(16) StepTile {
  int base;
  float frac, A_hi, A_lo, Q_hi, Q_lo;
  float X;   // f_a / df
  float s;   // 1 / (tau + t_a - T0)
};
static_assert(sizeof(StepTile) == 32, "two 16-byte loads");

struct StepEvent {
  const void* rho;           // [D][n_seg][n_bin]
  const uint32_t* bits;      // number count: bit map (see EventDesc), else null
  const double* t_mid;
  const double* anchors;     // [Bpad][n_tiles][2] (exact thresholds)
  const StepTile* tiles;     // [Bpad][n_tiles]
  const double* f0;          // sorted bank [Bpad]
  const double* nbr;
  const int32_t* q;          // [n_chunks][n_seg][D][cpad]
  const int4* head;          // [n_chunks][n_seg][D][kStepHead]
  const uint32_t* tab;       // [n_chunks][n_seg][D][step_buckets(cpad)]
  const uint2* fast;         // [n_chunks][n_seg][D][step_buckets(cpad)]
  const longlong2* wfix;     // [n_seg][D]
  const long long* wtot;     // [kStepSlots][2]: partial sums of w and w^2 over the segments from T0 on
  const int16_t* order;      // [passes][n_chunks][cpad] sky (in the chunk) at a position; null for one pass
                             // in the sorted order itself
  const int16_t* remap;      // [passes][n_chunks][cpad] that sky's position in the pass before
  float* psi;                // [>= S][Bpad]
  float* S_out;              // optional
  float* W1_out;
  float* W2_out;
  double T0;
  double x_unit, w1_unit, w2_unit;   // value of one unit of the fixed-point sums
  float x_scale;                     // 2^-16 / x_unit
  float r_unit;                      // 2^24 x_unit / sqrt(w2_unit), a power of 2
  float w1_scale, w2_scale;          // 2^-22 / w1_unit, 2^-22 / w2_unit
  int n_seg, n_tiles, S, Bpad;
  int bit_pitch;
  int chunk, cpad, log_t;    // skies per chunk, of a row; templates of a block: 1 << log_t
  int n_chunks, pass_seg, passes;
  int sub_shift;             // segments of one warp's turn: 1 << sub_shift <= 16 and <= tile
};

struct StepParams {
  const StepEvent* events;
  const int4* items;         // {event, chunk, first template, template blocks}; null: every chunk of
                             // event 0 x runs of bank_chunk template blocks
  int n_items, n_chunks, bank_chunk;
  int n_det;
  unsigned* next;            // item counter, zero at launch
  int64_t n_bin;
  double f_min, df, inv_q;
  float q, inv_q_f;
  float eps;                 // bound of the fp32 thresholds' error, in bins
  int nterms, tile_shift;    // FP64 track series (> 0), anchor tiles
  float x_min_i, x_min_f;    // f_min / df: whole bins, fraction
  int amp_power;
  double nc_q;               // number count: q = exp(-rho_th), else 0
  int track_bins;
  int map_half;
  int4* slow;                // [grid][step_slow_bytes(1)]: the warps' lists of steps left for later
  longlong2* edge;           // [grid][2 kStepCells + 32]: W1, W2 steps at band edges (zero between
                             // launches), and room to reorder them
  unsigned long long* n_general;
};

struct StepRowsParams {
  const double* vel;         // [D][n_seg][3]
  const double* nhat;        // [>= S][3] sorted
  const float* weights;      // [D][n_seg]
  const double* t_mid;
  double T0;
  int n_det, n_seg, S, chunk, cpad, n_chunks, tile_shift;
  int dets_per_pass, pass_seg, passes;
  double inv_q;
  int eps_max;               // largest error of an fp32 threshold, in grid units
  double w1_scale, w2_scale; // 1 / w1_unit, 1 / w2_unit
  int16_t* order;            // written first when not null, with remap (see StepEvent)
  int16_t* remap;
  int32_t* q;
  int4* head;
  uint32_t* tab;
  uint2* fast;
  longlong2* wfix;
  unsigned long long* wtot;  // zero at launch
};

constexpr int kStepHead = 2;     // int4 words of a row's head
constexpr int kStepSlots = 64;   // partial weight sums of an event
// Two buckets of thresholds per sky: about half a sky is left to compare per threshold.
__host__ __device__ constexpr int step_buckets(int cpad) { return 2 * cpad; }

// Chunks of an event's sorted skies: the fewest chunks of at most
// kStepMaxChunk skies, of nearly equal size; 32 templates per block while the
// difference cells allow it (chunks of up to 512 skies), else 16 (see step_block).
struct StepGeometry {
  int n_chunks, chunk, cpad, log_t;
  int dets_per_pass, pass_seg, passes;
};
// v: velocities [D][n_seg][3] (host); split: one detector per pass even where all would do.
StepGeometry step_geometry(int64_t S, int D, int64_t n_seg, int tile, const double* v, bool split);
inline void set_step_geometry(StepEvent& e, const StepGeometry& g) {
  e.chunk = g.chunk;
  e.cpad = g.cpad;
  e.log_t = g.log_t;
  e.n_chunks = g.n_chunks;
  e.pass_seg = g.pass_seg;
  e.passes = g.passes;
}
inline void set_step_geometry(StepRowsParams& p, const StepGeometry& g) {
  p.chunk = g.chunk;
  p.cpad = g.cpad;
  p.n_chunks = g.n_chunks;
  p.dets_per_pass = g.dets_per_pass;
  p.pass_seg = g.pass_seg;
  p.passes = g.passes;
}
inline bool step_ordered(const StepGeometry& g) { return g.passes > 1; }
// Doppler rows of one chunk, in bytes: about 28 per sky of a (segment, detector).
inline size_t step_chunk_bytes(const StepGeometry& g, int64_t n_seg, int D) {
  return (size_t)n_seg * D *
         (g.cpad * sizeof(int32_t) + kStepHead * sizeof(int4) +
          step_buckets(g.cpad) * (sizeof(uint2) + sizeof(uint32_t)));
}
// Rows held at a time: a longer sky list is searched some chunks at a time (a chunk
// fills the chip for milliseconds).
constexpr size_t kStepRowsMax = (size_t)4 << 30;

// The fp32 track's tiles and error bound: tile = 1 << shift segments (at most
// `most`: twice the anchor tiles of the other kernels, as a tile here is laid out
// in FP64 and read once, so that fewer are better: 64 for 32 segments takes a
// search with one sky from 22.6 to 19.4 ms), the FP64 series' terms, and the thresholds' error; ok = false when no
// tile keeps it.  x_max: largest f/df of the bank; x_top: f/df at the top of the
// band; db: largest Doppler shift in bins.
struct StepTrack {
  bool ok = false;
  int shift = 0, nterms = 0;
  float eps = 0;             // bins
  int eps_max = 0;           // in grid units
};
StepTrack step_track(const double* t_mid, int64_t n_seg, double T0, int most, double tau_min, double r_max,
                     double x_max, double x_top, double db, double f_min, double df, double inv_q);
// p.f_min and p.df are set.
inline void set_step_track(StepParams& p, const StepTrack& t) {
  const double x = p.f_min / p.df, i = std::nearbyint(x);
  p.x_min_i = (float)i;      // below 2^23 where the track is ok
  p.x_min_f = (float)(x - i);
  p.eps = t.eps;
  p.nterms = t.nterms;
  p.tile_shift = t.shift;
}

// Tile anchors and track constants of one event for every sorted template.
struct StepTileParams {
  AnchorParams a;            // as for launch_anchors
  double f_min, df;
  StepTile* tiles;
};
cudaError_t launch_step_tiles(const StepTileParams& p, cudaStream_t st);

// What the fixed-point sums are scaled by.  A map's largest |rho|, and its level: the
// smallest maximum of |rho| over its runs of kLevelRun bins (0: every bin is 0), about
// the mean power of the quietest stretch (0.95 for noise of mean 1 over 2e8 bins; runs
// of 4 would give 0.01).  Runs of zeros don't count, and those at their edges, with
// fewer than half of the bins nonzero, only where they are more than 1 in 16.
constexpr int kLevelRun = 32;
constexpr int kMapWords = 5;   // words that launch_map_range writes
struct MapRange {
  float max = 0, level = 0;
};
MapRange map_range(const unsigned* out);   // from launch_map_range's words
// The segments' weights: smallest nonzero one, largest one, sum.
struct WeightRange {
  float min = INFINITY, max = 0;
  double sum = 0;
  void take(const std::vector<float>& w) {
    for (float x : w) {
      if (x > 0 && x < min) min = x;
      if (x > max) max = x;
      sum += x;
    }
  }
};

// Fixed-point scales of one event, or ok = false when the sums would not be
// at least as accurate as fp32 partial sums (see step_scales).
struct StepScales {
  bool ok = false;
  int x = 0, w1 = 0, w2 = 0;   // exponents: one unit is 2^-x (2^-w1, 2^-w2)
};
// bins: powers that a lookup adds; amp: amplitude weights, a_ref: their factor at a
// template's first lookups.
StepScales step_scales(const MapRange& map, int bins, const WeightRange& w, bool amp, double a_ref);

inline void set_step_scales(StepEvent& e, const StepScales& s) {
  e.x_unit = std::ldexp(1.0, -s.x);
  e.w1_unit = std::ldexp(1.0, -s.w1);
  e.w2_unit = std::ldexp(1.0, -s.w2);
  e.x_scale = std::ldexp(1.0f, s.x - 16);
  e.r_unit = std::ldexp(1.0f, 24 - s.x + s.w2 / 2);
  e.w1_scale = std::ldexp(1.0f, s.w1 - 22);
  e.w2_scale = std::ldexp(1.0f, s.w2 - 22);
}
// Segments of one warp's turn (as a shift): the longest run, a whole tile or
// less, that leaves few of the 32 warps idle in a pass's last round of turns.
inline int step_sub_shift(const StepGeometry& g, int64_t n_seg, int tile_shift) {
  const int64_t len = n_seg < g.pass_seg ? n_seg : g.pass_seg;
  int best = tile_shift < 3 ? tile_shift : 3;
  double best_busy = 0;
  for (int s = tile_shift < 4 ? tile_shift : 4; s >= 3; --s) {
    const double turns = (double)((len + (1 << s) - 1) >> s), busy = turns / (std::ceil(turns / 32.0) * 32.0);
    if (busy > best_busy + 0.05) {
      best = s;
      best_busy = busy;
    }
  }
  return best;
}
// Templates of a block (as log2) for a bank whose blocks may not fill the chip:
// blocks of 16 or 4 when their rounds over `grid` CTAs end sooner than those of
// the largest block that fits (bank_chunk blocks are one item).  A (template, row) takes 2.8 ns of a CTA in
// blocks of 32 and 3.9 in blocks of 16 (128 skies, where 626 of 32 in 5 rounds
// take 9.0 ms and 1251 of 16 in 9 rounds 11.0), about twice as much in blocks of
// 4 (the tables' rows serve fewer templates), and a pass's end some 20 us.
// 301 templates x 12 skies x 4002 rows: 10 blocks of 32, 511 us; 76 of 4, 322.
int step_block(const StepGeometry& g, int Bpad, int bank_chunk, int grid, double rows);
inline int step_cells(const StepGeometry& g) { return (g.cpad + 1) << g.log_t; }
size_t step_slow_bytes(int grid);
inline size_t step_edge_bytes(int grid) { return (size_t)grid * (2 * kStepCells + 32) * sizeof(longlong2); }
cudaError_t launch_step_rows(const StepRowsParams& p, cudaStream_t st);
// A form of the search kernel: detectors of a pass, templates of a block (log2), an
// FP16 map, number count or two-bin lookups (general), amplitude weights.
struct StepForm {
  int dets_per_pass, log_t;
  bool half, general, amp;
};
// Raises the kernel's shared-memory limit (also done at its first launch; call before a graph capture).
cudaError_t step_prepare(const StepForm& v);
// cells: the largest step_cells of the items' events, which are all of this form.
cudaError_t launch_step(const StepParams& p, const StepForm& v, int cells, int grid, cudaStream_t st);
// out[kMapWords] as map_range reads it; zero at launch.
cudaError_t launch_map_range(const void* rho, bool half, int64_t n, unsigned* out, cudaStream_t st);

}  // namespace tcw
