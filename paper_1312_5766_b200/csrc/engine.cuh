// Whole rounds in one cooperative launch (engine.cu): what the kernel keeps between rounds, and its launchers.
#pragma once
#include "strads_internal.cuh"

namespace strads {

// Device-resident state of the round engine, in the workspace.  Zero before the first launch.
struct EngineState {
  unsigned int bar_count;       // grid barrier: arrivals of the launch in flight
  unsigned int draw_bar_count;  // ... of the threads that draw while others walk
  unsigned int exit_count;      // CTAs of the launch that have left
  float t_cut;                  // draw: cutoff for the next scan (0: none)
  unsigned int amb_count[2];    // dense Gram: pairs the screen left open (two counters, in turns)
  unsigned int edge_count;      // CSC Gram: conflicting pairs listed
  int bucket_failed;            // CSC Gram: a bucket or a candidate's list of terms overflowed in this round
  int skip_window;              // the last whole-list walk shows that the window would have been too short again
  int n_kept, n_examined;       // result of the walk
  int walk_open;                // the walk could not finish: fewer than P kept inside a window, or chains too long
  int mend;                     // a draw's selection has to be mended
  int streak;                   // CSC: attempts with the row buckets in a row that overflowed (or left the walk open)
  int avoid;                    // CSC: rounds until they are tried again
  // rounds prepared by squads of CTAs (squads.cu): the round whose turn it is, and (in the first squad's) the turns
  unsigned int turn_moving;     // kept coefficients that move
  unsigned long long turn_dmax; // bits of the largest |change|
  unsigned int turn_count;      // arrivals: one per CTA of the launch at its start, then one per CTA of a squad whose turn is over
  unsigned int turn_exit;       // CTAs of the launch that have left
  int dirty;                    // strads_sample_static: the last call gave up and left the histogram as it was
};

// The coefficients that a scheduler draws from.
__host__ __device__ inline long long owned_count(const Problem& p) { return (p.J - p.part_index + p.part_count - 1) / p.part_count; }

// How the pairs of a list are cut into tiles of the dense Gram: kGramRows x cols, K in stages of 64 elements, `split` CTAs sharing a tile with `per` stages each.
constexpr int kGramRows = 128;
struct GramPlan { int cols, col_blocks, tiles, split, steps, per; };
__host__ __device__ inline GramPlan gram_plan(long long N, int n, int n_ctas) {
  GramPlan best = {};
  float cost = 0.f;
  const int k = 64;
  const int row_blocks = (n + kGramRows - 1) / kGramRows, steps = (int)((N + k - 1) / k);
  for (int cols = 64; cols <= 128; cols += 64) {
    GramPlan pl;
    const int per_row = kGramRows / cols;
    pl.cols = cols;
    pl.col_blocks = (n + cols - 1) / cols;
    // row block i meets the column blocks that start before its end
    pl.tiles = 0;
    for (int i = 1; i <= row_blocks; ++i) pl.tiles += i * per_row < pl.col_blocks ? i * per_row : pl.col_blocks;
    pl.steps = steps;
    pl.split = n_ctas / pl.tiles;
    if (pl.split > 16) pl.split = 16;
    if (pl.split > steps) pl.split = steps;
    if (pl.split < 1) pl.split = 1;
    pl.per = (steps + pl.split - 1) / pl.split;
    pl.split = (steps + pl.per - 1) / pl.per;             // (no part without a stage)
    const int waves = (pl.tiles * pl.split + n_ctas - 1) / n_ctas;
    // microseconds: 0.35 (64 columns) or 0.45 (128) a stage, and what sharing a tile costs
    const float c = (float)waves * ((float)pl.per * (cols == 64 ? 0.35f : 0.45f) + (pl.split > 1 ? (cols == 64 ? 2.5f : 3.f) : 0.5f));
    if (cols == 64 || c < cost) { cost = c; best = pl; }
  }
  return best;
}

// What a launch needs beside the Problem.
struct Engine {
  EngineState* es;
  unsigned int* hist;           // [kHistBins] zero between scans
  unsigned int* bin_cur;        // [kHistBins] append cursors of the winners' groups
  unsigned long long* win;      // [cap_win] the winners of a draw, grouped by bin
  int cap_win, cap_boundary;
  unsigned long long* surv;     // [ctas][cap_surv] keys below the scan's cutoff, and how many each CTA saved
  unsigned int* saved;          // [ctas]
  unsigned int cap_surv;
  int n_list;                   // winners a draw made one round ahead collects: P' + P (at most J); 0: draws are made at the round's start
  int window;                   // candidates of the first attempt
  // dense
  unsigned short* xb;           // [n_cand][xb_pitch] BF16 high parts of the candidate columns, then (at lo_off) the low parts
  long long xb_pitch, lo_off;   // elements
  double* norm;                 // [n_cand] dense: norms of the candidates' columns as the rho test sees them
  float* norm_f;                // [n_cand] CSC: their squares, rounded
  float* part;                  // [ctas][128 * 128] partial Gram tiles
  unsigned int* tile_ticket;    // [tiles of 64 x 64] zero between rounds
  GramPlan plan[2];             // for the window and for the whole list
  int grid;                     // CTAs of the launch
};


cudaError_t prepare_engine(const Problem& p, Engine& e);     // grid and plans (window and n_list are set)
size_t engine_smem(const Problem& p, bool ahead);
// n_rounds rounds; have_list: this round's candidates are in p.cand; draw_next: leave the next round's there.
// out (device pointers or null): the last round's candidates, kept list, changes and counts.
// Tensor maps over the BF16 copies (dense; two of 128 bytes, 64-byte aligned).
cudaError_t encode_engine_maps(const Problem& p, const Engine& e, void* out_256_bytes);
cudaError_t launch_engine(const Problem& p, const Engine& e, const void* maps, int n_rounds, bool have_list, bool draw_next,
                          const strads_round_out_t* out, cudaStream_t s);

// The draw of p (as launch_sample's) in one launch of a thread-block cluster of e.grid CTAs; e: es, hist (zero before and after), bin_cur, win,
// surv, saved.  *ctas: its size on the current device (0: none).
cudaError_t prepare_draw_cluster(int* ctas);
cudaError_t launch_draw_cluster(const Problem& p, const Engine& e, int* cand_out, cudaStream_t s);

// CSC rounds whose blocks do not wait for one another's updates: several schedulers, or the static schedule.  As many squads of CTAs as
// there are blocks under way; problem i / engine i: the i-th squad's, which takes the rounds t with t mod n == i.
constexpr int kMaxSquads = STRADS_MAX_SCHEDULERS;
struct SquadSet {
  Problem p[kMaxSquads];
  Engine e[kMaxSquads];
  int n, size;                  // squads, CTAs of each
};
cudaError_t prepare_squads();
// have_list: every squad's list for its next round is in place; draw_next: leave them so.
cudaError_t launch_squads(const SquadSet& set, int n_rounds, bool have_list, bool draw_next, cudaStream_t s);

// The draw alone: p.cand[0 .. p.n_cand) for round t from p.delta (e: es, hist, bin_cur and win).  The barrier in es is zero before
// and after, and hist unless es->dirty says otherwise.
cudaError_t prepare_draw();
cudaError_t launch_draw(const Problem& p, const Engine& e, unsigned long long t, cudaStream_t s);

}  // namespace strads
