// CSC rounds whose blocks (the kept list of a round) do not depend on the updates of the rounds just before them, in one
// cooperative launch: with S scheduler threads taking turns (Section 3) a scheduler's block of round t depends on updates up to
// round t - S only, as nobody else changes its coefficients' priorities; under the static schedule (equal weights, the rho test on X
// alone) no block depends on any update.
//
// The CTAs form squads, one per scheduler (or per block under way), and a squad makes rounds as engine.cu does with all CTAs --
// draw ahead, row buckets, inner products, walk -- with barriers of its own.  Only the update waits for its turn: the squads pass it on
// in the order of rounds.  So a round costs the longer of a block divided by the number of squads, and an update.  What bounds an update is its chain of
// hand-overs (turn, two barriers of the squad) with one far access or two between them, so that the squad brings its kept columns into
// shared memory while it waits, and everything that others need not wait for is done behind its turn.
//
// The steps are those of the rounds launched one by one, in the same order: same bits.
#include "engine_csc.cuh"

namespace strads {
namespace {

// The update of a squad's round in its turn: x_a^T r of the kept coefficients, their changes, beta, delta and the residual.
// A warp has the kept coefficients warp * size + rank + k * (warps of the squad), 32 of them at a time; the columns of the first 32
// wait in shared memory as far as there is room.
constexpr int kHeldEntries = 512;
struct HeldEntries { int row[kHeldEntries]; float val[kHeldEntries]; };      // a warp's
constexpr size_t kHeldSmem = sizeof(HeldEntries) * kWarps;
// Shared memory of a round's update and of what follows it.
__host__ __device__ inline size_t squad_smem(const Problem& p, bool ahead) {
  const size_t changes = (ahead ? 2 * sizeof(unsigned long long) * (size_t)p.n_keep : 0) + sizeof(ChangedByBin);
  return changes > kHeldSmem ? changes : kHeldSmem;
}

struct Turn {
  unsigned int* count;
  unsigned int target, n, limit;
  unsigned int* status;
};
// Until the update before is over.  False: it gave up.
__device__ bool await_turn(const Turn& turn) {
  __shared__ int s_ok;
  if (threadIdx.x == 0) {
    Grid g;
    g.count = turn.count; g.target = turn.target; g.n = turn.n; g.limit = turn.limit; g.status = turn.status;
    s_ok = grid_wait(g, true);
  }
  __syncthreads();
  return s_ok != 0;
}
__device__ __forceinline__ void pass_turn(const Turn& turn) {
  __syncthreads();
  if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(turn.count) : "memory");
}

// A warp's kept coefficients: lane k has the k-th.
struct Held {
  int n;                                   // kept coefficients of the warp, of which 32 at a time
  int a, pos, j, len, at;                  // place in the kept list and among the candidates, coefficient, entries, where they wait (-1: in X)
  long long q0;
};
// kept_at: their positions where they are in shared memory (else null).  ranked: the next candidates may be in the place of these.
__device__ __forceinline__ Held hold(const Squad& crew, const Problem& p, int nk, const unsigned short* kept_at, int chunk, HeldEntries* entry, bool ranked) {
  const int lane = threadIdx.x & 31, warp = (int)threadIdx.x >> 5;
  const int first = warp * crew.size() + crew.rank(), step = kWarps * crew.size();
  Held h;
  h.n = nk > first ? (nk - first + step - 1) / step : 0;
  const bool on = chunk * 32 + lane < h.n;
  h.a = first + (chunk * 32 + lane) * step; h.pos = 0; h.j = 0; h.len = 0; h.q0 = 0; h.at = -1;
  if (on) {
    h.pos = kept_at != nullptr ? (int)kept_at[h.a] : p.kept_pos[h.a];
    if (ranked) {
      h.j = p.kept[h.a]; h.q0 = p.xptr[h.j]; h.len = (int)(p.xptr[h.j + 1] - h.q0);
    } else {
      const WalkColumn col = p.walk_cols[h.pos];
      h.j = col.j; h.len = max(col.n, 0); h.q0 = col.q0;
      if (kept_at != nullptr) { p.kept[h.a] = h.j; p.kept_pos[h.a] = h.pos; }
    }
  }
  if (entry == nullptr) return h;
  int incl = h.len;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += v;
  }
  if (on && incl <= kHeldEntries) h.at = incl - h.len;
  const int m = min(32, h.n);
#pragma unroll 1
  for (int k = 0; k < m; ++k) {
    const int at = __shfl_sync(kFull, h.at, k), len = __shfl_sync(kFull, h.len, k);
    const long long q0 = __shfl_sync(kFull, h.q0, k);
    if (at < 0) continue;
    for (int q = lane; q < len; q += 32) {
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(&entry->row[at + q])), "l"(p.xrow + q0 + q) : "memory");
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(&entry->val[at + q])), "l"(p.xv + q0 + q) : "memory");
    }
  }
  return h;
}
// f(k, row, value) for the entries of the warp's columns for which want(k): whole warps, lanes side by side.
template <typename W, typename F>
__device__ __forceinline__ void for_held(const Problem& p, const Held& h, int chunk, const HeldEntries* entry, W&& want, F&& f) {
  const int lane = threadIdx.x & 31, m = min(32, h.n - chunk * 32);
#pragma unroll 1
  for (int k = 0; k < m; ++k) {
    const int at = __shfl_sync(kFull, h.at, k), len = __shfl_sync(kFull, h.len, k);
    const long long q0 = __shfl_sync(kFull, h.q0, k);
    if (!want(k)) continue;
    for (int q = lane; q < len; q += 32) {
      if (at >= 0) f(k, entry->row[at + q], entry->val[at + q]);
      else f(k, __ldg(p.xrow + q0 + q), __ldg(p.xv + q0 + q));
    }
  }
}

// False: a wait gave up.
// own: the walk was this CTA's own (kept_at, and notes to be made), else null.
__device__ __forceinline__ bool squad_update(const Squad& crew, const Problem& p, const Engine& e, unsigned char* sm, Grid& g, const Turn& turn, const Settled* own,
                                             const unsigned short* kept_at, unsigned long long t_next, bool want_keys) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  HeldEntries* entry = reinterpret_cast<HeldEntries*>(sm) + warp;
  EngineState* es = e.es;
  __syncthreads();                                       // (what lay there before)
  const int nk = own != nullptr ? own->kept : es->n_kept, examined = own != nullptr ? own->examined : es->n_examined;
  const Held h = hold(crew, p, nk, kept_at, 0, entry, false);
  double n2 = 0.0;
  float E = 0.f;
  const bool on0 = lane < h.n;
  if (on0) {
    n2 = p.n2[h.j];
    if (want_keys) E = exponential_of(p, t_next, (uint32_t)h.j);
  }
  const float x_max = p.st->x_abs_max;
  asm volatile("cp.async.wait_all;" ::: "memory");
  if (!await_turn(turn)) return false;                   // (a barrier of the CTA in it)
  // ---- x_a^T r and the changes ----
  double d0 = 0.0;                                       // of the lane's kept coefficient (the first 32 of the warp)
  unsigned long long dmax = 0ull;
  int moving = 0;
#pragma unroll 1
  for (int chunk = 0; chunk * 32 < h.n; ++chunk) {
    Held c = h;
    if (chunk > 0) c = hold(crew, p, nk, kept_at, chunk, nullptr, false);
    const bool on = chunk * 32 + lane < h.n;
    const int m = min(32, h.n - chunk * 32);
    float b_old = 0.f, d_old = 0.f;
    if (on) {
      b_old = p.beta[c.j]; d_old = p.delta[c.j];
      if (chunk > 0) {
        n2 = p.n2[c.j];
        if (want_keys) E = exponential_of(p, t_next, (uint32_t)c.j);
      }
    }
    double dot = 0.0;
    constexpr int kU = 4;                                // columns at a time
#pragma unroll 1
    for (int k0 = 0; k0 < m; k0 += kU) {
      int at[kU], len[kU], most = 0;
      long long q0[kU];
      double acc[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        at[u] = __shfl_sync(kFull, c.at, (k0 + u) & 31); len[u] = __shfl_sync(kFull, c.len, (k0 + u) & 31); q0[u] = __shfl_sync(kFull, c.q0, (k0 + u) & 31);
        if (k0 + u >= m) len[u] = 0;
        most = max(most, len[u]);
        acc[u] = 0.0;
      }
#pragma unroll 1
      for (int q = lane; q - lane < most; q += 64) {
        float v[kU][2], r[kU][2];
#pragma unroll
        for (int u = 0; u < kU; ++u)
#pragma unroll
          for (int y = 0; y < 2; ++y) {
            v[u][y] = 0.f; r[u][y] = 0.f;
            if (q + 32 * y < len[u]) {
              const int i = q + 32 * y;
              v[u][y] = at[u] >= 0 ? entry->val[at[u] + i] : __ldg(p.xv + q0[u] + i);
              r[u][y] = p.resid[at[u] >= 0 ? entry->row[at[u] + i] : __ldg(p.xrow + q0[u] + i)];
            }
          }
#pragma unroll
        for (int u = 0; u < kU; ++u)
#pragma unroll
          for (int y = 0; y < 2; ++y)
            if (q + 32 * y < len[u]) acc[u] += (double)v[u][y] * (double)r[u][y];
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        if (k0 + u >= m) break;
        const double s = warp_sum(acc[u]);
        if (lane == k0 + u) dot = s;
      }
    }
    if (on) {
      const Proposal q = propose_begin(p, c.j, n2, b_old, d_old, E, want_keys);
      const Change ch = propose_end(p, q, c.pos, c.j, dot, E, want_keys);
      p.beta[c.j] = ch.b_new;
      if (!want_keys) p.delta[c.j] = (float)fabs(ch.d);  // (else the draw may want it as it was: commit_deltas)
      p.dbeta[c.a] = (float)ch.d;
      if (!isfinite(ch.d)) atomicOr(&p.st->status, STRADS_STATUS_NONFINITE);
      moving += ch.d != 0.0;
      dmax = max(dmax, (unsigned long long)__double_as_longlong(fabs(ch.d)));
      if (chunk == 0) d0 = ch.d;
    }
    __syncwarp();
  }
  if (h.n > 0) {
    const unsigned int hi = (unsigned int)(dmax >> 32), most = __reduce_max_sync(kFull, hi);
    const unsigned int low = __reduce_max_sync(kFull, hi == most ? (unsigned int)dmax : 0u);
    moving = __reduce_add_sync(kFull, moving);
    if (lane == 0 && moving > 0) {
      atomicMax(&es->turn_dmax, ((unsigned long long)most << 32) | low);
      atomicAdd(&es->turn_moving, (unsigned)moving);
    }
  }
  if (!grid_sync(g)) return false;
  if (own != nullptr && crew.rank() == 0 && tid == 0) settle_note(e, *own);
  // ---- the residual: sums in fixed point (engine_csc.cuh), then every row once ----
  const unsigned long long largest = __ldcg(&es->turn_dmax);
  const int n_moving = (int)__ldcg(&es->turn_moving);
  const int shift = csc_shift(x_max, largest, nk);
  auto change_of = [&](const Held& c, int chunk) { return chunk == 0 ? d0 : (chunk * 32 + lane < h.n ? p.cand_dbeta64[c.pos] : 0.0); };
  if (shift != INT_MIN) {
#pragma unroll 1
    for (int chunk = 0; chunk * 32 < h.n; ++chunk) {
      Held c = h;
      if (chunk > 0) c = hold(crew, p, nk, kept_at, chunk, nullptr, false);
      const double d_lane = change_of(c, chunk);
      double d = 0.0;
      for_held(p, c, chunk, entry, [&](int k) { d = __shfl_sync(kFull, d_lane, k); return d != 0.0; }, [&](int, int row, float v) {
        const long long fx = __double2ll_rn(ldexp((double)v * d, shift));
        atomicAdd(reinterpret_cast<unsigned long long*>(p.resid_acc + row), (unsigned long long)fx);
      });
    }
  }
  if (!grid_sync(g)) return false;
  if (shift != INT_MIN) {
    // few moving entries against the rows: visit the entries' rows (the first visitor of a row takes its sum), else all rows
    if ((double)n_moving * (double)p.nnz * 4.0 < (double)p.N * (double)p.J) {
#pragma unroll 1
      for (int chunk = 0; chunk * 32 < h.n; ++chunk) {
        Held c = h;
        if (chunk > 0) c = hold(crew, p, nk, kept_at, chunk, nullptr, true);
        const double d_lane = change_of(c, chunk);
        const int m = min(32, h.n - chunk * 32);
        constexpr int kU = 4;                            // columns at a time
#pragma unroll 1
        for (int k0 = 0; k0 < m; k0 += kU) {
          int at[kU], len[kU], most = 0;
          long long q0[kU];
#pragma unroll
          for (int u = 0; u < kU; ++u) {
            const int k = (k0 + u) & 31;
            at[u] = __shfl_sync(kFull, c.at, k); q0[u] = __shfl_sync(kFull, c.q0, k);
            len[u] = k0 + u < m && __shfl_sync(kFull, d_lane, k) != 0.0 ? __shfl_sync(kFull, c.len, k) : 0;
            most = max(most, len[u]);
          }
#pragma unroll 1
          for (int q = lane; q - lane < most; q += 32) {
            long long row[kU], v[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
              row[u] = 0; v[u] = 0;
              if (q < len[u]) row[u] = at[u] >= 0 ? entry->row[at[u] + q] : __ldg(p.xrow + q0[u] + q);
              if (q < len[u]) v[u] = (long long)atomicExch(reinterpret_cast<unsigned long long*>(p.resid_acc + row[u]), 0ull);
            }
            apply_sums<kU>(p, row, v, shift);
          }
        }
      }
    } else {
      csc_apply_rows(crew, p, shift);
    }
  }
  if (crew.rank() == 0 && tid == 0) {
    DeviceState* st = p.st;
    st->counts[0] = p.n_cand; st->counts[1] = examined; st->counts[2] = nk; st->counts[3] = n_moving;
    st->totals[0] += 1; st->totals[1] += (unsigned)examined; st->totals[2] += (unsigned)nk; st->totals[3] += (unsigned)n_moving;
    st->round += (unsigned long long)p.part_count;
    es->turn_dmax = 0ull; es->turn_moving = 0u;
  }
  pass_turn(turn);
  for (int a = nk + tid * crew.size() + crew.rank(); a < p.n_keep; a += kT * crew.size()) { p.kept[a] = -1; p.dbeta[a] = 0.f; }
  return true;
}
__device__ __forceinline__ void commit_deltas(const Squad& crew, const Problem& p, int nk, const unsigned short* kept_at) {
  for (int a = (int)threadIdx.x * crew.size() + crew.rank(); a < nk; a += kT * crew.size())
    p.delta[p.kept[a]] = (float)fabs(p.cand_dbeta64[kept_at != nullptr ? (int)kept_at[a] : p.kept_pos[a]]);
}

__global__ void __launch_bounds__(kT, 1) k_squads(const __grid_constant__ SquadSet set, int n_rounds, int have_list, int draw_next) {
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ DrawShared ds;
  __shared__ TurnShared ts;
  __shared__ ChangeShared cs;
  __shared__ Settled walk;
  __shared__ Problem sp;                                 // copies for the functions that are called rarely and not inlined
  __shared__ Engine se;
  const int tid = threadIdx.x, squad = (int)blockIdx.x / set.size, n_squads = set.n;
  const Problem& p = set.p[squad];
  const Engine& e = set.e[squad];
  Squad crew;
  crew.r = (int)blockIdx.x - squad * set.size; crew.n = set.size;
  EngineState* es = e.es;
  // The first round of the launch: read before anybody's turn can change it, which is why every CTA arrives once before the first turn.
  unsigned long long t0 = ~0ull;
  for (int i = 0; i < n_squads; ++i) t0 = min(t0, __ldcg(&set.p[i].st->round));
  const unsigned int status = p.st->status;
  Turn turn;
  turn.count = &set.e[0].es->turn_count; turn.n = (unsigned)crew.n; turn.limit = p.wait_limit ? p.wait_limit : kSpinLimit; turn.status = &p.st->status;
  pass_turn(turn);
  // after a wait that expired nothing runs on this handle until strads_recover (the other squads wait for a turn that does not come)
  if (status & STRADS_STATUS_WAIT_EXPIRED) return;
  auto keep_parameters = [&]() {
    __syncthreads();
    if (tid == 0) { sp = p; se = e; }
    __syncthreads();
  };
  const bool walker = crew.r == crew.n - 1;
  Grid g;
  g.count = &es->bar_count; g.target = 0u; g.n = (unsigned)crew.n; g.limit = turn.limit; g.status = &p.st->status;
  Grid g_draw = g;
  g_draw.count = &es->draw_bar_count;
  const unsigned long long t_end = t0 + (unsigned long long)n_rounds;
  unsigned long long t = t0 + (unsigned long long)((squad - (int)(t0 % (unsigned)n_squads) + n_squads) % n_squads);
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(sm);
  ChangedByBin* cb = reinterpret_cast<ChangedByBin*>(sm + (e.n_list > 0 ? 2 * sizeof(unsigned long long) * (size_t)p.n_keep : 0));
  unsigned short* kept_at = reinterpret_cast<unsigned short*>(sm + kept_at_offset(p, squad_smem(p, e.n_list > 0)));
  const bool no_filter = (p.flags & STRADS_FLAG_NO_FILTER) != 0, uniform = (p.flags & STRADS_FLAG_UNIFORM_DRAW) != 0;
  const int n_total = p.n_cand;
  bool have = have_list != 0, ok = true;
  // One trip per round, and one for a draw that nothing was drawn ahead for (real: false).
  while (true) {
    if (t >= t_end && (have || !draw_next || e.n_list == 0)) break;
    const bool real = have;
    const bool draws = !real || (e.n_list > 0 && (t + (unsigned)n_squads < t_end || draw_next));
    const unsigned long long td = real ? t + (unsigned)n_squads : t;             // the round drawn for
    const unsigned int k = real ? (unsigned)e.n_list : (unsigned)n_total;
    bool scanned = !draws, collected = !draws, own = false;                // own: the kept list is this CTA's own
    const int n = no_filter ? p.n_keep : e.window;
    bool window = no_filter || (p.bucket_count != nullptr && !(n < n_total && es->skip_window) && es->avoid == 0);
    if (real && window && !no_filter) csc_norms_begin(p, e, sm, n);
    if (real) csc_enter(crew, p, e, window ? n : n_total, window && !no_filter);
    // ---- the block; once more over all candidates where a window does not do ----
    while (true) {
      const bool during_walk = real && !window && !scanned, ahead = real && !no_filter && window;
      if (ahead) grid_arrive(g);
      if (!scanned && !during_walk) { draw_scan(crew, p, e, ds, sm, td, true); scanned = true; }
      if (ahead) {
        csc_products_begin(sm, n);
        if (!(ok = grid_complete(g))) break;
      } else if (!(real && !window && !(p.flags & STRADS_FLAG_DYNAMIC_DEPS)) && !(ok = grid_sync(g))) {
        break;
      }
      if (no_filter && real && walker) {                 // keep the first P
        for (int i = tid; i < p.n_keep; i += kT) { p.kept[i] = p.cand[i]; p.kept_pos[i] = i; }
        if (tid == 0) { es->n_kept = p.n_keep; es->n_examined = p.n_keep; es->walk_open = 0; }
      }
      if (!collected && !ahead && !during_walk) { draw_gather<AllThreads>(crew, p, e, ds, k, false); collected = true; }
      if (real && !window) {
        int walked = 0;
        if (!(ok = csc_walk_and_draw(crew, p, sp, e, ds, sm, g, g_draw, during_walk, td, k, &walked))) break;
        if (during_walk) scanned = collected = true;
      } else if (ahead) {
        csc_products<false>(crew, p, e, ts, sm, n, false, true, td, draws);
      }
      if (!(ok = grid_sync(g))) break;
      if (!ahead) break;
      csc_settle(p, e, sm, kept_at, walk, n, [&]() {
        const ClearAhead rows = csc_clear_begin(crew, p, n);
        if (!collected) draw_gather<OtherThreads>(crew, p, e, ds, k, false);
        csc_clear_end(p, rows);
      });
      collected = true;
      if (!walk_is_open(p, walk, n)) { own = true; break; }              // (the update's barriers stand for one here)
      if (!(ok = grid_sync(g))) break;
      if (crew.r == 0 && tid == 0) settle_note(e, walk);
      csc_enter(crew, p, e, n_total, false);
      window = false;
    }
    if (!ok) break;
    // ---- the update in its turn, then the list of this squad's next round ----
    const int n_next = no_filter ? p.n_keep : (e.window < n_total && es->skip_window ? n_total : e.window);   // looked at first
    const unsigned short* at = own ? kept_at : nullptr;
    const int nk = own ? walk.kept : es->n_kept;
    if (real) {
      turn.target = gridDim.x + (unsigned)(t - t0) * (unsigned)crew.n;
      if (!(ok = squad_update(crew, p, e, sm, g, turn, own ? &walk : nullptr, at, td, draws && !uniform))) break;
      t += (unsigned)n_squads;
    }
    if (draws && es->mend) {
      keep_parameters();
      if (!(ok = draw_mend(crew, sp, se, ds, sm, td, k, g))) break;
    }
    int n_changed = 0;
    if (real && draws && !uniform) {                     // (equal weights: no key changes)
      gather_changes<false>(p, ds, nk, at, true, keys, cb, nullptr, cs);
      n_changed = cs.n_changed;
      commit_deltas(crew, p, nk, at);
    }
    if (draws) draw_rank<false>(crew, p, e, ds, keys, cb, n_changed, n_changed > 0 ? nk : 0, cs.rank_wsum, crew.n, n_next);
    have = draws;
    if (!(ok = grid_sync(g))) break;
  }
  if (!ok || tid != 0) return;
  if (atomicInc(&es->exit_count, (unsigned)crew.n - 1u) == (unsigned)crew.n - 1u) { es->bar_count = 0u; es->draw_bar_count = 0u; }
  EngineState* first = set.e[0].es;
  if (atomicInc(&first->turn_exit, gridDim.x - 1u) == gridDim.x - 1u) first->turn_count = 0u;
}

}  // namespace

cudaError_t prepare_squads() {
  int dev = 0, most = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  if ((err = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return err;
  cudaFuncAttributes a;
  if ((err = cudaFuncGetAttributes(&a, k_squads)) != cudaSuccess) return err;
  return cudaFuncSetAttribute(k_squads, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)a.sharedSizeBytes);
}

cudaError_t launch_squads(const SquadSet& set, int n_rounds, bool have_list, bool draw_next, cudaStream_t s) {
  size_t smem = engine_smem(set.p[0], set.e[0].n_list > 0);
  const size_t update = kept_at_offset(set.p[0], squad_smem(set.p[0], set.e[0].n_list > 0)) + sizeof(unsigned short) * (size_t)set.p[0].n_keep;
  if (smem < update) smem = update;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(set.n * set.size)); cfg.blockDim = dim3(kT); cfg.dynamicSmemBytes = smem; cfg.stream = s;
  cfg.attrs = attr; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_squads, set, n_rounds, have_list ? 1 : 0, draw_next ? 1 : 0);
}

}  // namespace strads
