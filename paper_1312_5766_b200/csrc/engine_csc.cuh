// Rounds in one launch, CSC: inner products from row buckets, the residual, the walk over all candidates.
#pragma once
#include "engine_draw.cuh"
#include "walk_pairs.cuh"

namespace strads {
namespace {

// ------------------------------------------------------------------------------------------------
// CSC, steps 1 and 2: the window's pairs that share a row, by row buckets as in gram_csc.cu -- but a warp per candidate
// (its terms in a list of the warp's own in shared memory: no barrier), no conflict bits (the walk works from the list
// of conflicting pairs or forms rows on demand), and x_c^T r with the same visit to the column.
// ------------------------------------------------------------------------------------------------
constexpr int kMet = 512;                                // candidates one candidate may meet
constexpr int kRing = 4;                                 // steps of terms under way, and the one at hand
constexpr int kReach = 1664;                             // candidates of a window for each of which a warp has a place: 1,024 kept
constexpr int kPlaces = 1024;                            // ... places where there are more: at most half of them in use
constexpr unsigned short kNobody = 0xffff;
constexpr int kPart = 64;                                // positions of a column at a time
constexpr int kWorkers = kWarps - 1;                     // warps that form products; the last one makes the would-be changes
struct __align__(16) MetTable {
  int4 entry[kPart];                     // of a position of the column: row, terms before it, value, its own place in the row's bucket
  union {
    float dot[kReach];                   // by candidate; zero between candidates
    struct { float of_place[kPlaces]; unsigned short who[kPlaces]; };    // more candidates than that: by place (the same dot[]), and whose it is
  };
  unsigned short met[kMet];              // the places in use
  unsigned char lane[kReach];            // that had a term of the candidate last
  unsigned char pos[kPart * kBucketSlots];   // position of a term
  int2 term[kRing][32];                  // terms of the next steps: candidate and its value
  float value[kRing][32];                // ... the column's
};
constexpr int kNear = 2048;                              // candidates whose norms a CTA keeps in shared memory
constexpr size_t kTermsSmem = sizeof(MetTable) * kWorkers + sizeof(float) * kNear;
static_assert(STRADS_MAX_CANDIDATES < 0xffff && kPart <= 256, "16 bits per candidate, 8 per position");
static_assert(kPlaces + kPlaces / 2 <= kReach && kMet + 32 < kPlaces, "in the same memory; a search ends");

// The place of candidate b among more than kReach, taken if it has none: the next free one from its own number on.  Lanes that want the same
// free place all write to it and read who has it.  (Going through a candidate's terms once for every kReach candidates instead: us per
// round, 200,000 x 1,000,000 of 50 entries, P = 2,048, window of 6,000 75.4 -> 59.7, of 3,200 43.5 -> 41.6; P = 1,025, of 1,792 36.2 -> 34.1.
// Places of their own need no search: P = 1,024, of 1,664, 33.3.)
__device__ __forceinline__ int place_of(MetTable& wt, int b, bool on) {
  int at = b & (kPlaces - 1);
  bool open = on;
#pragma unroll 1
  while (__any_sync(kFull, open)) {
    if (open && wt.who[at] == kNobody) wt.who[at] = (unsigned short)b;
    __syncwarp();
    if (open) {
      if (wt.who[at] == (unsigned short)b) open = false;
      else at = (at + 1) & (kPlaces - 1);
    }
  }
  return at;
}

// The entries of candidates [0, n) into the buckets of their rows.  Where the columns lie was noted when the candidates
// were ranked, but for the dependencies dropped at run time (coupling_n2 follows beta and delta).
template <typename Crew>
__device__ __forceinline__ void csc_enter(const Crew& crew, const Problem& p, const Engine& e, int n, bool buckets) {
  const int lane = threadIdx.x & 31;
  const bool dynamic = (p.flags & STRADS_FLAG_DYNAMIC_DEPS) != 0;
  if (!buckets && !dynamic) return;
  constexpr int kU = Crew::kTogether;                    // candidates at a time: their chains of far accesses side by side
#pragma unroll 1
  for (int a0 = ((int)threadIdx.x >> 5) * crew.size() + crew.rank(); a0 < n; a0 += kU * kWarps * crew.size()) {
    WalkColumn col[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int a = a0 + u * kWarps * crew.size();
      col[u] = {};
      if (a < n) col[u] = p.walk_cols[a];
    }
    int most = 0;
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int a = a0 + u * kWarps * crew.size();
      if (dynamic && lane == 0 && a < n) {
        const double n2 = coupling_n2(p, col[u].j);
        p.walk_cols[a].n2 = n2;
        e.norm_f[a] = (float)n2;
      }
      most = max(most, col[u].n);
    }
    if (!buckets) continue;
#pragma unroll 1
    for (int q = lane; q - lane < most; q += 32) {
      int r[kU];
      float v[kU];
      unsigned int slot[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        r[u] = q < col[u].n ? __ldg(p.xrow + col[u].q0 + q) : -1;
        v[u] = q < col[u].n ? __ldg(p.xv + col[u].q0 + q) : 0.f;
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) slot[u] = r[u] >= 0 ? atomicAdd(&p.bucket_count[r[u]], 1u) : (unsigned)kBucketSlots;
#pragma unroll
      for (int u = 0; u < kU; ++u)
        if (r[u] >= 0 && q < kPart) p.bucket_own[(size_t)(a0 + u * kWarps * crew.size()) * kPart + q] = (unsigned char)min(slot[u], 255u);
#pragma unroll
      for (int u = 0; u < kU; ++u)
        if (slot[u] < (unsigned)kBucketSlots)
          p.bucket_pairs[(size_t)r[u] * kBucketSlots + slot[u]] = make_int2(a0 + u * kWarps * crew.size(), __float_as_int(v[u]));
    }
  }
}

// Emptied again by the threads that do not walk meanwhile.  In two parts, so that what there is to fetch is under way while
// the winners are collected: the rows of a warp's first candidates, two per lane; the others at once.
constexpr int kClearAhead = 2;
struct ClearAhead { int row[kClearAhead][2]; };
template <typename Crew>
__device__ __forceinline__ ClearAhead csc_clear_begin(const Crew& crew, const Problem& p, int n) {
  constexpr int kClearing = OtherThreads::kN / 32;
  const int lane = threadIdx.x & 31, step = kClearing * crew.size();
  ClearAhead c;
  int a = (OtherThreads::tid() >> 5) * crew.size() + crew.rank();
#pragma unroll
  for (int k = 0; k < kClearAhead; ++k, a += step) {
    c.row[k][0] = c.row[k][1] = -1;
    if (a >= n) continue;
    const WalkColumn col = p.walk_cols[a];
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (lane + 32 * h < col.n) c.row[k][h] = __ldg(p.xrow + col.q0 + lane + 32 * h);
    for (int q = lane + 64; q < col.n; q += 32) p.bucket_count[__ldg(p.xrow + col.q0 + q)] = 0u;
  }
#pragma unroll 1
  for (; a < n; a += step) {
    const WalkColumn col = p.walk_cols[a];
    for (int q = lane; q < col.n; q += 32) p.bucket_count[__ldg(p.xrow + col.q0 + q)] = 0u;
  }
  return c;
}
__device__ __forceinline__ void csc_clear_end(const Problem& p, const ClearAhead& c) {
#pragma unroll
  for (int k = 0; k < kClearAhead; ++k)
#pragma unroll
    for (int h = 0; h < 2; ++h) if (c.row[k][h] >= 0) p.bucket_count[c.row[k][h]] = 0u;
}

// |x_a^T x_b| >= rho ||x_a|| ||x_b||, with limit_a = rho^2 ||x_a||^2 and n2b = ||x_b||^2 in binary32: for certain not (may_conflict), for
// certain, or to be decided in FP64 (near the threshold, or where binary32 does not reach; the errors of d2 and of the limit
// are below 2^-21).
__device__ __forceinline__ bool limit_counts(float limit_a, float n2b, float limit) { return fminf(fminf(limit_a, n2b), limit) > 1e-30f && limit < 1e37f; }
__device__ __forceinline__ bool may_conflict(float dot, float limit_a, float n2b) {
  const float limit = limit_a * n2b;
  return !(limit_counts(limit_a, n2b, limit) && dot * dot < 0.9999f * limit);
}
__device__ __forceinline__ bool conflict_exactly(float dot, double n2a, double n2b, double rho) {
  const double den = sqrt(n2a * n2b);
  return den > 0.0 && fabs((double)dot) >= rho * den;
}
__device__ __forceinline__ bool in_conflict(float dot, float limit_a, double n2a, double n2b, double rho) {
  const float y = (float)n2b, limit = limit_a * y;
  if (!may_conflict(dot, limit_a, y)) return false;
  if (limit_counts(limit_a, y, limit) && dot * dot > 1.0001f * limit) return true;
  return conflict_exactly(dot, n2a, n2b, rho);
}
// (the norm of b is fetched where it is needed)
__device__ __forceinline__ bool in_conflict(float dot, float limit_a, double n2a, float n2b, const WalkColumn* b, double rho) {
  const float limit = limit_a * n2b;
  if (!may_conflict(dot, limit_a, n2b)) return false;
  if (limit_counts(limit_a, n2b, limit) && dot * dot > 1.0001f * limit) return true;
  return conflict_exactly(dot, n2a, b->n2, rho);
}

// x_c^T r and the would-be changes (kDots) of candidates [0, count) (kept: of the kept ones), and with `pairs` their inner
// products with the later candidates that share a row with them.  The CTA's k-th entry is cta + k * ctas; a warp per entry.
// What bounds it is the chain of dependent far accesses -- column, row, bucket -- so each link's loads go out together,
// and then the number of instructions per term.  The terms of 64 positions are laid out in the order of positions and dealt to
// the lanes, however unevenly the buckets are filled; a term is added to its candidate's product in an array of the
// warp's, terms of one candidate within a warp's step one after the other.  Whether a step has such terms shows when every
// lane writes its number to its candidate's place and reads it back: 280 cycles a step of 32 terms, where matching all lanes and
// a table with 16-bit compare-and-swap took 650 (match 160, compare-and-swap 200).
// An entry's own place in its row's bucket is noted when it is entered and left out: 50 of a candidate's 133 terms at 50,000 x 1,000,000
// (35.3 -> 34.9 us per round; four schedulers 20.2 -> 19.8).
// The would-be changes are made by a warp of their own, which has what it needs of the candidates by the time x_c^T r are there.
// 50,000 x 1,000,000, 1,664 candidates of 50 entries: 37.4 -> 35.3 us per round; 5,000 x 100,003, 384 candidates: 29.3 -> 28.1.
// (the tables, and the norms where they do not follow beta and delta: before the barrier that the buckets wait for)
__device__ __forceinline__ void csc_norms(const Problem& p, const Engine& e, unsigned char* sm, int count) {
  float* norm_f = reinterpret_cast<float*>(sm + sizeof(MetTable) * kWorkers);
  for (int i = threadIdx.x; i < min(count, kNear); i += kT) norm_f[i] = __ldcg(e.norm_f + i);
}
// (behind the scan's shared memory and that of what comes before it, so that they come in beside both)
__device__ __forceinline__ void csc_norms_begin(const Problem& p, const Engine& e, unsigned char* sm, int count) {
  static_assert(sizeof(MetTable) * kWorkers >= kScanSmem, "the norms lie behind the scan's shared memory");
  if (p.flags & STRADS_FLAG_DYNAMIC_DEPS) return;
  const uint32_t norm_f = smem_u32(sm + sizeof(MetTable) * kWorkers);
  for (int i = threadIdx.x; i < min(count, kNear); i += kT)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(norm_f + 4u * (unsigned)i), "l"(e.norm_f + i) : "memory");
}
__device__ __forceinline__ void csc_products_begin(unsigned char* sm, int count) {
  MetTable& wt = reinterpret_cast<MetTable*>(sm)[threadIdx.x >> 5];
  asm volatile("cp.async.wait_all;" ::: "memory");       // (the norms)
  __syncthreads();                                       // (what lay there before)
  if (threadIdx.x < 32 * kWorkers)
    for (int i = threadIdx.x & 31; i < kReach / 4; i += 32)
      reinterpret_cast<float4*>(wt.dot)[i] = count > kReach && i >= kPlaces / 4 ? make_float4(__int_as_float(-1), __int_as_float(-1), __int_as_float(-1), __int_as_float(-1))
                                                                              : make_float4(0.f, 0.f, 0.f, 0.f);
}
template <bool kDots, typename Crew>
__device__ __forceinline__ void csc_products(const Crew& crew, const Problem& p, const Engine& e, TurnShared& ts, unsigned char* sm, int count, bool kept, bool pairs,
                                             unsigned long long t_next, bool want_keys) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int cta = crew.rank(), n_ctas = crew.size();
  const double rho = (double)p.rho;
  MetTable& wt = reinterpret_cast<MetTable*>(sm)[warp];
  float* norm_f = reinterpret_cast<float*>(sm + sizeof(MetTable) * kWorkers);
  const int mine = count > cta ? (count - cta + n_ctas - 1) / n_ctas : 0;
  const bool direct = count <= kReach;
  if (mine == 0) return;
  if (pairs && (p.flags & STRADS_FLAG_DYNAMIC_DEPS)) {
    csc_norms(p, e, sm, count);
    __syncthreads();
  }
#pragma unroll 1
  for (int k0 = 0; k0 < mine; k0 += kTurn) {
    const int turn = min(kTurn, mine - k0);
    if (k0 > 0) __syncthreads();
    if (warp == kWorkers) {
      if (!kDots) continue;
      int j_own = 0, pos_own = 0;
      float E = 0.f;
      Proposal prop = {};
      if (lane < turn) {
        const int a = cta + n_ctas * (k0 + lane);
        pos_own = kept ? p.kept_pos[a] : a;
        j_own = kept ? p.kept[a] : p.cand[a];
        const double n_own = p.n2[j_own];
        const float b_own = p.beta[j_own], d_own = p.delta[j_own];
        if (want_keys) E = exponential_of(p, t_next, (uint32_t)j_own);
        prop = propose_begin(p, j_own, n_own, b_own, d_own, E, want_keys);
      }
      asm volatile("bar.sync 4, %0;" ::"n"(kT) : "memory");              // x_c^T r are there
      if (lane < turn) propose_end(p, prop, pos_own, j_own, ts.dot[lane][0], E, want_keys);
      continue;
    }
    if (kDots && warp >= turn) asm volatile("bar.arrive 4, %0;" ::"n"(kT) : "memory");
#pragma unroll 1
    for (int k = warp; k < turn; k += kWorkers) {
      const int a = cta + n_ctas * (k0 + k);
      const WalkColumn col = p.walk_cols[kept ? p.kept_pos[a] : a];
      double acc = 0.0;
      auto tell = [&]() {                                // this candidate's x_c^T r; the last one of the warp's: all of them
        if (!kDots) return;
        acc = warp_sum(acc);
        if (lane == 0) ts.dot[k][0] = acc;
        if (k + kWorkers >= turn) {
          __threadfence_block();
          __syncwarp();
          asm volatile("bar.arrive 4, %0;" ::"n"(kT) : "memory");
        }
      };
      if (col.n <= 0) tell();
      {
        int n_met = 0;                                   // (the same in all lanes)
        bool failed = false;
#pragma unroll 1
        for (int q0 = 0; q0 < col.n; q0 += kPart) {
          int r[2];
          float v[2];
          unsigned int cnt[2];
          int own[2];                                    // the entry's own place in its row's bucket: no term (255: not known)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int q = q0 + 32 * h + lane;
            r[h] = q < col.n ? __ldg(p.xrow + col.q0 + q) : -1;
            v[h] = q < col.n ? __ldg(p.xv + col.q0 + q) : 0.f;
            own[h] = pairs && q < min(col.n, kPart) ? p.bucket_own[(size_t)a * kPart + q] : 255;
          }
          float x[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            x[h] = kDots && r[h] >= 0 ? p.resid[r[h]] : 0.f;
            cnt[h] = pairs && r[h] >= 0 ? p.bucket_count[r[h]] : 0u;
          }
#pragma unroll
          for (int h = 0; h < 2; ++h)
            if (kDots && r[h] >= 0) acc += (double)v[h] * (double)x[h];
          if (q0 + kPart >= col.n) tell();
          if (!pairs) continue;
#pragma unroll
          for (int h = 0; h < 2; ++h)
            if (cnt[h] > (unsigned)kBucketSlots) { failed = true; cnt[h] = 0u; }
#pragma unroll
          for (int h = 0; h < 2; ++h)
            if ((unsigned)own[h] < cnt[h]) --cnt[h];
          const unsigned int both = cnt[0] | (cnt[1] << 16);
          unsigned int incl = both;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const unsigned int u = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += u;
          }
          const unsigned int all = __shfl_sync(kFull, incl, 31);
          const int n0 = (int)(all & 0xffffu), n_terms = n0 + (int)(all >> 16);
          const int off[2] = {(int)((incl - both) & 0xffffu), n0 + (int)((incl - both) >> 16)};
          __syncwarp();
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            wt.entry[32 * h + lane] = make_int4(r[h], off[h], __float_as_int(v[h]), own[h]);
            for (unsigned int i = 0; i < cnt[h]; ++i) wt.pos[off[h] + i] = (unsigned char)(32 * h + lane);
          }
          __syncwarp();
          // The terms of the next steps are under way, straight into shared memory (a bucket is a line of the L2 of which nobody else
          // on this SM needs anything).  One copy of the loop's code, as it is fetched anew every round: with four steps unrolled, for
          // their loads to go out together, a step took 850 cycles.
          auto load = [&](int i) {
            const int at = i * 32 + lane;
            if (at < n_terms) {
              const int4 en = wt.entry[wt.pos[at]];
              wt.value[i % kRing][lane] = __int_as_float(en.z);
              const int slot = at - en.y + (at - en.y >= en.w ? 1 : 0);
              asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(&wt.term[i % kRing][lane])),
                           "l"(p.bucket_pairs + (size_t)en.x * kBucketSlots + slot) : "memory");
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
          };
          const int steps = (n_terms + 31) >> 5;
#pragma unroll 1
          for (int i = 0; i < kRing - 1; ++i) load(i);
#pragma unroll 1
          for (int i = 0; i < steps; ++i) {
            load(i + kRing - 1);
            asm volatile("cp.async.wait_group %0;" ::"n"(kRing - 1) : "memory");
            struct { int b; float fa, fb; } term = {-1, 0.f, 0.f};
            if (i * 32 + lane < n_terms) {               // (a lane reads what it brought in itself)
              const int2 m = wt.term[i % kRing][lane];
              term.b = m.x; term.fb = __int_as_float(m.y); term.fa = wt.value[i % kRing][lane];
            }
            const bool on = term.b > a && (direct || n_met <= kMet);
            const int b = direct ? (on ? term.b : 0) : place_of(wt, term.b, on);
            if (on) wt.lane[b] = (unsigned char)lane;
            __syncwarp();
            float old = 1.f;
            if (__all_sync(kFull, !on || wt.lane[b] == lane)) {
              if (on) { old = wt.dot[b]; wt.dot[b] = fmaf(term.fa, term.fb, old); }
            } else {                                   // several terms of a candidate within these 32: in their order
              const unsigned int peers = __match_any_sync(kFull, on ? b : ~lane);
              const int turn_of = on ? __popc(peers & ((1u << lane) - 1u)) : -1;
#pragma unroll 1
              for (int i = 0; __any_sync(kFull, turn_of >= i); ++i) {
                if (turn_of == i) {
                  const float was = wt.dot[b];
                  if (i == 0) old = was;
                  wt.dot[b] = fmaf(term.fa, term.fb, was);
                }
                __syncwarp();
              }
            }
            const unsigned int m = __ballot_sync(kFull, on && old == 0.f);       // (met for the first time, or its products cancel: listed twice)
            if (on && old == 0.f) {
              const int i = n_met + __popc(m & ((1u << lane) - 1u));
              if (i < kMet) wt.met[i] = (unsigned short)b;
            }
            n_met += __popc(m);
            __syncwarp();
          }
        }
        if (!pairs) continue;
        const bool overflow = __any_sync(kFull, failed) || n_met > kMet;
        if (overflow && lane == 0) e.es->bucket_failed = 1;
        // which of them conflict: those that may are gathered first, so that the far accesses are made for all of them at once
        const float limit_a = (float)(rho * rho * col.n2);
        int n_near = 0;
#pragma unroll 1
        for (int i0 = 0; i0 < min(n_met, kMet); i0 += 32) {
          bool on = i0 + lane < min(n_met, kMet);
          const int b = on ? wt.met[i0 + lane] : 0, c = direct ? b : wt.who[b];
          on = on && (direct || c != kNobody);           // (listed twice, and settled)
          const float dot = on ? wt.dot[b] : 0.f;
          const bool near = on && may_conflict(dot, limit_a, c < kNear ? norm_f[c] : __ldcg(e.norm_f + c));
          if (on && !near) { wt.dot[b] = 0.f; if (!direct) wt.who[b] = kNobody; }
          const unsigned int m = __ballot_sync(kFull, near);
          if (near) wt.met[n_near + __popc(m & ((1u << lane) - 1u))] = (unsigned short)b;      // (places that have been read)
          n_near += __popc(m);
          __syncwarp();
        }
#pragma unroll 1
        for (int i0 = 0; i0 < n_near; i0 += 32) {
          bool on = i0 + lane < n_near;
          const int b = on ? wt.met[i0 + lane] : 0, c = direct ? b : wt.who[b];
          on = on && (direct || c != kNobody);
          const float dot = on ? wt.dot[b] : 0.f;
          __syncwarp();
          bool conflict = false;
          if (on) {
            wt.dot[b] = 0.f;
            if (!direct) wt.who[b] = kNobody;
            conflict = dot != 0.f && in_conflict(dot, limit_a, col.n2, c < kNear ? norm_f[c] : __ldcg(e.norm_f + c), p.walk_cols + c, rho);
          }
          const unsigned int m = __ballot_sync(kFull, conflict);
          if (m == 0u) continue;
          unsigned int at = 0u;
          if (lane == 0) at = atomicAdd(&e.es->edge_count, (unsigned)__popc(m));
          at = __shfl_sync(kFull, at, 0) + (unsigned)__popc(m & ((1u << lane) - 1u));
          if (conflict && at < (unsigned)p.cap_edges) p.edges[at] = ((unsigned int)a << 16) | (unsigned)c;
        }
        __syncwarp();
        if (n_met > kMet) {                              // (places that were not listed)
          for (int i = lane; i < (direct ? kReach : kPlaces); i += 32) wt.dot[i] = 0.f;
          for (int i = lane; i < (direct ? 0 : kPlaces); i += 32) wt.who[i] = kNobody;
        }
        __syncwarp();
      }
    }
  }
}

// ------------------------------------------------------------------------------------------------
// CSC, step 4 and the next step 1: the residual.  Contributions are added as 64-bit fixed-point integers (unit 2^-shift, the
// same bits in any order) and every row with a non-zero accumulator is updated once behind the next barrier.
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ int csc_shift(float x_abs_max, unsigned long long dmax_bits, int nk) {
  const double m = __longlong_as_double((long long)dmax_bits);
  if (!(m > 0.0) || !isfinite(m)) return INT_MIN;
  int x = 0;
  frexp(m * (double)x_abs_max * (double)max(nk, 1), &x);
  return 61 - x;
}

template <typename F, typename Crew>
__device__ __forceinline__ void for_moving_entries(const Crew& crew, const Problem& p, int nk, F&& f) {
  const int lane = threadIdx.x & 31;
  for (int a = ((int)threadIdx.x >> 5) * crew.size() + crew.rank(); a < nk; a += kWarps * crew.size()) {
    const double d = p.cand_dbeta64[p.kept_pos[a]];
    if (d == 0.0) continue;
    const int j = p.kept[a];
    const long long q1 = p.xptr[j + 1];
    for (long long q = p.xptr[j] + lane; q < q1; q += 32) f(q, d);
  }
}

// A warp's kept columns (a mod warps of the crew): lane k has the k-th.  kept_at: positions of the kept candidates in shared memory, read
// before anybody can rank the next candidates over these, and entered into the lists in global memory; null: from there.
struct KeptColumns { int m, len; long long q0; double d; };
template <typename Crew>
__device__ __forceinline__ KeptColumns kept_columns(const Crew& crew, const Problem& p, int nk, const unsigned short* kept_at) {
  const int first = ((int)threadIdx.x >> 5) * crew.size() + crew.rank(), step = kWarps * crew.size();
  const int a = first + ((int)threadIdx.x & 31) * step;
  KeptColumns c;
  c.m = nk > first ? (nk - first + step - 1) / step : 0; c.len = 0; c.q0 = 0; c.d = 0.0;
  if (a >= nk) return c;
  if (kept_at != nullptr) {
    const int pos = kept_at[a];
    const WalkColumn col = p.walk_cols[pos];
    c.d = p.cand_dbeta64[pos]; c.q0 = col.q0; c.len = col.n;
    p.kept[a] = col.j; p.kept_pos[a] = pos;
  } else {
    const int j = p.kept[a];
    c.d = p.cand_dbeta64[p.kept_pos[a]]; c.q0 = p.xptr[j]; c.len = (int)(p.xptr[j + 1] - c.q0);
  }
  return c;
}
__device__ __forceinline__ void csc_scatter(const Problem& p, const KeptColumns& c, int shift) {
  if (shift == INT_MIN) return;
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int k = 0; k < c.m; ++k) {
    const double d = __shfl_sync(kFull, c.d, k);
    const long long q0 = __shfl_sync(kFull, c.q0, k);
    const int len = __shfl_sync(kFull, c.len, k);
    if (d == 0.0) continue;
    for (int q = lane; q < len; q += 32) {
      const long long fx = __double2ll_rn(ldexp((double)__ldg(p.xv + q0 + q) * d, shift));
      atomicAdd(reinterpret_cast<unsigned long long*>(p.resid_acc + __ldg(p.xrow + q0 + q)), (unsigned long long)fx);
    }
  }
}
static_assert(STRADS_MAX_CANDIDATES <= 32 * kWarps * 32, "a lane per kept column of a warp with 32 CTAs or more");

// Rows r[] by the sums in v[] (0: nothing to do), with what they are now under way together.
template <int kU>
__device__ __forceinline__ void apply_sums(const Problem& p, const long long (&r)[kU], const long long (&v)[kU], int shift) {
  const bool logistic = (p.flags & STRADS_FLAG_LOGISTIC) != 0;
  const float* now = logistic ? p.margin : p.resid;
  float x[kU];
#pragma unroll
  for (int u = 0; u < kU; ++u) x[u] = v[u] != 0 ? now[r[u]] : 0.f;
#pragma unroll
  for (int u = 0; u < kU; ++u)
    if (v[u] != 0) apply_row(p, r[u], x[u], ldexp((double)v[u], -shift));
}
template <typename Crew>
__device__ __forceinline__ void csc_apply_rows(const Crew& crew, const Problem& p, int shift) {
  for (long long r = (long long)crew.rank() * kT + threadIdx.x; r < p.N; r += (long long)crew.size() * kT) {
    const long long v = p.resid_acc[r];
    if (v != 0) {
      apply_row(p, r, ldexp((double)v, -shift));
      p.resid_acc[r] = 0;
    }
  }
}
template <typename Crew>
__device__ void csc_apply(const Crew& crew, const Problem& p, int nk, int n_moving, int shift) {
  if (shift == INT_MIN) return;
  // few moving entries against the rows: visit the entries' rows (the first visitor of a row takes its sum), else all rows
  if ((double)n_moving * (double)p.nnz * 4.0 < (double)p.N * (double)p.J) {
    for_moving_entries(crew, p, nk, [&](long long q, double) {
      const int r = __ldg(p.xrow + q);
      const long long v = (long long)atomicExch(reinterpret_cast<unsigned long long*>(p.resid_acc + r), 0ull);
      if (v != 0) apply_row(p, r, ldexp((double)v, -shift));
    });
    return;
  }
  csc_apply_rows(crew, p, shift);
}

// ------------------------------------------------------------------------------------------------
// CSC, step 3b: the walk over all candidates with conflict rows on demand (see walk_csc.cu for the scheme: batches of 32
// unblocked candidates, picked, multiplied with one another and decided by every CTA alike; then the kept members against
// all later unblocked candidates over the grid; one barrier per batch).  Here 32 consecutive candidates -- a word of the mask
// -- belong to CTA word mod ctas, which brings their columns into shared memory once per walk and publishes the whole word
// after every batch: no atomics, and nothing to clear.
//
// What bounds a batch is its chain of short steps, so products are not merges of two sorted lists (2 nnz dependent steps each)
// but look-ups: the rows of the batch's columns go into a hash table in shared memory, each with the mask of the members
// that have an entry there and their values side by side; a thread that has a pair goes through one column's
// entries, none of which waits for the one before.  Same products, added in the same order of rows.
//
// Once few survive, a batch each for the next 32 of them costs more than all their products: every CTA multiplies its share of
// the survivors with all of them, and behind one more barrier every CTA settles the rest from the bits.
//
// The chain leaves most of the SM's issue slots idle whatever the number of its warps, and the next draw up to the collection of
// its winners needs nothing else: half the warps walk, the other half draw, with barriers of their own.
//
// 10^7 columns of 20 entries, 16,384 candidates of which ~64 are kept: 65 us per round.  With merges, batches of 32 to the end
// (5.1 of them at 9.7 us) and all warps in both, the scan in the walk's waits and behind it, 101.
// ------------------------------------------------------------------------------------------------
constexpr int kWalkWarps = kWalkT / 32;
constexpr int kBatch = 32;
constexpr int kColCap = 64;                              // entries of a batch member's column that the table takes
constexpr int kRowBits = 12, kRowSlots = 1 << kRowBits;  // of the table: at most half full
constexpr int kFreeRow = -1;
constexpr unsigned int kNoSlot = 0xffff;
constexpr int kOwn = 256;                                // candidates a CTA can hold (more: their columns stay in global memory)
constexpr int kOwnEntries = 5120;                        // entries of their columns
// ... where there are more: without the values, which the few entries in rows of kept members then fetch.  What finds no room at all is read
// from global memory for every kept member (us per round, 10^6 x 10^6 by Zipf's law, 16,384 candidates of 60 / 50 entries, up to 7,680 / 6,400 to a CTA:
// 137 / 107 with a third / a fifth of them so, one entry after the other; 131 / 101 with eight at a time; 86 / 76 with all rows held).
constexpr int kOwnRows = kOwnEntries * 3 / 2;
constexpr int kRestEntries = kOwnEntries * 3 / 2;
// Survivors that are settled at once: as many as a thread pair of bits per walking thread holds, and while their entries, all of
// which every CTA goes through, are no more than these -- by the mean length of all columns: an estimate, the pieces they are gone through in make up
// for it -- (us per round for 1,500 / 2,600 / 4,096 / 7,000 / 12,288: 10^7 columns of 20
// entries 65.8 / 65.5 / 64.8 / 65.3 / 66.3, 300,000 of 30 34.9 / 35.5 / 37.0 / 39.8 / 41.1, 3,000,000 of 12 47.0 / 44.9 / 45.1 / 48.2 / 48.1).
constexpr int kLast = 512;
constexpr long long kLastEntries = 3072;
constexpr int kPerMember = kWalkT / kBatch, kEach = kColCap / kPerMember;      // threads of a batch member; its entries per thread
static_assert(kMaxWords <= 2 * kWalkT && kOwn == kT - kWalkT && kBatch == 4 * kWalkWarps && kBatch * kColCap * 2 <= kRowSlots,
              "two mask words per walking thread, a held candidate per other thread, four members per warp");

struct DemandShared {
  int pos[kBatch], col[kBatch], len[kBatch];             // the batch: position in the list, coefficient, entries
  long long ptr[kBatch];
  double n2[kBatch];
  float limit[kBatch];                                   // rho^2 n2
  unsigned int conf[kBatch];                             // conflicts with earlier members
  int kept_q[kBatch];                                    // members kept, in order
  int n_shared[kBatch];                                  // a member's entries in rows of later members
  int wsum[kWarps];
  int longest, n_vals, n_free;
  int kept, ok, drawn;                                   // results
  unsigned int target, draw_target;
  // rows of the batch's columns
  __align__(16) int row_key[kRowSlots];
  __align__(16) uint2 row_rec[kRowSlots];                              // members with an entry in the row (0: slot free), and where their values start
  float row_val[kBatch * kColCap];
  __align__(16) uint4 ent[kBatch][kColCap];              // ... those: members of the row, where their values start, the entry's value
  int survivor[kLast];
  __align__(16) unsigned int state[2][2][kLast / 32];    // the survivors undecided and kept, in turns
  // the CTA's words and candidates
  unsigned int own_word[kMaxWords], own_hit[kMaxWords];
  int own_at[kOwn + 1], own_free[kOwn], n_met[kOwn];
  long long own_q0[kOwn];
  double own_n2[kOwn];
  union {
    struct {
      int orow[kOwnEntries];
      float oval[kOwnEntries];
      unsigned int omet[kOwnEntries];                    // a candidate's entries in rows of kept members: slot, and entry << 16
    };
    struct { int only_row[kOwnRows]; unsigned int only_met[kOwnRows]; };
    struct { int rrow[kRestEntries]; float rval[kRestEntries]; };      // survivors' columns
  };
};

__device__ __forceinline__ unsigned int row_hash(int row) { return ((unsigned int)row * 2654435761u) >> (32 - kRowBits); }
// Slots of rows of the batch's columns; kNoSlot: none of the members in `want` has an entry there (kFreeRow: no row).  Their first
// places are looked at together.
template <int kU>
__device__ __forceinline__ void find_rows(const DemandShared& s, const int (&row)[kU], unsigned int want, unsigned int (&slot)[kU]) {
  int key[kU];
#pragma unroll
  for (int u = 0; u < kU; ++u) { slot[u] = row_hash(row[u]); key[u] = s.row_key[slot[u]]; }
  bool more;
  do {                                                   // (other rows in their places)
    more = false;
#pragma unroll
    for (int u = 0; u < kU; ++u)
      if (key[u] != row[u] && key[u] != kFreeRow) { slot[u] = (slot[u] + 1u) & (kRowSlots - 1); key[u] = s.row_key[slot[u]]; more = true; }
  } while (more);
#pragma unroll
  for (int u = 0; u < kU; ++u) {
    const unsigned int members = s.row_rec[slot[u]].x;
    if (row[u] == kFreeRow || key[u] == kFreeRow || !(members & want)) slot[u] = kNoSlot;
  }
}
// dot + the products of member q's entries with values v of a column in rows of the table (rec: their members, where the members'
// values start), one after the other.  Each is as many accesses deep whether q has an entry or not, so that they go out together.
template <int kU>
__device__ __forceinline__ float add_products(const DemandShared& s, int q, const uint2 (&rec)[kU], const float (&v)[kU], float dot) {
  float x[kU];
#pragma unroll
  for (int u = 0; u < kU; ++u) x[u] = s.row_val[(rec[u].x >> q) & 1u ? rec[u].y + (unsigned)__popc(rec[u].x & ((1u << q) - 1u)) : 0u];
#pragma unroll
  for (int u = 0; u < kU; ++u) dot = (rec[u].x >> q) & 1u ? fmaf(x[u], v[u], dot) : dot;
  return dot;
}
// The same over n rows; at(i, &rec, &value) for i < n.  most: the largest n of the warp.
template <typename At>
__device__ __forceinline__ float row_products(const DemandShared& s, int q, int n, int most, At&& at) {
  constexpr int kU = 8;
  float dot = 0.f;
#pragma unroll 1
  for (int i0 = 0; i0 < most; i0 += kU) {
    uint2 rec[kU];
    float v[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      rec[u] = make_uint2(0u, 0u); v[u] = 0.f;
      if (i0 + u < n) at(i0 + u, rec[u], v[u]);
    }
    dot = add_products<kU>(s, q, rec, v, dot);
  }
  return dot;
}
// The same over a column in global memory, entries side by side.  (Out of line: rare, and the hot code is fetched anew every round.)
__device__ __noinline__ float column_products(const int* rows, const float* vals, int n, const DemandShared& s, int q) {
  constexpr int kU = 8;
  float dot = 0.f;
#pragma unroll 1
  for (int x0 = 0; x0 < n; x0 += kU) {
    int row[kU];
    float v[kU];
    unsigned int sl[kU];
    uint2 rec[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const bool on = x0 + u < n;
      row[u] = on ? __ldg(rows + x0 + u) : kFreeRow;
      v[u] = on ? __ldg(vals + x0 + u) : 0.f;
    }
    find_rows<kU>(s, row, 1u << q, sl);
#pragma unroll
    for (int u = 0; u < kU; ++u) rec[u] = sl[u] != kNoSlot ? s.row_rec[sl[u]] : make_uint2(0u, 0u);
    dot = add_products<kU>(s, q, rec, v, dot);
  }
  return dot;
}
// The same over the entries of held candidate k in rows of kept members, their values fetched.  (Out of line like that: as a branch in the
// loop where the values are held it cost rounds whose columns all fit 7 %, 10^6 x 10^7 with 20 entries 61.9 -> 66.4 us, like this under 1 %.)
__device__ __noinline__ float fetched_products(const DemandShared& s, const float* vals, int k, int q) {
  const int met = s.n_met[k], from = s.own_at[k];
  vals += s.own_q0[k];
  return row_products(s, q, met, met, [&](int x, uint2& rec, float& v) {
    const unsigned int en = s.only_met[from + x];
    rec = s.row_rec[en & 0xffffu]; v = __ldg(vals + (en >> 16));
  });
}
// x_a^T x_b of two ascending row lists, products added in row order; no branch depends on the data.
__device__ __forceinline__ float merge_dot(const int* ar, const float* av, int na, const int* br, const float* bv, int nb) {
  float dot = 0.f;
  int i = 0, k = 0;
  while (i < na && k < nb) {
    const int ra = ar[i], rb = br[k];
    if (ra == rb) dot = fmaf(av[i], bv[k], dot);
    i += ra <= rb;
    k += rb <= ra;
  }
  return dot;
}

// (cold) A batch with a column longer than the table takes: its pairs, and its kept members against a candidate, by merges.
__device__ __noinline__ void merge_batch(const Problem& p, DemandShared& s, int m) {
  const double rho = (double)p.rho;
  for (int i = threadIdx.x; i < m * m; i += kWalkT) {
    const int qa = i / m, qb = i - qa * m;
    if (qa >= qb) continue;
    const float dot = merge_dot(p.xrow + s.ptr[qa], p.xv + s.ptr[qa], s.len[qa], p.xrow + s.ptr[qb], p.xv + s.ptr[qb], s.len[qb]);
    if (in_conflict(dot, s.limit[qa], s.n2[qa], s.n2[qb], rho)) atomicOr(&s.conf[qb], 1u << qa);
  }
}
__device__ __noinline__ float merge_columns(const Problem& p, long long qa, int na, long long qb, int nb) {
  return merge_dot(p.xrow + qa, p.xv + qa, na, p.xrow + qb, p.xv + qb, nb);
}

__device__ __forceinline__ void walk_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kWalkT) : "memory"); }

// Grid barrier of the walking threads.
__device__ __forceinline__ bool walk_barrier(DemandShared& s, Grid& g) {
  g.target += g.n;
  walk_sync();
  if (threadIdx.x == 0) s.ok = grid_wait(g);
  walk_sync();
  return s.ok != 0;
}

// (cold, see hold_columns)
__device__ __noinline__ void hold_rows(DemandShared& s, const int* rows, int i, int count, int* row, int room) {
  for (int k = i >> 3; k < count; k += kOwn / 8) {
    const int at = s.own_at[k], m = s.own_at[k + 1] - at;
    if (at + m <= room)
#pragma unroll 4
      for (int q = i & 7; q < m; q += 8) row[at + q] = __ldg(rows + s.own_q0[k] + q);
  }
}
// The columns of `count` candidates (thread i of kOwn has the i-th) into row / val, one behind the other, as far as there is room
// (room_rows > 0: if not for all, as far as there is without the values).  Bound by the lines a load touches, so several threads share a column.  Bar: the threads' barrier.
template <int kBar>
__device__ __forceinline__ void hold_columns(const Problem& p, DemandShared& s, int i, int count, const WalkColumn& col, int* row, float* val, int room,
                                             int room_rows) {
  const int lane = threadIdx.x & 31, warp = i >> 5;
  int* wsum = s.wsum + (kBar == 1 ? 0 : kWalkWarps);
  int incl = col.n;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) wsum[warp] = incl;
  asm volatile("bar.sync %0, %1;" ::"n"(kBar), "n"(kOwn) : "memory");
  int before = 0;
#pragma unroll
  for (int k = 0; k < kOwn / 32; ++k) if (k < warp) before += wsum[k];
  if (i == 0) s.own_at[0] = 0;
  s.own_at[i + 1] = before + incl;
  s.own_q0[i] = col.q0; s.own_n2[i] = col.n2;
  asm volatile("bar.sync %0, %1;" ::"n"(kBar), "n"(kOwn) : "memory");
  if (room_rows > 0 && s.own_at[count] > room) {
    hold_rows(s, p.xrow, i, count, row, room_rows);
    return;
  }
#pragma unroll 2
  for (int k = i >> 3; k < count; k += kOwn / 8) {
    const int at = s.own_at[k], m = s.own_at[k + 1] - at;
    const long long from = s.own_q0[k];
    if (at + m <= room)
#pragma unroll 4
      for (int q = i & 7; q < m; q += 8) { row[at + q] = __ldg(p.xrow + from + q); val[at + q] = __ldg(p.xv + from + q); }
  }
}

// The rest of a walk: the batch's m members are this CTA's share (cta, cta + ctas, ...) of the `total` candidates that are left
// (s.survivor, in list order); their conflicts with all earlier ones go to global memory, a row of bits per survivor, and
// behind a barrier every CTA settles them all: a survivor with a kept earlier neighbour is out, one whose earlier neighbours
// are all out is kept; a thread holds the rows of two survivors, and the passes are as many as the longest chain of such
// dependencies.  False: the barrier gave up.
template <typename Crew>
__device__ __forceinline__ bool settle_rest(const Crew& crew, const Problem& p, const Problem& sp, DemandShared& s, Grid& g, int total, int m, bool table, int& kept,
                                            int& examined) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, cta = crew.rank(), n_ctas = crew.size();
  const int W = (total + 31) >> 5, pitch = (W + 3) & ~3;
  const double rho = (double)p.rho;
  constexpr int kTogether = 4;                           // members at a time
  constexpr int kU = 8;                                  // entries of a candidate's column at a time
  const int behind = cta + (m - 1) * n_ctas;             // candidates before the last member
  for (int c0 = 0, here; c0 < behind; c0 += here) {      // as many at a time as there is room for
    const int count = min(behind - c0, kOwn);
    WalkColumn col = {};
    if (tid < count) col = p.walk_cols[s.survivor[c0 + tid]];
    hold_columns<1>(p, s, tid, count, col, s.rrow, s.rval, kRestEntries, 0);
    walk_sync();
    here = kOwn;                                         // whole words; of the first one whatever does not fit is read where it is
    while (here > 32 && s.own_at[here] > kRestEntries) here -= 32;
    const int c = c0 + tid, at = s.own_at[tid], n = tid < here ? s.own_at[tid + 1] - at : 0;
    const bool held = at + n <= kRestEntries;
    int met = 0;
    if (tid < here) {
      // the entries in rows of members move to the front of the candidate's stretch (its thread has read what lay there), each
      // with its row's slot: most rows are no member's, and products are four times the instructions of a look-up
      if (table) {
#pragma unroll 1
        for (int x0 = 0; x0 < (held ? n : 0); x0 += kU) {
          int row[kU];
          float v[kU];
          unsigned int sl[kU];
#pragma unroll
          for (int u = 0; u < kU; ++u) {
            const bool on = x0 + u < n;
            row[u] = on ? s.rrow[at + x0 + u] : kFreeRow;
            v[u] = on ? s.rval[at + x0 + u] : 0.f;
          }
          find_rows<kU>(s, row, kFull, sl);
#pragma unroll
          for (int u = 0; u < kU; ++u)
            if (sl[u] != kNoSlot) { s.rrow[at + met] = (int)sl[u]; s.rval[at + met] = v[u]; ++met; }
        }
        __syncwarp();
      }
      const int most = __reduce_max_sync(kFull, met);
#pragma unroll 1
      for (int g0 = 0; g0 < m; g0 += kTogether) {
        float dot[kTogether] = {};
        if (table) {
#pragma unroll 1
          for (int x0 = 0; x0 < most; x0 += kU) {
            float v[kU];
            uint2 rec[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
              const bool on = x0 + u < met;
              rec[u] = on ? s.row_rec[s.rrow[at + x0 + u]] : make_uint2(0u, 0u);
              v[u] = on ? s.rval[at + x0 + u] : 0.f;
            }
#pragma unroll
            for (int y = 0; y < kTogether; ++y)
              if (g0 + y < m) dot[y] = add_products<kU>(s, g0 + y, rec, v, dot[y]);
          }
          if (!held) {                                   // (no room for its column: one entry after the other)
            const unsigned int want = ((1u << kTogether) - 1u) << g0;
#pragma unroll 1
            for (int x = 0; x < n; ++x) {
              const int row[1] = {__ldg(p.xrow + col.q0 + x)};
              unsigned int sl[1];
              find_rows<1>(s, row, want, sl);
              if (sl[0] == kNoSlot) continue;
              const uint2 rec[1] = {s.row_rec[sl[0]]};
              const float v[1] = {__ldg(p.xv + col.q0 + x)};
#pragma unroll
              for (int y = 0; y < kTogether; ++y)
                if (g0 + y < m) dot[y] = add_products<1>(s, g0 + y, rec, v, dot[y]);
            }
          }
        } else {
#pragma unroll
          for (int y = 0; y < kTogether; ++y)
            if (g0 + y < m) dot[y] = merge_columns(sp, s.ptr[g0 + y], s.len[g0 + y], col.q0, col.n);
        }
#pragma unroll
        for (int y = 0; y < kTogether; ++y) {
          const int q = g0 + y, i = cta + q * n_ctas;    // the member's place among the survivors
          if (q >= m) break;
          const unsigned int word = __ballot_sync(kFull, c < i && in_conflict(dot[y], s.limit[q], s.n2[q], col.n2, rho));
          if (lane == 0 && (c >> 5) < W) __stcg(p.conflict + i * pitch + (c >> 5), word);
        }
      }
    }
    walk_sync();
  }
  if (tid < 2 * kLast / 32) {                            // undecided, kept
    const int w = tid % (kLast / 32), here = total - w * 32;
    s.state[0][tid / (kLast / 32)][w] = tid >= kLast / 32 || here <= 0 ? 0u : (here >= 32 ? kFull : (1u << here) - 1u);
  }
  if (!walk_barrier(s, g)) return false;
  static_assert(kLast == 2 * kWalkT && kLast / 32 == 2 * kWalkWarps, "two survivors per thread, two words per warp");
  uint4 row[2][kLast / 128];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int w = 0; w < kLast / 128; ++w) {
      const int i = tid + h * kWalkT;
      row[h][w] = make_uint4(0u, 0u, 0u, 0u);            // (nothing was written behind the survivor's own place)
      if (i < total && 128 * w < i) {
        const uint4 r = __ldcg(reinterpret_cast<const uint4*>(p.conflict + i * pitch) + w);
        auto before = [&](int word) { const int k = i - 128 * w - 32 * word; return k >= 32 ? kFull : (k <= 0 ? 0u : (1u << k) - 1u); };
        row[h][w] = make_uint4(r.x & before(0), r.y & before(1), r.z & before(2), r.w & before(3));
      }
    }
  unsigned int here = 1u;
#pragma unroll 1
  for (int pass = 0; here != 0u; ++pass) {
    const uint4* und = reinterpret_cast<const uint4*>(s.state[pass & 1][0]);
    const uint4* kep = reinterpret_cast<const uint4*>(s.state[pass & 1][1]);
    unsigned int wait[2] = {0u, 0u}, out[2] = {0u, 0u}, left = 0u;
#pragma unroll
    for (int w = 0; w < kLast / 128; ++w) {
      if (4 * w >= W) break;
      const uint4 u = und[w], k = kep[w];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint4 r = row[h][w];
        wait[h] |= (r.x & u.x) | (r.y & u.y) | (r.z & u.z) | (r.w & u.w);
        out[h] |= (r.x & k.x) | (r.y & k.y) | (r.z & k.z) | (r.w & k.w);
      }
      left |= u.x | u.y | u.z | u.w;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int w = warp + h * kWalkWarps;
      const unsigned int mine = s.state[pass & 1][0][w];
      const unsigned int gone = __ballot_sync(kFull, out[h] != 0u) & mine, fresh = __ballot_sync(kFull, out[h] == 0u && wait[h] == 0u) & mine;
      if (lane == 0) {
        s.state[(pass + 1) & 1][0][w] = mine & ~(gone | fresh);
        s.state[(pass + 1) & 1][1][w] = s.state[pass & 1][1][w] | fresh;
      }
    }
    here = left;
    walk_sync();
  }
  // (the last pass changed nothing: both copies hold the kept ones)
  const int room = p.n_keep - kept;
  int before[2] = {0, 0}, all = 0;
#pragma unroll
  for (int w = 0; w < kLast / 32; ++w) {
    const int c = __popc(s.state[0][1][w]);
#pragma unroll
    for (int h = 0; h < 2; ++h) if (w < warp + h * kWalkWarps) before[h] += c;
    all += c;
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const unsigned int word = s.state[0][1][warp + h * kWalkWarps];
    const int r = before[h] + __popc(word & ((1u << lane) - 1u));
    if (((word >> lane) & 1u) && r < room) {             // stop exactly at P
      const int at = s.survivor[tid + h * kWalkT];
      if (r == room - 1) s.n_free = at;
      if ((kept + r) % n_ctas == cta) { p.kept[kept + r] = p.cand[at]; p.kept_pos[kept + r] = at; }
    }
  }
  walk_sync();
  if (all >= room) examined = s.n_free + 1;
  kept += min(all, room);
  return true;
}

// The columns of all candidates lie where p.walk_cols says (written behind the last barrier's far side).  draw(): what the other
// threads do meanwhile, with the grid barrier g_draw; false: it gave up.  Every CTA leaves the places of the kept list that it
// owns (a mod ctas) and, in *n_kept, their number.  False: a barrier gave up.
// Nobody need have met before: others may still be applying the last round's changes to the residual, or reading how this round is to be
// made, which CTA 0 decides anew at the end.  A walk without a barrier -- its first batch was the last one -- has one there.
template <typename Draw, typename Crew>
__device__ __forceinline__ bool csc_walk_on_demand(const Crew& crew, const Problem& p, Problem& sp, const Engine& e, unsigned char* sm, Grid& g, Grid& g_draw, int* n_kept,
                                                   Draw&& draw) {
  DemandShared& s = *reinterpret_cast<DemandShared*>(sm);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int cta = crew.rank(), n_ctas = crew.size(), n = p.n_cand, W = (n + 31) >> 5;
  // this CTA's words of the mask: cta, cta + n_ctas, ...; its k-th candidate is bit k & 31 of the (k / 32)-th of them
  const int own_words = W > cta ? (W - cta + n_ctas - 1) / n_ctas : 0, n_own = own_words * 32, n_here = min(n_own, kOwn);
  auto own_index = [&](int k) { return ((cta + (k >> 5) * n_ctas) << 5) | (k & 31); };
  const unsigned int begun = g.target;
  __syncthreads();
  if (warp >= kWalkWarps) {
    for (int w = tid - kWalkT; w < own_words; w += kT - kWalkT) s.own_word[w] = s.own_hit[w] = 0u;
    {
      const int i = tid - kWalkT;
      WalkColumn col = {};
      if (i < n_here && own_index(i) < n) col = p.walk_cols[own_index(i)];
      hold_columns<2>(p, s, i, n_here, col, s.orow, s.oval, kOwnEntries, kOwnRows);
    }
    asm volatile("bar.arrive 3, %0;" ::"n"(kT) : "memory");
    const bool drawn = draw();
    if (tid == kWalkT) { s.drawn = drawn; s.draw_target = g_draw.target; }
  } else {
    const double rho = (double)p.rho;
    for (int i = tid; i < kRowSlots / 4; i += kWalkT) reinterpret_cast<int4*>(s.row_key)[i] = make_int4(kFreeRow, kFreeRow, kFreeRow, kFreeRow);
    for (int i = tid; i < kRowSlots / 2; i += kWalkT) reinterpret_cast<uint4*>(s.row_rec)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (tid == 0) { s.longest = 0; s.n_vals = 0; s.n_free = 0; }
    int cursor = 0, kept = 0, examined = n, mask_at = 0;
    bool ok = true, held = false;
#pragma unroll 1
    for (unsigned int batch = 0u;; ++batch) {
      // ---- A: the next <= 32 unblocked candidates at or after the cursor ----
      int total = n;
      bool last = false;
      if (batch == 0u) {
        if (tid < kBatch) s.pos[tid] = tid;
      } else {
        const int first = tid << 6;
        unsigned int f[2] = {0u, 0u};
        if (first + 64 > cursor && first < n) {
          const uint2 b = __ldcg(reinterpret_cast<const uint2*>(p.walk_blocked + mask_at) + tid);
          f[0] = ~b.x; f[1] = ~b.y;
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int at = first + 32 * u;
            if (at + 32 <= cursor || at >= n) f[u] = 0u;
            else {
              if (at < cursor) f[u] &= kFull << (cursor - at);
              if (at + 32 > n) f[u] &= kFull >> (at + 32 - n);
            }
          }
        }
        const int c = __popc(f[0]) + __popc(f[1]);
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_up_sync(kFull, incl, o);
          if (lane >= o) incl += v;
        }
        if (lane == 31) s.wsum[warp] = incl;
        walk_sync();
        int idx = incl - c;
        total = 0;
#pragma unroll
        for (int k = 0; k < kWalkWarps; ++k) { const int v = s.wsum[k]; if (k < warp) idx += v; total += v; }
        if (total == 0) break;                           // list exhausted (the same in every CTA)
        last = total > kBatch && total <= kLast && total <= n_ctas * kBatch && (long long)total * p.nnz <= kLastEntries * p.J;
        int* list = last ? s.survivor : s.pos;
        const int most = last ? kLast : kBatch;
#pragma unroll 1
        for (; (f[0] | f[1]) != 0u && idx < most; ++idx) {
          const int u = f[0] != 0u ? 0 : 1;
          const unsigned int x = u ? f[1] : f[0];
          list[idx] = first + 32 * u + __ffs((int)x) - 1;
          if (u) f[1] &= f[1] - 1u; else f[0] &= f[0] - 1u;
        }
      }
      // (last: the members are this CTA's share of the survivors)
      const int m = !last ? min(kBatch, total) : (total > cta ? (total - cta + n_ctas - 1) / n_ctas : 0);
      walk_sync();
      // ---- B: the members' rows into the table, kPerMember threads each ----
      const int q = tid / kPerMember, l = tid % kPerMember;
      unsigned int slot[kEach];
      float val[kEach];
      {
        WalkColumn col = {};
        if (q < m) col = p.walk_cols[last ? s.survivor[cta + q * n_ctas] : s.pos[q]];
        if (l == 0) {
          s.col[q] = col.j; s.ptr[q] = col.q0; s.n2[q] = col.n2; s.limit[q] = (float)(rho * rho * col.n2); s.len[q] = col.n; s.conf[q] = 0u;
          if (col.n > kColCap) s.longest = col.n;        // (any of them will do)
        }
        const int len = min(col.n, kColCap), turns = (__reduce_max_sync(kFull, len) + kPerMember - 1) / kPerMember;
        int row[kEach], key[kEach];
#pragma unroll
        for (int u = 0; u < kEach; ++u) {
          row[u] = kFreeRow; val[u] = 0.f; slot[u] = kNoSlot;
          if (l + kPerMember * u < len) { row[u] = __ldg(p.xrow + col.q0 + l + kPerMember * u); val[u] = __ldg(p.xv + col.q0 + l + kPerMember * u); }
        }
#pragma unroll
        for (int u = 0; u < kEach; ++u) {                // (all of them under way together; another row in the place is rare)
          if (u >= turns) break;
          if (row[u] != kFreeRow) { slot[u] = row_hash(row[u]); key[u] = atomicCAS(&s.row_key[slot[u]], kFreeRow, row[u]); }
        }
#pragma unroll
        for (int u = 0; u < kEach; ++u) {
          if (u >= turns) break;
          if (row[u] == kFreeRow) continue;
#pragma unroll 1
          while (key[u] != kFreeRow && key[u] != row[u]) {
            slot[u] = (slot[u] + 1u) & (kRowSlots - 1);
            key[u] = atomicCAS(&s.row_key[slot[u]], kFreeRow, row[u]);
          }
          atomicOr(&s.row_rec[slot[u]].x, 1u << q);
        }
      }
      walk_sync();
      const bool table = s.longest == 0;                 // (the same in every CTA, but for the last batch)
      if (!table) {
        if (tid == 0) sp = p;                            // (for the functions that merge)
        walk_sync();
      }
      if (table) {
        // the values of a row side by side, in the order of the members: its first member takes the places
        unsigned int members[kEach];
        int want = 0;
#pragma unroll
        for (int u = 0; u < kEach; ++u) {
          members[u] = slot[u] != kNoSlot ? s.row_rec[slot[u]].x : 0u;
          if ((members[u] & ((1u << q) - 1u)) == 0u) want += __popc(members[u]);
        }
        int incl = want;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_up_sync(kFull, incl, o);
          if (lane >= o) incl += v;
        }
        int at = 0;
        if (lane == 31) at = atomicAdd(&s.n_vals, incl);
        at = __shfl_sync(kFull, at, 31) + incl - want;
#pragma unroll
        for (int u = 0; u < kEach; ++u)
          if (members[u] != 0u && (members[u] & ((1u << q) - 1u)) == 0u) { s.row_rec[slot[u]].y = (unsigned)at; at += __popc(members[u]); }
        walk_sync();
        int n_shared = 0;
        const unsigned int group = ((1u << kPerMember) - 1u) << (lane & ~(kPerMember - 1));
#pragma unroll
        for (int u = 0; u < kEach; ++u) {
          if (!__any_sync(kFull, members[u] != 0u)) break;
          const unsigned int start = members[u] != 0u ? s.row_rec[slot[u]].y : 0u;
          if (members[u] != 0u) s.row_val[start + (unsigned)__popc(members[u] & ((1u << q) - 1u))] = val[u];
          const bool later = (members[u] >> q) > 1u;
          const unsigned int mine = __ballot_sync(kFull, later) & group;
          if (later) s.ent[q][n_shared + __popc(mine & ((1u << lane) - 1u))] = make_uint4(members[u], start, __float_as_uint(val[u]), 0u);
          n_shared += __popc(mine);
        }
        if (l == 0) s.n_shared[q] = n_shared;
        walk_sync();
        // the pairs among them, one per lane: member w with those behind it and member 31 - w likewise
        if (!last) {
#pragma unroll 1
          for (int w = warp; w < kBatch / 2; w += kWalkWarps) {
            const int a = lane > w ? w : kBatch - 1 - w, b = lane > w ? lane : kBatch - 1 - lane;
            const float dot = row_products(s, b, lane == w ? 0 : s.n_shared[a], max(s.n_shared[w], s.n_shared[kBatch - 1 - w]),
                                           [&](int i, uint2& rec, float& v) { const uint4 en = s.ent[a][i]; rec = make_uint2(en.x, en.y); v = __uint_as_float(en.z); });
            if (lane != w && b < m && in_conflict(dot, s.limit[a], s.n2[a], s.n2[b], rho)) atomicOr(&s.conf[b], 1u << a);
          }
        }
      } else if (!last) {
        merge_batch(sp, s, m);
      }
      if (last) {
        ok = settle_rest(crew, p, sp, s, g, total, m, table, kept, examined);
        break;
      }
      walk_sync();
      // ---- C: decide the batch (lane = member; the same in every warp and CTA) ----
      unsigned int keep = 0u;
      {
        const unsigned int earlier = s.conf[lane];
        unsigned int und = m >= 32 ? kFull : ((1u << m) - 1u);
#pragma unroll 1
        while (und != 0u) {                              // (the first undecided one is kept every time)
          const unsigned int fresh = __ballot_sync(kFull, (earlier & (und | keep)) == 0u) & und;
          keep |= fresh;
          und &= ~(fresh | __ballot_sync(kFull, (earlier & fresh) != 0u));
        }
      }
      const int open = p.n_keep - kept;
      const bool done = __popc(keep) >= open;            // stop exactly at P: drop the surplus from the back
      while (__popc(keep) > open) keep &= ~(1u << (31 - __clz((int)keep)));
      if (warp < 2 && ((keep >> lane) & 1u)) {
        const int r = __popc(keep & ((1u << lane) - 1u));
        if (warp == 0) {
          s.kept_q[r] = lane;
        } else if ((kept + r) % n_ctas == cta) {
          p.kept[kept + r] = s.col[lane];
          p.kept_pos[kept + r] = s.pos[lane];
        }
      }
      const int n_new = __popc(keep);
      kept += n_new;
      cursor = s.pos[m - 1] + 1;
      if (done) examined = s.pos[31 - __clz((int)keep)] + 1;
      if (done || total <= kBatch) break;                // P kept: what they block no longer matters; or nobody comes later
      // ---- D: the kept members against this CTA's later unblocked candidates ----
      mask_at = walk_mask_at(batch, p.mask_words);
      if (!held) { held = true; asm volatile("bar.sync 3, %0;" ::"n"(kT) : "memory"); }        // their columns are there
      const bool values = s.own_at[n_here] <= kOwnEntries;
      const int room = values ? kOwnEntries : kOwnRows;
      unsigned int* omet = values ? s.omet : s.only_met;
      for (int k0 = 0; k0 < n_own; k0 += kOwn) {         // (a turn of at most kOwn candidates; one turn as a rule)
        if (k0 > 0) { walk_sync(); if (tid == 0) s.n_free = 0; walk_sync(); }
        for (int k = k0 + tid; k < min(n_own, k0 + kOwn); k += kWalkT) {
          const int b = own_index(k);
          if (b < n && b >= cursor && !((s.own_word[k >> 5] >> (k & 31)) & 1u)) s.own_free[atomicAdd(&s.n_free, 1)] = k;
        }
        walk_sync();
        const int n_free = s.n_free;
        if (table && k0 == 0) {                          // their entries in rows of kept members
          int share = 5;                                 // threads per candidate
          while (share > 0 && (n_free << share) > kWalkT) --share;
          const int c = tid >> share, sub = tid & ((1 << share) - 1);
          const unsigned int group = (share == 5 ? kFull : ((1u << (1 << share)) - 1u)) << (lane - sub);
          int k = 0, from = 0, end = 0, met = 0;
          if (c < n_free) {
            k = s.own_free[c]; from = s.own_at[k]; end = s.own_at[k + 1];
            if (end > room) end = from;
          }
#pragma unroll 1
          for (int i0 = from + sub; __any_sync(kFull, i0 < end + sub); i0 += 4 << share) {
            int row[4];
            unsigned int sl[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) row[u] = i0 + (u << share) < end ? s.orow[i0 + (u << share)] : kFreeRow;
            find_rows<4>(s, row, keep, sl);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const unsigned int mine = __ballot_sync(kFull, sl[u] != kNoSlot) & group;
              if (sl[u] != kNoSlot) omet[from + met + __popc(mine & ((1u << lane) - 1u))] = sl[u] | (unsigned)(i0 + (u << share) - from) << 16;
              met += __popc(mine);
            }
          }
          if (c < n_free && sub == 0) s.n_met[k] = met;
          walk_sync();
        }
        const unsigned int per = ((1u << 20) + (unsigned)n_new - 1u) / (unsigned)n_new;        // i / n_new = i per >> 20 (i < 2^13, n_new <= 32)
        for (int i = tid; i < n_free * n_new; i += kWalkT) {
          const int c = (int)((unsigned)i * per >> 20), qk = s.kept_q[i - c * n_new], k = s.own_free[c];
          float dot = 0.f;
          double n2b;
          if (table && k < kOwn && s.own_at[k + 1] <= room) {
            n2b = s.own_n2[k];
            if (values) {
              const int met = s.n_met[k], from = s.own_at[k];
              dot = row_products(s, qk, met, met, [&](int x, uint2& rec, float& v) {
                const unsigned int en = s.omet[from + x];
                rec = s.row_rec[en & 0xffffu]; v = s.oval[from + (int)(en >> 16)];
              });
            } else {
              dot = fetched_products(s, p.xv, k, qk);
            }
          } else if (table) {                            // (no room for its column)
            const WalkColumn cb = p.walk_cols[own_index(k)];
            n2b = cb.n2;
            dot = column_products(p.xrow + cb.q0, p.xv + cb.q0, cb.n, s, qk);
          } else {
            const WalkColumn cb = p.walk_cols[own_index(k)];
            n2b = cb.n2;
            dot = merge_columns(sp, s.ptr[qk], s.len[qk], cb.q0, cb.n);
          }
          if (in_conflict(dot, s.limit[qk], s.n2[qk], n2b, rho)) atomicOr(&s.own_hit[k >> 5], 1u << (k & 31));
        }
      }
      walk_sync();
      for (int w = tid; w < own_words; w += kWalkT) {    // the words as they are now
        const unsigned int v = s.own_word[w] | s.own_hit[w];
        s.own_word[w] = v;
        s.own_hit[w] = 0u;
        p.walk_blocked[mask_at + cta + w * n_ctas] = v;
      }
      // the table as the next batch expects it
#pragma unroll
      for (int u = 0; u < kEach; ++u)
        if (slot[u] != kNoSlot) { s.row_key[slot[u]] = kFreeRow; s.row_rec[slot[u]].x = 0u; }
      if (tid == 0) { s.longest = 0; s.n_vals = 0; s.n_free = 0; }
      if (!(ok = walk_barrier(s, g))) break;
    }
    if (!held) asm volatile("bar.sync 3, %0;" ::"n"(kT) : "memory");
    if (ok && walk_to_meet(begun, g.target)) ok = walk_barrier(s, g);
    if (tid == 0) {
      s.kept = kept; s.ok = ok; s.target = g.target;
      if (cta == 0 && ok) {
        EngineState* es = e.es;
        es->n_kept = kept; es->n_examined = examined; es->walk_open = 0;
        if (es->avoid > 0) es->avoid -= 1;
        if (e.window < n) es->skip_window = kept == p.n_keep && examined <= e.window ? 0 : 1;
      }
    }
  }
  __syncthreads();
  g.target = s.target; g_draw.target = s.draw_target;
  *n_kept = s.kept;
  return s.ok != 0 && s.drawn != 0;
}

// The walk from the list of the window's conflicting pairs, by every CTA for itself with half its threads -- what it needs is in L2 for all of
// them behind the barrier, and nobody then waits for one of them -- while the others do what else there is (`meanwhile`).  The kept
// candidates' positions go to kept_at (shared memory, not among the walk's own); whoever fetches their columns leaves the lists in global memory.
// All threads of the CTA; settle_note makes the notes behind a barrier.
struct WalkThreads {
  static constexpr int kN = kWalkT;
  static __device__ __forceinline__ void sync() { asm volatile("bar.sync 1, %0;" ::"n"(kN) : "memory"); }
  static __device__ __forceinline__ bool any(int x) {
    int r;
    asm volatile("{ .reg .pred p, q; setp.ne.s32 p, %1, 0; bar.red.or.pred q, 1, %2, p; selp.s32 %0, 1, 0, q; }" : "=r"(r) : "r"(x), "n"(kN) : "memory");
    return r != 0;
  }
};
struct Settled { int kept, examined, settled; };
// Where kept_at can lie: behind the walk's own, and behind step 4's (`changes` bytes).
__host__ __device__ inline size_t kept_at_offset(const Problem& p, size_t changes) {
  const size_t walk = walk_pairs_smem(p.n_cand, (unsigned)p.cap_edges);
  return ((walk > changes ? walk : changes) + 15) & ~(size_t)15;
}
template <typename F>
__device__ __forceinline__ void csc_settle(const Problem& p, const Engine& e, unsigned char* sm, unsigned short* kept_at, Settled& out, int n,
                                           F&& meanwhile) {
  const int tid = threadIdx.x;
  __syncthreads();                                       // (what lay there before)
  if (tid >= kWalkT) {
    meanwhile();
  } else {
    const unsigned int edges = e.es->edge_count;
    const int failed = e.es->bucket_failed;
    if (tid == 0) { out.kept = 0; out.examined = n; }
    WalkThreads::sync();
    bool settled = !failed && edges <= (unsigned)p.cap_edges;
    if (settled)
      settled = walk_pairs<WalkThreads>(p, nullptr, n, edges, sm, &out.kept, &out.examined, [&](int a, int i, int) { kept_at[a] = (unsigned short)i; });
    if (tid == 0) out.settled = settled;
  }
  __syncthreads();
}
__device__ __forceinline__ bool walk_is_open(const Problem& p, const Settled& w, int n) { return !w.settled || (w.kept < p.n_keep && n < p.n_cand); }
// One thread, when everybody has read what it changes.
__device__ __forceinline__ void settle_note(const Engine& e, const Settled& w) {
  EngineState* es = e.es;
  // after an overflow the buckets are left alone: for a round, then twice as long after every further one, to 64
  // (a count of rounds, not the round to wait for: strads_set_round may go back); this round's walk counts too
  if (!w.settled) es->avoid = 1 + (1 << es->streak);
  es->streak = w.settled ? 0 : min(es->streak + 1, 6);
  es->bucket_failed = 0; es->edge_count = 0u;
}

// The walk over all candidates by half the warps, with `draws` the draw of round td up to the collection of its k winners by the
// others.  False: a barrier gave up.
template <typename Crew>
__device__ __forceinline__ bool csc_walk_and_draw(const Crew& crew, const Problem& p, Problem& sp, const Engine& e, DrawShared& ds, unsigned char* sm, Grid& g,
                                                  Grid& g_draw, bool draws, unsigned long long td, unsigned int k, int* n_kept) {
  const int warp = (int)threadIdx.x >> 5;
  unsigned char* sm_scan = sm + sizeof(DemandShared);
  unsigned int* sh = reinterpret_cast<unsigned int*>(sm_scan);
  const float cut = draws ? scan_open(crew, e, ds, sm_scan, true) : 0.f;
  const Binning bins = binning_of(cut);
  const WeightForm wf = weight_form(p);
  auto draw = [&]() {
    if (!draws) return true;
    WarpScan scan = begin_scan(cut, scan_queue(sm_scan), (warp - kWalkWarps) * crew.size() + crew.rank(), (kWarps - kWalkWarps) * crew.size());
    scan_all<Crew::kParts>(p, td, wf, scan, [&](unsigned long long key, bool on) { scan_found(crew, e, ds, sh, bins, key, on); });
    scan_close<OtherThreads>(crew, e, ds, sm_scan);
    __shared__ int s_over;
    g_draw.target += g_draw.n;
    OtherThreads::sync();
    if (OtherThreads::tid() == 0) s_over = grid_wait(g_draw);
    OtherThreads::sync();
    if (!s_over) return false;
    draw_gather<OtherThreads>(crew, p, e, ds, k, false);
    return true;
  };
  return csc_walk_on_demand(crew, p, sp, e, sm, g, g_draw, n_kept, draw);
}

}  // namespace
}  // namespace strads
