// Whole rounds of Algorithm 1 in one cooperative launch: one CTA of 512 threads per SM, the steps of a round
// separated by a grid barrier instead of by kernel boundaries.
//
// A round is a chain of short dependent steps over a few MB at most, so what bounds it is the number of times the
// whole grid has to hand over to itself and what every hand-over costs.  As separate launches a round took 11 to 17
// kernels, each with its launch, its ramp and the drain of the one before; here it takes four barriers of 2 to 3 us, and the
// draw of the next round runs in the shadow of the steps of this one:
//
//   step           dense                                          CSC
//   1  (all CTAs)  BF16 copies of the candidates' columns,        last round's residual applied; candidates entered
//                  x_c^T r and would-be changes; scan of the      into the row buckets; scan of the keys of round t + 1
//                  keys of round t + 1
//   2  (all CTAs)  Gram tiles on the tensor cores, then the      inner products from the buckets, x_c^T r and would-be
//                  pairs they leave open                          changes
//  (2b)            open pairs that their CTA had no room for
//   3              greedy walk (last CTA); keys of round t + 1    greedy walk by half the threads of every CTA; buckets emptied,
//                  below the boundary collected (the others)      keys of round t + 1 collected by the others
//  (3b)            all candidates instead of the window           walk over all candidates with conflict rows on demand by half the
//                                                                 warps, the draw of round t + 1 by the others
//   4  (all CTAs)  residual, beta, delta; the winners of the draw ranked, corrected for this round's changes
//
// Drawing ahead is exact: the draw of round t + 1 collects the P' + P smallest keys by the priorities of round t's
// start; the update changes at most P priorities, so every candidate of round t + 1 that is not one of those is among
// them, and its rank follows from its rank in the early list, the old keys of the changed coefficients below it and
// their new keys below it.
//
// The results are those of the kernels used one by one (split-phase calls): same keys, same order of the FP64 sums of
// CSC columns, same decisions; dense inner products are pairs of floats as in the pack kernel, in another order.
// No floating-point atomics.  Every barrier wait has an iteration limit (STRADS_STATUS_WAIT_EXPIRED).
#include <cuda.h>
#include <cuda_bf16.h>

#include "engine_csc.cuh"

namespace strads {
namespace {

struct RoundOutputs { int* cand; int* kept; float* dbeta; int* counts; };

__device__ void commit_changes(const Problem& p, int examined, int nk, int n_moving, const RoundOutputs& out, bool last) {
  const int tid = threadIdx.x;
  DeviceState* st = p.st;
  for (int a = tid * (int)gridDim.x + (int)blockIdx.x; a < p.n_keep; a += kT * (int)gridDim.x) {
    float d32 = 0.f;
    int j = -1;
    if (a < nk) {
      const int pos = p.kept_pos[a];
      const double d = p.cand_dbeta64[pos];
      j = p.kept[a];
      p.beta[j] = p.cand_bnew[pos];
      p.delta[j] = (float)fabs(d);
      d32 = (float)d;
      if (!isfinite(d)) atomicOr(&st->status, STRADS_STATUS_NONFINITE);
    }
    p.dbeta[a] = d32;
    if (a >= nk) p.kept[a] = -1;
    if (last && out.kept != nullptr) out.kept[a] = j;
    if (last && out.dbeta != nullptr) out.dbeta[a] = d32;
  }
  if (last && out.cand != nullptr)                       // (the candidates of this round; the draw ahead would overwrite them)
    for (int i = tid * (int)gridDim.x + (int)blockIdx.x; i < p.n_cand; i += kT * (int)gridDim.x) out.cand[i] = p.cand[i];
  if (blockIdx.x == 0 && tid == 0) {
    st->counts[0] = p.n_cand; st->counts[1] = examined; st->counts[2] = nk; st->counts[3] = n_moving;
    if (last && out.counts != nullptr) { out.counts[0] = p.n_cand; out.counts[1] = examined; out.counts[2] = nk; out.counts[3] = n_moving; }
    st->totals[0] += 1; st->totals[1] += (unsigned)examined; st->totals[2] += (unsigned)nk; st->totals[3] += (unsigned)n_moving;
    st->round += (unsigned long long)p.part_count;
  }
}

// ------------------------------------------------------------------------------------------------
// Dense, step 1: BF16 copies of the candidates' columns (operands of the Gram's screen), x_c^T r and the would-be
// changes.  Candidate lo + cta + k * ctas is the CTA's k-th; `group` warps share a column (a function of N alone, so
// that a product's bits do not depend on the number of candidates).
//
// The candidates are scattered over X (a page each), so what counts is how much is under way per SM: the columns come
// into shared memory by bulk copies, up to four whole columns of a group ahead, instead of through registers trip by trip.
// Every thread holds its rows of r in registers for the whole step.  1,024 candidates of 463 rows: 3.6 us (their columns
// were prefetched into L2 when they were ranked).
// ------------------------------------------------------------------------------------------------
struct PackBars { unsigned long long full[kWarps]; unsigned int uses[kWarps]; };

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint32_t limit) {
  for (uint32_t it = 0; it < limit; ++it) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    if (ok) return true;
  }
  return false;
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// acc += x * r with acc = hi + lo a pair of floats, product and sum errors kept exactly: ~2^-46 of the summed magnitudes.
__device__ __forceinline__ void dot_step(float x, float r, float& hi, float& lo) {
  const float pr = __fmul_rn(x, r);
  const float pe = __fmaf_rn(x, r, -pr);
  const float s = __fadd_rn(hi, pr);
  const float bb = __fsub_rn(s, hi);
  const float se = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(pr, bb));
  hi = s;
  lo = __fadd_rn(lo, __fadd_rn(se, pe));
}

__device__ __forceinline__ unsigned int bf16x2_bits(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const unsigned int*>(&v);
}
__device__ __forceinline__ float bf16_residue(float x) { return x - __bfloat162float(__float2bfloat16_rn(x)); }
__device__ __forceinline__ void store_parts(uint2* bhi, uint2* blo, const float4& x) {
  *bhi = make_uint2(bf16x2_bits(x.x, x.y), bf16x2_bits(x.z, x.w));
  *blo = make_uint2(bf16x2_bits(bf16_residue(x.x), bf16_residue(x.y)), bf16x2_bits(bf16_residue(x.z), bf16_residue(x.w)));
}

constexpr int kHeld = 4;                   // groups of four rows of r a thread holds: a group has a lane per 16 rows or more (pack_group)
constexpr size_t kPackSmem = 160 * 1024;

__device__ __forceinline__ int pack_group(int n4) {
  int group = 1;
  while (group < kWarps && n4 >= group * 2 * 64) group *= 2;            // (at least two 16-byte groups per lane)
  return group;
}

// Four rows of r from group gi on; zero past the end.
__device__ __forceinline__ float4 resid4(const Problem& p, int gi, int n4, int n4_whole) {
  float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
  if (gi < n4_whole) {
    r = reinterpret_cast<const float4*>(p.resid)[gi];
  } else if (gi < n4) {
    const long long i = (long long)gi << 2;
    r.x = p.resid[i];
    if (i + 1 < p.N) r.y = p.resid[i + 1];
    if (i + 2 < p.N) r.z = p.resid[i + 2];
  }
  return r;
}
// Rows past N do not exist (the padding of a column may hold anything).
__device__ __forceinline__ void mask_rows(const Problem& p, int gi, float4& x) {
  const long long i = (long long)gi << 2;
  if (i + 1 >= p.N) x.y = 0.f;
  if (i + 2 >= p.N) x.z = 0.f;
  x.w = 0.f;
}

__device__ void dense_pack(const Problem& p, const Engine& e, unsigned char* sm, TurnShared& ts, PackBars& bars, int lo, int hi,
                           unsigned long long t_next, bool want_keys, uint32_t wait_limit) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int cta = (int)blockIdx.x, n_ctas = (int)gridDim.x;
  const int n4 = (int)((p.N + 3) >> 2), n4_whole = (int)(p.N >> 2);
  const int group = pack_group(n4), part = warp & (group - 1), grp = warp / group, groups = kWarps / group;
  const int mine = hi - lo > cta ? (hi - lo - cta + n_ctas - 1) / n_ctas : 0;
  // columns of a group under way at once
  const uint32_t col_bytes = (uint32_t)n4 * 16u;
  int depth = (int)min((size_t)4, kPackSmem / ((size_t)groups * col_bytes));
  depth = min(depth, kWarps / groups);                   // (a barrier per column under way)
  const uint32_t slots = smem_u32(sm) + (uint32_t)(grp * depth) * col_bytes;
  const int at0 = part * 32 + lane, step = 32 * group;
  float4 rv[kHeld];
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");           // what this CTA last did with the slots is over
  __syncthreads();
  if (part == 0 && lane == 0)
    for (int i = 0; i < depth && grp + i * groups < mine; ++i) {
      const uint32_t bar = smem_u32(&bars.full[grp * depth + i]);
      mbar_expect(bar, col_bytes);
      bulk_load(slots + (uint32_t)i * col_bytes, p.xv + (long long)p.cand[lo + cta + n_ctas * (grp + i * groups)] * p.ld, col_bytes, bar);
    }
#pragma unroll
  for (int u = 0; u < kHeld; ++u) rv[u] = u * step + at0 < n4 ? resid4(p, u * step + at0, n4, n4_whole) : make_float4(0.f, 0.f, 0.f, 0.f);
  int seen = 0;                                          // columns this group has been through
  for (int k0 = 0; k0 < mine; k0 += kTurn) {
    const int turn = min(kTurn, mine - k0);
    // what the end of the turn needs of a candidate, by the lanes of the last warp
    int j_own = 0;
    float E = 0.f;
    Proposal prop = {};
    bool dormant = false;
    if (warp == kWarps - 1 && lane < turn) {
      j_own = p.cand[lo + cta + n_ctas * (k0 + lane)];
      const double n_own = p.n2[j_own];
      const float b_own = p.beta[j_own], d_own = p.delta[j_own];
      if (want_keys) E = exponential_of(p, t_next, (uint32_t)j_own);
      prop = propose_begin(p, j_own, n_own, b_own, d_own, E, want_keys);
      dormant = (p.flags & STRADS_FLAG_DYNAMIC_DEPS) && b_own == 0.f && d_own == 0.f;      // (coupling_n2)
    }
    int k = seen * groups + grp - k0;                    // this group's next column, counted from the turn's first
    for (; k < turn; k += groups, ++seen) {
      const int a = lo + cta + n_ctas * (k0 + k);
      uint2* bhi = reinterpret_cast<uint2*>(e.xb + (long long)a * e.xb_pitch);
      uint2* blo = reinterpret_cast<uint2*>(e.xb + (long long)a * e.xb_pitch + e.lo_off);
      float h0 = 0.f, l0 = 0.f, h1 = 0.f, l1 = 0.f;
      const int slot = seen % depth, b = grp * depth + slot;
      const uint32_t ph = (bars.uses[b] + (unsigned)(seen / depth)) & 1u;
      if (!mbar_wait(smem_u32(&bars.full[b]), ph, wait_limit) && lane == 0) atomicOr(&p.st->status, STRADS_STATUS_WAIT_EXPIRED);
      const uint32_t src = slots + (uint32_t)slot * col_bytes;
#pragma unroll
      for (int u = 0; u < kHeld; ++u) {
        const int gi = u * step + at0;
        if (gi >= n4) break;
        float4 x;
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w) : "r"(src + (uint32_t)gi * 16u) : "memory");
        if (gi >= n4_whole) mask_rows(p, gi, x);
        store_parts(bhi + gi, blo + gi, x);
        dot_step(x.x, rv[u].x, h0, l0); dot_step(x.y, rv[u].y, h1, l1);
        dot_step(x.z, rv[u].z, h0, l0); dot_step(x.w, rv[u].w, h1, l1);
      }
      const int nxt = grp + (seen + depth) * groups;   // the column that comes into this slot next
      if (nxt < mine) {
        if (group > 1) asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "r"(32 * group) : "memory");
        else __syncwarp();
        if (part == 0 && lane == 0) {
          const uint32_t bar = smem_u32(&bars.full[b]);
          mbar_expect(bar, col_bytes);
          bulk_load(src, p.xv + (long long)p.cand[lo + cta + n_ctas * nxt] * p.ld, col_bytes, bar);
        }
      }
      const double v = warp_sum(((double)h0 + (double)l0) + ((double)h1 + (double)l1));
      if (lane == 0) ts.dot[k][part] = v;
    }
    __syncthreads();
    if (warp == kWarps - 1 && lane < turn) {
      const int a = lo + cta + n_ctas * (k0 + lane);
      double gsum = 0.0;
      for (int w = 0; w < group; ++w) gsum += ts.dot[lane][w];
      e.norm[a] = dormant ? 0.0 : sqrt(prop.n);
      propose_end(p, prop, a, j_own, gsum, E, want_keys);
    }
    __syncthreads();
  }
  __syncthreads();
  if (part == 0 && lane == 0)                            // every slot's barrier has completed this many more phases
    for (int i = 0; i < depth; ++i) bars.uses[grp * depth + i] += (unsigned)((seen - i + depth - 1) / depth);
  // the copies are read by bulk tensor copies (another proxy) behind the next barrier
  asm volatile("fence.proxy.async;" ::: "memory");
}

// ------------------------------------------------------------------------------------------------
// Dense, step 2: conflict bits of all candidate pairs on the tensor cores: tiles of 128 rows x 64 or 128 columns of the
// lower triangle, BF16 operands by TMA (128-byte swizzle) into a ring in shared memory, tcgen05.mma into tensor memory.
// As in gram_dense_tc.cu the result is a screen: pairs closer to rho than its error bound go to a list and are decided
// from exact products.  The columns are short, so their correlations scatter widely (standard deviation N^-1/2) and the
// error band of a product of BF16 roundings (2^-8) would leave percents of all pairs open: three products, hi.hi + hi.lo
// + lo.hi, off by at most 3 * 2^-18.
// What bounds it is bringing operands from L2 to shared memory (~110 GB/s an SM), so K is split until every CTA has a
// share; the CTAs of a tile leave their partial sums in global memory, wait for one another (they all run at once) and
// each adds up and thresholds its share of the rows.  A tile of 128 columns reads fewer operand bytes per product, one
// of 64 leaves half the partial sums: gram_plan takes the cheaper.
// ------------------------------------------------------------------------------------------------
constexpr int kRowsT = kGramRows;                        // rows of a tile
constexpr int kRingBytes = 192 * 1024;
constexpr int kMaxStages = 4;
constexpr size_t kGramSmem = (size_t)kRingBytes + 1024;
constexpr uint32_t kTmemCols = 128;

// A stage holds the high and the low parts of 64 elements of K for both operands.  Its size depends on the tile's width alone, so there is a set of barriers per width.
constexpr unsigned int kOwnOpen = 64;                    // open pairs of its own that a CTA decides itself (a warp each)
struct GramShared {
  unsigned long long full[2][kMaxStages], empty[2][kMaxStages], done;
  uint32_t tmem;
  int abort_;
  double norm_a[kRowsT], norm_b[128];
  float norm_af[kRowsT], norm_bf[128];
  unsigned int n_open, open[kOwnOpen];
};
// Phases of the barriers so far (the same in all threads of a CTA).
struct GramCount { unsigned int stages[2], units; };

// Conflict bits here: a candidate's with all earlier ones, as the walk wants them.  Four words (128 earlier candidates) of
// consecutive candidates lie side by side, so that a warp whose lanes want a candidate each reads whole lines.
__device__ __forceinline__ unsigned int* conflict_word(const Problem& p, int a, int w) { return p.conflict + ((size_t)(w >> 2) * p.n_cand + a) * 4 + (w & 3); }

__device__ __forceinline__ double engine_band(long long N) { return 1.0 / 32768.0 + 3.0 * (double)N * (1.0 / 33554432.0); }

__device__ __forceinline__ void tma_box(uint32_t dst, const void* tmap, int x, int y, uint32_t bar) {
  asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
               ::"r"(dst), "l"(tmap), "r"(x), "r"(y), "r"(bar) : "memory");
}
// K-major operand, rows of 128 bytes with the 128-byte swizzle, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t operand_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
               ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_load16(uint32_t addr, uint32_t (&v)[16]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]),
                 "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]) : "r"(addr) : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Exact decision of one pair by a warp.
__device__ __forceinline__ void decide_exactly(const Problem& p, const Engine& e, int a, int b) {
  const int lane = threadIdx.x & 31;
  const float* xa = p.xv + (long long)p.cand[a] * p.ld;
  const float* xb = p.xv + (long long)p.cand[b] * p.ld;
  const int n4 = (int)(p.N >> 2);
  double acc = 0.0;
  for (int g = lane; g < n4; g += 32) {
    const float4 u = __ldg(reinterpret_cast<const float4*>(xa) + g), w = __ldg(reinterpret_cast<const float4*>(xb) + g);
    acc += (double)u.x * w.x + (double)u.y * w.y + (double)u.z * w.z + (double)u.w * w.w;
  }
  const long long i = ((long long)n4 << 2) + lane;
  if (i < p.N) acc += (double)xa[i] * xb[i];
  acc = warp_sum(acc);
  if (lane == 0) {
    const double den = e.norm[a] * e.norm[b];
    if (den > 0.0 && fabs(acc) >= (double)p.rho * den) atomicOr(conflict_word(p, a, b >> 5), 1u << (b & 31));
  }
}

__device__ __forceinline__ void dense_gram(const Problem& p, const Engine& e, const GramPlan& pl, const void* tmap_rows, const void* tmap_cols,
                                           unsigned char* sm, GramShared& gs, GramCount& gc, int n, unsigned int* amb_count,
                                           uint32_t wait_limit) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int units = pl.tiles * pl.split;
  if ((int)blockIdx.x >= units) return;
  const int set = pl.cols == 128 ? 1 : 0;
  const uint32_t a_bytes = kRowsT * 128, b_bytes = (uint32_t)pl.cols * 128, stage_bytes = 2u * (a_bytes + b_bytes);
  const unsigned int stages = set ? 3u : 4u;
  const uint32_t ring = (smem_u32(sm) + 1023u) & ~1023u;
  float* tile_sm = reinterpret_cast<float*>(sm + (ring - smem_u32(sm)));   // the finished tile (no split), over the ring
  const double rho = (double)p.rho, band = engine_band(p.N);
  const float quick = (float)((rho - band) * 0.99999);   // |g| below quick ||a|| ||b||: certainly no conflict
  const int cols4 = pl.cols >> 2, cols_log = set ? 7 : 6;
  if (tid == 0) gs.n_open = 0u;                          // (used behind a barrier of the CTA)

  for (int unit = (int)blockIdx.x; unit < units; unit += (int)gridDim.x) {
    const int tile = unit / pl.split, sp = unit - tile * pl.split;
    int ri = 0, rem = tile, len = kRowsT >> cols_log;    // row block i meets the column blocks that start before its end
    while (rem >= min(len, pl.col_blocks)) { rem -= min(len, pl.col_blocks); len += kRowsT >> cols_log; ++ri; }
    const int row0 = ri * kRowsT, col0 = rem << cols_log;
    const int s0 = min(pl.steps, sp * pl.per), count = min(pl.steps, s0 + pl.per) - s0;
    const unsigned int slot0 = gc.stages[set] % stages, ph0 = (gc.stages[set] / stages) & 1u;
    if (warp == 0) {
      // ---- operands (one lane) ----
      if (lane == 0) {
        unsigned int slot = slot0, ph = ph0;
        const int x_step = 64, second = (int)e.lo_off;
        int x = s0 * x_step;
#pragma unroll 1
        for (int st = 0; st < count; ++st, x += x_step) {
          if (!mbar_wait(smem_u32(&gs.empty[set][slot]), ph ^ 1u, wait_limit)) {
            gs.abort_ = 1; atomicOr(&p.st->status, STRADS_STATUS_WAIT_EXPIRED);
            break;
          }
          const uint32_t bar = smem_u32(&gs.full[set][slot]), dst = ring + slot * stage_bytes;
          mbar_expect(bar, stage_bytes);
          tma_box(dst, tmap_rows, x, row0, bar);
          tma_box(dst + 2 * a_bytes, set ? tmap_rows : tmap_cols, x, col0, bar);
          tma_box(dst + a_bytes, tmap_rows, x + second, row0, bar);
          tma_box(dst + 2 * a_bytes + b_bytes, set ? tmap_rows : tmap_cols, x + second, col0, bar);
          if (++slot == stages) { slot = 0; ph ^= 1u; }
        }
      }
      __syncwarp();
    } else if (warp == 1) {
      // ---- multiplication (one lane): FP32 accumulator, both operands BF16 and K-major, M = 128, N = cols ----
      if (lane == 0) {
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(pl.cols >> 3) << 17) | ((uint32_t)(kRowsT >> 4) << 24);
        const uint32_t tmem = gs.tmem;
        unsigned int slot = slot0, ph = ph0;
        uint32_t acc = 0u;
#pragma unroll 1
        for (int st = 0; st < count; ++st) {
          if (*(volatile int*)&gs.abort_ || !mbar_wait(smem_u32(&gs.full[set][slot]), ph, wait_limit)) {
            gs.abort_ = 1; atomicOr(&p.st->status, STRADS_STATUS_WAIT_EXPIRED);
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t sb = ring + slot * stage_bytes;
          const uint64_t a0 = operand_desc(sb), a1 = operand_desc(sb + a_bytes);
          const uint64_t b0 = operand_desc(sb + 2 * a_bytes), b1 = operand_desc(sb + 2 * a_bytes + b_bytes);
#pragma unroll
          for (uint64_t o = 0; o < 8; o += 2) {          // 16 elements of K per instruction
            mma_f16(tmem, a0 + o, b0 + o, idesc, acc);
            acc = 1u;
            mma_f16(tmem, a0 + o, b1 + o, idesc, 1u);
            mma_f16(tmem, a1 + o, b0 + o, idesc, 1u);
          }
          mma_commit(smem_u32(&gs.empty[set][slot]));
          if (++slot == stages) { slot = 0; ph ^= 1u; }
        }
        mma_commit(smem_u32(&gs.done));
      }
      __syncwarp();
    } else if (tid >= 256) {                             // the norms of the tile, meanwhile
      const int i = tid - 256;
      if (i < kRowsT) {
        const double v = row0 + i < n ? e.norm[row0 + i] : 0.0;
        gs.norm_a[i] = v; gs.norm_af[i] = (float)v;
      } else if (i - kRowsT < pl.cols) {
        const double v = col0 + i - kRowsT < n ? e.norm[col0 + i - kRowsT] : 0.0;
        gs.norm_b[i - kRowsT] = v; gs.norm_bf[i - kRowsT] = (float)v;
      }
    }
    const bool ok = mbar_wait(smem_u32(&gs.done), gc.units & 1u, wait_limit);
    if (!ok && lane == 0) { gs.abort_ = 1; atomicOr(&p.st->status, STRADS_STATUS_WAIT_EXPIRED); }
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    gc.stages[set] += (unsigned)count;
    gc.units += 1u;
    {
      // warp w reads the rows of its quarter of tensor memory, 16 columns at a time
      const int row = (warp & 3) * 32 + lane;
#pragma unroll 1
      for (int c = (warp >> 2) * 16; c < pl.cols; c += 64) {
        uint32_t v[16];
        if (count > 0) {
          tmem_load16(gs.tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c, v);
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = 0u;
        }
        // into shared memory, where the operands were; group q of four columns of row r lies at q ^ (r & 15): no bank conflicts
        // either way
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int q = ((c >> 2) + i) ^ (row & 15);
          *reinterpret_cast<uint4*>(tile_sm + (row << cols_log) + 4 * q) = make_uint4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    }
    int r_lo = 0, r_hi = kRowsT;
    __syncthreads();
    if (pl.split > 1) {
      // as it lies there to global memory (from the accumulator's registers each thread would touch lines of its own row only:
      // 4,096 of them, 2 us)
      uint4* dst = reinterpret_cast<uint4*>(e.part + (size_t)unit * (kRowsT * 128));
#pragma unroll 4
      for (int i = tid; i < kRowsT * cols4; i += kT) __stcg(dst + i, *reinterpret_cast<const uint4*>(tile_sm + 4 * i));
      __syncthreads();
      if (tid == 0) {                                    // wait for the other parts of the tile
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(e.tile_ticket + tile) : "memory");
        unsigned int v = 0u;
        uint32_t it = 0u;
        do {
          asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(e.tile_ticket + tile) : "memory");
        } while (v < (unsigned)pl.split && ++it < wait_limit);
        if (v < (unsigned)pl.split) atomicOr(&p.st->status, STRADS_STATUS_WAIT_EXPIRED);
      }
      r_lo = sp * kRowsT / pl.split;
      r_hi = (sp + 1) * kRowsT / pl.split;
      __syncthreads();
    }
    const int total = (r_hi - r_lo) * cols4;
#pragma unroll 1
    for (int i0 = 0; i0 < total; i0 += kT) {
      const int i = i0 + tid;
      const bool in = i < total;
      const int r = r_lo + ((in ? i : 0) >> (cols_log - 2)), q = i & (cols4 - 1);
      float4 g4 = make_float4(0.f, 0.f, 0.f, 0.f);
      if (pl.split > 1) {
        const float4* src = reinterpret_cast<const float4*>(e.part + (size_t)tile * pl.split * (kRowsT * 128) + (r << cols_log)) + (q ^ (r & 15));
        for (int k0 = 0; k0 < pl.split; k0 += 4) {       // in split order
          float4 u[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) u[k] = in && k0 + k < pl.split ? __ldcg(src + (size_t)(k0 + k) * (kRowsT * 128 / 4)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int k = 0; k < 4; ++k) { g4.x += u[k].x; g4.y += u[k].y; g4.z += u[k].z; g4.w += u[k].w; }
        }
      } else if (in) {
        g4 = *reinterpret_cast<const float4*>(tile_sm + (r << cols_log) + 4 * (q ^ (r & 15)));
      }
      const int a = row0 + r, b0 = col0 + 4 * q;
      const float gv[4] = {g4.x, g4.y, g4.z, g4.w};
      const float lim = quick * gs.norm_af[r];
      bool near = false;
#pragma unroll
      for (int c = 0; c < 4; ++c) near |= fabsf(gv[c]) >= lim * gs.norm_bf[4 * q + c];
      unsigned int hits = 0u, open = 0u;
      if (in && near) {
        const double norm_a = gs.norm_a[r];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const double den = norm_a * gs.norm_b[4 * q + c], gx = fabs((double)gv[c]);
          const bool live = den > 0.0 && b0 + c < a;
          if (live && fabs(gx - rho * den) <= band * den) open |= 1u << c;
          else if (live && gx >= rho * den) hits |= 1u << c;
        }
      }
      unsigned int word = hits << ((lane & 7) * 4);      // eight lanes make one word of the row's bits
      word |= __shfl_xor_sync(kFull, word, 1);
      word |= __shfl_xor_sync(kFull, word, 2);
      word |= __shfl_xor_sync(kFull, word, 4);
      if (in && (lane & 7) == 0 && a < n && (b0 >> 5) < p.mask_words) *conflict_word(p, a, b0 >> 5) = word;
      if (__any_sync(kFull, open)) {                     // too close to call: listed
        const int cnt = __popc(open);
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int u = __shfl_up_sync(kFull, incl, o);
          if (lane >= o) incl += u;
        }
        unsigned int at = 0u;
        if (lane == 31) at = atomicAdd(&gs.n_open, (unsigned)incl);
        at = __shfl_sync(kFull, at, 31) + (unsigned)(incl - cnt);
        for (; open; open &= open - 1u, ++at) {
          const unsigned int pair = ((unsigned)a << 16) | (unsigned)(b0 + __ffs((int)open) - 1);
          if (at < kOwnOpen) { gs.open[at] = pair; continue; }
          const unsigned int over = atomicAdd(amb_count, 1u);
          if (over < (unsigned)p.cap_amb) p.amb_pairs[over] = pair;
        }
      }
    }
    if (unit + (int)gridDim.x < units) {                 // (the tile in shared memory, before the next operands)
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      if (__syncthreads_or(*(volatile int*)&gs.abort_)) return;
    }
  }
  // the pairs left open, by the CTA that found them; a list and a barrier for all of them took 4.6 us at 463 rows
  __syncthreads();
#pragma unroll 1
  for (unsigned int i = warp; i < min(gs.n_open, kOwnOpen); i += kWarps) decide_exactly(p, e, (int)(gs.open[i] >> 16), (int)(gs.open[i] & 0xffffu));
}

// ------------------------------------------------------------------------------------------------
// Dense, step 3: first-fit over the conflict bits, by one CTA, 1,024 candidates at a time.  A thread holds the bits of two
// candidates with the earlier ones of the piece in registers (those with earlier pieces are looked at once), and a piece is settled in
// passes: a candidate with no undecided earlier neighbour is kept, and those it conflicts with are out.  The passes are
// as many as the longest chain of such dependencies, five to six where 1,024 candidates of 463 rows leave 110; bound by the
// ANDs (half the lanes' rate for logic).  One warp
// going through the words one after the other took 0.7 us a word of 32 candidates, 21.7 us of 463 x 508,999's 56 per round; this
// takes 6.2 of 36: 1.7 to bring in the rows, 0.7 a pass.
// (Passes that OR the rows of undecided candidates in shared memory: 2 us each, bound by reading the rows.)
// ------------------------------------------------------------------------------------------------
constexpr int kPiece = 2 * kT, kPieceWords = kPiece / 32;
struct WalkShared {
  __align__(16) unsigned int state[2][kPieceWords];      // of the piece: undecided, kept in this pass
  __align__(16) unsigned int kept[kMaxWords + kPieceWords];      // of all pieces so far
  int ex;
};
__device__ __forceinline__ unsigned int any_of(const uint4& a, const uint4& b) { return (a.x & b.x) | (a.y & b.y) | (a.z & b.z) | (a.w & b.w); }

// Whether the thread's two candidates (of words `warp` and warp + kWarps) have neighbours among `mask`: what lies before them only.
__device__ __forceinline__ void touch(const uint4 (&row)[2][kPieceWords / 4], const unsigned int* mask, int warp, unsigned int (&met)[2]) {
#pragma unroll
  for (int q = 0; q < kPieceWords / 4; ++q) {
    if (q > (warp + kWarps) / 4) break;
    const uint4 m = reinterpret_cast<const uint4*>(mask)[q];
    if (q <= (kWarps - 1) / 4 && q <= warp / 4) met[0] |= any_of(row[0][q], m);
    met[1] |= any_of(row[1][q], m);
  }
}

__device__ __forceinline__ void dense_walk(const Problem& p, const Engine& e, unsigned char* sm, int n, int n_total) {
  WalkShared& s = *reinterpret_cast<WalkShared*>(sm);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kQuads = kPieceWords / 4;
  const uint4* rows = reinterpret_cast<const uint4*>(p.conflict);
  int kept = 0, examined = n;
  bool done = false;
  __syncthreads();
#pragma unroll 1
  for (int r0 = 0; r0 < n && !done; r0 += kPiece) {
    uint4 row[2][kQuads];
    bool out0[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int a = r0 + tid + h * kT, own = a - r0;
#pragma unroll
      for (int q = 0; q < kQuads; ++q)
        row[h][q] = a < n && 128 * q < own ? __ldcg(rows + (size_t)(r0 / 128 + q) * p.n_cand + a) : make_uint4(0u, 0u, 0u, 0u);
      out0[h] = a >= n;
    }
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
      const int a = r0 + tid + h * kT;
      unsigned int hit = 0u;
      if (a < n) {
#pragma unroll 4
        for (int q = 0; q < r0 / 128; ++q) hit |= any_of(__ldcg(rows + (size_t)q * p.n_cand + a), reinterpret_cast<const uint4*>(s.kept)[q]);
      }
      if (hit) out0[h] = true;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int own = tid + h * kT;
      // (of the last four words only the bits before the candidate's own place mean anything)
#pragma unroll
      for (int q = 0; q < kQuads; ++q)
        if (128 * q < own && own < 128 * (q + 1)) {
          auto before = [&](int word) { const int k = own - 128 * q - 32 * word; return k >= 32 ? kFull : (k <= 0 ? 0u : (1u << k) - 1u); };
          row[h][q].x &= before(0); row[h][q].y &= before(1); row[h][q].z &= before(2); row[h][q].w &= before(3);
        }
      const unsigned int und = __ballot_sync(kFull, !out0[h]);
      if (lane == 0) s.state[0][warp + h * kWarps] = und;
    }
    __syncthreads();
    unsigned int und[2] = {s.state[0][warp], s.state[0][warp + kWarps]}, keep[2] = {0u, 0u};     // (this warp's words)
#pragma unroll 1
    for (bool open = true; open;) {
      // kept: those with no undecided earlier neighbour (decided ones are out of everybody's way: kept or not)
      unsigned int fresh[2] = {0u, 0u};
      if (und[0] | und[1]) {
        unsigned int wait[2] = {0u, 0u};
        touch(row, s.state[0], warp, wait);
#pragma unroll
        for (int h = 0; h < 2; ++h) { fresh[h] = __ballot_sync(kFull, wait[h] == 0u) & und[h]; keep[h] |= fresh[h]; }
      }
      if (lane == 0) { s.state[1][warp] = fresh[0]; s.state[1][warp + kWarps] = fresh[1]; }
      __syncthreads();
      // out: those with one of them before
      if (und[0] | und[1]) {
        unsigned int out[2] = {0u, 0u};
        touch(row, s.state[1], warp, out);
#pragma unroll
        for (int h = 0; h < 2; ++h) und[h] &= ~(fresh[h] | __ballot_sync(kFull, out[h] != 0u));
        if (lane == 0) { s.state[0][warp] = und[0]; s.state[0][warp + kWarps] = und[1]; }
      }
      open = __syncthreads_or((und[0] | und[1]) != 0u) != 0;
    }
    if (lane == 0) { s.kept[r0 / 32 + warp] = keep[0]; s.kept[r0 / 32 + warp + kWarps] = keep[1]; }
    __syncthreads();
    // numbered, up to P
    const int c = __popc(s.kept[r0 / 32 + lane]);
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += v;
    }
    const int total = __shfl_sync(kFull, incl, 31), room = p.n_keep - kept;
    static_assert(kPieceWords == 32, "a word per lane");
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const unsigned int word = keep[h];
      const int r = __shfl_sync(kFull, incl - c, warp + h * kWarps) + __popc(word & ((1u << lane) - 1u)), a = r0 + tid + h * kT;
      if (((word >> lane) & 1u) && r < room) {           // stop exactly at P
        p.kept[kept + r] = p.cand[a];
        p.kept_pos[kept + r] = a;
        if (r == room - 1) s.ex = a + 1;
      }
    }
    __syncthreads();
    done = total >= room;
    if (done) examined = s.ex;
    kept += min(total, room);
  }
  if (tid == 0) {
    EngineState* es = e.es;
    es->n_kept = kept; es->n_examined = examined;
    es->walk_open = kept < p.n_keep && n < n_total ? 1 : 0;
    // would the window have done?  (the next round goes straight to the whole list if not)
    if (n == n_total && e.window < n_total) es->skip_window = kept == p.n_keep && examined <= e.window ? 0 : 1;
  }
}

// ------------------------------------------------------------------------------------------------
// Dense, step 4: r <- r - sum_a x_a dbeta_a.  The rows are dealt out evenly, a stretch of 16-byte groups per CTA (four of
// them at 2,048 rows on 148 CTAs); a thread takes one group of one column at a time (the moving columns dealt out over
// kT / groups teams), six loads under way, and the teams' FP64 sums are added in a fixed order.  Few rows, few columns that
// move: 0.8 us at 463 rows, latency.
// ------------------------------------------------------------------------------------------------
__device__ void dense_apply(const Problem& p, const Moving& mv, double* part, int nk, int n_moving) {
  const int tid = threadIdx.x;
  const int n4 = (int)((p.N + 3) >> 2), per = (n4 + (int)gridDim.x - 1) / (int)gridDim.x;
  const int g_lo = (int)blockIdx.x * per, g_hi = min(n4, g_lo + per);
  if (g_lo >= n4 || n_moving == 0) return;
  const int g0 = g_lo, width = g_hi - g_lo, teams = kT / width;          // (at most 2,048 rows: width <= kT)
  const int team = tid / width, q = tid - team * width;
  double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
  const float* x0 = p.xv + ((long long)(g0 + q) << 2);
  constexpr int kU = 6;
  auto add = [&](const float4& x, double d) { s0 += (double)x.x * d; s1 += (double)x.y * d; s2 += (double)x.z * d; s3 += (double)x.w * d; };
  if (team < teams) {
    const int here = min(n_moving, kStage);
    for (int a0 = team; a0 < here; a0 += teams * kU) {
      float4 x[kU];
      double d[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int a = a0 + u * teams;
        d[u] = a < here ? mv.d[a] : 0.0;
        x[u] = a < here ? __ldg(reinterpret_cast<const float4*>(x0 + mv.off[a])) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) add(x[u], d[u]);
    }
    if (n_moving > kStage) {                           // beyond what was staged: found again in the kept list
      int seen = 0;
      for (int a = 0; a < nk; ++a) {
        const double d = p.cand_dbeta64[p.kept_pos[a]];
        if (d == 0.0) continue;
        if (seen >= kStage && seen % teams == team) add(__ldg(reinterpret_cast<const float4*>(x0 + (long long)p.kept[a] * p.ld)), d);
        ++seen;
      }
    }
    double* at = part + ((size_t)team * width + q) * 4;
    at[0] = s0; at[1] = s1; at[2] = s2; at[3] = s3;
  }
  __syncthreads();
  const int rows = width * 4;
  int tpr = 1;                                         // threads per row
  while (tpr < 32 && tpr * 2 * rows <= kT) tpr *= 2;
  for (int r0 = 0; r0 < rows; r0 += kT / tpr) {
    const int r = r0 + tid / tpr, sub = tid & (tpr - 1);
    double s = 0.0;
    if (r < rows)
      for (int t = sub; t < teams; t += tpr) s += part[(size_t)t * rows + r];
    for (int o = tpr >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
    const long long row = ((long long)g0 << 2) + r;
    if (sub == 0 && r < rows && row < p.N && s != 0.0) apply_row(p, row, s);
  }
  __syncthreads();
}

constexpr unsigned int kFewOpen = 48;                    // open pairs the walking CTA decides itself

// (cold) Data whose products cluster at rho leave more pairs open than the list holds: all pairs of the first n candidates
// exactly, tiles of 32 x 128 of the lower triangle.  32 rows of the tile's columns at a time lie in shared memory as
// binary64, and a thread adds up 2 x 4 products: bound by reading the operands there (a warp's step takes 9 cycles of shared
// memory and 4 of the FP64 pipe).  A warp per pair, both columns read again for every pair and the lower triangle stepped
// through as well, took 9.7 ms per round at 4,096 candidates of 900 rows, this takes 2.2 (the launch chain's 3xTF32 pass, list
// included, 4.2 to 4.8).  4 x 4 products take 1.5, but need registers that the rest of the kernel then spills: rounds
// that never come here 2 % slower.
constexpr int kExactRows = 32, kExactCols = 128, kExactK = 32;
struct ExactTile { double a[kExactK][kExactRows], b[kExactK][kExactCols], norm[kExactRows + kExactCols]; const float* col[kExactRows + kExactCols]; };

__device__ __noinline__ void decide_all(const Problem& p, const Engine& e, int n) {
  extern __shared__ __align__(1024) unsigned char sm[];
  ExactTile& s = *reinterpret_cast<ExactTile*>(sm);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  static_assert(kWarps * 2 == kExactRows && 32 * 4 == kExactCols, "2 x 4 products a thread");
  constexpr int kBoth = kExactRows + kExactCols, kStaged = (kBoth * (kExactK / 4) + kT - 1) / kT;         // columns; groups of four rows a thread brings in
  const int n4 = (int)((p.N + 3) >> 2), row_tiles = (n + kExactRows - 1) / kExactRows;
  unsigned int tile = 0u;
  for (int r = 0; r < row_tiles; ++r) {
    for (int c = 0; c <= r * kExactRows / kExactCols; ++c) {
      if (tile++ % gridDim.x != blockIdx.x) continue;
      const int row0 = r * kExactRows, col0 = c * kExactCols;
      __syncthreads();                                   // (the tile before)
      if (tid < kBoth) {
        const int i = tid < kExactRows ? row0 + tid : col0 + tid - kExactRows;
        s.norm[tid] = i < n ? e.norm[i] : 0.0;
        s.col[tid] = i < n ? p.xv + (long long)p.cand[i] * p.ld : nullptr;
      }
      __syncthreads();
      double acc[2][4] = {};
      for (int g0 = 0; g0 < n4; g0 += kExactK / 4) {
        float4 v[kStaged];
#pragma unroll
        for (int u = 0; u < kStaged; ++u) {
          const int g = g0 + (tid + u * kT) / kBoth;
          const float4* src = reinterpret_cast<const float4*>(s.col[(tid + u * kT) % kBoth]);
          v[u] = src != nullptr && g < n4 && g < g0 + kExactK / 4 ? __ldg(src + g) : make_float4(0.f, 0.f, 0.f, 0.f);
          if (4ll * g + 3 >= p.N && g < n4) mask_rows(p, g, v[u]);
        }
        __syncthreads();                                 // (the rows before)
#pragma unroll
        for (int u = 0; u < kStaged; ++u) {
          const int i = (tid + u * kT) % kBoth, k = (tid + u * kT) / kBoth * 4;
          if (k >= kExactK) continue;
          double* dst = i < kExactRows ? &s.a[k][i] : &s.b[k][i - kExactRows];
          const int pitch = i < kExactRows ? kExactRows : kExactCols;
          dst[0] = v[u].x; dst[pitch] = v[u].y; dst[2 * pitch] = v[u].z; dst[3 * pitch] = v[u].w;
        }
        __syncthreads();
#pragma unroll 4
        for (int k = 0; k < kExactK; ++k) {
          const double2 a = *reinterpret_cast<const double2*>(&s.a[k][warp * 2]);
#pragma unroll
          for (int y = 0; y < 4; ++y) {
            const double b = s.b[k][lane + 32 * y];
#pragma unroll
            for (int x = 0; x < 2; ++x) acc[x][y] = fma(x ? a.y : a.x, b, acc[x][y]);
          }
        }
      }
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const int a = row0 + warp * 2 + x;
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          const double den = s.norm[warp * 2 + x] * s.norm[kExactRows + lane + 32 * y];
          const unsigned int word = __ballot_sync(kFull, col0 + lane + 32 * y < a && den > 0.0 && fabs(acc[x][y]) >= (double)p.rho * den);
          if (lane == 0 && a < n && (col0 >> 5) + y < p.mask_words) *conflict_word(p, a, (col0 >> 5) + y) = word;
        }
      }
    }
  }
}

// ------------------------------------------------------------------------------------------------
// The rounds.  Every step is called from one place, so that the loop's code stays within the instruction cache (with each
// variant of a round written out, 750 KB of it, every step ran from L2 and took two to three times as long).
// ------------------------------------------------------------------------------------------------
struct Pending { int nk, n_moving, shift; };             // CSC: the residual's changes of the last round, still in the accumulators

struct EngineMaps { CUtensorMap rows, cols; };           // boxes of 64 elements x 128 and 64 candidates

template <bool kDense>
__global__ void __launch_bounds__(kT, 1) k_engine(const __grid_constant__ Problem p, const __grid_constant__ Engine e,
                                                  const __grid_constant__ EngineMaps maps, int n_rounds, int have_list, int draw_next,
                                                  RoundOutputs out) {
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ DrawShared ds;
  __shared__ TurnShared ts;
  __shared__ ChangeShared cs;
  __shared__ __align__(8) PackBars pb;
  __shared__ __align__(16) GramShared gs;
  __shared__ Settled walk;
  // Copies for the functions that are called rarely and not inlined, made when they are: a reference to the parameters themselves would make
  // every access to them, in the hot code too, a load from memory.
  __shared__ Problem sp;
  __shared__ Engine se;
  // after a wait that expired nothing runs on this handle until strads_recover (CTAs that disagree on the bit only
  // meet a barrier that gives up)
  if (p.st->status & STRADS_STATUS_WAIT_EXPIRED) return;
  const int tid = threadIdx.x, warp = tid >> 5, cta = (int)blockIdx.x, n_ctas = (int)gridDim.x;
  auto keep_parameters = [&]() {                         // (where one of those functions is called: one thread takes 2.7 us for it)
    __syncthreads();
    if (tid == 0) { sp = p; se = e; }
    __syncthreads();
  };
  const bool walker = cta == n_ctas - 1;                 // the CTA that walks
  const uint32_t limit = p.wait_limit ? p.wait_limit : 1u << 24;
  GramCount gc = {};
  if (kDense) {
    if (tid == 0) {
      for (int i = 0; i < kWarps; ++i) { mbar_init(smem_u32(&pb.full[i]), 1); pb.uses[i] = 0u; }
      for (int s = 0; s < 2; ++s)
        for (int i = 0; i < kMaxStages; ++i) { mbar_init(smem_u32(&gs.full[s][i]), 1); mbar_init(smem_u32(&gs.empty[s][i]), 1); }
      mbar_init(smem_u32(&gs.done), 1);
      gs.abort_ = 0;
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < 32) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&gs.tmem)), "r"(kTmemCols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    }
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  }
  Grid g;
  g.count = &e.es->bar_count; g.target = 0u; g.n = gridDim.x; g.limit = p.wait_limit ? p.wait_limit : kSpinLimit; g.status = &p.st->status;
  Grid g_draw = g;                                       // (CSC: of the threads that draw while the others walk)
  g_draw.count = &e.es->draw_bar_count;
  EngineState* es = e.es;
  unsigned long long t = p.st->round;
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(sm);
  unsigned char* behind_keys = sm + (e.n_list > 0 ? 2 * sizeof(unsigned long long) * (size_t)p.n_keep : 0);
  Moving* mv = reinterpret_cast<Moving*>(behind_keys);
  double* part = reinterpret_cast<double*>(behind_keys + sizeof(Moving));
  ChangedByBin* cb = reinterpret_cast<ChangedByBin*>(behind_keys + (kDense ? sizeof(Moving) + sizeof(double) * 4 * kT : 0));
  unsigned short* kept_at = reinterpret_cast<unsigned short*>(sm + kept_at_offset(p, (size_t)(behind_keys - sm) + sizeof(ChangedByBin)));
  const bool no_filter = (p.flags & STRADS_FLAG_NO_FILTER) != 0;
  const int n_total = p.n_cand;
  Pending last;
  last.nk = 0; last.n_moving = 0; last.shift = INT_MIN;
  unsigned int attempts = 0u;                            // dense: Gram passes so far
  bool have = have_list != 0, ok = true;
  int left = n_rounds;
  // One trip per round, and one for a draw that nothing was drawn ahead for (real: false).  CSC ends with a trip that only
  // applies the last round's changes to the residual.
  while (true) {
    if (!kDense) {
      csc_apply(WholeGrid(), p, last.nk, last.n_moving, last.shift);
      last.shift = INT_MIN;
    }
    if (left == 0) break;
    const bool real = have, final_round = real && left == 1;
    const bool draws = !real || (e.n_list > 0 && (!final_round || draw_next));
    const unsigned long long td = real ? t + 1 : t;      // the round drawn for
    const unsigned int k = real ? (unsigned)e.n_list : (unsigned)n_total;
    bool scanned = !draws, collected = !draws;
    bool spare = kDense && real && !no_filter;           // the last CTA leaves the draw's winners to the others
    int n = no_filter ? p.n_keep : e.window, packed = 0;
    bool window = true, pending = false;                   // pending: a barrier to be met, and the kept list is this CTA's own
    if (kDense) {
      if (n < n_total && es->skip_window && !no_filter) n = n_total;
    } else {
      window = no_filter || (p.bucket_count != nullptr && !(n < n_total && es->skip_window) && es->avoid == 0);
      if (real && window && !no_filter) csc_norms_begin(p, e, sm, n);
      if (real) csc_enter(WholeGrid(), p, e, window ? n : n_total, window && !no_filter);
    }
    // ---- steps 1 to 3, once more over all candidates where a window does not do ----
    while (true) {
      const GramPlan& pl = e.plan[n == n_total ? 1 : 0];
      if (kDense && real) {
        if (!no_filter)
          for (int i = cta * kT + tid; i < pl.tiles; i += n_ctas * kT) e.tile_ticket[i] = 0u;
        dense_pack(p, e, sm, ts, pb, packed, n, t + 1, draws, limit);
      }
      // a walk on demand leaves the SMs mostly idle, at its barriers above all: the scan is made there
      const bool during_walk = !kDense && real && !window && !scanned;
      // The scan's counts are wanted behind the barrier after the next one, where there is one: it lies between arriving and
      // waiting, and the wait is over when it ends (50,000 x 1,000,000: 38.0 -> 37.4 us per round).
      const bool ahead = real && !no_filter && (kDense || window);
      if (ahead) grid_arrive(g);
      if (!scanned && !during_walk) { draw_scan(WholeGrid(), p, e, ds, sm, td, true); scanned = true; }
      if (kDense) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // (the Gram's operands come in over it)
      // (the walk needs nothing of what is before it but the norms that follow beta and delta)
      if (ahead) {
        if (!kDense) csc_products_begin(sm, n);
        if (!(ok = grid_complete(g))) break;
      } else if (!(!kDense && real && !window && !(p.flags & STRADS_FLAG_DYNAMIC_DEPS)) && !(ok = grid_sync(g))) {
        break;
      }
      if (kDense && real && !no_filter) {
        unsigned int* amb = &es->amb_count[attempts & 1u];
        if (cta == 0 && tid == 0) es->amb_count[(attempts + 1u) & 1u] = 0u;
        ++attempts;
        dense_gram(p, e, pl, &maps.rows, &maps.cols, sm, gs, gc, n, amb, limit);
        if (!(ok = grid_sync(g, p.stall != 0))) break;
        const unsigned int open = *amb;
        const bool listed = open <= (unsigned)p.cap_amb;
        if (!listed) {
          if (cta == 0 && tid == 0) atomicOr(&p.st->status, STRADS_STATUS_GRAM_FALLBACK);
          keep_parameters();
          decide_all(sp, se, n);
        }
        if (listed && open > 0u && (open > kFewOpen || walker)) {
          const unsigned int first = open > kFewOpen ? (unsigned)(warp * n_ctas + cta) : (unsigned)warp;
          for (unsigned int i = first; i < open; i += open > kFewOpen ? (unsigned)(kWarps * n_ctas) : (unsigned)kWarps) {
            const unsigned int pr = __ldcg(p.amb_pairs + i);
            decide_exactly(p, e, (int)(pr >> 16), (int)(pr & 0xffffu));
          }
          __threadfence();
        }
        if (open > kFewOpen && !(ok = grid_sync(g))) break;
        if (walker) dense_walk(p, e, sm, n, n_total);
      }
      if (no_filter && real && walker) {                 // keep the first P
        for (int i = tid; i < p.n_keep; i += kT) { p.kept[i] = p.cand[i]; p.kept_pos[i] = i; }
        if (tid == 0) { es->n_kept = p.n_keep; es->n_examined = p.n_keep; es->walk_open = 0; }
      }
      // the winners of the draw: by every CTA but the one that walks; CSC in step 3 as well, unless there is none
      const bool csc_window = !kDense && real && window && !no_filter;
      if (!collected && !csc_window && !during_walk) { draw_gather<AllThreads>(WholeGrid(), p, e, ds, k, spare); collected = true; }
      if (!kDense && real) {
        if (!window) {
          int walked = 0;
          if (!(ok = csc_walk_and_draw(WholeGrid(), p, sp, e, ds, sm, g, g_draw, during_walk, td, k, &walked))) break;
          if (during_walk) scanned = collected = true;
          csc_products<true>(WholeGrid(), p, e, ts, sm, walked, true, false, t + 1, draws);
        } else {
          csc_products<true>(WholeGrid(), p, e, ts, sm, n, false, csc_window, t + 1, draws);
        }
      }
      if (!(ok = grid_sync(g))) break;
      if (!real || no_filter) break;
      if (!kDense) {
        if (!window) break;
        csc_settle(p, e, sm, kept_at, walk, n, [&]() {
          const ClearAhead rows = csc_clear_begin(WholeGrid(), p, n);
          if (!collected) draw_gather<OtherThreads>(WholeGrid(), p, e, ds, k, false);
          csc_clear_end(p, rows);
        });
        collected = true;
        if (!walk_is_open(p, walk, n)) { pending = true; break; }
        if (!(ok = grid_sync(g))) break;
        if (cta == 0 && tid == 0) settle_note(e, walk);
        csc_enter(WholeGrid(), p, e, n_total, false);
        window = false;
      } else {
        if (!es->walk_open) break;
        packed = n; n = n_total;
      }
    }
    if (!ok) break;
    // ---- step 4 ----
    int n_moving = 0, nk = 0, examined = 0;
    const int n_next = no_filter ? p.n_keep : (e.window < n_total && es->skip_window ? n_total : e.window);   // looked at first
    if (real) {
      nk = pending ? walk.kept : es->n_kept;
      examined = pending ? walk.examined : es->n_examined;
      KeptColumns kept;
      if (!kDense) kept = kept_columns(WholeGrid(), p, nk, pending ? kept_at : nullptr);
      if (pending) grid_arrive(g);
      n_moving = gather_changes<kDense>(p, ds, nk, pending ? kept_at : nullptr, draws, keys, cb, mv, cs);
      last.nk = nk; last.n_moving = n_moving;
      if (!kDense) {
        last.shift = csc_shift(p.st->x_abs_max, cs.dmax, nk);
        csc_scatter(p, kept, last.shift);
      }
    }
    if (pending) {
      if (!(ok = grid_complete(g))) break;
      if (cta == 0 && tid == 0) settle_note(e, walk);
    }
    // (the priorities as they were, and nothing of this round's changes in shared memory)
    if (draws && es->mend) {
      keep_parameters();
      if (!(ok = draw_mend(WholeGrid(), sp, se, ds, sm, td, k, g))) break;
      if (real) gather_again<kDense>(sp, ds, nk, keys, cb, mv, cs);
    }
    if (real) {
      commit_changes(p, examined, nk, n_moving, out, final_round);
      --left;
      ++t;
    }
    if (draws) draw_rank<kDense>(WholeGrid(), p, e, ds, keys, cb, real ? cs.n_changed : 0, nk, cs.rank_wsum, spare ? max(1, n_ctas - 1) : n_ctas, n_next);
    if (kDense && real) dense_apply(p, *mv, part, nk, last.n_moving);
    have = draws;
    if (left == 0 && kDense) break;
    if (!(ok = grid_sync(g))) break;
  }
  if (kDense) {
    __syncthreads();
    if (tid < 32) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(gs.tmem), "r"(kTmemCols) : "memory");
    }
  }
  if (!ok) return;
  if (tid == 0 && atomicInc(&e.es->exit_count, gridDim.x - 1u) == gridDim.x - 1u) {
    e.es->bar_count = 0u; e.es->draw_bar_count = 0u;
    if (kDense) { e.es->amb_count[0] = 0u; e.es->amb_count[1] = 0u; }
  }
}

// ------------------------------------------------------------------------------------------------
// The draw alone (strads_sample_static), all of it in one launch: keys computed once and kept in shared memory, histogram,
// selection, collection and ranking with two grid barriers between them.  Bound by the launch and the barriers: 22.6 us
// as six launches (clear, round index, two passes, ordering), each waiting for the one before, at J = 100,000, P' = 2,048;
// one launch 16.4, and 14.3 since its parameters are copied to shared memory only where a rare path wants them.  It leaves its scratch clear.
// A call whose wait runs out leaves -1 in the places of the list that it did not come to, and says so to the next one
// (EngineState::dirty), which then clears the histogram behind a barrier of its own: every CTA leaves through the same few
// lines, and the one that leaves last sets the barrier back and knows from their count whether any of them gave up.
// A grid of no more CTAs than have keys or winners to go through: the barriers cost less among few.
// ------------------------------------------------------------------------------------------------
constexpr size_t kDrawKeys = 144 * 1024;   // keys a CTA keeps in shared memory (more: computed again to collect the winners)

// (cold; out of line, as the kernel runs from a cold instruction cache)  False: a wait gave up.
__device__ __noinline__ bool clear_histogram(const Engine& e, Grid& g) {
  for (int b = (int)blockIdx.x * kT + (int)threadIdx.x; b < kHistBins; b += (int)gridDim.x * kT) e.hist[b] = 0u;
  return grid_sync(g);
}

// False: a wait gave up.
__device__ __forceinline__ bool draw_alone(const Problem& p, const Engine& e, DrawShared& ds, Problem& sp, Engine& se, unsigned char* sm, unsigned long long t,
                                           int kept_groups, int stall) {
  unsigned int* sh = reinterpret_cast<unsigned int*>(sm);
  unsigned long long* held = reinterpret_cast<unsigned long long*>(sm + kScanSmem);      // [kept_groups][4][kT]
  const int tid = threadIdx.x;
  const long long groups = (p.J + 3) >> 2, whole = p.J >> 2;
  const WeightForm wf = weight_form(p);
  const Binning bins = binning_of(0.f);
  for (int b = tid; b < kHistBins; b += kT) sh[b] = 0u;
  static_assert(STRADS_STATIC_MAX_CANDIDATES <= kHistBins, "a place of the list per bin");
  for (int b = (int)blockIdx.x * kT + tid; b < kHistBins; b += (int)gridDim.x * kT) {
    e.bin_cur[b] = 0u;
    if (b < p.n_cand) p.cand[b] = -1;
  }
  const int dirty = e.es->dirty;
  if (tid == 0) ds.cut = 0.f;
  __syncthreads();
  // (for the functions that are called rarely; made where they are: one thread takes 2.7 us for it, before the first key 16.5 -> 15.1 us
  // per call at J = 100,000)
  auto keep_parameters = [&]() {
    __syncthreads();
    if (tid == 0) { sp = p; se = e; }
    __syncthreads();
  };
  Grid g;
  g.count = &e.es->bar_count; g.target = 0u; g.n = gridDim.x; g.limit = p.wait_limit ? p.wait_limit : kSpinLimit; g.status = &p.st->status;
  int turn = 0;
  for (long long gi = (long long)blockIdx.x * kT + tid; gi < groups; gi += (long long)gridDim.x * kT, ++turn) {
    float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
    if (gi < whole) {
      d = __ldg(reinterpret_cast<const float4*>(p.delta) + gi);
    } else {
      const long long j = gi << 2;
      d.x = p.delta[j];
      if (j + 1 < p.J) d.y = p.delta[j + 1];
      if (j + 2 < p.J) d.z = p.delta[j + 2];
    }
    uint32_t w[4];
    philox4x32_10((uint32_t)gi, (uint32_t)t, (uint32_t)(t >> 32), 0u, (uint32_t)p.seed, (uint32_t)(p.seed >> 32), w);
    const float dd[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const long long j = (gi << 2) + i;
      const unsigned long long key = j < p.J ? key_of(wf, dd[i], w[i], (uint32_t)j) : ~0ull;
      if (j < p.J) atomicAdd(&sh[bin_of(bins, (unsigned int)(key >> 32))], 1u);
      if (turn < kept_groups) held[((size_t)turn * 4 + i) * kT + tid] = key;
    }
  }
  __syncthreads();
  if (dirty) {                                           // (the same in every CTA: it changes when the last one leaves)
    keep_parameters();
    if (!clear_histogram(se, g)) return false;
  }
  for (int b = tid; b < kHistBins; b += kT)
    if (sh[b]) atomicAdd(&e.hist[b], sh[b]);
  if (!grid_sync(g, stall != 0 && blockIdx.x == 0)) return false;
  draw_select<AllThreads>(e, ds, (unsigned)p.n_cand);
  if (ds.bnd_count > (unsigned)e.cap_boundary) {
    keep_parameters();
    if (!draw_refine(WholeGrid(), sp, se, ds, sm, t, (unsigned)p.n_cand, g)) return false;
  }
  if (kept_groups > 0) {
    for (int k = 0; k < turn; ++k)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const unsigned long long key = held[((size_t)k * 4 + i) * kT + tid];
        if (key != ~0ull) take_winner(e, ds, bins, key);
      }
  } else {
    keep_parameters();
    draw_collect_all(WholeGrid(), sp, se, ds, sm, t);
  }
  if (!grid_sync(g)) return false;
  draw_rank<true>(WholeGrid(), p, e, ds, nullptr, nullptr, 0, 0, nullptr, (int)gridDim.x, 0);       // (leaves the histogram clear)
  return true;
}

__global__ void __launch_bounds__(kT, 1) k_draw(const __grid_constant__ Problem p, const __grid_constant__ Engine e, unsigned long long t, int kept_groups,
                                                int stall) {
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ DrawShared ds;
  __shared__ Problem sp;
  __shared__ Engine se;
  const bool ok = draw_alone(p, e, ds, sp, se, sm, t, kept_groups, stall);
  if (threadIdx.x != 0) return;
  constexpr unsigned int kGaveUp = 1u << 16;             // (fewer CTAs than that)
  const unsigned int left = atomicAdd(&e.es->exit_count, ok ? 1u : 1u + kGaveUp);
  if ((left & (kGaveUp - 1u)) != gridDim.x - 1u) return;
  e.es->exit_count = 0u;
  e.es->bar_count = 0u;
  e.es->dirty = !ok || left >= kGaveUp ? 1 : 0;
}

size_t smem_of(const Problem& p, bool ahead) {
  const bool dense = p.layout == STRADS_DENSE_COLMAJOR;
  const int n_keep = p.n_keep;
  size_t need = kScanSmem;
  const size_t keys = ahead ? 2 * sizeof(unsigned long long) * (size_t)n_keep : 0;
  auto at_least = [&](size_t v) { if (need < v) need = v; };
  at_least(keys);
  if (dense) {
    at_least(kPackSmem);
    at_least(kGramSmem);
    at_least(sizeof(WalkShared));
    at_least(keys + sizeof(Moving) + sizeof(double) * 4 * kT + (ahead ? sizeof(ChangedByBin) : 0));
  } else {
    at_least(kTermsSmem);
    at_least(sizeof(DemandShared) + kScanSmem);
    at_least(kept_at_offset(p, keys + sizeof(ChangedByBin)) + sizeof(unsigned short) * (size_t)n_keep);
  }
  return need;
}

}  // namespace

size_t engine_smem(const Problem& p, bool ahead) { return smem_of(p, ahead); }

// The grid: one CTA per SM.  (A single thread-block cluster of 16 CTAs for small problems, whose barriers cost a fifth, was
// slower all the same: c1 41.6 us per round instead of 36.6, every CTA having nine times the candidates to go through.)
cudaError_t prepare_engine(const Problem& p, Engine& e) {
  const bool dense = p.layout == STRADS_DENSE_COLMAJOR;
  const void* fn = dense ? reinterpret_cast<const void*>(k_engine<true>) : reinterpret_cast<const void*>(k_engine<false>);
  int dev = 0, most = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  if ((err = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return err;
  cudaFuncAttributes a;
  if ((err = cudaFuncGetAttributes(&a, fn)) != cudaSuccess) return err;
  // the largest any handle can need
  if ((err = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)a.sharedSizeBytes)) != cudaSuccess) return err;
  e.grid = p.sm_count;
  if (dense) {
    e.plan[0] = gram_plan(p.N, e.window, e.grid);
    e.plan[1] = gram_plan(p.N, p.n_cand, e.grid);
  }
  return cudaSuccess;
}

cudaError_t prepare_draw() { return cudaFuncSetAttribute(k_draw, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kScanSmem + kDrawKeys)); }

cudaError_t launch_draw(const Problem& p, const Engine& e, unsigned long long t, cudaStream_t s) {
  const long long groups = (p.J + 3) / 4;
  const long long need = (groups + kT - 1) / kT, rank = ((long long)e.cap_win * 8 + kT - 1) / kT;
  long long grid = need > rank ? need : rank;
  if (grid > p.sm_count) grid = p.sm_count;
  const long long turns = (groups + grid * kT - 1) / (grid * kT);
  const bool held = (size_t)turns * 4 * kT * sizeof(unsigned long long) <= kDrawKeys;
  const size_t smem = kScanSmem + (held ? (size_t)turns * 4 * kT * sizeof(unsigned long long) : 0);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid); cfg.blockDim = dim3(kT); cfg.dynamicSmemBytes = smem; cfg.stream = s;
  cfg.attrs = attr; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_draw, p, e, t, held ? (int)turns : 0, p.stall);
}

cudaError_t encode_engine_maps(const Problem& p, const Engine& e, void* out) {
  static_assert(sizeof(EngineMaps) == 256, "two tensor maps");
  EngineMaps* maps = static_cast<EngineMaps*>(out);
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  const cudaError_t err = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres);
  if (err != cudaSuccess) return err;
  if (fn == nullptr || qres != cudaDriverEntryPointSuccess) return cudaErrorNotSupported;
  using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  const cuuint64_t dims[2] = {(cuuint64_t)e.xb_pitch, (cuuint64_t)p.n_cand}, strides[1] = {(cuuint64_t)e.xb_pitch * 2};
  const cuuint32_t estr[2] = {1, 1};
  for (int i = 0; i < 2; ++i) {
    const cuuint32_t box[2] = {64, i ? 64u : (cuuint32_t)kRowsT};
    const CUresult r = reinterpret_cast<EncodeFn>(fn)(i ? &maps->cols : &maps->rows, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, e.xb, dims, strides, box,
                                                      estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                                      CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
  }
  return cudaSuccess;
}

cudaError_t launch_engine(const Problem& p, const Engine& e, const void* maps, int n_rounds, bool have_list, bool draw_next,
                          const strads_round_out_t* out, cudaStream_t s) {
  const bool dense = p.layout == STRADS_DENSE_COLMAJOR;
  const EngineMaps& tm = *static_cast<const EngineMaps*>(maps);
  RoundOutputs o = {};
  if (out != nullptr) { o.cand = out->cand; o.kept = out->kept; o.dbeta = out->dbeta; o.counts = out->counts; }
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)e.grid); cfg.blockDim = dim3(kT); cfg.dynamicSmemBytes = engine_smem(p, e.n_list > 0); cfg.stream = s;
  cfg.attrs = attr; cfg.numAttrs = 1;
  const int have = have_list ? 1 : 0, next = draw_next ? 1 : 0;
  return dense ? cudaLaunchKernelEx(&cfg, k_engine<true>, p, e, tm, n_rounds, have, next, o)
               : cudaLaunchKernelEx(&cfg, k_engine<false>, p, e, tm, n_rounds, have, next, o);
}

}  // namespace strads
