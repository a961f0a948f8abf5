// Whole rounds of Algorithm 1 in one cooperative launch: one CTA of 512 threads per SM, the steps of a round
// separated by a grid barrier instead of by kernel boundaries.
//
// A round is a chain of short dependent steps over a few MB at most, so what bounds it is the number of times the
// whole grid has to hand over to itself and what every hand-over costs.  As separate launches a round took 11 to 17
// kernels, each with its launch, its ramp and the drain of the one before; here it takes four barriers of ~1.5 us, and the
// draw of the next round runs in the shadow of the steps of this one:
//
//   step           dense                                          CSC
//   1  (all CTAs)  BF16 copies of the candidates' columns,        last round's residual applied; candidates entered
//                  x_c^T r and would-be changes; scan of the      into the row buckets; scan of the keys of round t + 1
//                  keys of round t + 1
//   2  (all CTAs)  Gram tiles on the tensor cores, then the      inner products from the buckets, x_c^T r and would-be
//                  pairs they leave open                          changes
//  (2b)            open pairs that their CTA had no room for
//   3              greedy walk (last CTA); keys of round t + 1    the same; buckets emptied (the others)
//                  below the boundary collected (the others)
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
#include <climits>

#include <cuda.h>
#include <cuda_bf16.h>

#include "engine.cuh"
#include "walk_pairs.cuh"

namespace strads {
namespace {

constexpr int kT = 512;                    // threads of a CTA, one CTA per SM
constexpr int kWarps = kT / 32;
constexpr unsigned int kFull = 0xffffffffu;
constexpr unsigned int kSpinLimit = 1u << 22;

// ------------------------------------------------------------------------------------------------
// Grid barrier: one counter that only grows during a launch.  A CTA may pass when all have arrived target / n times;
// no CTA can be more than one barrier ahead, so the counter lies within [target, target + n) then -- an arrival count
// outside that range (strads_inject_stall plants one) never lets anybody pass.
// ------------------------------------------------------------------------------------------------
struct Grid {
  unsigned int* count;
  unsigned int target, n, limit;
  unsigned int* status;
};

// Arrives and waits (one thread; what its CTA wrote is ordered by a barrier before).  False: it gave up.
__device__ __forceinline__ bool grid_wait(const Grid& g, bool withhold = false) {
  if (!withhold) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(g.count) : "memory");
  unsigned int v, it = 0;
  bool ok;
  do {
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(g.count) : "memory");
    ok = v - g.target < g.n;
  } while (!ok && ++it < g.limit);
  if (!ok) atomicOr(g.status, STRADS_STATUS_WAIT_EXPIRED);
  return ok;
}

// withhold: this CTA does not arrive (an injected stall: everybody's wait runs out).
__device__ bool grid_sync(Grid& g, bool withhold = false) {
  __shared__ int s_ok;
  g.target += g.n;
  __syncthreads();
  if (threadIdx.x == 0) s_ok = grid_wait(g, withhold);
  __syncthreads();
  return s_ok != 0;
}
// The same in two parts, with work between them that nobody waits for.
__device__ __forceinline__ void grid_arrive(Grid& g) {
  g.target += g.n;
  __syncthreads();
  if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(g.count) : "memory");
}
__device__ bool grid_complete(const Grid& g) {
  __shared__ int s_ok;
  if (threadIdx.x == 0) s_ok = grid_wait(g, true);
  __syncthreads();
  return s_ok != 0;
}

// The threads of a CTA that do a step together: all of them, or those that do not walk while the others do (below).
constexpr int kWalkT = 256;                // threads that walk
struct AllThreads {
  static constexpr int kN = kT;
  static __device__ __forceinline__ int tid() { return threadIdx.x; }
  static __device__ __forceinline__ void sync() { __syncthreads(); }
};
struct OtherThreads {
  static constexpr int kN = kT - kWalkT;
  static __device__ __forceinline__ int tid() { return (int)threadIdx.x - kWalkT; }
  static __device__ __forceinline__ void sync() { asm volatile("bar.sync 2, %0;" ::"n"(kN) : "memory"); }
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// ------------------------------------------------------------------------------------------------
// The draw (SAP step 1; the keys and their order are those of sampler.cu).
//
// scan     every key below the cutoff carried over from the last draw is binned and saved (by each CTA in a stretch of
//          its own: one counter for all was 2,400 additions to one address, 3.5 us); the others are recognised
//          from a few operations (T >= v / w with v = (x + 1/2) 2^-32) and not computed.  Without a cutoff all keys
//          are computed and binned by their top 12 bits.
// select   every CTA reads the 4,096 counts, scans them and finds the bin that holds the n_list-th key -- the same in
//          all of them, so nothing has to be published.
// collect  the keys up to that bin, saved ones if the scan saved them all, go to `win`, grouped by bin.
// rank     a key's rank is the start of its group plus the smaller keys inside it.
//
// With a cutoff the bins are 128 per octave for the 24 octaves below it and 16 per octave for 64 more, by the distance of
// the time's bits from the cutoff's: the winners of an exponential race spread over the top octaves, so a group holds
// P' / 256 keys or fewer where 8 bins per octave (the unguided scan) leave P' / 16; the coarse ones are for rounds in which
// coefficients never touched (times 10^14 times smaller) and coefficients at rest are drawn together.
// ------------------------------------------------------------------------------------------------
constexpr unsigned int kFineSpan = 24u << 23;            // bits of time: 24 octaves, 3,072 bins
constexpr int kCoarseBins = kHistBins - 3072;
struct Binning { unsigned int cut; };                    // bits of the cutoff; 0: none
__device__ __forceinline__ Binning binning_of(float cut) {
  Binning b;
  b.cut = cut > 0.f ? __float_as_uint(cut) : 0u;
  return b;
}
__device__ __forceinline__ unsigned int bin_of(const Binning& b, unsigned int bits) {
  if (b.cut == 0u) return min(bits >> (32 - kHistBits), (unsigned)(kHistBins - 1));
  if (bits >= b.cut) return kHistBins - 1;
  const unsigned int d = b.cut - bits;
  if (d < kFineSpan) return kHistBins - 1 - (d >> 16);
  const unsigned int c = (d - kFineSpan) >> 19;
  return c < (unsigned)kCoarseBins ? kCoarseBins - 1 - c : 0u;
}

constexpr int kQueue = 192;                // survivors of a warp waiting for their keys; a step appends at most 128

// Place of a bin in an array in shared memory: a gap every 32 words, so that threads that own eight consecutive bins
// each do not meet in the same banks.
__device__ __forceinline__ int pad(int b) { return b + (b >> 5); }

// What a CTA knows about the draw in progress (shared memory).
struct DrawShared {
  unsigned int off[kHistBins + (kHistBins >> 5) + 1];      // winners before each bin, at pad(bin)
  unsigned int wsum[kWarps];
  int bnd, refined;                        // the bin of the n_list-th key; whether it had to be cut further
  unsigned int bnd_count, total;
  unsigned long long prefix;               // refined: keys of the boundary bin whose top `bits` bits exceed it are no winners
  int bits;
  float cut;                               // cutoff of the scan
  unsigned int saved;                      // keys below it that this CTA saved
};

// w_j = fma(x, y, z) for every importance distribution: (|d|, |d|, eta), (|d|, 1, eta) or (0, 0, 1) -- the same bits as
// priority_weight, and one sequence of instructions for all three.
struct WeightForm { bool square, uniform; float one, z; };
__device__ __forceinline__ WeightForm weight_form(const Problem& p) {
  const int mode = weight_mode_of(p.flags);
  WeightForm f;
  f.square = mode == kWeightSquare; f.uniform = mode == kWeightUniform;
  f.one = f.uniform ? 0.f : 1.f; f.z = f.uniform ? 1.f : p.eta;
  return f;
}
__device__ __forceinline__ float weight_of(const WeightForm& f, float d) {
  const float x = f.uniform ? 0.f : fabsf(d);
  return __fmaf_rn(x, f.square ? x : f.one, f.z);
}
__device__ __forceinline__ unsigned long long key_of(const WeightForm& f, float d, uint32_t word, uint32_t j) {
  return ((unsigned long long)__float_as_uint(__fdiv_rn(unit_exponential_rn(word), weight_of(f, d))) << 32) | j;
}

// A warp's share of a scan, step by step: 128 coefficients at a time; those whose keys may lie below the cutoff wait in a
// queue of the warp's in shared memory until there are enough of them for all lanes.  f(key, active) is called by whole warps.
struct WarpScan {
  uint2* queue;
  long long next, step;                    // Philox block of the warp's next step, and between two
  int n;                                   // in the queue
  float k;                                 // x 2^-32 > 1.02 cut w implies T > cut: the computed E is never below (x + 1/2) 2^-32 up to rounding
};
__device__ __forceinline__ WarpScan begin_scan(float cut, uint2* queue, int warp0, int n_warps) {
  WarpScan s;
  s.queue = queue; s.next = (long long)warp0 * 32; s.step = (long long)n_warps * 32; s.n = 0;
  s.k = cut > 0.f ? __fmul_rn(cut, 1.02f * 4294967296.0f) : __uint_as_float(0x7f800000u);
  return s;
}
// One step; past the end it only empties the queue.  Whether there was anything to do.
template <typename F>
__device__ __forceinline__ bool scan_step(const Problem& p, unsigned long long t, const WeightForm& wf, WarpScan& s, F&& f) {
  const int lane = threadIdx.x & 31;
  const long long groups = (p.J + 3) >> 2, whole = p.J >> 2, g = s.next + lane;
  const bool more = s.next < groups;
  if (!more && s.n == 0) return false;
  if (more) {
    float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
    if (g < whole) {
      d = __ldcg(reinterpret_cast<const float4*>(p.delta) + g);
    } else if (g < groups) {
      const long long j = g << 2;
      d.x = p.delta[j];
      if (j + 1 < p.J) d.y = p.delta[j + 1];
      if (j + 2 < p.J) d.z = p.delta[j + 2];
    }
    uint32_t w[4];
    philox4x32_10((uint32_t)g, (uint32_t)t, (uint32_t)(t >> 32), 0u, (uint32_t)p.seed, (uint32_t)(p.seed >> 32), w);
    const float dd[4] = {d.x, d.y, d.z, d.w};
    bool in[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) in[i] = !(__uint2float_rn(w[i]) > __fmul_rn(s.k, weight_of(wf, dd[i])));
    if (g >= whole) {
#pragma unroll
      for (int i = 0; i < 4; ++i) in[i] = in[i] && (g << 2) + i < p.J;
    }
    s.next += s.step;
    if (!__any_sync(kFull, in[0] | in[1] | in[2] | in[3])) return true;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const unsigned int m = __ballot_sync(kFull, in[i]);
      if (in[i]) s.queue[s.n + __popc(m & ((1u << lane) - 1u))] = make_uint2((uint32_t)(g << 2) + i, w[i]);
      s.n += __popc(m);
    }
  }
  if (s.n > kQueue - 128 || !more) {                     // the keys of the survivors, computed by all lanes together
    __syncwarp();
#pragma unroll 1
    for (int i = 0; i < s.n; i += 32) {
      const bool on = i + lane < s.n;
      const uint2 e = on ? s.queue[i + lane] : make_uint2(0u, 0u);
      f(on ? key_of(wf, p.delta[e.x], e.y, e.x) : ~0ull, on);
    }
    __syncwarp();
    s.n = 0;
  }
  return true;
}
template <typename F>
__device__ __forceinline__ void scan_keys(const Problem& p, unsigned long long t, float cut, uint2* queue, int warp0, int n_warps, F&& f) {
  const WeightForm wf = weight_form(p);
  WarpScan s = begin_scan(cut, queue, warp0, n_warps);
#pragma unroll 1
  while (scan_step(p, t, wf, s, f)) {}
}

// Shared memory of a scan: the CTA's histogram, then a queue per warp.
constexpr size_t kScanSmem = sizeof(unsigned int) * kHistBins + sizeof(uint2) * kQueue * kWarps;

// A scan in parts: it can be made in the waits of other work.  guided: with the cutoff es->t_cut (if there is one).
__device__ __forceinline__ float scan_open(const Engine& e, DrawShared& ds, unsigned char* sm, bool guided) {
  unsigned int* sh = reinterpret_cast<unsigned int*>(sm);
  const int tid = threadIdx.x;
  const float cut = guided ? e.es->t_cut : 0.f;
  __syncthreads();
  for (int b = tid; b < kHistBins; b += kT) sh[b] = 0u;
  for (int b = (int)blockIdx.x * kT + tid; b < kHistBins; b += (int)gridDim.x * kT) e.bin_cur[b] = 0u;     // the cursors of the groups
  if (tid == 0) { ds.cut = cut; ds.saved = 0u; }
  __syncthreads();
  return cut;
}
__device__ __forceinline__ void scan_found(const Engine& e, DrawShared& ds, unsigned int* sh, const Binning& bins, unsigned long long key, bool on) {
  const unsigned int bits = (unsigned int)(key >> 32);
  if (!on || (bins.cut != 0u && bits >= bins.cut)) return;
  atomicAdd(&sh[bin_of(bins, bits)], 1u);
  if (bins.cut != 0u) {
    const unsigned int at = atomicAdd(&ds.saved, 1u);
    if (at < e.cap_surv) e.surv[(size_t)blockIdx.x * e.cap_surv + at] = key;
  }
}
template <typename Team>
__device__ __forceinline__ void scan_close(const Engine& e, const DrawShared& ds, unsigned char* sm) {
  const unsigned int* sh = reinterpret_cast<const unsigned int*>(sm);
  Team::sync();
  if (Team::tid() == 0) e.saved[blockIdx.x] = ds.saved;
  for (int b = Team::tid(); b < kHistBins; b += Team::kN) {
    const unsigned int v = sh[b];
    if (v) atomicAdd(&e.hist[b], v);
  }
}
__device__ __forceinline__ uint2* scan_queue(unsigned char* sm) {
  return reinterpret_cast<uint2*>(sm + sizeof(unsigned int) * kHistBins) + (threadIdx.x >> 5) * kQueue;
}

// (a warp takes its steps round-robin over the CTAs: a few thousand coefficients already use every SM)
__device__ __forceinline__ void draw_scan(const Problem& p, const Engine& e, DrawShared& ds, unsigned char* sm, unsigned long long t, bool guided) {
  unsigned int* sh = reinterpret_cast<unsigned int*>(sm);
  const float cut = scan_open(e, ds, sm, guided);
  const Binning bins = binning_of(cut);
  scan_keys(p, t, cut, scan_queue(sm), (int)(threadIdx.x >> 5) * (int)gridDim.x + (int)blockIdx.x, kWarps * (int)gridDim.x,
            [&](unsigned long long key, bool on) { scan_found(e, ds, sh, bins, key, on); });
  scan_close<AllThreads>(e, ds, sm);
}

// The bin b with before(b) < k <= before(b) + count(b), and the winners before every bin (ds.total < k: there is none).
template <typename Team>
__device__ __forceinline__ void draw_select(const Engine& e, DrawShared& ds, unsigned int k) {
  const int tid = Team::tid(), lane = tid & 31, warp = tid >> 5;
  constexpr int kPer = kHistBins / Team::kN, kTeamWarps = Team::kN / 32;
  static_assert(kPer % 4 == 0, "16-byte loads");
  unsigned int c[kPer], mine = 0u;
#pragma unroll
  for (int u = 0; u < kPer / 4; ++u) {
    const uint4 v = __ldcg(reinterpret_cast<const uint4*>(e.hist) + tid * (kPer / 4) + u);
    c[4 * u] = v.x; c[4 * u + 1] = v.y; c[4 * u + 2] = v.z; c[4 * u + 3] = v.w;
  }
#pragma unroll
  for (int u = 0; u < kPer; ++u) mine += c[u];
  unsigned int incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int v = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += v;
  }
  Team::sync();
  if (lane == 31) ds.wsum[warp] = incl;
  if (tid == 0) ds.refined = 0;
  Team::sync();
  unsigned int before = 0u, total = 0u;
#pragma unroll
  for (int w = 0; w < kTeamWarps; ++w) { const unsigned int v = ds.wsum[w]; if (w < warp) before += v; total += v; }
  unsigned int run = before + incl - mine;
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    ds.off[pad(tid * kPer + u)] = run;
    if (run < k && k <= run + c[u]) { ds.bnd = tid * kPer + u; ds.bnd_count = c[u]; }
    run += c[u];
  }
  if (tid == 0) { ds.off[pad(kHistBins)] = total; ds.total = total; }
  Team::sync();
}
// (for the cold paths)
__device__ __noinline__ void draw_select_all(const Engine& e, DrawShared& ds, unsigned int k) { draw_select<AllThreads>(e, ds, k); }

// Upper edge of the boundary bin, as the bits of a binary32 time.
__device__ __forceinline__ unsigned int boundary_edge(const DrawShared& ds) {
  const Binning b = binning_of(ds.cut);
  const unsigned int bin = (unsigned)ds.bnd;
  unsigned long long x;
  if (b.cut == 0u) x = (unsigned long long)(bin + 1u) << (32 - kHistBits);
  else if (bin >= (unsigned)kCoarseBins) x = b.cut - ((kHistBins - 1u - bin) << 16) + 1u;
  else x = b.cut - kFineSpan - ((kCoarseBins - 1u - bin) << 19) + 1u;
  return x < 0x7f800000ull ? (unsigned int)x : 0x7f800000u;
}

__device__ __forceinline__ void take_winner(const Engine& e, const DrawShared& ds, const Binning& bins, unsigned long long key) {
  const unsigned int bin = bin_of(bins, (unsigned int)(key >> 32)), bnd = (unsigned)ds.bnd;
  if (bin > bnd || (bin == bnd && ds.refined && (key >> (64 - ds.bits)) > ds.prefix)) return;
  const unsigned int at = ds.off[pad((int)bin)] + atomicAdd(&e.bin_cur[bin], 1u);
  if (at < (unsigned)e.cap_win) e.win[at] = key;
}

// (cold) the winners from all J keys
__device__ __noinline__ void draw_collect_all(const Problem& p, const Engine& e, const DrawShared& ds, unsigned char* sm, unsigned long long t) {
  const int warp = (int)threadIdx.x >> 5;
  const Binning bins = binning_of(ds.cut);
  const unsigned int edge = boundary_edge(ds);
  uint2* queue = reinterpret_cast<uint2*>(sm + sizeof(unsigned int) * kHistBins) + warp * kQueue;
  __syncthreads();
  scan_keys(p, t, edge < 0x7f800000u ? __uint_as_float(edge) : 0.f, queue, warp * (int)gridDim.x + (int)blockIdx.x, kWarps * (int)gridDim.x,
            [&](unsigned long long key, bool on) { if (on) take_winner(e, ds, bins, key); });
}

// ... from the keys the scan saved: every CTA its own (the first of each thread in `key`), and a share of the last one's where that
// has other work.
template <typename Team>
__device__ __forceinline__ void draw_collect(const Engine& e, const DrawShared& ds, unsigned long long key, bool spare_last) {
  const Binning bins = binning_of(ds.cut);
  const unsigned int own = ds.saved, more = spare_last ? __ldcg(e.saved + gridDim.x - 1u) : 0u;
  const unsigned long long* mine = e.surv + (size_t)blockIdx.x * e.cap_surv;
  const unsigned long long* its = e.surv + (size_t)(gridDim.x - 1u) * e.cap_surv;
#pragma unroll 1
  for (unsigned int i = Team::tid(); i < own;) {
    take_winner(e, ds, bins, key);
    i += Team::kN;
    if (i < own) key = __ldcg(mine + i);
  }
#pragma unroll 1
  for (unsigned int i = Team::tid() * (gridDim.x - 1u) + blockIdx.x; i < more; i += Team::kN * (gridDim.x - 1u)) take_winner(e, ds, bins, __ldcg(its + i));
}

// Rare: more keys share the boundary bin than there is room for (thousands of tied times).  The grid cuts the bin
// further, digit by digit, over all J keys.  False: a barrier gave up.
__device__ __noinline__ bool draw_refine(const Problem& p, const Engine& e, DrawShared& ds, unsigned char* sm, unsigned long long t, unsigned int k, Grid& g) {
  const int tid = threadIdx.x, warp = tid >> 5;
  unsigned int* sh = reinterpret_cast<unsigned int*>(sm);
  uint2* queue = reinterpret_cast<uint2*>(sm + sizeof(unsigned int) * kHistBins) + warp * kQueue;
  const Binning bins = binning_of(ds.cut);
  const unsigned int bnd = (unsigned)ds.bnd;
  unsigned int sure = ds.off[pad((int)bnd)];                       // winners before the keys still in question
  unsigned long long prefix = 0ull;
  int bits = 0;
  if (blockIdx.x == 0 && tid == 0) atomicOr(&p.st->status, STRADS_STATUS_SAMPLER_REFINED);
  __shared__ int s_digit;
  __shared__ unsigned int s_before, s_here, s_w[kWarps];
  for (unsigned int here = ds.bnd_count; here > (unsigned)e.cap_boundary && bits < 64;) {
    const int width = min(kHistBits, 64 - bits);
    if (!grid_sync(g)) return false;                     // everybody has read the counts
    for (int b = (int)blockIdx.x * kT + tid; b < kHistBins; b += (int)gridDim.x * kT) e.hist[b] = 0u;
    for (int b = tid; b < kHistBins; b += kT) sh[b] = 0u;
    if (!grid_sync(g)) return false;
    const int up = 64 - bits - width;
    scan_keys(p, t, 0.f, queue, warp * (int)gridDim.x + (int)blockIdx.x, kWarps * (int)gridDim.x, [&](unsigned long long key, bool on) {
      if (on && bin_of(bins, (unsigned int)(key >> 32)) == bnd && (bits == 0 || (key >> (64 - bits)) == prefix))
        atomicAdd(&sh[(key >> up) & ((1u << width) - 1u)], 1u);
    });
    __syncthreads();
    for (int b = tid; b < kHistBins; b += kT) if (sh[b]) atomicAdd(&e.hist[b], sh[b]);
    if (!grid_sync(g)) return false;
    // the digit that holds the k-th key
    unsigned int c[kHistBins / kT], mine = 0u;
#pragma unroll
    for (int u = 0; u < kHistBins / kT; ++u) { c[u] = __ldcg(e.hist + tid * (kHistBins / kT) + u); mine += c[u]; }
    unsigned int incl = mine;
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int v = __shfl_up_sync(kFull, incl, o);
      if ((tid & 31) >= o) incl += v;
    }
    if ((tid & 31) == 31) s_w[warp] = incl;
    __syncthreads();
    unsigned int run = sure + incl - mine;
    for (int w = 0; w < warp; ++w) run += s_w[w];
#pragma unroll
    for (int u = 0; u < kHistBins / kT; ++u) {
      if (run < k && k <= run + c[u]) { s_digit = tid * (kHistBins / kT) + u; s_before = run; s_here = c[u]; }
      run += c[u];
    }
    __syncthreads();
    prefix = (prefix << width) | (unsigned long long)s_digit;
    bits += width;
    sure = s_before;
    here = s_here;
    __syncthreads();
  }
  if (tid == 0) { ds.refined = 1; ds.prefix = prefix; ds.bits = bits; }
  __syncthreads();
  return true;
}

// Selection and collection.  Where the selection needs mending (fewer keys than wanted, or too many that tie) the CTAs
// that see it say so, and all of them meet in draw_mend behind the next barrier.
template <typename Team>
__device__ __forceinline__ void draw_gather(const Problem& p, const Engine& e, DrawShared& ds, unsigned int k, bool spare_last) {
  if (spare_last && gridDim.x > 1 && blockIdx.x == gridDim.x - 1) return;
  const unsigned int at = Team::tid();                    // (under way meanwhile)
  const unsigned long long key = at < min(ds.saved, e.cap_surv) ? __ldcg(e.surv + (size_t)blockIdx.x * e.cap_surv + at) : ~0ull;
  draw_select<Team>(e, ds, k);
  // (a stretch that overflowed is seen by its owner alone: the others' winners are collected all the same, and again)
  const bool too_many = ds.saved > e.cap_surv || (spare_last && blockIdx.x == 0 && __ldcg(e.saved + gridDim.x - 1u) > e.cap_surv);
  if (ds.total < k || ds.bnd_count > (unsigned)e.cap_boundary || ds.cut == 0.f || too_many) {
    if (Team::tid() == 0 && (blockIdx.x == 0 || too_many)) e.es->mend = 1;
    return;
  }
  draw_collect<Team>(e, ds, key, spare_last);
}

// (cold) by all CTAs.  False: a barrier gave up.
__device__ __noinline__ bool draw_mend(const Problem& p, const Engine& e, DrawShared& ds, unsigned char* sm, unsigned long long t, unsigned int k, Grid& g) {
  draw_select_all(e, ds, k);
  if (!grid_sync(g)) return false;                       // everybody has read the counts and the flag
  if (blockIdx.x == 0 && threadIdx.x == 0) e.es->mend = 0;
  if (ds.total < k) {
    // the cutoff was too low (the weights collapsed: the end of the first sweep, say): once more, all keys
    for (int b = (int)blockIdx.x * kT + (int)threadIdx.x; b < kHistBins; b += (int)gridDim.x * kT) e.hist[b] = 0u;
    if (!grid_sync(g)) return false;
    draw_scan(p, e, ds, sm, t, false);
    if (!grid_sync(g)) return false;
    draw_select_all(e, ds, k);
  }
  if (ds.bnd_count > (unsigned)e.cap_boundary && !draw_refine(p, e, ds, sm, t, k, g)) return false;
  for (int b = (int)blockIdx.x * kT + (int)threadIdx.x; b < kHistBins; b += (int)gridDim.x * kT) e.bin_cur[b] = 0u;
  if (!grid_sync(g)) return false;
  draw_collect_all(p, e, ds, sm, t);
  return grid_sync(g);
}

// ------------------------------------------------------------------------------------------------
// This round's changes, as every CTA needs them in step 4.
// ------------------------------------------------------------------------------------------------
struct ChangeShared {
  int n_changed;                           // kept coefficients whose key of the next round changed
  int wsum[kWarps], rank_wsum[kWarps];
  unsigned long long dmax;                 // bits of the largest |change|
};

// Shared memory of step 4: the changed keys (old [n_keep], new [n_keep]), then either the moving columns (dense:
// residual) or the changed keys indexed by bin (draw_rank).
constexpr int kStage = 4096;               // moving columns staged at a time
struct Moving { double d[kStage]; long long off[kStage]; };
struct ChangedByBin { int before[kHistBins + (kHistBins >> 5)]; int head[kHistBins]; unsigned short next[2 * kStage]; };

// The kept coefficients' changes: how many move, the largest, the keys that change (in any order), and for dense X the
// moving columns in list order.  Returns the number that move.
constexpr int kFewChanged = 48;            // kept coefficients up to which draw_rank counts through all changed keys
template <bool kDense>
__device__ int gather_changes(const Problem& p, const Binning& bins, int nk, bool want_keys, unsigned long long* keys, ChangedByBin* cb, Moving* mv,
                              ChangeShared& cs) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool indexed = want_keys && nk > kFewChanged;
  __syncthreads();
  if (tid == 0) { cs.n_changed = 0; cs.dmax = 0ull; }
  if (indexed) {
    static_assert(sizeof(cb->before) % 16 == 0 && sizeof(cb->head) % 16 == 0, "cleared 16 bytes at a time");
    for (int i = tid; i < (int)(sizeof(cb->before) / 16); i += kT) reinterpret_cast<int4*>(cb->before)[i] = make_int4(0, 0, 0, 0);
    for (int i = tid; i < (int)(sizeof(cb->head) / 16); i += kT) reinterpret_cast<int4*>(cb->head)[i] = make_int4(-1, -1, -1, -1);
  }
  __syncthreads();
  const int per = (nk + kT - 1) / kT, a_lo = min(tid * per, nk), a_hi = min(a_lo + per, nk);
  unsigned long long dmax = 0ull;
  double d_first = 0.0;
  int moving = 0;
  for (int a = a_lo; a < a_hi; ++a) {
    const int pos = p.kept_pos[a];
    const double d = p.cand_dbeta64[pos];
    unsigned long long o = 0ull, w = 0ull;
    if (want_keys) { o = p.cand_keys[pos]; w = p.cand_keys[p.n_cand + pos]; }
    if (a == a_lo) d_first = d;
    moving += d != 0.0;
    dmax = max(dmax, (unsigned long long)__double_as_longlong(fabs(d)));
    if (o != w) {
      const int at = atomicAdd(&cs.n_changed, 1);
      keys[at] = o;
      keys[p.n_keep + at] = w;
      if (indexed) {                                     // by bin: a count for the prefix sum, and a list
        const unsigned int bo = bin_of(bins, (unsigned int)(o >> 32)), bw = bin_of(bins, (unsigned int)(w >> 32));
        atomicAdd(&cb->before[pad((int)bo)], -1);
        atomicAdd(&cb->before[pad((int)bw)], 1);
        cb->next[2 * at] = (unsigned short)atomicExch(&cb->head[bo], 2 * at);
        cb->next[2 * at + 1] = (unsigned short)atomicExch(&cb->head[bw], 2 * at + 1);
      }
    }
  }
  int incl = moving;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += v;
  }
  if (!kDense) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dmax = max(dmax, __shfl_xor_sync(kFull, dmax, o));
    if (lane == 0 && dmax) atomicMax(&cs.dmax, dmax);
  }
  if (lane == 31) cs.wsum[warp] = incl;
  __syncthreads();
  int before = 0, total = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) { const int v = cs.wsum[w]; if (w < warp) before += v; total += v; }
  if (kDense) {
    int rank = before + incl - moving;
    for (int a = a_lo; a < a_hi && rank < kStage; ++a) {
      const double d = a == a_lo ? d_first : p.cand_dbeta64[p.kept_pos[a]];
      if (d == 0.0) continue;
      mv->d[rank] = d;
      mv->off[rank] = (long long)p.kept[a] * p.ld;
      ++rank;
    }
    __syncthreads();
  }
  return total;
}

// [from, to) towards L2: the groups of 16 bytes that any of it lies in.
__device__ __forceinline__ void prefetch_l2(const void* from, const void* to) {
  const unsigned long long lo = (unsigned long long)from & ~15ull, hi = ((unsigned long long)to + 15ull) & ~15ull;
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(lo), "r"((unsigned)(hi - lo)) : "memory");
}

// Winners ranked; with changes, corrected for the kept coefficients' changed priorities (keys[0 .. n_changed) old,
// keys[p.n_keep ..) new).  A key's place among the changed ones: those in lower bins from a prefix sum over the bins, those
// in its own bin one by one (a list per bin); a plain count while they are few.
// Leaves the draw's buffers as the next scan expects them.
template <bool kDense>
__device__ __forceinline__ void draw_rank(const Problem& p, const Engine& e, const DrawShared& ds, const unsigned long long* keys, ChangedByBin* cb, int n_changed,
                          int nk, int* wsum, int n_rank, int n_prefetch) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if ((int)blockIdx.x >= n_rank) return;
  const Binning bins = binning_of(ds.cut);
  const unsigned int bnd = (unsigned)ds.bnd;
  unsigned int total = ds.off[pad((int)bnd)] + (ds.refined ? __ldcg(e.bin_cur + bnd) : ds.bnd_count);
  total = min(total, (unsigned)e.cap_win);
  const unsigned long long* old_k = keys;
  const unsigned long long* new_k = keys + p.n_keep;
  const bool indexed = nk > kFewChanged;                 // (gather_changes made the lists)
  if (indexed) {
    constexpr int kPer = kHistBins / kT;
    int c[kPer], mine = 0;
#pragma unroll
    for (int u = 0; u < kPer; ++u) { c[u] = cb->before[pad(tid * kPer + u)]; mine += c[u]; }
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += v;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    int run = incl - mine;
    for (int w = 0; w < warp; ++w) run += wsum[w];
#pragma unroll
    for (int u = 0; u < kPer; ++u) { cb->before[pad(tid * kPer + u)] = run; run += c[u]; }
    __syncthreads();
  }
  const int items = (int)total + (n_changed > 0 ? nk : 0);   // (new keys by place in the kept list: the order of `keys` is each CTA's own)
  const int shift = 64 - ds.bits;
  // lanes per winner: two where there are too many, eight for the larger groups of an unguided draw
  const int share = items * 4 > n_rank * kT ? 1 : (bins.cut == 0u && items * 8 <= n_rank * kT ? 3 : 2);
  const int lanes = 1 << share, slice = lane & (lanes - 1), per_warp = 32 >> share;
#pragma unroll 1
  for (int i0 = (warp * n_rank + (int)blockIdx.x) * per_warp; i0 < items; i0 += kWarps * n_rank * per_warp) {
    const int i = i0 + (lane >> share);
    const bool fresh = i >= (int)total;
    unsigned long long key = 0ull;
    bool on = i < items;
    if (on && !fresh) key = __ldcg(e.win + i);
    if (on && fresh) {
      const int pos = p.kept_pos[i - (int)total];
      key = p.cand_keys[p.n_cand + pos];
      on = key != p.cand_keys[pos];
    }
    const int j = (int)(key & 0xffffffffull);
    long long q0 = 0, q1 = 0;                            // CSC: where the column lies, under way meanwhile
    double n2 = 0.0;
    if (!kDense && on && slice == 0) { q0 = p.xptr[j]; q1 = p.xptr[j + 1]; n2 = p.n2[j]; }
    const unsigned int bin = bin_of(bins, (unsigned int)(key >> 32));
    // (a new key behind the boundary ranks behind all candidates: the winners before it are more than P')
    // -- unless the winners are all there are
    const bool behind = fresh && (bin > bnd || (bin == bnd && ds.refined && (key >> shift) > ds.prefix));
    if (behind && total < (unsigned long long)p.J) on = false;
    unsigned int first = 0u, count = 0u;
    if (on) { first = behind ? total : ds.off[pad((int)bin)]; count = behind ? 0u : (bin < bnd ? ds.off[pad((int)bin + 1)] : total) - first; }
    int below = 0, struck = 0;
#pragma unroll 1
    for (unsigned int k0 = slice; k0 < count; k0 += 8 * lanes) {
      unsigned long long v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = k0 + lanes * u < count ? __ldcg(e.win + first + k0 + lanes * u) : ~0ull;
#pragma unroll
      for (int u = 0; u < 8; ++u) below += v[u] < key;
    }
    if (!indexed) {
#pragma unroll 1
      for (int a = slice; a < n_changed; a += lanes) {
        const unsigned long long o = old_k[a];
        below -= o < key;
        struck |= o == key;
        below += new_k[a] < key;
      }
    } else if (on && slice == 0) {
      below += cb->before[pad((int)bin)];
      for (int n = cb->head[bin]; n >= 0 && n != 0xffff; n = cb->next[n]) {
        if (n & 1) {
          below += new_k[n >> 1] < key;
        } else {
          const unsigned long long o = old_k[n >> 1];
          below -= o < key;
          struck |= o == key;
        }
      }
    }
#pragma unroll 1
    for (int o = 1; o < lanes; o <<= 1) {
      below += __shfl_xor_sync(kFull, below, o);
      struck |= __shfl_xor_sync(kFull, struck, o);
    }
    const int rank = (int)first + below;
    if (on && slice == 0 && (fresh || !struck) && (unsigned)rank < (unsigned)p.n_cand) {
      p.cand[rank] = j;
      // the columns of the next round's window start towards L2 while this round's changes are applied
      if (kDense) {
        if (rank < n_prefetch)
          asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p.xv + (long long)j * p.ld), "r"((unsigned)((p.N + 3) >> 2) * 16u) : "memory");
      } else {
        WalkColumn col;
        col.q0 = q0; col.n = (int)(q1 - q0); col.j = j; col.n2 = n2; col.unused = 0.0;
        p.walk_cols[rank] = col;
        e.norm_f[rank] = (float)n2;
        if (rank < n_prefetch) {
          if (q1 > q0) { prefetch_l2(p.xrow + q0, p.xrow + q1); prefetch_l2(p.xv + q0, p.xv + q1); }
        }
      }
    }
  }
  // the next scan's buffers and cutoff (everybody read them before the last barrier)
  for (int b = (int)blockIdx.x * kT + tid; b < kHistBins; b += (int)gridDim.x * kT) e.hist[b] = 0u;
  if (blockIdx.x == 0 && tid == 0) {
    // twice the boundary, which changes little from round to round; more where few winners let it scatter
    const unsigned int edge = boundary_edge(ds);
    e.es->t_cut = edge < 0x7f800000u ? __fmul_rn(p.n_cand < 64 ? 8.0f : 2.0f, __uint_as_float(edge)) : 0.f;
  }
}

// ------------------------------------------------------------------------------------------------
// Would-be changes (Eq. 2): for the candidate at position `pos` with coefficient j, n = ||x_j||^2 and g = x_j^T r.
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ float exponential_of(const Problem& p, unsigned long long t, uint32_t j) {
  uint32_t w[4];
  philox4x32_10(j >> 2, (uint32_t)t, (uint32_t)(t >> 32), 0u, (uint32_t)p.seed, (uint32_t)(p.seed >> 32), w);
  return unit_exponential_rn((j & 2u) ? ((j & 1u) ? w[3] : w[2]) : ((j & 1u) ? w[1] : w[0]));
}

// In two parts: what does not depend on g is made while the products are under way.
struct Proposal { double n, threshold; float b_old; unsigned long long old_key; };
__device__ __forceinline__ Proposal propose_begin(const Problem& p, int j, double n, float b_old, float d_old, float E, bool want_keys) {
  Proposal q;
  q.n = n; q.b_old = b_old;
  q.threshold = n > 0.0 ? step_scale(p) * (double)p.lambda / n : 0.0;
  q.old_key = want_keys ? race_key_from(E, d_old, p.eta, (uint32_t)j, weight_mode_of(p.flags)) : 0ull;
  return q;
}
__device__ __forceinline__ void propose_end(const Problem& p, const Proposal& q, int pos, int j, double g, float E, bool want_keys) {
  float b_new = q.b_old;
  if (q.n > 0.0) {
    const double z = (double)q.b_old + step_scale(p) * g / q.n;
    const double m = fabs(z) - q.threshold;
    b_new = (float)(m <= 0.0 ? 0.0 : (z > 0.0 ? m : -m));
  }
  const double d = isfinite(g) ? (double)b_new - (double)q.b_old : g - g;      // a non-finite product shows as NaN
  p.cand_bnew[pos] = b_new;
  p.cand_dbeta64[pos] = d;
  if (want_keys) {
    p.cand_keys[pos] = q.old_key;
    p.cand_keys[p.n_cand + pos] = race_key_from(E, (float)fabs(d), p.eta, (uint32_t)j, weight_mode_of(p.flags));
  }
}

constexpr int kMaxWords = STRADS_MAX_CANDIDATES / 32;
constexpr int kTurn = 32;                  // candidates a CTA handles per turn of step 1 (dense) / 2 (CSC)

struct RoundOutputs { int* cand; int* kept; float* dbeta; int* counts; };

__device__ void commit_changes(const Problem& p, const Engine& e, int nk, int n_moving, const RoundOutputs& out, bool last) {
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
    const int examined = e.es->n_examined;
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
struct TurnShared { double dot[kTurn][kWarps]; };
struct PackBars { unsigned long long full[kWarps]; unsigned int uses[kWarps]; };

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
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
// CSC, steps 1 and 2: the window's pairs that share a row, by row buckets as in gram_csc.cu -- but a warp per candidate
// (its terms in a list of the warp's own in shared memory: no barrier), no conflict bits (the walk works from the list
// of conflicting pairs or forms rows on demand), and x_c^T r with the same visit to the column.
// ------------------------------------------------------------------------------------------------
constexpr int kMet = 512;                                // candidates one candidate may meet (of kReach)
constexpr int kRing = 4;                                 // steps of terms under way, and the one at hand
constexpr int kReach = 1664;                             // candidates a warp has a place for at a time: a window of 1,024 kept
constexpr int kPart = 64;                                // positions of a column at a time
constexpr int kWorkers = kWarps - 1;                     // warps that form products; the last one makes the would-be changes
struct __align__(16) MetTable {
  int4 entry[kPart];                     // of a position of the column: row, terms before it, value
  float dot[kReach];                     // by candidate; zero between candidates
  unsigned short met[kMet];              // the places in use
  unsigned char lane[kReach];            // that had a term of the candidate last
  unsigned char pos[kPart * kBucketSlots];   // position of a term
  int2 term[kRing][32];                  // terms of the next steps: candidate and its value
  float value[kRing][32];                // ... the column's
};
constexpr int kNear = 2048;                              // candidates whose norms a CTA keeps in shared memory
constexpr size_t kTermsSmem = sizeof(MetTable) * kWorkers + sizeof(float) * kNear;
static_assert(STRADS_MAX_CANDIDATES < 0xffff && kPart <= 256, "16 bits per candidate, 8 per position");

// The entries of candidates [0, n) into the buckets of their rows.  Where the columns lie was noted when the candidates
// were ranked, but for the dependencies dropped at run time (coupling_n2 follows beta and delta).
__device__ __forceinline__ void csc_enter(const Problem& p, const Engine& e, int n, bool buckets) {
  const int lane = threadIdx.x & 31;
  const bool dynamic = (p.flags & STRADS_FLAG_DYNAMIC_DEPS) != 0;
  if (!buckets && !dynamic) return;
#pragma unroll 1
  for (int a = ((int)threadIdx.x >> 5) * (int)gridDim.x + (int)blockIdx.x; a < n; a += kWarps * (int)gridDim.x) {
    const WalkColumn col = p.walk_cols[a];
    if (dynamic && lane == 0) {
      const double n2 = coupling_n2(p, col.j);
      p.walk_cols[a].n2 = n2;
      e.norm_f[a] = (float)n2;
    }
    if (!buckets) continue;
    for (int q = lane; q < col.n; q += 32) {
      const int r = __ldg(p.xrow + col.q0 + q);
      const float v = __ldg(p.xv + col.q0 + q);
      const unsigned int slot = atomicAdd(&p.bucket_count[r], 1u);
      if (slot < (unsigned)kBucketSlots) p.bucket_pairs[(size_t)r * kBucketSlots + slot] = make_int2(a, __float_as_int(v));
    }
  }
}

// Emptied again by all CTAs but the last, which walks meanwhile.  In two parts, so that what there is to fetch is under way while
// the winners are collected: the rows of a warp's first candidate, two per lane; the others at once.
struct ClearAhead { int row[2]; };
__device__ __forceinline__ ClearAhead csc_clear_begin(const Problem& p, int n) {
  const int cta = (int)blockIdx.x, n_ctas = max(1, (int)gridDim.x - 1), lane = threadIdx.x & 31;
  ClearAhead c = {{-1, -1}};
  if (cta >= n_ctas) return c;
  const int first = ((int)threadIdx.x >> 5) * n_ctas + cta;
  for (int a = first; a < n; a += kWarps * n_ctas) {
    const WalkColumn col = p.walk_cols[a];
    if (a == first) {
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (lane + 32 * h < col.n) c.row[h] = __ldg(p.xrow + col.q0 + lane + 32 * h);
    }
    for (int q = lane + (a == first ? 64 : 0); q < col.n; q += 32) p.bucket_count[__ldg(p.xrow + col.q0 + q)] = 0u;
  }
  return c;
}
__device__ __forceinline__ void csc_clear_end(const Problem& p, const ClearAhead& c) {
#pragma unroll
  for (int h = 0; h < 2; ++h) if (c.row[h] >= 0) p.bucket_count[c.row[h]] = 0u;
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

// x_c^T r and the would-be changes of candidates [0, count) (kept: of the kept ones), and with `pairs` their inner
// products with the later candidates that share a row with them.  The CTA's k-th entry is cta + k * ctas; a warp per entry.
// What bounds it is the chain of dependent far accesses -- column, row, bucket -- so each link's loads go out together,
// and then the number of instructions per term.  The terms of 64 positions are laid out in the order of positions and dealt to
// the lanes, however unevenly the buckets are filled; a term is added to its candidate's product in an array of the
// warp's, terms of one candidate within a warp's step one after the other.  Whether a step has such terms shows when every
// lane writes its number to its candidate's place and reads it back: 280 cycles a step of 32 terms, where matching all lanes and
// a table with 16-bit compare-and-swap took 650 (match 160, compare-and-swap 200).
// The would-be changes are made by a warp of their own, which has what it needs of the candidates by the time x_c^T r are there.
// 50,000 x 1,000,000, 1,664 candidates of 50 entries: 37.4 -> 35.3 us per round; 5,000 x 100,003, 384 candidates: 29.3 -> 28.1.
// (the tables, and the norms where they do not follow beta and delta: before the barrier that the buckets wait for)
__device__ __forceinline__ void csc_norms(const Problem& p, const Engine& e, unsigned char* sm, int count) {
  float* norm_f = reinterpret_cast<float*>(sm + sizeof(MetTable) * kWorkers);
  for (int i = threadIdx.x; i < min(count, kNear); i += kT) norm_f[i] = __ldcg(e.norm_f + i);
}
__device__ __forceinline__ void csc_products_begin(const Problem& p, const Engine& e, unsigned char* sm, int count) {
  MetTable& wt = reinterpret_cast<MetTable*>(sm)[threadIdx.x >> 5];
  __syncthreads();                                       // (what lay there before)
  if (threadIdx.x < 32 * kWorkers)
    for (int i = threadIdx.x & 31; i < kReach / 4; i += 32) reinterpret_cast<float4*>(wt.dot)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (!(p.flags & STRADS_FLAG_DYNAMIC_DEPS)) csc_norms(p, e, sm, count);
}
__device__ __forceinline__ void csc_products(const Problem& p, const Engine& e, TurnShared& ts, unsigned char* sm, int count, bool kept, bool pairs,
                                             unsigned long long t_next, bool want_keys) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int cta = (int)blockIdx.x, n_ctas = (int)gridDim.x;
  const double rho = (double)p.rho;
  MetTable& wt = reinterpret_cast<MetTable*>(sm)[warp];
  float* norm_f = reinterpret_cast<float*>(sm + sizeof(MetTable) * kWorkers);
  const int mine = count > cta ? (count - cta + n_ctas - 1) / n_ctas : 0;
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
    if (warp >= turn) asm volatile("bar.arrive 4, %0;" ::"n"(kT) : "memory");
#pragma unroll 1
    for (int k = warp; k < turn; k += kWorkers) {
      const int a = cta + n_ctas * (k0 + k);
      const WalkColumn col = p.walk_cols[kept ? p.kept_pos[a] : a];
      double acc = 0.0;
      auto tell = [&]() {                                // this candidate's x_c^T r; the last one of the warp's: all of them
        acc = warp_sum(acc);
        if (lane == 0) ts.dot[k][0] = acc;
        if (k + kWorkers >= turn) {
          __threadfence_block();
          __syncwarp();
          asm volatile("bar.arrive 4, %0;" ::"n"(kT) : "memory");
        }
      };
      if (col.n <= 0) tell();
      const int reach0 = pairs ? a / kReach * kReach : 0;
#pragma unroll 1
      for (int reach = reach0; reach == reach0 || reach < count; reach += kReach) {      // (one trip up to a window of kReach)
        int n_met = 0;                                   // (the same in all lanes)
        bool failed = false;
#pragma unroll 1
        for (int q0 = 0; q0 < col.n; q0 += kPart) {
          int r[2];
          float v[2];
          unsigned int cnt[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int q = q0 + 32 * h + lane;
            r[h] = q < col.n ? __ldg(p.xrow + col.q0 + q) : -1;
            v[h] = q < col.n ? __ldg(p.xv + col.q0 + q) : 0.f;
          }
          float x[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            x[h] = r[h] >= 0 && reach == reach0 ? p.resid[r[h]] : 0.f;
            cnt[h] = pairs && r[h] >= 0 ? p.bucket_count[r[h]] : 0u;
          }
          if (reach == reach0) {
#pragma unroll
            for (int h = 0; h < 2; ++h)
              if (r[h] >= 0) acc += (double)v[h] * (double)x[h];
            if (q0 + kPart >= col.n) tell();
          }
          if (!pairs) continue;
#pragma unroll
          for (int h = 0; h < 2; ++h)
            if (cnt[h] > (unsigned)kBucketSlots) { failed = true; cnt[h] = 0u; }
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
            wt.entry[32 * h + lane] = make_int4(r[h], off[h], __float_as_int(v[h]), 0);
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
              asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(&wt.term[i % kRing][lane])),
                           "l"(p.bucket_pairs + (size_t)en.x * kBucketSlots + (at - en.y)) : "memory");
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
            const bool on = term.b > a && (unsigned)(term.b - reach) < (unsigned)kReach;
            const int b = on ? term.b - reach : 0;
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
        if (!pairs) break;
        const bool overflow = __any_sync(kFull, failed) || n_met > kMet;
        if (overflow && lane == 0) e.es->bucket_failed = 1;
        // which of them conflict: those that may are gathered first, so that the far accesses are made for all of them at once
        const float limit_a = (float)(rho * rho * col.n2);
        int n_near = 0;
#pragma unroll 1
        for (int i0 = 0; i0 < min(n_met, kMet); i0 += 32) {
          const bool on = i0 + lane < min(n_met, kMet);
          const int b = on ? wt.met[i0 + lane] : 0;
          const float dot = on ? wt.dot[b] : 0.f;
          const bool near = on && may_conflict(dot, limit_a, b + reach < kNear ? norm_f[b + reach] : __ldcg(e.norm_f + b + reach));
          if (on && !near) wt.dot[b] = 0.f;
          const unsigned int m = __ballot_sync(kFull, near);
          if (near) wt.met[n_near + __popc(m & ((1u << lane) - 1u))] = (unsigned short)b;      // (places that have been read)
          n_near += __popc(m);
          __syncwarp();
        }
#pragma unroll 1
        for (int i0 = 0; i0 < n_near; i0 += 32) {
          const bool on = i0 + lane < n_near;
          const int b = on ? wt.met[i0 + lane] : 0;
          const float dot = on ? wt.dot[b] : 0.f;
          __syncwarp();
          bool conflict = false;
          if (on) {
            wt.dot[b] = 0.f;
            conflict = dot != 0.f && in_conflict(dot, limit_a, col.n2, b + reach < kNear ? norm_f[b + reach] : __ldcg(e.norm_f + b + reach), p.walk_cols + b + reach, rho);
          }
          const unsigned int m = __ballot_sync(kFull, conflict);
          if (m == 0u) continue;
          unsigned int at = 0u;
          if (lane == 0) at = atomicAdd(&e.es->edge_count, (unsigned)__popc(m));
          at = __shfl_sync(kFull, at, 0) + (unsigned)__popc(m & ((1u << lane) - 1u));
          if (conflict && at < (unsigned)p.cap_edges) p.edges[at] = ((unsigned int)a << 16) | (unsigned)(b + reach);
        }
        __syncwarp();
        if (n_met > kMet)                                // (places that were not listed)
          for (int i = lane; i < kReach; i += 32) wt.dot[i] = 0.f;
        __syncwarp();
      }
    }
  }
}

// ------------------------------------------------------------------------------------------------
// CSC, step 4 and the next step 1: the residual.  Contributions are added as 64-bit fixed-point integers (unit 2^-shift, the
// same bits in any order) and every row with a non-zero accumulator is updated once behind the next barrier.
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ int csc_shift(const Problem& p, unsigned long long dmax_bits, int nk) {
  const double m = __longlong_as_double((long long)dmax_bits);
  if (!(m > 0.0) || !isfinite(m)) return INT_MIN;
  int x = 0;
  frexp(m * (double)p.st->x_abs_max * (double)max(nk, 1), &x);
  return 61 - x;
}

template <typename F>
__device__ __forceinline__ void for_moving_entries(const Problem& p, int nk, F&& f) {
  const int lane = threadIdx.x & 31;
  for (int a = ((int)threadIdx.x >> 5) * (int)gridDim.x + (int)blockIdx.x; a < nk; a += kWarps * (int)gridDim.x) {
    const double d = p.cand_dbeta64[p.kept_pos[a]];
    if (d == 0.0) continue;
    const int j = p.kept[a];
    const long long q1 = p.xptr[j + 1];
    for (long long q = p.xptr[j] + lane; q < q1; q += 32) f(q, d);
  }
}

__device__ void csc_scatter(const Problem& p, int nk, int shift) {
  if (shift == INT_MIN) return;
  for_moving_entries(p, nk, [&](long long q, double d) {
    const long long fx = __double2ll_rn(ldexp((double)__ldg(p.xv + q) * d, shift));
    atomicAdd(reinterpret_cast<unsigned long long*>(p.resid_acc + __ldg(p.xrow + q)), (unsigned long long)fx);
  });
}

__device__ void csc_apply(const Problem& p, int nk, int n_moving, int shift) {
  if (shift == INT_MIN) return;
  // few moving entries against the rows: visit the entries' rows (the first visitor of a row takes its sum), else all rows
  if ((double)n_moving * (double)p.nnz * 4.0 < (double)p.N * (double)p.J) {
    for_moving_entries(p, nk, [&](long long q, double) {
      const int r = __ldg(p.xrow + q);
      const long long v = (long long)atomicExch(reinterpret_cast<unsigned long long*>(p.resid_acc + r), 0ull);
      if (v != 0) apply_row(p, r, ldexp((double)v, -shift));
    });
    return;
  }
  for (long long r = (long long)blockIdx.x * kT + threadIdx.x; r < p.N; r += (long long)gridDim.x * kT) {
    const long long v = p.resid_acc[r];
    if (v != 0) {
      apply_row(p, r, ldexp((double)v, -shift));
      p.resid_acc[r] = 0;
    }
  }
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
constexpr int kRestEntries = kOwnEntries * 3 / 2;
// Survivors that are settled at once: as many as a thread pair of bits per walking thread holds, and while their entries, all of
// which every CTA goes through, are no more than these (us per round for 1,500 / 2,600 / 4,096 / 7,000 / 12,288: 10^7 columns of 20
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

// The columns of `count` candidates (thread i of kOwn has the i-th) into row / val, one behind the other, as far as there is room.
// Bound by the lines a load touches, so several threads share a column.  Bar: the threads' barrier.
template <int kBar>
__device__ __forceinline__ void hold_columns(const Problem& p, DemandShared& s, int i, int count, const WalkColumn& col, int* row, float* val, int room) {
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
__device__ __forceinline__ bool settle_rest(const Problem& p, const Problem& sp, DemandShared& s, Grid& g, int total, int m, bool table, int& kept,
                                            int& examined) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, cta = (int)blockIdx.x, n_ctas = (int)gridDim.x;
  const int W = (total + 31) >> 5, pitch = (W + 3) & ~3;
  const double rho = (double)p.rho;
  constexpr int kTogether = 4;                           // members at a time
  constexpr int kU = 8;                                  // entries of a candidate's column at a time
  const int behind = cta + (m - 1) * n_ctas;             // candidates before the last member
  for (int c0 = 0, here; c0 < behind; c0 += here) {      // as many at a time as there is room for
    const int count = min(behind - c0, kOwn);
    WalkColumn col = {};
    if (tid < count) col = p.walk_cols[s.survivor[c0 + tid]];
    hold_columns<1>(p, s, tid, count, col, s.rrow, s.rval, kRestEntries);
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
template <typename Draw>
__device__ __forceinline__ bool csc_walk_on_demand(const Problem& p, Problem& sp, const Engine& e, unsigned char* sm, Grid& g, Grid& g_draw, int* n_kept,
                                                   Draw&& draw) {
  DemandShared& s = *reinterpret_cast<DemandShared*>(sm);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int cta = (int)blockIdx.x, n_ctas = (int)gridDim.x, n = p.n_cand, W = (n + 31) >> 5;
  // this CTA's words of the mask: cta, cta + n_ctas, ...; its k-th candidate is bit k & 31 of the (k / 32)-th of them
  const int own_words = W > cta ? (W - cta + n_ctas - 1) / n_ctas : 0, n_own = own_words * 32, n_here = min(n_own, kOwn);
  auto own_index = [&](int k) { return ((cta + (k >> 5) * n_ctas) << 5) | (k & 31); };
  __syncthreads();
  if (warp >= kWalkWarps) {
    for (int w = tid - kWalkT; w < own_words; w += kT - kWalkT) s.own_word[w] = s.own_hit[w] = 0u;
    {
      const int i = tid - kWalkT;
      WalkColumn col = {};
      if (i < n_here && own_index(i) < n) col = p.walk_cols[own_index(i)];
      hold_columns<2>(p, s, i, n_here, col, s.orow, s.oval, kOwnEntries);
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
        ok = settle_rest(p, sp, s, g, total, m, table, kept, examined);
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
      const int room = p.n_keep - kept;
      const bool done = __popc(keep) >= room;            // stop exactly at P: drop the surplus from the back
      while (__popc(keep) > room) keep &= ~(1u << (31 - __clz((int)keep)));
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
            if (end > kOwnEntries) end = from;
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
              if (sl[u] != kNoSlot) s.omet[from + met + __popc(mine & ((1u << lane) - 1u))] = sl[u] | (unsigned)(i0 + (u << share) - from) << 16;
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
          if (table && k < kOwn && s.own_at[k + 1] <= kOwnEntries) {
            n2b = s.own_n2[k];
            const int met = s.n_met[k], from = s.own_at[k];
            dot = row_products(s, qk, met, met, [&](int x, uint2& rec, float& v) {
              const unsigned int en = s.omet[from + x];
              rec = s.row_rec[en & 0xffffu]; v = s.oval[from + (int)(en >> 16)];
            });
          } else if (table) {                            // (no room for its column)
            const WalkColumn cb = p.walk_cols[own_index(k)];
            n2b = cb.n2;
            for (int x = 0; x < cb.n; ++x) {
              const int row[1] = {__ldg(p.xrow + cb.q0 + x)};
              unsigned int sl[1];
              find_rows<1>(s, row, 1u << qk, sl);
              const uint2 rec[1] = {s.row_rec[sl[0] != kNoSlot ? sl[0] : 0u]};
              const float v[1] = {__ldg(p.xv + cb.q0 + x)};
              if (sl[0] != kNoSlot) dot = add_products<1>(s, qk, rec, v, dot);
            }
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
  __shared__ int s_kept, s_examined;
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
      csc_apply(p, last.nk, last.n_moving, last.shift);
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
    bool window = true;
    if (kDense) {
      if (n < n_total && es->skip_window && !no_filter) n = n_total;
    } else {
      window = no_filter || (p.bucket_count != nullptr && !(n < n_total && es->skip_window) && es->avoid == 0);
      if (real) csc_enter(p, e, window ? n : n_total, window && !no_filter);
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
      if (!scanned && !during_walk) { draw_scan(p, e, ds, sm, td, true); scanned = true; }
      if (kDense) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // (the Gram's operands come in over it)
      // (the walk needs nothing of what is before it but the norms that follow beta and delta)
      if (ahead) {
        if (!kDense) csc_products_begin(p, e, sm, n);
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
      if (!collected && !csc_window && !during_walk) { draw_gather<AllThreads>(p, e, ds, k, spare); collected = true; }
      if (!kDense && real) {
        if (!window) {
          unsigned char* sm_scan = sm + sizeof(DemandShared);
          unsigned int* sh = reinterpret_cast<unsigned int*>(sm_scan);
          const float cut = during_walk ? scan_open(e, ds, sm_scan, true) : 0.f;
          const Binning bins = binning_of(cut);
          const WeightForm wf = weight_form(p);
          auto draw = [&]() {
            if (!during_walk) return true;
            WarpScan scan = begin_scan(cut, scan_queue(sm_scan), (warp - kWalkWarps) * n_ctas + cta, (kWarps - kWalkWarps) * n_ctas);
#pragma unroll 1
            while (scan_step(p, td, wf, scan, [&](unsigned long long key, bool on) { scan_found(e, ds, sh, bins, key, on); })) {}
            scan_close<OtherThreads>(e, ds, sm_scan);
            __shared__ int s_over;
            g_draw.target += g_draw.n;
            OtherThreads::sync();
            if (OtherThreads::tid() == 0) s_over = grid_wait(g_draw);
            OtherThreads::sync();
            if (!s_over) return false;
            draw_gather<OtherThreads>(p, e, ds, k, false);
            return true;
          };
          int walked = 0;
          if (!(ok = csc_walk_on_demand(p, sp, e, sm, g, g_draw, &walked, draw))) break;
          if (during_walk) scanned = collected = true;
          csc_products(p, e, ts, sm, walked, true, false, t + 1, draws);
        } else {
          csc_products(p, e, ts, sm, n, false, csc_window, t + 1, draws);
        }
      }
      if (!(ok = grid_sync(g))) break;
      if (!real || no_filter) break;
      if (!kDense) {
        if (!window) break;
        if (walker) {
          const unsigned int edges = es->edge_count;
          const int failed = es->bucket_failed;
          if (tid == 0) { s_kept = 0; s_examined = n; }
          __syncthreads();
          bool settled = !failed && edges <= (unsigned)p.cap_edges;
          if (settled) settled = walk_from_pair_list<kT>(p, p.cand, n, edges, sm, p.kept, &s_kept, &s_examined);
          __syncthreads();
          if (tid == 0) {
            es->n_kept = s_kept; es->n_examined = s_examined;
            es->walk_open = !settled || (s_kept < p.n_keep && n < n_total) ? 1 : 0;
            // after an overflow the buckets are left alone: for a round, then twice as long after every further one, to 64
            // (a count of rounds, not the round to wait for: strads_set_round may go back); this round's walk counts too
            if (!settled) es->avoid = 1 + (1 << es->streak);
            es->streak = settled ? 0 : min(es->streak + 1, 6);
            es->bucket_failed = 0; es->edge_count = 0u;
          }
        }
        const ClearAhead rows = csc_clear_begin(p, n);
        if (!collected) { draw_gather<AllThreads>(p, e, ds, k, true); collected = true; spare = true; }
        csc_clear_end(p, rows);
        if (!(ok = grid_sync(g))) break;
        if (!es->walk_open) break;
        csc_enter(p, e, n_total, false);
        window = false;
      } else {
        if (!es->walk_open) break;
        packed = n; n = n_total;
      }
    }
    if (!ok) break;
    if (draws && es->mend) {
      keep_parameters();
      if (!(ok = draw_mend(sp, se, ds, sm, td, k, g))) break;
    }
    // ---- step 4 ----
    int n_changed = 0, nk = 0;
    const int n_next = no_filter ? p.n_keep : (e.window < n_total && es->skip_window ? n_total : e.window);   // looked at first
    if (real) {
      nk = es->n_kept;
      const int n_moving = gather_changes<kDense>(p, binning_of(ds.cut), nk, draws, keys, cb, mv, cs);
      n_changed = cs.n_changed;
      commit_changes(p, e, nk, n_moving, out, final_round);
      last.nk = nk; last.n_moving = n_moving;
      if (!kDense) {
        last.shift = csc_shift(p, cs.dmax, nk);
        csc_scatter(p, nk, last.shift);
      }
      --left;
      ++t;
    }
    if (draws) draw_rank<kDense>(p, e, ds, keys, cb, n_changed, nk, cs.rank_wsum, spare ? max(1, n_ctas - 1) : n_ctas, n_next);
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
// one launch and a clear before it still took 16.4, so the kernel leaves its scratch clear instead.
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
    if (!draw_refine(sp, se, ds, sm, t, (unsigned)p.n_cand, g)) return false;
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
    draw_collect_all(sp, se, ds, sm, t);
  }
  if (!grid_sync(g)) return false;
  draw_rank<true>(p, e, ds, nullptr, nullptr, 0, 0, nullptr, (int)gridDim.x, 0);       // (leaves the histogram clear)
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

size_t smem_of(bool dense, int n_keep, bool ahead, int n_cand) {
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
    at_least(walk_pairs_smem(n_cand, 8192));
    if (ahead) at_least(keys + sizeof(ChangedByBin));
  }
  return need;
}

}  // namespace

size_t engine_smem(const Problem& p, bool ahead) { return smem_of(p.layout == STRADS_DENSE_COLMAJOR, p.n_keep, ahead, p.n_cand); }

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
