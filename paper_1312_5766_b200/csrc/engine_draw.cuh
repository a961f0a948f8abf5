// Rounds in one launch: the grid barrier, the draw, and a round's changes as the draw of a later one needs them (engine.cu has the
// order of the steps).
#pragma once
#include <climits>

#include "engine.cuh"

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

// The CTAs that make a round together: all of them, or as many of them as prepare the rounds whose turn is theirs (squads.cu).
struct WholeGrid {
  static constexpr bool kParts = false;    // all coefficients
  static constexpr bool kKeys = false;     // the winners' keys are not wanted beside the list
  static constexpr int kTogether = 1;      // entries of a list that a warp goes through side by side: it has one as a rule
  __device__ __forceinline__ int rank() const { return (int)blockIdx.x; }
  __device__ __forceinline__ int size() const { return (int)gridDim.x; }
};
struct Squad {
  static constexpr bool kParts = true;     // a scheduler's
  static constexpr bool kKeys = false;
  static constexpr int kTogether = 4;
  int r, n;
  __device__ __forceinline__ int rank() const { return r; }
  __device__ __forceinline__ int size() const { return n; }
};

// The CTAs of a launch of one thread-block cluster (draw_cluster.cu), and their barrier.
struct ClusterCrew {
  static constexpr bool kParts = true, kKeys = true;
  static constexpr int kTogether = 1;
  __device__ __forceinline__ int rank() const { return (int)blockIdx.x; }
  __device__ __forceinline__ int size() const { return (int)gridDim.x; }
};
struct ClusterGrid {};
__device__ __forceinline__ bool grid_sync(ClusterGrid&) {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  return true;
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

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

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
// The keys of the coefficients in the queue, computed by all lanes together.
template <typename F>
__device__ __forceinline__ void scan_flush(const Problem& p, const WeightForm& wf, WarpScan& s, F&& f) {
  const int lane = threadIdx.x & 31;
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
// A step over a scheduler's coefficients, 64 of them or 32 groups of four.  With four schedulers or more a group has one coefficient of
// each at most, so that the coefficients are enumerated (a Philox block each, 1 / S of them all); with two or three a group has two at most.
template <typename F>
__device__ __forceinline__ bool scan_step_part(const Problem& p, unsigned long long t, const WeightForm& wf, WarpScan& s, F&& f) {
  const int lane = threadIdx.x & 31;
  const unsigned int S = (unsigned)p.part_count, idx = (unsigned)p.part_index;
  const bool each = S >= 4u;
  const long long units = each ? (owned_count(p) + 1) >> 1 : (p.J + 3) >> 2;
  const bool more = s.next < units;
  if (!more && s.n == 0) return false;
  if (more) {
    long long j[2];
    uint32_t word[2];
    if (each) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        j[u] = idx + (long long)S * (2 * s.next + 32 * u + lane);
        uint32_t w[4];
        philox4x32_10((uint32_t)(j[u] >> 2), (uint32_t)t, (uint32_t)(t >> 32), 0u, (uint32_t)p.seed, (uint32_t)(p.seed >> 32), w);
        word[u] = (j[u] & 2) ? ((j[u] & 1) ? w[3] : w[2]) : ((j[u] & 1) ? w[1] : w[0]);
      }
    } else {
      const long long g = s.next + lane;
      uint32_t w[4];
      philox4x32_10((uint32_t)g, (uint32_t)t, (uint32_t)(t >> 32), 0u, (uint32_t)p.seed, (uint32_t)(p.seed >> 32), w);
      const unsigned int m = S == 3u ? (uint32_t)g % 3u : 0u;            // 4 g mod S
      const unsigned int i = idx >= m ? idx - m : idx + S - m;
      j[0] = (g << 2) + i;
      word[0] = i == 0u ? w[0] : (i == 1u ? w[1] : w[2]);
      j[1] = i + S < 4u ? j[0] + S : p.J;
      word[1] = i + S == 2u ? w[2] : w[3];
    }
    s.next += s.step;
    bool in[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const float d = j[u] < p.J ? __ldcg(p.delta + j[u]) : 0.f;
      in[u] = j[u] < p.J && !(__uint2float_rn(word[u]) > __fmul_rn(s.k, weight_of(wf, d)));
    }
    if (!__any_sync(kFull, in[0] | in[1])) return true;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const unsigned int m = __ballot_sync(kFull, in[u]);
      if (in[u]) s.queue[s.n + __popc(m & ((1u << lane) - 1u))] = make_uint2((uint32_t)j[u], word[u]);
      s.n += __popc(m);
    }
  }
  if (s.n > kQueue - 128 || !more) scan_flush(p, wf, s, f);
  return true;
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
  if (s.n > kQueue - 128 || !more) scan_flush(p, wf, s, f);
  return true;
}
template <bool kParts, typename F>
__device__ __forceinline__ void scan_all(const Problem& p, unsigned long long t, const WeightForm& wf, WarpScan& s, F&& f) {
  if (kParts && p.part_count > 1) {
#pragma unroll 1
    while (scan_step_part(p, t, wf, s, f)) {}
  } else {
#pragma unroll 1
    while (scan_step(p, t, wf, s, f)) {}
  }
}
template <bool kParts, typename F>
__device__ __forceinline__ void scan_keys(const Problem& p, unsigned long long t, float cut, uint2* queue, int warp0, int n_warps, F&& f) {
  const WeightForm wf = weight_form(p);
  WarpScan s = begin_scan(cut, queue, warp0, n_warps);
  scan_all<kParts>(p, t, wf, s, f);
}

// Shared memory of a scan: the CTA's histogram, then a queue per warp.
constexpr size_t kScanSmem = sizeof(unsigned int) * kHistBins + sizeof(uint2) * kQueue * kWarps;

// A scan in parts: it can be made in the waits of other work.  guided: with the cutoff es->t_cut (if there is one).
template <typename Crew>
__device__ __forceinline__ float scan_open(const Crew& crew, const Engine& e, DrawShared& ds, unsigned char* sm, bool guided) {
  unsigned int* sh = reinterpret_cast<unsigned int*>(sm);
  const int tid = threadIdx.x;
  const float cut = guided ? e.es->t_cut : 0.f;
  __syncthreads();
  for (int b = tid; b < kHistBins; b += kT) sh[b] = 0u;
  for (int b = crew.rank() * kT + tid; b < kHistBins; b += crew.size() * kT) e.bin_cur[b] = 0u;     // the cursors of the groups
  if (tid == 0) { ds.cut = cut; ds.saved = 0u; }
  __syncthreads();
  return cut;
}
template <typename Crew>
__device__ __forceinline__ void scan_found(const Crew& crew, const Engine& e, DrawShared& ds, unsigned int* sh, const Binning& bins, unsigned long long key, bool on) {
  const unsigned int bits = (unsigned int)(key >> 32);
  if (!on || (bins.cut != 0u && bits >= bins.cut)) return;
  atomicAdd(&sh[bin_of(bins, bits)], 1u);
  if (bins.cut != 0u) {
    const unsigned int at = atomicAdd(&ds.saved, 1u);
    if (at < e.cap_surv) e.surv[(size_t)crew.rank() * e.cap_surv + at] = key;
  }
}
template <typename Team, typename Crew>
__device__ __forceinline__ void scan_close(const Crew& crew, const Engine& e, const DrawShared& ds, unsigned char* sm) {
  const unsigned int* sh = reinterpret_cast<const unsigned int*>(sm);
  Team::sync();
  if (Team::tid() == 0) e.saved[crew.rank()] = ds.saved;
  for (int b = Team::tid(); b < kHistBins; b += Team::kN) {
    const unsigned int v = sh[b];
    if (v) atomicAdd(&e.hist[b], v);
  }
}
__device__ __forceinline__ uint2* scan_queue(unsigned char* sm) {
  return reinterpret_cast<uint2*>(sm + sizeof(unsigned int) * kHistBins) + (threadIdx.x >> 5) * kQueue;
}

// (a warp takes its steps round-robin over the CTAs: a few thousand coefficients already use every SM)
template <typename Crew>
__device__ __forceinline__ void draw_scan(const Crew& crew, const Problem& p, const Engine& e, DrawShared& ds, unsigned char* sm, unsigned long long t, bool guided) {
  unsigned int* sh = reinterpret_cast<unsigned int*>(sm);
  const float cut = scan_open(crew, e, ds, sm, guided);
  const Binning bins = binning_of(cut);
  scan_keys<Crew::kParts>(p, t, cut, scan_queue(sm), (int)(threadIdx.x >> 5) * crew.size() + crew.rank(), kWarps * crew.size(),
            [&](unsigned long long key, bool on) { scan_found(crew, e, ds, sh, bins, key, on); });
  scan_close<AllThreads>(crew, e, ds, sm);
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
template <typename Crew>
__device__ __noinline__ void draw_collect_all(const Crew& crew, const Problem& p, const Engine& e, const DrawShared& ds, unsigned char* sm, unsigned long long t) {
  const int warp = (int)threadIdx.x >> 5;
  const Binning bins = binning_of(ds.cut);
  const unsigned int edge = boundary_edge(ds);
  uint2* queue = reinterpret_cast<uint2*>(sm + sizeof(unsigned int) * kHistBins) + warp * kQueue;
  __syncthreads();
  scan_keys<Crew::kParts>(p, t, edge < 0x7f800000u ? __uint_as_float(edge) : 0.f, queue, warp * crew.size() + crew.rank(), kWarps * crew.size(),
            [&](unsigned long long key, bool on) { if (on) take_winner(e, ds, bins, key); });
}

// ... from the keys the scan saved: every CTA its own (the first of each thread in `key`), and a share of the last one's where that
// has other work.
template <typename Team, typename Crew>
__device__ __forceinline__ void draw_collect(const Crew& crew, const Engine& e, const DrawShared& ds, unsigned long long key, bool spare_last) {
  const Binning bins = binning_of(ds.cut);
  const unsigned int own = ds.saved, more = spare_last ? __ldcg(e.saved + crew.size() - 1) : 0u;
  const unsigned long long* mine = e.surv + (size_t)crew.rank() * e.cap_surv;
  const unsigned long long* its = e.surv + (size_t)(crew.size() - 1) * e.cap_surv;
#pragma unroll 1
  for (unsigned int i = Team::tid(); i < own;) {
    take_winner(e, ds, bins, key);
    i += Team::kN;
    if (i < own) key = __ldcg(mine + i);
  }
#pragma unroll 1
  for (unsigned int i = Team::tid() * (crew.size() - 1) + crew.rank(); i < more; i += Team::kN * (crew.size() - 1)) take_winner(e, ds, bins, __ldcg(its + i));
}

// Rare: more keys share the boundary bin than there is room for (thousands of tied times).  The grid cuts the bin
// further, digit by digit, over all J keys.  False: a barrier gave up.
template <typename Crew, typename G>
__device__ __noinline__ bool draw_refine(const Crew& crew, const Problem& p, const Engine& e, DrawShared& ds, unsigned char* sm, unsigned long long t, unsigned int k, G& g) {
  const int tid = threadIdx.x, warp = tid >> 5;
  unsigned int* sh = reinterpret_cast<unsigned int*>(sm);
  uint2* queue = reinterpret_cast<uint2*>(sm + sizeof(unsigned int) * kHistBins) + warp * kQueue;
  const Binning bins = binning_of(ds.cut);
  const unsigned int bnd = (unsigned)ds.bnd;
  unsigned int sure = ds.off[pad((int)bnd)];                       // winners before the keys still in question
  unsigned long long prefix = 0ull;
  int bits = 0;
  if (crew.rank() == 0 && tid == 0) atomicOr(&p.st->status, STRADS_STATUS_SAMPLER_REFINED);
  __shared__ int s_digit;
  __shared__ unsigned int s_before, s_here, s_w[kWarps];
  for (unsigned int here = ds.bnd_count; here > (unsigned)e.cap_boundary && bits < 64;) {
    const int width = min(kHistBits, 64 - bits);
    if (!grid_sync(g)) return false;                     // everybody has read the counts
    for (int b = crew.rank() * kT + tid; b < kHistBins; b += crew.size() * kT) e.hist[b] = 0u;
    for (int b = tid; b < kHistBins; b += kT) sh[b] = 0u;
    if (!grid_sync(g)) return false;
    const int up = 64 - bits - width;
    scan_keys<Crew::kParts>(p, t, 0.f, queue, warp * crew.size() + crew.rank(), kWarps * crew.size(), [&](unsigned long long key, bool on) {
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
template <typename Team, typename Crew>
__device__ __forceinline__ void draw_gather(const Crew& crew, const Problem& p, const Engine& e, DrawShared& ds, unsigned int k, bool spare_last) {
  if (spare_last && crew.size() > 1 && crew.rank() == crew.size() - 1) return;
  const unsigned int at = Team::tid();                    // (under way meanwhile)
  const unsigned long long key = at < min(ds.saved, e.cap_surv) ? __ldcg(e.surv + (size_t)crew.rank() * e.cap_surv + at) : ~0ull;
  draw_select<Team>(e, ds, k);
  // (a stretch that overflowed is seen by its owner alone: the others' winners are collected all the same, and again)
  const bool too_many = ds.saved > e.cap_surv || (spare_last && crew.rank() == 0 && __ldcg(e.saved + crew.size() - 1) > e.cap_surv);
  if (ds.total < k || ds.bnd_count > (unsigned)e.cap_boundary || ds.cut == 0.f || too_many) {
    if (Team::tid() == 0 && (crew.rank() == 0 || too_many)) e.es->mend = 1;
    return;
  }
  draw_collect<Team>(crew, e, ds, key, spare_last);
}

// (cold) by all CTAs.  False: a barrier gave up.
template <typename Crew, typename G>
__device__ __noinline__ bool draw_mend(const Crew& crew, const Problem& p, const Engine& e, DrawShared& ds, unsigned char* sm, unsigned long long t, unsigned int k, G& g) {
  draw_select_all(e, ds, k);
  if (!grid_sync(g)) return false;                       // everybody has read the counts and the flag
  if (crew.rank() == 0 && threadIdx.x == 0) e.es->mend = 0;
  if (ds.total < k) {
    // the cutoff was too low (the weights collapsed: the end of the first sweep, say): once more, all keys
    for (int b = crew.rank() * kT + (int)threadIdx.x; b < kHistBins; b += crew.size() * kT) e.hist[b] = 0u;
    if (!grid_sync(g)) return false;
    draw_scan(crew, p, e, ds, sm, t, false);
    if (!grid_sync(g)) return false;
    draw_select_all(e, ds, k);
  }
  if (ds.bnd_count > (unsigned)e.cap_boundary && !draw_refine(crew, p, e, ds, sm, t, k, g)) return false;
  for (int b = crew.rank() * kT + (int)threadIdx.x; b < kHistBins; b += crew.size() * kT) e.bin_cur[b] = 0u;
  if (!grid_sync(g)) return false;
  draw_collect_all(crew, p, e, ds, sm, t);
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
// kept_at: the positions of the kept candidates, where they are in shared memory (else null).
template <bool kDense>
__device__ __forceinline__ int gather_changes(const Problem& p, const DrawShared& ds, int nk, const unsigned short* kept_at, bool want_keys, unsigned long long* keys,
                                              ChangedByBin* cb, Moving* mv, ChangeShared& cs) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool indexed = want_keys && nk > kFewChanged;
  const Binning bins = binning_of(ds.cut);
  // Keys behind the boundary's bin concern no rank -- unless the winners are all there are -- and are not entered: most new keys are
  // there, those beyond the cutoff all in one bin, one after the other (50,000 x 1,000,000: a step of 3 us of 34).
  const int last_bin = (long long)ds.total >= (p.part_count > 1 ? owned_count(p) : p.J) ? kHistBins : ds.bnd;
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
  constexpr int kU = kDense ? 1 : 2;                     // entries of a thread at a time (dense: rarely more than one)
#pragma unroll 1
  for (int i0 = 0; i0 < per; i0 += kU) {
    double d[kU];
    unsigned long long o[kU], w[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int a = a_lo + i0 + u;
      d[u] = 0.0; o[u] = w[u] = 0ull;
      if (i0 + u < per && a < a_hi) {
        const int pos = !kDense && kept_at != nullptr ? (int)kept_at[a] : p.kept_pos[a];
        d[u] = p.cand_dbeta64[pos];
        if (want_keys) { o[u] = p.cand_keys[pos]; w[u] = p.cand_keys[p.n_cand + pos]; }
      }
    }
    if (i0 == 0) d_first = d[0];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      moving += d[u] != 0.0;
      dmax = max(dmax, (unsigned long long)__double_as_longlong(fabs(d[u])));
      const unsigned int changed = __ballot_sync(kFull, o[u] != w[u]);
      if (changed == 0u) continue;
      int at = 0;                                        // (one addition per warp: they all go to one address)
      if (lane == 0) at = atomicAdd(&cs.n_changed, __popc(changed));
      at = __shfl_sync(kFull, at, 0) + __popc(changed & ((1u << lane) - 1u));
      if (o[u] == w[u]) continue;
      keys[at] = o[u];
      keys[p.n_keep + at] = w[u];
      if (indexed) {                                     // by bin: a count for the prefix sum, and a list
        const int bo = (int)bin_of(bins, (unsigned int)(o[u] >> 32)), bw = (int)bin_of(bins, (unsigned int)(w[u] >> 32));
        if (bo <= last_bin) {
          atomicAdd(&cb->before[pad(bo)], -1);
          cb->next[2 * at] = (unsigned short)atomicExch(&cb->head[bo], 2 * at);
        }
        if (bw <= last_bin) {
          atomicAdd(&cb->before[pad(bw)], 1);
          cb->next[2 * at + 1] = (unsigned short)atomicExch(&cb->head[bw], 2 * at + 1);
        }
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

// (cold)
template <bool kDense>
__device__ __noinline__ int gather_again(const Problem& p, const DrawShared& ds, int nk, unsigned long long* keys, ChangedByBin* cb, Moving* mv, ChangeShared& cs) {
  return gather_changes<kDense>(p, ds, nk, nullptr, true, keys, cb, mv, cs);
}

// Winners ranked; with changes, corrected for the kept coefficients' changed priorities (keys[0 .. n_changed) old,
// keys[p.n_keep ..) new).  A key's place among the changed ones: those in lower bins from a prefix sum over the bins, those
// in its own bin one by one (a list per bin); a plain count while they are few.
// Leaves the draw's buffers as the next scan expects them.
template <bool kDense, typename Crew>
__device__ __forceinline__ void draw_rank(const Crew& crew, const Problem& p, const Engine& e, const DrawShared& ds, const unsigned long long* keys, ChangedByBin* cb, int n_changed,
                          int nk, int* wsum, int n_rank, int n_prefetch) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (crew.rank() >= n_rank) return;
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
  for (int i0 = (warp * n_rank + crew.rank()) * per_warp; i0 < items; i0 += kWarps * n_rank * per_warp) {
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
    if (behind && total < (unsigned long long)(Crew::kParts ? owned_count(p) : p.J)) on = false;
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
      if (Crew::kKeys && p.keys_out != nullptr) p.keys_out[rank] = key;
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
  for (int b = crew.rank() * kT + tid; b < kHistBins; b += crew.size() * kT) e.hist[b] = 0u;
  if (crew.rank() == 0 && tid == 0) {
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
struct Change { double d; float b_new; };
__device__ __forceinline__ Change propose_end(const Problem& p, const Proposal& q, int pos, int j, double g, float E, bool want_keys) {
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
  return {d, b_new};
}

constexpr int kMaxWords = STRADS_MAX_CANDIDATES / 32;
constexpr int kTurn = 32;                  // candidates a CTA handles per turn of step 1 (dense) / 2 (CSC)
struct TurnShared { double dot[kTurn][kWarps]; };

}  // namespace
}  // namespace strads
