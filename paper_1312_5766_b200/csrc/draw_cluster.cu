// The draw (SAP step 1) of rounds made launch by launch, in one launch of one thread-block cluster: the steps of rounds in one launch
// (engine_draw.cuh: keys below the cutoff carried over, selection, collection, ranks) with the cluster's barrier between them.
//
// A draw of some 10^5 coefficients is a chain of hand-overs, not work: as three launches (sampler.cu: histogram, collection, ranks) each waits for
// the one before, every CTA of the first clears and merges a histogram of its own and the last one makes the selection alone.  One
// cluster has all its CTAs running by definition, so nothing waits for a grid, and it leaves the other SMs to the round's Gram beside it.
#include <mutex>

#include "engine_draw.cuh"

namespace strads {
namespace {

constexpr int kMaxClusterCtas = 16;        // (eight are portable)

__global__ void __launch_bounds__(kT, 2) k_draw_cluster(const __grid_constant__ Problem p, const __grid_constant__ Engine e) {
  chain_begin();
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ DrawShared ds;
  __shared__ Problem sp;                                 // copies for the functions that are called rarely and not inlined
  __shared__ Engine se;
  const ClusterCrew crew;
  ClusterGrid g;
  const unsigned long long t = *p.round_ptr + (unsigned long long)p.round_ahead;
  const unsigned int k = (unsigned)p.n_cand;
  draw_scan(crew, p, e, ds, sm, t, true);
  grid_sync(g);
  draw_gather<AllThreads>(crew, p, e, ds, k, false);
  grid_sync(g);
  if (__ldcg(&e.es->mend)) {
    __syncthreads();
    if (threadIdx.x == 0) { sp = p; se = e; }
    __syncthreads();
    draw_mend(crew, sp, se, ds, sm, t, k, g);
  }
  draw_rank<true>(crew, p, e, ds, nullptr, nullptr, 0, 0, nullptr, crew.size(), 0);
  if (crew.rank() == 0 && threadIdx.x == 0) p.st->counts[0] = p.n_cand;
}

}  // namespace

// CTAs of the cluster on each device (0: not asked yet, -1: none fits).
constexpr int kMaxDevices = 64;
static int g_cluster_ctas[kMaxDevices];
static std::mutex g_cluster_mutex;

static cudaLaunchConfig_t cluster_config(int ctas, cudaLaunchAttribute* attr) {
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)ctas; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)ctas); cfg.blockDim = dim3(kT); cfg.dynamicSmemBytes = kScanSmem;
  cfg.attrs = attr; cfg.numAttrs = 1;
  return cfg;
}

// Sixteen CTAs, the most there can be, where the device takes such a cluster, else eight (us per draw of 2,048 from 100,000, 4,096 from 400,000: 10.6,
// 18.3 and 13.9, 27.9; three launches 16.4, 20.9).
cudaError_t prepare_draw_cluster(int* ctas) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  *ctas = 0;
  if (dev < 0 || dev >= kMaxDevices) return cudaSuccess;
  std::lock_guard<std::mutex> lock(g_cluster_mutex);
  if (g_cluster_ctas[dev] == 0) {
    if ((e = cudaFuncSetAttribute(k_draw_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kScanSmem)) != cudaSuccess) return e;
    const bool large = cudaFuncSetAttribute(k_draw_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    g_cluster_ctas[dev] = -1;
    for (int size = large ? kMaxClusterCtas : kMaxClusterCtas / 2; size >= kMaxClusterCtas / 2; size /= 2) {
      cudaLaunchAttribute attr[1];
      const cudaLaunchConfig_t cfg = cluster_config(size, attr);
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, k_draw_cluster, &cfg) == cudaSuccess && n > 0) { g_cluster_ctas[dev] = size; break; }
    }
    cudaGetLastError();                                  // (a size the device refuses is simply not used)
  }
  *ctas = g_cluster_ctas[dev] > 0 ? g_cluster_ctas[dev] : 0;
  return cudaSuccess;
}

cudaError_t launch_draw_cluster(const Problem& p, const Engine& e, int* cand_out, cudaStream_t s) {
  Problem q = p;
  q.cand = cand_out;
  return launch_chained_cluster(k_draw_cluster, (unsigned)e.grid, kT, kScanSmem, s, e.grid, q, e);
}

}  // namespace strads
