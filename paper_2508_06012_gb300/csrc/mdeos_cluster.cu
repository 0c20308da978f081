// Cluster form of the batch kernel: few boxes, each on a thread-block cluster.  A translation
// unit of its own: its CTAs have few warps with work, so its force passes fetch their lists
// further ahead (MDEOS_LIST_AHEAD, mdeos_device.cuh).
#define MDEOS_LIST_AHEAD 3
#include <array>
#include <map>
#include <mutex>

#include "mdeos_big.cuh"

namespace mdeos {

// Cluster form for batches too small to fill the GPU: one box per thread-block
// cluster of csize CTAs (cluster c runs item c, one box, the whole CTA as its group).
// Shared-memory boxes: every CTA holds the box and advances it alike; each computes
// the forces and lists of its share of the atoms and sends the forces to the others
// (run_box with Group::csize > 1).  Boxes above the shared-memory limit: one state in
// the scratch of the cluster's first CTA, each CTA owning a slab of its slots
// (run_big with csize > 1).  All CTAs of a cluster take the same path through the
// box, so they meet at the same cluster barriers; the last one below keeps every CTA
// alive until no other can still store into its shared memory.
__global__ void __launch_bounds__(kCtaThreads, 1)
    eos_cluster_kernel(const BoxDesc* __restrict__ boxes, const WorkItem* __restrict__ items,
                       int nitems, mdeos_result* __restrict__ results, uint16_t* nl_scratch,
                       long long nl_elems_per_cta, RunParams rp, int* ready) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  unsigned char* smem = align_smem(smem_raw);
  const int csize = cluster_size(), crank = cluster_rank();
  const int it = blockIdx.x / csize;
  uint16_t* nl_cta = nl_scratch + (long long)blockIdx.x * nl_elems_per_cta;
  if (it < nitems && items[it].big) {
    const BoxDesc& bd = boxes[items[it].box[0]];
    uint16_t* box_scratch = nl_scratch + (long long)(blockIdx.x - crank) * nl_elems_per_cta;
    run_big(reinterpret_cast<unsigned char*>(box_scratch), reinterpret_cast<BigShared*>(smem), bd,
            rp, results + bd.out_index, crank, csize);
    if (ready != nullptr && crank == 0 && threadIdx.x == 0) {
      __threadfence_system();
      reinterpret_cast<volatile int*>(ready)[bd.out_index] = 1;
    }
  } else if (it < nitems) {
    const WorkItem wi = items[it];
    const BoxDesc& bd = boxes[wi.box[0]];
    Group g = make_group(smem, threadIdx.x, wi.warps_per_box, wi.apt, wi.ncell_cap, 1, nl_cta);
    g.crank = crank;
    g.csize = csize;
    mdeos_result* out = results + bd.out_index;
    switch (wi.apt) {
      case 1: run_box_path<1>(g, bd, rp, out); break;
      case 2: run_box_path<2>(g, bd, rp, out); break;
      default: run_box_path<4>(g, bd, rp, out); break;
    }
    if (ready != nullptr && crank == 0 && g.tid == 0) {
      __threadfence_system();
      reinterpret_cast<volatile int*>(ready)[bd.out_index] = 1;
    }
  }
  cluster_sync();
}

cudaError_t set_cluster_attributes(int dyn) {
  return cudaFuncSetAttribute(eos_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn);
}

// Clusters of `cluster` full-size CTAs (one per SM) that the current device holds at once: a
// property of the device and the launch, so it is asked once per process (50 us a question,
// a fifth of creating a handle for three of them).
cudaError_t max_resident_clusters(int cluster, int smem, int* n) {
  static std::mutex mu;
  static std::map<std::array<int, 3>, int> known;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  const std::array<int, 3> key{dev, cluster, smem};
  const auto it = known.find(key);
  if (it != known.end()) {
    *n = it->second;
    return cudaSuccess;
  }
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3((unsigned)cluster, 1, 1);
  lc.blockDim = dim3(kCtaThreads, 1, 1);
  lc.dynamicSmemBytes = (size_t)smem + kSmemAlign;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cluster;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  e = cudaOccupancyMaxActiveClusters(n, eos_cluster_kernel, &lc);
  if (e == cudaSuccess) known[key] = *n;
  return e;
}

cudaError_t launch_eos_cluster(const BoxDesc* boxes, const WorkItem* items, int nitems,
                               mdeos_result* results, uint16_t* nl, long long nl_elems_per_cta,
                               const RunParams& rp, int grid, int smem, cudaStream_t st, int* ready,
                               int cluster, int threads) {
  // grid = nitems * cluster CTAs of `threads` in clusters of `cluster`
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3((unsigned)grid, 1, 1);
  lc.blockDim = dim3((unsigned)threads, 1, 1);
  lc.dynamicSmemBytes = (size_t)smem + kSmemAlign;
  lc.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cluster;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  return cudaLaunchKernelEx(&lc, eos_cluster_kernel, boxes, items, nitems, results, nl,
                            nl_elems_per_cta, rp, ready);
}

}  // namespace mdeos
