// ns_inst.cu -- instantiates the per-dimension kernels for one register
// class (compiled once per class with -DNS_DMAX=<class>, so the classes
// build in parallel; the wide classes in parts, -DNS_PART=<bits>: 1 the group
// walkers' run kernel, 2 the thread walkers', 4 the rest).
#include "ns_run.cuh"

#ifndef NS_DMAX
#error "compile with -DNS_DMAX=<register class>"
#endif

#ifndef NS_PART
#define NS_PART 7
#endif

namespace nsd {

#define NS_CAT2(a, b) a##b
#define NS_CAT(a, b) NS_CAT2(a, b)

// Launches n runs as clusters of `cluster` blocks (blocks r*cluster ..
// r*cluster + cluster - 1 are run r's).
template <class K>
static cudaError_t launch_runs(K* kernel, const RunDesc* runs, const int* ids, int n, int block, size_t smem, int chunk,
                               int vb, int cluster, int room, cudaStream_t s) {
  cudaError_t e = allow_smem(kernel, smem);
  if (e != cudaSuccess) return e;
  if (cluster <= 1) {
    kernel<<<n, block, smem, s>>>(runs, ids, chunk, vb, room);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(n * cluster), 1, 1);
  cfg.blockDim = dim3((unsigned)block, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, runs, ids, chunk, vb, room);
}

template <class K>
static cudaError_t occupancy(K* kernel, int block, size_t smem, int* blocks_per_sm) {
  cudaError_t e = allow_smem(kernel, smem);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, kernel, block, smem);
}

// One run kernel's launch, or (n = 0) its occupancy, by mode.
using RunFn = cudaError_t(const RunDesc* runs, const int* ids, int n, int block, size_t smem, int chunk, int vb,
                          int cluster, int room, int* blocks_per_sm, cudaStream_t s);
RunFn NS_CAT(run_group_, NS_DMAX), NS_CAT(run_thread_, NS_DMAX);

#if NS_PART & 1
cudaError_t NS_CAT(run_group_, NS_DMAX)(const RunDesc* runs, const int* ids, int n, int block, size_t smem, int chunk,
                                        int vb, int cluster, int room, int* blocks_per_sm, cudaStream_t s) {
  if (n == 0) return occupancy(k_run<NS_DMAX, kModeGroup>, block, smem, blocks_per_sm);
  return launch_runs(k_run<NS_DMAX, kModeGroup>, runs, ids, n, block, smem, chunk, vb, cluster, room, s);
}
#endif

#if NS_PART & 2
cudaError_t NS_CAT(run_thread_, NS_DMAX)(const RunDesc* runs, const int* ids, int n, int block, size_t smem, int chunk,
                                         int vb, int, int room, int* blocks_per_sm, cudaStream_t s) {
  if (n == 0) return occupancy(k_run<NS_DMAX, kModeThread>, block, smem, blocks_per_sm);
  return launch_runs(k_run<NS_DMAX, kModeThread>, runs, ids, n, block, smem, chunk, vb, 1, room, s);
}
#endif

#if NS_PART & 4
cudaError_t NS_CAT(launch_run_, NS_DMAX)(const RunDesc* runs, const int* ids, int n, int block, size_t smem,
                                         int chunk, int vb, int group, int cluster, int room, cudaStream_t s) {
  return (group ? NS_CAT(run_group_, NS_DMAX) : NS_CAT(run_thread_, NS_DMAX))(runs, ids, n, block, smem, chunk, vb,
                                                                             cluster, room, nullptr, s);
}

cudaError_t NS_CAT(occupancy_run_, NS_DMAX)(int block, size_t smem, int group, int* blocks_per_sm) {
  return (group ? NS_CAT(run_group_, NS_DMAX) : NS_CAT(run_thread_, NS_DMAX))(nullptr, nullptr, 0, block, smem, 0, 0, 1,
                                                                             0, blocks_per_sm, nullptr);
}

cudaError_t NS_CAT(launch_loglike_, NS_DMAX)(const LikParams& P, int n, const float* x, float* out,
                                             cudaStream_t s) {
  k_loglike<NS_DMAX><<<(n + 127) / 128, 128, 0, s>>>(P, n, x, out);
  return cudaGetLastError();
}

cudaError_t NS_CAT(launch_slice_, NS_DMAX)(const LikParams& P, const SliceCfg& SC, int m, int n_pad,
                                           int correction, const float* live_x, const float* live_l,
                                           const int* seed_slot, const float* W, const float* chol, const int* cid,
                                           float* new_x, float* new_l, float* hist_l, float* hist_x, int* hist_len,
                                           long long* evals, int* flags, float* dir_scratch, int warp,
                                           cudaStream_t s) {
  if (warp) {  // four walkers (warps) per block
    k_slice_warp<NS_DMAX><<<(m + 3) / 4, 128, 0, s>>>(P, SC, m, n_pad, correction, live_x, live_l, seed_slot, W, chol,
                                                      cid, new_x, new_l, hist_l, hist_x, hist_len, evals, flags,
                                                      dir_scratch);
    return cudaGetLastError();
  }
  k_slice<NS_DMAX><<<(m + kSliceWalkers - 1) / kSliceWalkers, kSliceThreads,
                     sizeof(float) * kSliceWalkers * group_floats(NS_DMAX), s>>>(
      P, SC, m, n_pad, correction, live_x, live_l, seed_slot, W, chol, cid, new_x, new_l, hist_l, hist_x, hist_len,
      evals, flags, dir_scratch);
  return cudaGetLastError();
}

#if NS_DMAX == 32
// MLP runs (any d <= 32) use the widest class with the lock-step walkers.
// cluster > 1: each run is a cluster of that many CTAs (blocks r*cluster ..
// r*cluster + cluster - 1), which share its tensor-core evaluations.
cudaError_t launch_run_mlp(const RunDesc* runs, const int* ids, int n, int block, size_t smem, int chunk, int cluster,
                           cudaStream_t s) {
  return launch_runs(k_run<32, kModeMlp>, runs, ids, n, block, smem, chunk, block, cluster, (int)kRunSmemBudget, s);
}
#endif
#endif

}  // namespace nsd
