// Set-up and launches of the attention kernel (attend.cuh).
#include <mutex>

#include "attend.cuh"

namespace sva {
namespace {

// One-time per-device set-up of the kernel instances (shared-memory limit,
// register check), done under a lock so that two host threads launching on
// the same device for the first time cannot race.
template <int D>
cudaError_t configure_d(int dev) {
  static std::mutex mu;
  static bool configured[64] = {};
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  if (configured[dev]) return cudaSuccess;
  // setmaxnreg.inc waits until the block's register pool can serve it: a
  // build whose launch register count leaves the split short would never
  // proceed, so such a build is refused here.
  for (AttendKernel k :
       {attend_dense_kernel(D), attend_masked_kernel(D, false), attend_masked_kernel(D, true),
        attend_cluster_kernel(D, false, false), attend_cluster_kernel(D, true, false),
        attend_cluster_kernel(D, true, true)}) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         AttnCfg<D>::kSmemBytes);
    if (e != cudaSuccess) return e;
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, k);
    if (e != cudaSuccess) return e;
    if (fa.numRegs * kThreads < AttnRegs<D>::kPool) return cudaErrorInvalidConfiguration;
  }
  configured[dev] = true;
  return cudaSuccess;
}

template <int D>
cudaError_t launch_d(const AttnParams& p, int grid, cudaStream_t s) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = configure_d<D>(dev);
  if (e != cudaSuccess) return e;
  const bool token = p.masked && (p.own_mask != nullptr || p.hist_mask != nullptr);
  LaunchConfig l(dim3((unsigned)grid), kThreads, AttnCfg<D>::kSmemBytes, s,
                 p.cluster ? p.n_split : 0);
  AttendKernel k = p.cluster  ? attend_cluster_kernel(D, p.masked, token)
                   : p.masked ? attend_masked_kernel(D, token)
                              : attend_dense_kernel(D);
  return cudaLaunchKernelEx(&l.cfg, k, p);
}

// Clusters of `size` CTAs (one CTA per SM) that can be resident at once on the
// current device, looked up once per device and size.
template <int D>
cudaError_t max_clusters_d(int size, int* out) {
  static std::mutex mu;
  static int known[64][kMaxClusterSplit + 1] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = configure_d<D>(dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  if (known[dev][size] == 0) {
    LaunchConfig l(dim3((unsigned)size), kThreads, AttnCfg<D>::kSmemBytes, nullptr, size);
    int n = 0;
    e = cudaOccupancyMaxActiveClusters(&n, attend_cluster_kernel(D, false, false), &l.cfg);
    if (e != cudaSuccess) return e;
    known[dev][size] = n + 1;
  }
  *out = known[dev][size] - 1;
  return cudaSuccess;
}

}  // namespace

cudaError_t launch_attend(const AttnParams& p, int head_dim, int grid, cudaStream_t s) {
  if (head_dim == 128) return launch_d<128>(p, grid, s);
  if (head_dim == 64) return launch_d<64>(p, grid, s);
  return cudaErrorInvalidValue;
}

cudaError_t attend_max_clusters(int head_dim, int size, int* clusters) {
  if (size < 2 || size > kMaxClusterSplit) return cudaErrorInvalidValue;
  if (head_dim == 128) return max_clusters_d<128>(size, clusters);
  if (head_dim == 64) return max_clusters_d<64>(size, clusters);
  return cudaErrorInvalidValue;
}

}  // namespace sva
