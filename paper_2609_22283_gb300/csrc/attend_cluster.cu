// The attention instances whose units are split over thread-block clusters
// (see attend.cuh).
#include "attend.cuh"

namespace sva {

AttendKernel attend_cluster_kernel(int head_dim, bool masked, bool token) {
  if (head_dim == 128)
    return token ? attend_kernel<128, true, true, true>
                 : (masked ? attend_kernel<128, true, false, true> : attend_kernel<128, false, false, true>);
  return token ? attend_kernel<64, true, true, true>
               : (masked ? attend_kernel<64, true, false, true> : attend_kernel<64, false, false, true>);
}

}  // namespace sva
