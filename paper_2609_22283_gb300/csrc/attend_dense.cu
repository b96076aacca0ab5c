// The dense attention instances (see attend.cuh).
#include "attend.cuh"

namespace sva {

AttendKernel attend_dense_kernel(int head_dim) {
  return head_dim == 128 ? attend_kernel<128, false, false, false>
                         : attend_kernel<64, false, false, false>;
}

}  // namespace sva
