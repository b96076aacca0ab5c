// The attention instances with a block-sparse tile mask and with token masks
// (see attend.cuh).
#include "attend.cuh"

namespace sva {

AttendKernel attend_masked_kernel(int head_dim, bool token) {
  if (head_dim == 128)
    return token ? attend_kernel<128, true, true, false> : attend_kernel<128, true, false, false>;
  return token ? attend_kernel<64, true, true, false> : attend_kernel<64, true, false, false>;
}

}  // namespace sva
