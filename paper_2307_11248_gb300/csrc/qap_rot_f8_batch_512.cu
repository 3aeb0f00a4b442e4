// Rotation-layout batch kernels, int8 flows, 512 threads per walk.
#include "qap_rotation.cuh"

namespace qapk {

BatchKernelFn rot_batch_f8_512(int c) {
  switch (c) {
    case 1: return rot_batch_kernel<512, 1>;
    case 2: return rot_batch_kernel<512, 2>;
    case 3: return rot_batch_kernel<512, 3>;
    case 5: return rot_batch_kernel<512, 5>;
    case 7: return rot_batch_kernel<512, 7>;
    case 8: return rot_batch_kernel<512, 8>;
    case 11: return rot_batch_kernel<512, 11>;
    case 13: return rot_batch_kernel<512, 13>;
    default: return nullptr;
  }
}

}  // namespace qapk
