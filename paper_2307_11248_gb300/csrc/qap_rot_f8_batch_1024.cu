// Rotation-layout batch kernels, int8 flows, 1024 threads per walk.
#include "qap_rotation.cuh"

namespace qapk {

BatchKernelFn rot_batch_f8_1024(int c) {
  switch (c) {
    case 2: return rot_batch_kernel<1024, 2>;
    case 4: return rot_batch_kernel<1024, 4>;
    case 5: return rot_batch_kernel<1024, 5>;
    case 6: return rot_batch_kernel<1024, 6>;
    default: return nullptr;
  }
}

}  // namespace qapk
