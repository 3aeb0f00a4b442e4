// Rotation-layout kernels, int8 flows, 128 threads per walk.
#include "qap_rotation.cuh"

namespace qapk {

BatchKernelFn rot_f8_128(int c) {
  switch (c) {
    case 1: return rot_kernel<128, 1, int8_t>;
    case 2: return rot_kernel<128, 2, int8_t>;
    case 4: return rot_kernel<128, 4, int8_t>;
    case 7: return rot_kernel<128, 7, int8_t>;
    default: return nullptr;
  }
}

}  // namespace qapk
