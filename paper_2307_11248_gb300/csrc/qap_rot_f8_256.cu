// Rotation-layout kernels, int8 flows, 256 threads per walk.
#include "qap_rotation.cuh"

namespace qapk {

BatchKernelFn rot_f8_256(int c) {
  switch (c) {
    case 1: return rot_kernel<256, 1, int8_t>;
    case 2: return rot_kernel<256, 2, int8_t>;
    case 3: return rot_kernel<256, 3, int8_t>;
    case 4: return rot_kernel<256, 4, int8_t>;
    default: return nullptr;
  }
}

}  // namespace qapk
