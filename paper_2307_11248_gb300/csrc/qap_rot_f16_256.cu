// Rotation-layout kernels, int16 flows, 256 threads per walk.
#include "qap_rotation.cuh"

namespace qapk {

BatchKernelFn rot_f16_256(int c) {
  switch (c) {
    case 1: return rot_kernel<256, 1, int16_t>;
    case 2: return rot_kernel<256, 2, int16_t>;
    case 3: return rot_kernel<256, 3, int16_t>;
    case 4: return rot_kernel<256, 4, int16_t>;
    default: return nullptr;
  }
}

}  // namespace qapk
