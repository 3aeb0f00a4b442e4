// Rotation-layout kernels, int16 flows, 256 threads per walk.
#include "qap_rotation.cuh"

namespace qapk {

BatchKernelFn rot_f16_256w(int c) {
  switch (c) {
    case 6: return rot_kernel<256, 6, int16_t>;
    case 7: return rot_kernel<256, 7, int16_t>;
    case 12: return rot_kernel<256, 12, int16_t>;
    case 13: return rot_kernel<256, 13, int16_t>;
    default: return nullptr;
  }
}

}  // namespace qapk
