// Rotation-layout kernels, int16 flows, 512 threads per walk.
#include "qap_rotation.cuh"

namespace qapk {

BatchKernelFn rot_f16_512w(int c) {
  switch (c) {
    case 5: return rot_kernel<512, 5, int16_t>;
    case 7: return rot_kernel<512, 7, int16_t>;
    case 8: return rot_kernel<512, 8, int16_t>;
    case 12: return rot_kernel<512, 12, int16_t>;
    case 13: return rot_kernel<512, 13, int16_t>;
    default: return nullptr;
  }
}

}  // namespace qapk
