// Rotation-layout kernels, int16 flows, 512 threads per walk.
#include "qap_rotation.cuh"

namespace qapk {

BatchKernelFn rot_f16_512(int c) {
  switch (c) {
    case 1: return rot_kernel<512, 1, int16_t>;
    case 2: return rot_kernel<512, 2, int16_t>;
    case 3: return rot_kernel<512, 3, int16_t>;
    default: return nullptr;
  }
}

}  // namespace qapk
