// Rotation-layout kernels, int16 flows, 1024 threads per walk.
#include "qap_rotation.cuh"

namespace qapk {

BatchKernelFn rot_f16_1024(int c) {
  switch (c) {
    case 2: return rot_kernel<1024, 2, int16_t>;
    case 4: return rot_kernel<1024, 4, int16_t>;
    default: return nullptr;
  }
}

}  // namespace qapk
