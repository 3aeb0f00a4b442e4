// Rotation-layout kernels, int8 flows, 1024 threads per walk.
#include "qap_rotation.cuh"

namespace qapk {

BatchKernelFn rot_f8_1024(int c) {
  switch (c) {
    case 2: return rot_kernel<1024, 2, int8_t>;
    case 4: return rot_kernel<1024, 4, int8_t>;
    default: return nullptr;
  }
}

}  // namespace qapk
