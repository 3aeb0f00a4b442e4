// Rotation-layout walk kernels, int8 flows, 128 threads per walk.
#include "qap_rotation.cuh"

namespace qapk {

WalkKernelFn rot_walk_f8_128(int c) {
  switch (c) {
    case 1: return rot_walk_kernel<128, 1>;
    case 2: return rot_walk_kernel<128, 2>;
    case 4: return rot_walk_kernel<128, 4>;
    case 7: return rot_walk_kernel<128, 7>;
    default: return nullptr;
  }
}

}  // namespace qapk
