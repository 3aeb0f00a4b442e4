// Rotation-layout walk kernels, int8 flows, 256 threads per walk.
#include "qap_rotation.cuh"

namespace qapk {

WalkKernelFn rot_walk_f8_256(int c) {
  switch (c) {
    case 1: return rot_walk_kernel<256, 1>;
    case 2: return rot_walk_kernel<256, 2>;
    case 3: return rot_walk_kernel<256, 3>;
    case 4: return rot_walk_kernel<256, 4>;
    case 6: return rot_walk_kernel<256, 6>;
    case 7: return rot_walk_kernel<256, 7>;
    case 11: return rot_walk_kernel<256, 11>;
    case 13: return rot_walk_kernel<256, 13>;
    default: return nullptr;
  }
}

}  // namespace qapk
