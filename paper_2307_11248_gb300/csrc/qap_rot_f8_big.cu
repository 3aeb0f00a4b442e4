// Rotation-layout kernels, int8 flows, large n (M in the CTA's workspace).
#include "qap_rotation.cuh"

namespace qapk {

BatchKernelFn rot_f8_big(int c) {
  switch (c) {
    case 10: return rot_kernel<kRotBig, 10, int8_t>;
    case 12: return rot_kernel<kRotBig, 12, int8_t>;
    case 17: return rot_kernel<kRotBig, 17, int8_t>;
    case 19: return rot_kernel<kRotBig, 19, int8_t>;
    case 21: return rot_kernel<kRotBig, 21, int8_t>;
    case 22: return rot_kernel<kRotBig, 22, int8_t>;
    default: return nullptr;
  }
}

}  // namespace qapk
