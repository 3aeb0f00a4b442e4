// The rotation-layout kernel for a flow width, a thread count and a number of
// partner blocks per thread.  qap_rot_*_*.cu hold the instantiations, several
// translation units so that they compile in parallel.
#include "qap_rotation.cuh"

namespace qapk {

BatchKernelFn rot_f8_128(int c);
BatchKernelFn rot_f8_256(int c);
BatchKernelFn rot_f8_256w(int c);
BatchKernelFn rot_f8_512(int c);
BatchKernelFn rot_f8_512w(int c);
BatchKernelFn rot_f8_1024(int c);
BatchKernelFn rot_f8_big(int c);
BatchKernelFn rot_f16_128(int c);
BatchKernelFn rot_f16_256(int c);
BatchKernelFn rot_f16_256w(int c);
BatchKernelFn rot_f16_512(int c);
BatchKernelFn rot_f16_512w(int c);
BatchKernelFn rot_f16_1024(int c);

BatchKernelFn rot_kernel_of(int fbytes, int nt, int c) {
  const bool w = c >= 5;
  if (nt == kRotBig) return fbytes == 1 ? rot_f8_big(c) : nullptr;
  if (fbytes == 1)
    return nt == 128   ? rot_f8_128(c)
           : nt == 256 ? (w ? rot_f8_256w(c) : rot_f8_256(c))
           : nt == 512 ? (w ? rot_f8_512w(c) : rot_f8_512(c))
                       : rot_f8_1024(c);
  return nt == 128   ? rot_f16_128(c)
         : nt == 256 ? (w ? rot_f16_256w(c) : rot_f16_256(c))
         : nt == 512 ? (w ? rot_f16_512w(c) : rot_f16_512(c))
                     : rot_f16_1024(c);
}

}  // namespace qapk
