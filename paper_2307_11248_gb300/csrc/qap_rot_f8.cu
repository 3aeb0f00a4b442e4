// The rotation-layout kernels with int8 flows: the one for a thread count and
// a number of partner blocks per thread.  qap_rot_f8_*.cu hold the
// instantiations, one translation unit per kernel and thread count so that
// they compile in parallel.
#include "qap_rotation.cuh"

namespace qapk {

WalkKernelFn rot_walk_f8_128(int c);
WalkKernelFn rot_walk_f8_256(int c);
WalkKernelFn rot_walk_f8_512(int c);
WalkKernelFn rot_walk_f8_1024(int c);
BatchKernelFn rot_batch_f8_128(int c);
BatchKernelFn rot_batch_f8_256(int c);
BatchKernelFn rot_batch_f8_512(int c);
BatchKernelFn rot_batch_f8_1024(int c);

WalkKernelFn rot_walk_kernel_f8(int nt, int c) {
  return nt == 128   ? rot_walk_f8_128(c)
         : nt == 256 ? rot_walk_f8_256(c)
         : nt == 512 ? rot_walk_f8_512(c)
                     : rot_walk_f8_1024(c);
}

BatchKernelFn rot_batch_kernel_f8(int nt, int c) {
  return nt == 128   ? rot_batch_f8_128(c)
         : nt == 256 ? rot_batch_f8_256(c)
         : nt == 512 ? rot_batch_f8_512(c)
                     : rot_batch_f8_1024(c);
}

}  // namespace qapk
