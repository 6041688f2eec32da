// fcs_batch_k3.cu -- batch class kernels for FFT lengths P = 16384 and 32768
// on the row-pair engine.
#include "fcs_batch_kernels.cuh"

namespace fcs {

ClassKernel class_kernel_13(int L, int ipc, int sb) {
  return L == 14 ? pair_class_kernel<32>(ipc, sb) : pair_class_kernel<16>(ipc, sb);
}

}  // namespace fcs
