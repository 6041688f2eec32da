// fcs_batch_k2.cu -- batch class kernels for FFT length P = 8192
// (log2 M = 12): the slot FFT at both thread multipliers, and the row-pair
// engine.
#include "fcs_batch_kernels.cuh"

namespace fcs {

ClassKernel class_kernel_12(int eng, int ntm, int ipc, int64_t Imax, int sb) {
  if (eng == 1) return pair_class_kernel<8>(ipc, sb);
  return class_kernel_l<12>(ntm, ipc, Imax, sb);
}

}  // namespace fcs
