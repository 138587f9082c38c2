// Register-resident transforms: forward transform only.
#include "reg_fft.cuh"

namespace spectre {

int reg_forward(const spectre_ctx* ctx, cudaStream_t st, RegParams p, int M, int nslab, int dtype) {
  p.nslab = nslab;
  SPECTRE_IO_DISPATCH(dtype, return (reg_launch_tokens<T, kRegForward>(ctx, p, M, p.src2 ? 2 * nslab : nslab, st)));
}

}  // namespace spectre
