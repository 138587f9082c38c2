// Register-resident transforms: inverse transform from gated half spectra.
#include "reg_fft.cuh"

namespace spectre {

int reg_inverse(const spectre_ctx* ctx, cudaStream_t st, RegParams p, int M, int nslab, bool ws, int dtype) {
  if (ws) return reg_launch_ws<kRegInverse>(ctx, p, M, nslab, st);
  SPECTRE_IO_DISPATCH(dtype, return (reg_launch_tokens<T, kRegInverse>(ctx, p, M, nslab, st)));
}

}  // namespace spectre
