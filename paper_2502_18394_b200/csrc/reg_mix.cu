// Register-resident transforms: forward transform, gate, inverse transform.
#include "reg_fft.cuh"

namespace spectre {

int reg_mix(const spectre_ctx* ctx, cudaStream_t st, RegParams p, int M, int nslab, bool ws, int dtype) {
  if (ws) return reg_launch_ws<kRegMix>(ctx, p, M, nslab, st);
  SPECTRE_IO_DISPATCH(dtype, return (reg_launch_tokens<T, kRegMix>(ctx, p, M, nslab, st)));
}

bool reg_supported(int M) {
#define SPECTRE_REG_IS(R1, R2) M == R1 * R2 ||
  return SPECTRE_REG_TWO_STEP(SPECTRE_REG_IS) M == 2048;
#undef SPECTRE_REG_IS
}

int reg_parts(int M, int D) {
  const int ntile = (D / 2 + kRegPairs - 1) / kRegPairs;
  return M == 2048 ? ntile * (kRegPairs / 4) : ntile;
}

// ---- twiddle tables ----
// Two steps: [a < R1 / 2][b < R1] of (W^{2a b}, W^{(2a + 1) b}), W = exp(-j 2 pi / M), b = a lane's digit: the lanes of
// a warp read consecutive float4.  2048: the same with a < 16, b < 64, then W_64^{a b} for a, b < 8.
static int table_entries(int R1, int M) { return M == 2048 ? 16 * 64 + 32 : R1 / 2 * R1; }

__global__ void __launch_bounds__(256) reg_table_kernel(float4* __restrict__ tab, int na, int nb, int M) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < na * nb) {
    const int a = i / nb, b = i - a * nb;
    const float2 w0 = twiddle_fwd((unsigned)(2 * a * b % M), (unsigned)M), w1 = twiddle_fwd((unsigned)((2 * a + 1) * b % M), (unsigned)M);
    tab[i] = make_float4(w0.x, w0.y, w1.x, w1.y);
  }
}
__global__ void reg_table64_kernel(float2* __restrict__ tab) {
  const int i = threadIdx.x;
  tab[i] = twiddle_fwd((unsigned)((i >> 3) * (i & 7)), 64u);
}

size_t reg_table_bytes() {
  size_t n = 0;
#define SPECTRE_REG_SUM(R1, R2) n += table_entries(R1, R1 * R2);
  SPECTRE_REG_TWO_STEP(SPECTRE_REG_SUM)
#undef SPECTRE_REG_SUM
  return (n + table_entries(32, 2048)) * sizeof(float4);
}

const float4* reg_table(const spectre_ctx* ctx, int M) {
  const float4* t = reinterpret_cast<const float4*>(ctx->tw_reg);
#define SPECTRE_REG_AT(R1, R2) if (M == R1 * R2) return t; t += table_entries(R1, R1 * R2);
  SPECTRE_REG_TWO_STEP(SPECTRE_REG_AT)
#undef SPECTRE_REG_AT
  return t;
}

int reg_build_tables(void* tab, cudaStream_t st) {
  float4* t = reinterpret_cast<float4*>(tab);
#define SPECTRE_REG_BUILD(R1, R2)                                                                     \
  reg_table_kernel<<<(R1 / 2 * R1 + 255) / 256, 256, 0, st>>>(t, R1 / 2, R1, R1 * R2);                \
  t += table_entries(R1, R1 * R2);
  SPECTRE_REG_TWO_STEP(SPECTRE_REG_BUILD)
#undef SPECTRE_REG_BUILD
  reg_table_kernel<<<4, 256, 0, st>>>(t, 16, 64, 2048);
  reg_table64_kernel<<<1, 64, 0, st>>>(reinterpret_cast<float2*>(t + 16 * 64));
  SPECTRE_LAUNCH_OK("reg_table_kernel");
  return SPECTRE_OK;
}

}  // namespace spectre
