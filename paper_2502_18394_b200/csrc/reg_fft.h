// Host interface of the register-resident fp32 transforms (reg_fft.cuh).
#pragma once
#include "common.cuh"

namespace spectre {

// The complex workspace of the multi-pass transforms: [sequence][tile of 8 column pairs][M rows][pairs of the tile].  Neighbouring rows
// of a tile, which a warp stores together, are contiguous; as rows of all D/2 pairs every 64 bytes were a line, and a cycle of the
// load/store unit, of their own.
constexpr int kWsPairs = 8;
__host__ __device__ inline int ws_width(int half, int pair) { const int left = half - (pair & ~(kWsPairs - 1)); return left < kWsPairs ? left : kWsPairs; }
__host__ __device__ inline size_t ws_at(int half, int M, size_t seq, int row, int pair) {
  return (seq * half + (pair & ~(kWsPairs - 1))) * M + (size_t)row * ws_width(half, pair) + (pair & (kWsPairs - 1));
}

struct RegParams {
  const void* src;          // tokens [B, L, H, D]
  const void* src2;         // second tensor: of the gradient; forward: its nslab sequences follow the first one's in the launch (NULL: none)
  void* dst;                // tokens out
  float2* ws;               // complex rows (ws_at), sequences slab_local N1 + k1: input and / or output
  float2* ws2;              // forward: rows of the second tensor
  const float2* g;          // gate [B*H][K]
  const float2* spec;       // half spectra [B*H][K][D] (inverse)
  float2* sums;             // gradient: partial sums [slab_local][parts][n]; NULL: not wanted
  void* ring;               // forward: dense [B][n][H][D] copy of the zero-padded input, or NULL
  const float4* tw;         // twiddles of the plan
  int64_t s_sb, s_sl, s_sh;
  int64_t s2_sb, s2_sl, s2_sh;
  int64_t d_sb, d_sl, d_sh;
  int batch, H, D, L, n, K;
  int* status;              // host-mapped status word (bounded waits)
  int N1;                   // outer factor of n = N1 M; a CTA's sequence is k1 of N1
  int decim;                // forward, from tokens: element j of sequence k1 is token N1 j + k1
  int slab0, ntile, nslab;
  float scale;              // 1/n, folded into the gate
};

// Lengths M that one CTA transforms: the powers of two 64 ... 2048 and, for patch grids, the square of every even side from 8 to 32
// whose prime factors are 2, 3, 5, 7 (the others are no supported lengths).  Even, because the twiddle tables hold pairs of
// factors; the first step is at least the second and a multiple of it, so that a thread holds as many points on either side of
// the exchange: odd sides and most rectangles have no such plan and run on onchip_kernel.  Mixer of 12.6 M elements there and
// here, fp32 / bf16, us: 100 89 / 106 -> 28 / 25, 144 102 / 113 -> 25 / 20, 324 129 / 149 -> 33 / 30, 900 119 / 135 -> 36 / 35 (its backward
// 236 ... 368 -> 38 ... 62), one sequence of 900 19 -> 7; what stays there: 225 96 / 111, 441 113 / 130, 192 71 / 88, 384 86 / 105.
#define SPECTRE_REG_TWO_STEP(X)                                  \
  X(8, 8) X(16, 8) X(16, 16) X(32, 16) X(32, 32) X(10, 10)       \
  X(12, 12) X(14, 14) X(18, 18) X(20, 20) X(24, 24) X(28, 28) X(30, 30)
bool reg_supported(int M);
constexpr int kRegWsM = 1024;    // the length whose rows may also come from the complex workspace
// partial sums per (batch, head) and bin that the gradient leaves, one per group of pairs summed inside a warp
int reg_parts(int M, int D);

// One launch over nslab slabs (p.tw and p.ntile are filled in); `ws`: rows of the complex workspace (M = kRegWsM)
// instead of tokens of type dtype.
int reg_mix(const spectre_ctx* ctx, cudaStream_t st, RegParams p, int M, int nslab, bool ws, int dtype);
int reg_forward(const spectre_ctx* ctx, cudaStream_t st, RegParams p, int M, int nslab, int dtype);   // with src2: of either tensor
int reg_inverse(const spectre_ctx* ctx, cudaStream_t st, RegParams p, int M, int nslab, bool ws, int dtype);
int reg_grad(const spectre_ctx* ctx, cudaStream_t st, RegParams p, int M, int nslab, int dtype);

// Twiddle tables of all plans: built once per context.
size_t reg_table_bytes();
int reg_build_tables(void* tab, cudaStream_t st);
const float4* reg_table(const spectre_ctx* ctx, int M);

}  // namespace spectre
