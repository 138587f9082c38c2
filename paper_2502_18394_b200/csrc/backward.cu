// Backward of the spectral mixer (Eq. 3-4 are real-linear in V and in (Re g, Im g); Sec. 3.7
// asks for differentiability).  With Vhat = R_n(pad V), Ghat = R_n(pad dY):
//   dV   = R_n^{-1}( conj(g) Ghat )              -> the forward mixer on dY with the conjugate gate
//   dg_k = (w_k / n) sum_c conj(Vhat_{k,c}) Ghat_{k,c},   w_0 = w_{n/2} = 1, else 2
// The gate gradient needs both spectra at once: a forward-only pass of the fp32 transform
// kernels over either tensor into the workspace (pair-packed columns, Z = fft(a + jb)), then one reduction over the
// column pairs that uses  conj(A^V) A^G + conj(B^V) B^G = ( conj(Z^V_k) Z^G_k + Z^V_{n-k} conj(Z^G_{n-k}) ) / 2.
// Beyond one CTA's 2048 rows the passes leave the spectra of the N1 decimated sequences and the reduction
// runs the last radix-N1 step itself.
#include "fft_reg.cuh"
#include "reg_fft.h"

namespace spectre {

// from mixer.cu
int forward_decimated(const spectre_ctx* ctx, cudaStream_t st, const spectre_act* v, const spectre_act* with, int n, int slab0, int cnt,
                      float2* ws, float2* ws_with, int* N1_out, int* M_out, int N1_max, void* ring, int* ring_done);
bool transform_supported(const spectre_ctx* ctx, int n);
size_t transform_slab_bytes(int n, int D);
int mixer_check(const spectre_ctx* ctx, const spectre_act* v, const float* g, const spectre_act* y, int n_fft, const void* workspace,
                size_t workspace_bytes);

__global__ void __launch_bounds__(256) conj_gate_kernel(const float2* g, float2* gc, size_t total) {
  after_previous();
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < total) {
    float2 v = g[i];
    gc[i] = make_float2(v.x, -v.y);
  }
}

// dg from the partial sums S_k = sum over the pairs of conj(Z^V_k) Z^G_k of all n bins, which the transform kernels
// leave per group of pairs: dg_k = (w_k / 2n) (S_k + conj(S_{n-k})).
__global__ void __launch_bounds__(256) gate_grad_sum_kernel(const float2* sums, float2* dg, int n, int K,
                                                            int parts, int slab0, int nslab) {
  after_previous();
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (size_t)nslab * K) return;
  const int k = (int)(i % K), slab_local = (int)(i / K), km = k == 0 ? 0 : n - k;
  const float2* s = sums + (size_t)slab_local * parts * n;
  float2 acc = make_float2(0.f, 0.f);
#pragma unroll 4
  for (int p = 0; p < parts; ++p) {
    const float2 a = s[(size_t)p * n + k], b = s[(size_t)p * n + km];
    acc.x += a.x + b.x;
    acc.y += a.y - b.y;
  }
  const float w = ((k == 0 || 2 * k == n) ? 0.5f : 1.0f) / (float)n;
  dg[(size_t)(slab0 + slab_local) * K + k] = cscale(acc, w);
}

// One warp per (slab, bin): lanes over the column pairs, both workspaces hold the spectrum itself,
// a sequence per slab (transforms that fit one CTA).
__global__ void __launch_bounds__(256) gate_grad_kernel(const float2* wsV, const float2* wsG,
                                                        float2* dg, int n, int K, int D, int slab0, int nslab) {
  after_previous();
  const size_t wid = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (wid >= (size_t)nslab * K) return;
  const int k = (int)(wid % K), slab_local = (int)(wid / K);
  const int km = (n - k) % n;
  const int half = D / 2;
  float2 acc = make_float2(0.f, 0.f);
  for (int c = lane; c < half; c += 32) {
    const size_t rk = ws_at(half, n, (size_t)slab_local, k, c), rm = ws_at(half, n, (size_t)slab_local, km, c);
    const float2 vk = wsV[rk], vm = wsV[rm], gk = wsG[rk], gm = wsG[rm];
    acc = cadd(acc, cmulc(gk, vk));          // conj(Z^V_k) Z^G_k
    acc = cadd(acc, cmulc(vm, gm));          // Z^V_{n-k} conj(Z^G_{n-k})
  }
  for (int o = 16; o > 0; o >>= 1) {
    acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
    acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
  }
  if (lane == 0) {
    const float w = ((k == 0 || 2 * k == n) ? 1.0f : 2.0f) * 0.5f / (float)n;
    dg[(size_t)(slab0 + slab_local) * K + k] = cscale(acc, w);
  }
}

// Longer transforms, n = N1 M with token t = N1 n2 + n1: the workspaces hold Y[n1][k2], the M-point spectra of
// the N1 decimated sequences (workspace sequence slab_local N1 + n1), and Z[k2 + M k1] = sum_n1 W_N1^{n1 k1} W_n^{n1 k2} Y[n1][k2].
// A warp per (slab, k2 <= M/2).  Lanes 0-15 form Z of both tensors at k2 + M k1, lanes 16-31 at m2 + M k1, m2 = M - k2: each
// family holds the mirror bins n - k of the other.  A lane takes two column pairs (16-byte loads), sums
// S[k1] = conj(Z^V) Z^G over its pairs, the half-warp over its lanes, and dg_k = (w_k / 2n)(S_k + conj(S_{n-k})) takes one
// exchange between the halves.  Bound by HBM; with both families and tensors in one lane (256 registers of spectra at
// N1 = 8) the pass over 134 MB took 43 us.
template <int N1>
__global__ void __launch_bounds__(256, N1 <= 8 ? 2 : 1) gate_grad_combine_kernel(const float2* wsV, const float2* wsG,
                                                                float2* dg, int n, int K, int D, int M,
                                                                int slab0, int nslab) {
  after_previous();
  const size_t wid = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31, sub = lane & 15, s = sub % N1;
  const int nk2 = M / 2 + 1, half = D / 2;
  if (wid >= (size_t)nslab * nk2) return;
  const int slab_local = (int)(wid / nk2), k2 = (int)(wid % nk2), m2 = (M - k2) % M;
  const int mine = lane < 16 ? k2 : m2;
  float2 w[N1];
  w[0] = make_float2(1.f, 0.f);
#pragma unroll
  for (int q = 1; q < N1; ++q) w[q] = (q == 1) ? twiddle_fwd((unsigned)mine, (unsigned)n) : cmul(w[q / 2], w[q - q / 2]);
  float2 acc[N1];
#pragma unroll
  for (int k1 = 0; k1 < N1; ++k1) acc[k1] = make_float2(0.f, 0.f);
  for (int c = 2 * sub; c < half; c += 32) {                   // D is a multiple of 8: whole 16-byte pieces
    float2 v[2][N1], g[2][N1];
    const size_t first = ws_at(half, M, (size_t)slab_local * N1, mine, c), step = (size_t)M * half;
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1) {
      const size_t at = first + n1 * step;
      const float4 tv = __ldcs(reinterpret_cast<const float4*>(wsV + at)), tg = __ldcs(reinterpret_cast<const float4*>(wsG + at));
      v[0][n1] = make_float2(tv.x, tv.y); v[1][n1] = make_float2(tv.z, tv.w);
      g[0][n1] = make_float2(tg.x, tg.y); g[1][n1] = make_float2(tg.z, tg.w);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
#pragma unroll
      for (int q = 1; q < N1; ++q) {
        v[i][q] = cmul(v[i][q], w[q]);
        g[i][q] = cmul(g[i][q], w[q]);
      }
      RegDft<N1, false>::run(v[i]);
      RegDft<N1, false>::run(g[i]);
#pragma unroll
      for (int k1 = 0; k1 < N1; ++k1) acc[k1] = cadd(acc[k1], cmulc(g[i][k1], v[i][k1]));
    }
  }
  // lane s of the half-warp: the sum of value s over its 16 lanes
#pragma unroll
  for (int h = N1 / 2; h >= 1; h >>= 1) {
    const bool up = s & h;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const float2 send = up ? acc[i] : acc[i + h], keep = up ? acc[i + h] : acc[i];
      acc[i] = make_float2(keep.x + __shfl_xor_sync(0xffffffffu, send.x, h), keep.y + __shfl_xor_sync(0xffffffffu, send.y, h));
    }
  }
#pragma unroll
  for (int h = N1; h < 16; h <<= 1) {
    acc[0].x += __shfl_xor_sync(0xffffffffu, acc[0].x, h);
    acc[0].y += __shfl_xor_sync(0xffffffffu, acc[0].y, h);
  }
  // the mirror of bin s of a family is bin N1 - 1 - s of the other, at k2 = 0 bin (N1 - s) % N1 of the same one
  const int from = k2 == 0 ? (N1 - s) % N1 : (lane ^ 16) - s + (N1 - 1 - s);
  const float mx = __shfl_sync(0xffffffffu, acc[0].x, from), my = __shfl_sync(0xffffffffu, acc[0].y, from);
  const int k = mine + M * s;
  const bool write = sub < N1 && (k2 == 0 ? lane < 16 && s <= N1 / 2 : s < N1 / 2 && (lane < 16 || k2 != m2));
  if (write) {
    const float wt = ((k == 0 || 2 * k == n) ? 0.5f : 1.0f) / (float)n;      // bins other than 0 and n/2 count twice
    dg[(size_t)(slab0 + slab_local) * K + k] = make_float2((acc[0].x + mx) * wt, (acc[0].y - my) * wt);
  }
}

template <int N1>
static void launch_gate_grad_combine(cudaStream_t st, const float2* wsV, const float2* wsG, float2* dg, int n, int K, int D,
                                     int M, int slab0, int cnt) {
  const size_t nwarps = (size_t)cnt * (M / 2 + 1);
  (void)launch_after(gate_grad_combine_kernel<N1>, (unsigned)((nwarps * 32 + 255) / 256), 256, 0, st, wsV, wsG, dg, n, K, D, M, slab0,
                     cnt);                                     // the caller asks for the error
}

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }
static const size_t kSpectrumCap = (size_t)128 << 20;      // per spectrum buffer

static size_t spectrum_group(int n, int D, int nslab) {
  size_t per = transform_slab_bytes(n, D);
  size_t g = kSpectrumCap / per;
  if (g < 1) g = 1;
  if (g > (size_t)nslab) g = (size_t)nslab;
  return g;
}

// Lengths one CTA transforms: dg, and dv with it, from one kernel over both tensors.
static size_t grad_slab_bytes(int n, int D) { return (size_t)reg_parts(n, D) * n * sizeof(float2); }
static int backward_reg(const spectre_ctx* ctx, cudaStream_t st, const spectre_act* v, const spectre_act* dy, const float* g,
                        const spectre_act* dv, float* dg, int n, void* ws, size_t ws_bytes) {
  const int nslab = v->B * v->H, K = n / 2 + 1, parts = reg_parts(n, v->D);
  RegParams p = {};
  p.n = n; p.K = K; p.H = v->H; p.D = v->D; p.L = v->L; p.N1 = 1;
  p.scale = 1.0f / (float)n;
  p.g = reinterpret_cast<const float2*>(g);
  p.src = v->ptr; p.s_sb = v->stride_b; p.s_sl = v->stride_l; p.s_sh = v->stride_h;
  p.src2 = dy->ptr; p.s2_sb = dy->stride_b; p.s2_sl = dy->stride_l; p.s2_sh = dy->stride_h;
  if (dv) { p.dst = dv->ptr; p.d_sb = dv->stride_b; p.d_sl = dv->stride_l; p.d_sh = dv->stride_h; }
  p.sums = reinterpret_cast<float2*>(ws);
  size_t group = ws_bytes / grad_slab_bytes(n, v->D);
  if (group > (size_t)nslab) group = (size_t)nslab;
  for (int s0 = 0; s0 < nslab; s0 += (int)group) {
    const int cnt = nslab - s0 < (int)group ? nslab - s0 : (int)group;
    p.slab0 = s0;
    int rc = reg_grad(ctx, st, p, n, cnt, v->dtype);
    if (rc != SPECTRE_OK) return rc;
    SPECTRE_CUDA_OK(launch_after(gate_grad_sum_kernel, (unsigned)(((size_t)cnt * K + 255) / 256), 256, 0, st, p.sums,
                                 reinterpret_cast<float2*>(dg), n, K, parts, s0, cnt));
    SPECTRE_LAUNCH_OK("gate_grad_sum_kernel");
  }
  return SPECTRE_OK;
}

}  // namespace spectre

using namespace spectre;

extern "C" size_t spectre_mixer_backward_workspace_bytes(const spectre_ctx* ctx, int32_t B, int32_t L, int32_t H, int32_t D,
                                                         int32_t n_fft, int32_t dtype) {
  if (!ctx || B < 1 || H < 1 || D < 8 || !transform_supported(ctx, n_fft)) return 0;
  const size_t K = (size_t)n_fft / 2 + 1;
  return align256((size_t)B * H * K * sizeof(float2)) +
         align256(spectre_mixer_workspace_bytes(ctx, B, L, H, D, n_fft, dtype)) +
         2 * spectrum_group(n_fft, D, B * H) * transform_slab_bytes(n_fft, D);
}

extern "C" int spectre_mixer_backward(spectre_ctx* ctx, void* stream, const spectre_act* v, const spectre_act* dy,
                                      const float* g, const spectre_act* dv, float* dg, int32_t n_fft, void* workspace,
                                      size_t workspace_bytes) {
  if (!ctx) return fail(SPECTRE_ERR_INVALID_ARG, "ctx is NULL");
  int rc = check_act(v, "v");
  if (rc != SPECTRE_OK) return rc;
  rc = check_act(dy, "dy");
  if (rc != SPECTRE_OK) return rc;
  if (dv) {
    rc = check_act(dv, "dv");
    if (rc != SPECTRE_OK) return rc;
    if (dv->B != v->B || dv->L != v->L || dv->H != v->H || dv->D != v->D || dv->dtype != v->dtype)
      return fail(SPECTRE_ERR_INVALID_ARG, "dv differs from v in shape or dtype");
  }
  if (dy->B != v->B || dy->L != v->L || dy->H != v->H || dy->D != v->D || dy->dtype != v->dtype)
    return fail(SPECTRE_ERR_INVALID_ARG, "dy differs from v in shape or dtype");
  if (!dv && !dg) return fail(SPECTRE_ERR_INVALID_ARG, "neither dv nor dg requested");
  if (!g || (reinterpret_cast<uintptr_t>(g) & 7)) return fail(SPECTRE_ERR_INVALID_ARG, "g is NULL or not 8-byte aligned");
  if (dg && (reinterpret_cast<uintptr_t>(dg) & 7)) return fail(SPECTRE_ERR_INVALID_ARG, "dg not 8-byte aligned");
  if (n_fft < v->L) return fail(SPECTRE_ERR_INVALID_ARG, "n_fft smaller than L");
  if (!transform_supported(ctx, n_fft)) return fail(SPECTRE_ERR_UNSUPPORTED, "n_fft outside the supported set");
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 15))
    return fail(SPECTRE_ERR_WORKSPACE, "workspace is NULL or not 16-byte aligned");
  const int B = v->B, H = v->H, D = v->D, nslab = B * H;
  const size_t K = (size_t)n_fft / 2 + 1;
  const size_t gc_bytes = align256((size_t)nslab * K * sizeof(float2));
  const size_t mix_bytes = align256(spectre_mixer_workspace_bytes(ctx, B, v->L, H, D, n_fft, v->dtype));
  const size_t per = transform_slab_bytes(n_fft, D);
  if (workspace_bytes < gc_bytes + mix_bytes + 2 * per) return fail(SPECTRE_ERR_WORKSPACE, "backward workspace too small");
  unsigned char* base = reinterpret_cast<unsigned char*>(workspace);
  auto pitch_ok = [](const spectre_act* a) { return !a || (a->stride_l >= 0 && a->stride_l <= (1 << 18)); };   // 32-bit row offsets
  const bool one_kernel = dg && reg_supported(n_fft) && pitch_ok(v) && pitch_ok(dy) && pitch_ok(dv);
  if (dv && !one_kernel) {                   // a mixer that would be refused below must not leave dg written
    rc = mixer_check(ctx, dy, reinterpret_cast<const float*>(base), dv, n_fft, mix_bytes ? base + gc_bytes : nullptr, mix_bytes);
    if (rc != SPECTRE_OK) return rc;
  }
  SPECTRE_CUDA_OK(cudaSetDevice(ctx->device));
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (one_kernel)
    return backward_reg(ctx, st, v, dy, g, dv, dg, n_fft, base + gc_bytes + mix_bytes, workspace_bytes - gc_bytes - mix_bytes);
  if (dg) {                                  // first: dv may alias dy, which this reads
    size_t group = (workspace_bytes - gc_bytes - mix_bytes) / (2 * per);
    if (group > (size_t)nslab) group = (size_t)nslab;
    float2* wsV = reinterpret_cast<float2*>(base + gc_bytes + mix_bytes);
    float2* wsG = reinterpret_cast<float2*>(base + gc_bytes + mix_bytes + group * per);
    for (int s0 = 0; s0 < nslab; s0 += (int)group) {
      const int cnt = nslab - s0 < (int)group ? nslab - s0 : (int)group;
      int N1 = 1, M = n_fft;
      int no_ring = 0;
      rc = forward_decimated(ctx, st, v, dy, n_fft, s0, cnt, wsV, wsG, &N1, &M, 16, nullptr, &no_ring);
      if (rc != SPECTRE_OK) return rc;
      float2* dgc = reinterpret_cast<float2*>(dg);
      switch (N1) {
        case 1: {
          const size_t nwarps = (size_t)cnt * K;
          SPECTRE_CUDA_OK(launch_after(gate_grad_kernel, (unsigned)((nwarps * 32 + 255) / 256), 256, 0, st, wsV, wsG, dgc, n_fft, (int)K,
                                       D, s0, cnt));
          break;
        }
        case 2: launch_gate_grad_combine<2>(st, wsV, wsG, dgc, n_fft, (int)K, D, M, s0, cnt); break;
        case 4: launch_gate_grad_combine<4>(st, wsV, wsG, dgc, n_fft, (int)K, D, M, s0, cnt); break;
        case 8: launch_gate_grad_combine<8>(st, wsV, wsG, dgc, n_fft, (int)K, D, M, s0, cnt); break;
        case 16: launch_gate_grad_combine<16>(st, wsV, wsG, dgc, n_fft, (int)K, D, M, s0, cnt); break;
        default: return fail(SPECTRE_ERR_UNSUPPORTED, "outer factor not supported");
      }
      SPECTRE_LAUNCH_OK("gate_grad kernel");
    }
  }
  if (dv) {
    float2* gc = reinterpret_cast<float2*>(base);
    const size_t total = (size_t)nslab * K;
    SPECTRE_CUDA_OK(launch_after(conj_gate_kernel, (unsigned)((total + 255) / 256), 256, 0, st, reinterpret_cast<const float2*>(g), gc, total));
    SPECTRE_LAUNCH_OK("conj_gate_kernel");
    rc = spectre_mixer_forward(ctx, stream, dy, reinterpret_cast<const float*>(gc), dv, n_fft, nullptr,
                               mix_bytes ? base + gc_bytes : nullptr, mix_bytes);
    if (rc != SPECTRE_OK) return rc;
  }
  return SPECTRE_OK;
}
