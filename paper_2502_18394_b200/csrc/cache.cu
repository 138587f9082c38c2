// Prefix-FFT cache (Sec. 3.3, Eq. 5, Alg. 1): prefill, per-token append, and the whole decode
// step with single-row read-out.
#include "reg_fft.h"

namespace spectre {

// from mixer.cu / gate.cu
int forward_decimated(const spectre_ctx* ctx, cudaStream_t st, const spectre_act* v, const spectre_act* with, int n, int slab0, int cnt,
                      float2* ws, float2* ws_with, int* N1_out, int* M_out, int N1_max, void* ring, int* ring_done);
bool transform_supported(const spectre_ctx* ctx, int n);
size_t transform_slab_bytes(int n, int D);
int pool_sum_ring(const spectre_ctx* ctx, cudaStream_t st, const spectre_act* q, float* sums, void* ring, int N);
size_t gate_min_workspace(int B, int H, int D, int n_fft, int r);
int gate_check(const spectre_ctx* ctx, const spectre_act* q, const float* sum_q, int B, int H, int D, float inv_count,
               const spectre_gate_params* gp, int n_fft, const float* g_out, const void* workspace, size_t workspace_bytes);
int gate_call(spectre_ctx* ctx, void* stream, const spectre_act* q, const float* sum_q, int B, int H, int D, float inv_count,
              const spectre_gate_params* gp, int n_fft, const int64_t* shift, int64_t shift_all, float* g_out, float* qbar_out,
              void* workspace, size_t workspace_bytes, bool early, const GateToken* tok);
size_t inverse_workspace_bytes(const spectre_ctx* ctx, int n, int D, int nslab);
int inverse_from_spectrum(const spectre_ctx* ctx, cudaStream_t st, const float* spec, const float* g, const spectre_act* y,
                          int n, void* ws, size_t ws_bytes);

// ---- prefill -----------------------------------------------------------------
// With Z = fft_n(a + jb) for each column pair (a, b), the half spectra of the two real columns follow
// from Hermitian symmetry (App. B):
//   A_k = (Z_k + conj(Z_{n-k})) / 2,   B_k = (Z_k - conj(Z_{n-k})) / (2j).
__device__ __forceinline__ void store_split(float* prefix, size_t slab, int K, int D, int k, int c, float2 z,
                                            float2 zm) {
  float4 out;
  out.x = 0.5f * (z.x + zm.x);
  out.y = 0.5f * (z.y - zm.y);
  out.z = 0.5f * (z.y + zm.y);
  out.w = -0.5f * (z.x - zm.x);
  *reinterpret_cast<float4*>(prefix + ((slab * K + k) * D + 2 * c) * 2) = out;
}

// Transforms that fit the on-chip kernel (N1 = 1) leave Z in the workspace, a sequence per slab.  A thread takes
// kSplitBins consecutive bins of one column pair, all their loads in flight together.
constexpr int kSplitBins = 4;
__global__ void __launch_bounds__(256) split_kernel(const float2* ws, float* prefix, int n,
                                                    int K, int D, int slab0, int nslab) {
  after_previous();
  const int half = D / 2;
  const int kblocks = (K + kSplitBins - 1) / kSplitBins;
  const size_t total = (size_t)nslab * kblocks * half;
  size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= total) return;
  const int c = (int)(idx % half);
  const size_t r = idx / half;
  const int k0 = (int)(r % kblocks) * kSplitBins;
  const int slab_local = (int)(r / kblocks);
  const float2* col = ws + ws_at(half, n, (size_t)slab_local, 0, c);
  const int w = ws_width(half, c);
  float2 z[kSplitBins], zm[kSplitBins];
#pragma unroll
  for (int u = 0; u < kSplitBins; ++u) {
    const int k = min(k0 + u, K - 1), km = (n - k) % n;
    z[u] = col[(size_t)k * w];
    zm[u] = col[(size_t)km * w];
  }
#pragma unroll
  for (int u = 0; u < kSplitBins; ++u) {
    const int k = k0 + u;
    if (k < K) store_split(prefix, (size_t)(slab0 + slab_local), K, D, k, c, z[u], zm[u]);
  }
}

// Longer transforms, n = N1 M with token t = N1 n2 + n1: the forward pass leaves the M-point spectra of the
// N1 decimated sequences, Y[n1][k2] in workspace sequence slab_local N1 + n1, and the last radix-N1 step runs here,
//   Z[k2 + M k1] = sum_n1 W_N1^{n1 k1} ( W_n^{n1 k2} Y[n1][k2] ).
// Z[n - k] for k = k2 + M k1 is Z[(M - k2) + M (N1 - 1 - k1)] (k2 > 0), so the thread that owns k2 and
// M - k2 of one column pair holds both sides of every Hermitian pair it stores: the bins k2 + M k1 and
// (M - k2) + M k1 for k1 < N1/2 (and, at k2 = 0, bin n/2); the packed spectrum never goes back to memory.
template <int N1>
__global__ void __launch_bounds__(256) combine_split_kernel(const float2* ws, float* prefix, int n,
                                                            int K, int D, int M, int slab0) {
  after_previous();
  // a CTA: 32 neighbouring k2 of one workspace tile, 2 KB of each sequence and 128 bytes of every row of the result (32 sequences of 64 heads:
  // 196 us; 8 k2 of the four tiles of a head 206, one k2 a warp 211)
  const int half = D / 2, ntile = (half + kWsPairs - 1) / kWsPairs;
  const int nk2 = M / 2 + 1, nq = (nk2 + 31) / 32;
  const int c = (int)(blockIdx.x % ntile) * kWsPairs + threadIdx.x % kWsPairs;
  const int r = blockIdx.x / ntile;
  const int k2 = (r % nq) * 32 + threadIdx.x / kWsPairs;
  const int slab_local = r / nq;
  if (c >= half || k2 >= nk2) return;
  const int m2 = (M - k2) % M;
  float2 xa[N1], xb[N1];
  const float2* col = ws + ws_at(half, M, (size_t)slab_local * N1, 0, c);
  const size_t step = (size_t)M * half;                         // from one sequence to the next
  const int w = ws_width(half, c);
#pragma unroll
  for (int n1 = 0; n1 < N1; ++n1) {
    xa[n1] = col[n1 * step + (size_t)k2 * w];
    xb[n1] = col[n1 * step + (size_t)m2 * w];
  }
  const float2 wa1 = twiddle_fwd((unsigned)k2, (unsigned)n), wb1 = twiddle_fwd((unsigned)m2, (unsigned)n);
  float2 wa[N1], wb[N1];
  wa[0] = wb[0] = make_float2(1.f, 0.f);
#pragma unroll
  for (int q = 1; q < N1; ++q) {
    wa[q] = (q == 1) ? wa1 : cmul(wa[q / 2], wa[q - q / 2]);
    wb[q] = (q == 1) ? wb1 : cmul(wb[q / 2], wb[q - q / 2]);
    xa[q] = cmul(xa[q], wa[q]);
    xb[q] = cmul(xb[q], wb[q]);
  }
  Dft<N1, false>::run(xa);
  Dft<N1, false>::run(xb);
  const size_t slab = (size_t)(slab0 + slab_local);
  const bool own = k2 == 0 || k2 == m2;       // k2 = 0 and k2 = M/2 are their own mirror
#pragma unroll
  for (int k1 = 0; k1 < N1 / 2; ++k1) {
    store_split(prefix, slab, K, D, k2 + M * k1, c, xa[k1], k2 == 0 ? xa[(N1 - k1) % N1] : xb[N1 - 1 - k1]);
    if (!own) store_split(prefix, slab, K, D, m2 + M * k1, c, xb[k1], xa[N1 - 1 - k1]);
  }
  if (k2 == 0) store_split(prefix, slab, K, D, M * (N1 / 2), c, xa[N1 / 2], xa[N1 / 2]);
}

template <int N1>
static void launch_combine_split(cudaStream_t st, const float2* ws, float* prefix, int n, int K, int D, int M, int slab0,
                                 int cnt) {
  const size_t blocks = (size_t)cnt * ((M / 2 + 32) / 32) * ((D / 2 + kWsPairs - 1) / kWsPairs);
  (void)launch_after(combine_split_kernel<N1>, (unsigned)blocks, 256, 0, st, ws, prefix, n, K, D, M, slab0);    // the caller asks for the error
}

// Ring buffers: rows 0..L-1 <- tokens, rows L..N-1 <- 0 (Alg. 1 PreFill).  A CTA copies kRingRows
// consecutive rows of one batch entry, a thread one 16-byte piece of each with all of them in flight.
constexpr int kRingRows = 8;
template <typename T>
__global__ void __launch_bounds__(256) ring_fill_kernel(const T* src, int64_t sb, int64_t sl, int64_t sh,
                                                        T* buf, int B, int N, int H, int D, int L) {
  after_previous();
  constexpr int V = 16 / sizeof(T);
  const int vec_per_row = H * D / V;
  const int chunks = (N + kRingRows - 1) / kRingRows;
  const int b = blockIdx.x / chunks, r0 = (blockIdx.x - b * chunks) * kRingRows;
  for (int vi = threadIdx.x; vi < vec_per_row; vi += blockDim.x) {
    const int e = vi * V, h = e / D, c = e - h * D;
    const T* s = src + b * sb + h * sh + c;
    T* d = buf + (((size_t)b * N + r0) * H + h) * D + c;
    uint4 val[kRingRows];
#pragma unroll
    for (int u = 0; u < kRingRows; ++u)
      val[u] = (r0 + u < L) ? __ldcs(reinterpret_cast<const uint4*>(s + (int64_t)(r0 + u) * sl)) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int u = 0; u < kRingRows; ++u)
      if (r0 + u < N) __stcs(reinterpret_cast<uint4*>(d + (size_t)u * H * D), val[u]);
  }
}

// ---- append ------------------------------------------------------------------
// A warp owns 32 consecutive bins of one (batch, head): lane l evaluates the
// twiddle of bin k0 + l once, then the warp walks the 32 bins with every lane
// updating 2 channels (one 16-byte complex pair) of the bin's contiguous row.
template <typename T>
__global__ void __launch_bounds__(256) append_spectrum_kernel(float* prefix, const T* V_buf, const T* v_t, int H, int D, int N, int K,
                                                              int slot, unsigned tm, int evict, int warps_per_slab,
                                                              size_t nwarps_total) {
  after_previous();
  const size_t wid = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (wid >= nwarps_total) return;
  const int slab = (int)(wid / warps_per_slab);
  const int k0 = (int)(wid % warps_per_slab) * 32;
  const int b = slab / H, h = slab - b * H;
  const int half = D / 2, nb = min(32, K - k0);
  float* base = prefix + (((size_t)slab * K + k0) * D) * 2;
  // four bins per round, their loads issued together (the compiler cannot move a load of this array
  // above the store before it)
  float4 v[4];
  auto fetch = [&](int i0, int c) {
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (c < half && i0 + u < nb) v[u] = *reinterpret_cast<const float4*>(base + ((size_t)(i0 + u) * D + 2 * c) * 2);
  };
  T tok[2], old[2];                            // as loaded, so that nothing waits for them yet
  auto token = [&](int c) {
    if (c >= half) return;
    const T *a = v_t + (size_t)slab * D + 2 * c, *o = evict ? V_buf + (((size_t)b * N + slot) * H + h) * D + 2 * c : a;
    tok[0] = a[0]; tok[1] = a[1];
    old[0] = o[0]; old[1] = o[1];
  };
  token(lane);
  fetch(0, lane);
  // twiddle exp(-j 2 pi k t / N) of bin k0 + lane, angle reduced in integers
  float2 my = make_float2(1.f, 0.f);
  if (k0 + lane < K) {
    unsigned kk = (unsigned)(((unsigned long long)(k0 + lane) * tm) % (unsigned)N);
    my = twiddle_fwd(kk, (unsigned)N);
  }
  for (int c0 = 0; c0 < half; c0 += 32) {      // uniform trip count: every lane takes part in the shuffles
    const int c = c0 + lane;
    const bool live = c < half;
    if (c0 > 0) token(c);
    float d0 = 0.f, d1 = 0.f;
    if (live) {
      d0 = io<T>::load1(tok) - (evict ? io<T>::load1(old) : 0.f);
      d1 = io<T>::load1(tok + 1) - (evict ? io<T>::load1(old + 1) : 0.f);
    }
    for (int i0 = 0; i0 < nb; i0 += 4) {
      if (c0 + i0 > 0) fetch(i0, c);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = min(i0 + u, 31);
        const float wr = __shfl_sync(0xffffffffu, my.x, i), wi = __shfl_sync(0xffffffffu, my.y, i);
        if (live && i0 + u < nb) {
          v[u].x = fmaf(d0, wr, v[u].x); v[u].y = fmaf(d0, wi, v[u].y);
          v[u].z = fmaf(d1, wr, v[u].z); v[u].w = fmaf(d1, wi, v[u].w);
          *reinterpret_cast<float4*>(base + ((size_t)(i0 + u) * D + 2 * c) * 2) = v[u];
        }
      }
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(256) append_ring_kernel(T* V_buf, T* Q_buf,
                                                          float* sum_q, const T* q_t, const T* v_t, int B, int H, int D, int N,
                                                          int slot, int evict) {
  after_previous();
  const int total = B * H * D;
  int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= total) return;
  int b = idx / (H * D), hd = idx - b * (H * D);
  size_t o = ((size_t)b * N + slot) * H * D + hd;
  const T q = q_t[idx], v = v_t[idx];          // all loads in front of the stores, which none may pass
  const float s = sum_q[idx], qo = evict ? io<T>::load1(Q_buf + o) : 0.f;
  sum_q[idx] = s + (io<T>::load1(&q) - qo);
  Q_buf[o] = q;
  V_buf[o] = v;
}


// ---- decode step -------------------------------------------------------------
struct DecodeRows { int r[SPECTRE_DECODE_MAX_ROWS]; };

// One pass over the spectrum: P_k += delta exp(-j 2 pi k t / N) (Eq. 5) and, from the updated
// value, with delta = v_t - v_old, the NR read-out rows  V~[r] = (1/N) sum_k w_k Re(g_k P_k exp(+j 2 pi k r / N)),
// w_0 = w_{N/2} = 1, else 2 (Sec. 3.3.2 step e at one output index).  A CTA takes 256
// consecutive bins of one (batch, head), a warp 32 of them: lane l evaluates bin k0 + l's
// update twiddle and its NR read-out coefficients once, then the warp walks the 32 bins with
// every lane holding 2 channels.  Row sums are reduced over the CTA and written as one
// partial per (slab, bin block); the CTA that finishes a slab last adds its partials in a fixed order (a kernel of its
// own for that took 10 us behind the 650 us pass of 256 x 32k slabs and 2.7 us of a short window's 19).  The same CTA moves
// the slab's part of ring buffers and running sum on by the token: every other one has read the evicted row then, and the gate in front
// took the token from where it came (a kernel of its own for it in front of
// the gate: step of a 4k window 14.1 -> 15.8 us, of two 2k windows 15.2 -> 16.4).
// TAKE false: the cache holds the token already, the pass only reads out.
// Bound by HBM (16 bytes per bin and channel).  Launched as a programmatic dependent of the gate kernel, which waited for the caller's work:
// the first bins and the token are on their way before the gate is complete.
template <typename T, int NR, bool TAKE>
__global__ void __launch_bounds__(256) decode_spectrum_kernel(float* prefix, T* V_buf, T* Q_buf, float* sum_q, const T* q_t, const T* v_t,
                                                              int slot, int evict, const float2* g, float* partial, int* done, T* y, int H, int D, int N, int K,
                                                              unsigned tm, DecodeRows rows, int nrows, int nblk) {
  __shared__ float red[8][NR][64];
  __shared__ int last;
  const int slab = blockIdx.x / nblk, blk = blockIdx.x - slab * nblk;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k0 = (blk * 8 + warp) * 32, k = k0 + lane;
  const int nb = max(0, min(32, K - k0));
  const int half = D / 2;
  float* base = prefix + (((size_t)slab * K + k0) * D) * 2;
  // eight bins per round, their loads issued together (the compiler cannot move a load of this array above the store
  // before it)
  float4 v[8];
  auto fetch = [&](int i0, int c) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (c < half && i0 + u < nb) v[u] = *reinterpret_cast<const float4*>(base + ((size_t)(i0 + u) * D + 2 * c) * 2);
    }
  };
  const int b = slab / H, h = slab - b * H;
  const size_t ring = (((size_t)b * N + slot) * H + h) * D;
  T tok[2], old[2];                            // as loaded, so that nothing waits for them yet
  auto token = [&](int c) {
    if (c >= half || !TAKE) return;
    const T *a = v_t + (size_t)slab * D + 2 * c, *o = evict ? V_buf + ring + 2 * c : a;
    tok[0] = a[0]; tok[1] = a[1];
    old[0] = o[0]; old[1] = o[1];
  };
  token(lane);
  fetch(0, lane);
  float2 my = make_float2(1.f, 0.f);
  float2 coef[NR];
  const float wk = ((k == 0 || 2 * k == N) ? 1.0f : 2.0f) / (float)N;
#pragma unroll
  for (int r = 0; r < NR; ++r) coef[r] = make_float2(0.f, 0.f);
  if (k < K) {
    my = twiddle_fwd((unsigned)(((unsigned long long)k * tm) % (unsigned)N), (unsigned)N);
#pragma unroll
    for (int r = 0; r < NR; ++r)
      coef[r] = cscale(twiddle_fwd((unsigned)(((unsigned long long)k * (unsigned)rows.r[r]) % (unsigned)N), (unsigned)N), wk);
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");      // g
  if (k < K) {
    const float2 gk = g[(size_t)slab * K + k];
#pragma unroll
    for (int r = 0; r < NR; ++r) coef[r] = cmulc(gk, coef[r]);   // g_k exp(+j theta) w_k / N
  }
  for (int c0 = 0; c0 < half; c0 += 32) {               // uniform trip count: every lane takes part in the shuffles
    const int c = c0 + lane;
    const bool live = c < half;
    if (c0 > 0) token(c);
    float d0 = 0.f, d1 = 0.f;
    if (live && TAKE) {
      d0 = io<T>::load1(tok) - (evict ? io<T>::load1(old) : 0.f);
      d1 = io<T>::load1(tok + 1) - (evict ? io<T>::load1(old + 1) : 0.f);
    }
    float acc[NR][2];
#pragma unroll
    for (int r = 0; r < NR; ++r) acc[r][0] = acc[r][1] = 0.f;
    for (int i0 = 0; i0 < nb; i0 += 8) {
      if (i0 + c0 > 0) fetch(i0, c);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int i = min(i0 + u, 31);
        const bool in = i0 + u < nb;                          // uniform over the warp
        const float wr = __shfl_sync(0xffffffffu, my.x, i), wi = __shfl_sync(0xffffffffu, my.y, i);
        if (live && in) {
          v[u].x = fmaf(d0, wr, v[u].x); v[u].y = fmaf(d0, wi, v[u].y);
          v[u].z = fmaf(d1, wr, v[u].z); v[u].w = fmaf(d1, wi, v[u].w);
          *reinterpret_cast<float4*>(base + ((size_t)(i0 + u) * D + 2 * c) * 2) = v[u];
        }
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          const float cr = __shfl_sync(0xffffffffu, coef[r].x, i), ci = __shfl_sync(0xffffffffu, coef[r].y, i);
          if (in) {
            acc[r][0] = fmaf(cr, v[u].x, fmaf(-ci, v[u].y, acc[r][0]));
            acc[r][1] = fmaf(cr, v[u].z, fmaf(-ci, v[u].w, acc[r][1]));
          }
        }
      }
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      red[warp][r][2 * lane] = acc[r][0];
      red[warp][r][2 * lane + 1] = acc[r][1];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < NR * 64; e += 256) {
      const int r = e >> 6, cc = e & 63;
      if (2 * c0 + cc < D) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) s += red[w][r][cc];
        partial[(((size_t)slab * nblk + blk) * NR + r) * D + 2 * c0 + cc] = s;
      }
    }
    __syncthreads();
  }
  // the slab's last block: partials of all blocks, four threads per output
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(done + slab, 1) == nblk - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int c = TAKE ? (int)threadIdx.x : D; c < D; c += 256) {  // ring buffers and running sum of this slab
    const size_t at = (size_t)slab * D + c;
    const T q = q_t[at], v = v_t[at];                       // all loads in front of the stores, which none may pass
    const float s = sum_q[at], qo = evict ? io<T>::load1(Q_buf + ring + c) : 0.f;
    sum_q[at] = s + (io<T>::load1(&q) - qo);
    Q_buf[ring + c] = q;
    V_buf[ring + c] = v;
  }
  const int part = threadIdx.x & 3;
  for (int o0 = 0; o0 < nrows * D; o0 += 64) {                 // uniform trip count for the shuffles
    const int o = o0 + (int)(threadIdx.x >> 2), r = o / D, c = o - r * D;
    const bool in = o < nrows * D;
    const float* p = partial + ((size_t)slab * nblk * NR + r) * D + c;
    float s = 0.f;
    for (int j0 = part; j0 < nblk; j0 += 32) {
      float t[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) t[u] = in && j0 + 4 * u < nblk ? __ldcg(p + (size_t)(j0 + 4 * u) * NR * D) : 0.f;
#pragma unroll
      for (int u = 0; u < 8; ++u) s += t[u];
    }
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    if (NR == 1 && o0 == 0) __syncthreads();                   // one row may take the token's own place: all of it has been read
    if (in && part == 0) io<T>::store1(y + (((size_t)b * nrows + r) * H + h) * D + c, s);
  }
}

// The append: spectrum, then ring buffers and running sum
static int append_call(cudaStream_t st, const spectre_cache* cache, const void* q_t, const void* v_t, int64_t t) {
  const int B = cache->B, H = cache->H, D = cache->D, N = cache->N_max, K = N / 2 + 1;
  const int slot = (int)(t % N);
  const int evict = t >= N ? 1 : 0;
  const int wps = (K + 31) / 32;
  const size_t nwarps = (size_t)B * H * wps;
  const unsigned blocks = (unsigned)((nwarps * 32 + 255) / 256);
  const unsigned blocks2 = (unsigned)(((size_t)B * H * D + 255) / 256);
  SPECTRE_IO_DISPATCH(cache->buf_dtype, {
    SPECTRE_CUDA_OK(launch_after(append_spectrum_kernel<T>, blocks, 256, 0, st, cache->prefix_fft,
                                 reinterpret_cast<const T*>(cache->V_buf), reinterpret_cast<const T*>(v_t), H, D, N, K, slot,
                                 (unsigned)slot, evict, wps, nwarps));
    SPECTRE_CUDA_OK(launch_after(append_ring_kernel<T>, blocks2, 256, 0, st, reinterpret_cast<T*>(cache->V_buf),
                                 reinterpret_cast<T*>(cache->Q_buf), cache->sum_q, reinterpret_cast<const T*>(q_t),
                                 reinterpret_cast<const T*>(v_t), B, H, D, N, slot, evict));
  });
  SPECTRE_LAUNCH_OK("append kernels");
  return SPECTRE_OK;
}

// any byte in common
static bool overlap(const void* a, size_t na, const void* b, size_t nb) {
  const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
  return x < y + nb && y < x + na;
}

static int check_cache(const spectre_cache* c) {
  if (!c) return fail(SPECTRE_ERR_INVALID_ARG, "cache descriptor is NULL");
  if (c->B < 1 || c->H < 1 || c->D < 1 || c->N_max < 2) return fail(SPECTRE_ERR_INVALID_ARG, "cache extents");
  if (c->D % 8) return fail(SPECTRE_ERR_UNSUPPORTED, "cache D must be a multiple of 8");
  if (!is_io_dtype(c->buf_dtype)) return fail(SPECTRE_ERR_INVALID_ARG, "cache dtype");
  if (!c->prefix_fft || !c->V_buf || !c->Q_buf || !c->sum_q) return fail(SPECTRE_ERR_INVALID_ARG, "cache pointer is NULL");
  if ((reinterpret_cast<uintptr_t>(c->prefix_fft) | reinterpret_cast<uintptr_t>(c->V_buf) |
       reinterpret_cast<uintptr_t>(c->Q_buf)) & 15)
    return fail(SPECTRE_ERR_INVALID_ARG, "cache buffers must be 16-byte aligned");
  return SPECTRE_OK;
}

// Group size cap for the prefill scratch.  Larger groups measured faster (fewer, fuller launches; the partial
// spectra do not stay in L2 at any useful group size): 3.0 ms at 32-64 MB, 2.58 ms at 256 MB, 2.49 ms at 1 GiB, 2.47 ms
// with all 256 heads of the c4 window in one group (2.15 GB).
static const size_t kPrefillWsCap = (size_t)1 << 30;

}  // namespace spectre

using namespace spectre;

extern "C" size_t spectre_prefill_workspace_bytes(const spectre_ctx* ctx, int32_t B, int32_t H, int32_t D, int32_t N_max) {
  if (!ctx || B < 1 || H < 1 || D < 8 || !transform_supported(ctx, N_max)) return 0;
  size_t per = transform_slab_bytes(N_max, D);
  size_t g = kPrefillWsCap / per;
  if (g < 1) g = 1;
  if (g > (size_t)B * H) g = (size_t)B * H;
  return g * per;
}

extern "C" int spectre_prefix_cache_prefill(spectre_ctx* ctx, void* stream, const spectre_cache* cache,
                                            const spectre_act* q, const spectre_act* v, void* workspace,
                                            size_t workspace_bytes) {
  if (!ctx) return fail(SPECTRE_ERR_INVALID_ARG, "ctx is NULL");
  int rc = check_cache(cache);
  if (rc != SPECTRE_OK) return rc;
  rc = check_act(q, "q");
  if (rc != SPECTRE_OK) return rc;
  rc = check_act(v, "v");
  if (rc != SPECTRE_OK) return rc;
  const int B = cache->B, H = cache->H, D = cache->D, N = cache->N_max;
  if (q->B != B || q->H != H || q->D != D || v->B != B || v->H != H || v->D != D || q->L != v->L)
    return fail(SPECTRE_ERR_INVALID_ARG, "q / v shape differs from the cache");
  if (q->dtype != cache->buf_dtype || v->dtype != cache->buf_dtype)
    return fail(SPECTRE_ERR_INVALID_ARG, "q / v dtype differs from buf_dtype");
  if (v->L > N) return fail(SPECTRE_ERR_INVALID_ARG, "prompt longer than N_max");
  if (!transform_supported(ctx, N)) return fail(SPECTRE_ERR_UNSUPPORTED, "N_max outside the supported transform lengths");
  const size_t per = transform_slab_bytes(N, D);
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 15))
    return fail(SPECTRE_ERR_WORKSPACE, "workspace is NULL or not 16-byte aligned");
  if (workspace_bytes < per) return fail(SPECTRE_ERR_WORKSPACE, "prefill workspace smaller than one (batch, head) slab");
  // limits of the kernels behind the transforms, in front of the first launch
  if (B > 65535) return fail(SPECTRE_ERR_UNSUPPORTED, "B exceeds 65535");
  const size_t nblocks = (size_t)B * ((N + kRingRows - 1) / kRingRows);
  if (nblocks > 0x7fffffffu) return fail(SPECTRE_ERR_UNSUPPORTED, "B * N_max too large for the ring copy");
  SPECTRE_CUDA_OK(cudaSetDevice(ctx->device));
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int nslab = B * H, K = N / 2 + 1;
  size_t gmax = workspace_bytes / per;
  if (gmax > (size_t)nslab) gmax = (size_t)nslab;
  const int ngroups = (nslab + (int)gmax - 1) / (int)gmax;
  const int group = (nslab + ngroups - 1) / ngroups;             // equal groups rather than full ones and a remainder
  float2* ws = reinterpret_cast<float2*>(workspace);
  int v_ring_done = 0;                 // the transform's load pass can fill V_buf on its way
  for (int s0 = 0; s0 < nslab; s0 += group) {
    int cnt = nslab - s0 < group ? nslab - s0 : group;
    int N1 = 1, M = N;
    rc = forward_decimated(ctx, st, v, nullptr, N, s0, cnt, ws, nullptr, &N1, &M, 32, cache->V_buf, &v_ring_done);
    if (rc != SPECTRE_OK) return rc;
    switch (N1) {
      case 1: {
        size_t total = (size_t)cnt * ((K + kSplitBins - 1) / kSplitBins) * (D / 2);
        SPECTRE_CUDA_OK(launch_after(split_kernel, (unsigned)((total + 255) / 256), 256, 0, st, ws, cache->prefix_fft, N, K, D, s0, cnt));
        break;
      }
      case 2: launch_combine_split<2>(st, ws, cache->prefix_fft, N, K, D, M, s0, cnt); break;
      case 4: launch_combine_split<4>(st, ws, cache->prefix_fft, N, K, D, M, s0, cnt); break;
      case 8: launch_combine_split<8>(st, ws, cache->prefix_fft, N, K, D, M, s0, cnt); break;
      case 16: launch_combine_split<16>(st, ws, cache->prefix_fft, N, K, D, M, s0, cnt); break;
      case 32: launch_combine_split<32>(st, ws, cache->prefix_fft, N, K, D, M, s0, cnt); break;
      default: return fail(SPECTRE_ERR_UNSUPPORTED, "outer factor not supported");
    }
    SPECTRE_LAUNCH_OK("split kernel");
  }
  if (!v_ring_done) {
    const unsigned blocks = (unsigned)nblocks;
    SPECTRE_IO_DISPATCH(cache->buf_dtype, {
      SPECTRE_CUDA_OK(launch_after(ring_fill_kernel<T>, blocks, 256, 0, st, reinterpret_cast<const T*>(v->ptr), v->stride_b, v->stride_l,
                                   v->stride_h, reinterpret_cast<T*>(cache->V_buf), B, N, H, D, v->L));
    });
    SPECTRE_LAUNCH_OK("ring_fill_kernel");
  }
  // q is read once: its sum over the sequence and its ring copy come from the same pass
  return pool_sum_ring(ctx, st, q, cache->sum_q, cache->Q_buf, N);
}

extern "C" int spectre_prefix_cache_append(spectre_ctx* ctx, void* stream, const spectre_cache* cache, const void* q_t,
                                           const void* v_t, int64_t t) {
  if (!ctx) return fail(SPECTRE_ERR_INVALID_ARG, "ctx is NULL");
  int rc = check_cache(cache);
  if (rc != SPECTRE_OK) return rc;
  if (!q_t || !v_t) return fail(SPECTRE_ERR_INVALID_ARG, "token pointer is NULL");
  if (t < 0) return fail(SPECTRE_ERR_INVALID_ARG, "t must be >= 0");
  if ((size_t)cache->B * cache->H * cache->D > (size_t)1 << 30) return fail(SPECTRE_ERR_UNSUPPORTED, "B*H*D too large");
  SPECTRE_CUDA_OK(cudaSetDevice(ctx->device));
  return append_call(reinterpret_cast<cudaStream_t>(stream), cache, q_t, v_t, t);
}

static size_t round256(size_t x) { return (x + 255) & ~(size_t)255; }
static int decode_nr(int nrows) { return nrows <= 1 ? 1 : (nrows <= 2 ? 2 : SPECTRE_DECODE_MAX_ROWS); }

extern "C" size_t spectre_decode_workspace_bytes(const spectre_ctx* ctx, int32_t B, int32_t H, int32_t D, int32_t N_max,
                                                 int32_t nrows, int32_t toeplitz_r) {
  (void)ctx;
  if (B < 1 || H < 1 || D < 1 || N_max < 2 || nrows < 1 || nrows > SPECTRE_DECODE_MAX_ROWS || toeplitz_r < 0) return 0;
  const int K = N_max / 2 + 1, nblk = (K + 255) / 256;
  return round256((size_t)B * H * nblk * decode_nr(nrows) * D * 4) + round256((size_t)B * H * sizeof(int)) +
         gate_min_workspace(B, H, D, N_max, toeplitz_r);
}

extern "C" int spectre_prefix_cache_decode_step(spectre_ctx* ctx, void* stream, const spectre_cache* cache, const void* q_t,
                                                const void* v_t, int64_t t, const spectre_gate_params* params,
                                                const int32_t* rows, int32_t nrows, void* y_rows, float* g_out,
                                                void* workspace, size_t workspace_bytes) {
  if (!ctx) return fail(SPECTRE_ERR_INVALID_ARG, "ctx is NULL");
  int rc = check_cache(cache);
  if (rc != SPECTRE_OK) return rc;
  if (!q_t || !v_t || !y_rows || !g_out) return fail(SPECTRE_ERR_INVALID_ARG, "token, output or gate pointer is NULL");
  if (!params) return fail(SPECTRE_ERR_INVALID_ARG, "gate parameters are NULL");
  if (t < 0) return fail(SPECTRE_ERR_INVALID_ARG, "t must be >= 0");
  if (!rows || nrows < 1 || nrows > SPECTRE_DECODE_MAX_ROWS)
    return fail(SPECTRE_ERR_INVALID_ARG, "rows is NULL or nrows outside 1..SPECTRE_DECODE_MAX_ROWS");
  const int B = cache->B, H = cache->H, D = cache->D, N = cache->N_max;
  for (int i = 0; i < nrows; ++i)
    if (rows[i] < 0 || rows[i] >= N) return fail(SPECTRE_ERR_INVALID_ARG, "read-out row outside [0, N_max)");
  if ((size_t)B * H * D > (size_t)1 << 30) return fail(SPECTRE_ERR_UNSUPPORTED, "B*H*D too large");
  const int K = N / 2 + 1, nblk = (K + 255) / 256, NR = decode_nr(nrows);
  if ((size_t)B * H * nblk > (size_t)0x7fffffff) return fail(SPECTRE_ERR_UNSUPPORTED, "B*H*K too large");
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 15))
    return fail(SPECTRE_ERR_WORKSPACE, "workspace is NULL or not 16-byte aligned");
  const size_t part_bytes = round256((size_t)B * H * nblk * NR * D * 4);
  const size_t done_bytes = round256((size_t)B * H * sizeof(int));
  const size_t gate_bytes = gate_min_workspace(B, H, D, N, params->toeplitz_r < 0 ? 0 : params->toeplitz_r);
  if (workspace_bytes < part_bytes + done_bytes + gate_bytes) return fail(SPECTRE_ERR_WORKSPACE, "decode workspace too small");
  float* partial = reinterpret_cast<float*>(workspace);
  int* done = reinterpret_cast<int*>(reinterpret_cast<unsigned char*>(workspace) + part_bytes);
  void* gate_ws = reinterpret_cast<unsigned char*>(workspace) + part_bytes + done_bytes;
  // a gate that would be refused below must not leave the cache with the token in it
  rc = gate_check(ctx, nullptr, cache->sum_q, B, H, D, 1.0f / (float)N, params, N, g_out, gate_ws, gate_bytes);
  if (rc != SPECTRE_OK) return rc;
  SPECTRE_CUDA_OK(cudaSetDevice(ctx->device));
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int slot = (int)(t % N);
  const int evict = t >= N ? 1 : 0;
  // The token is read until the pass over the spectrum ends, by the CTAs of its own slab.  One row written over it is written by the last
  // of them; outputs that meet it in any other way wait until the cache has it (its spectrum goes through memory twice then).
  const size_t es = io_elem_bytes(cache->buf_dtype), tok_bytes = (size_t)B * H * D * es;
  auto meets = [&](const void* x) {
    return overlap(g_out, (size_t)B * H * K * sizeof(float2), x, tok_bytes) ||
           (overlap(y_rows, nrows * tok_bytes, x, tok_bytes) && !(nrows == 1 && y_rows == x));
  };
  const bool first = meets(q_t) || meets(v_t);
  if (first) {
    SPECTRE_CUDA_OK(cudaMemsetAsync(done, 0, (size_t)B * H * sizeof(int), st));
    rc = append_call(st, cache, q_t, v_t, t);
    if (rc != SPECTRE_OK) return rc;
  }
  // (c)-(d) gate from the running sum with the token in it, phase p = t
  const size_t row = (size_t)slot * H * D * es;
  const GateToken tok = {q_t, evict ? static_cast<const char*>(static_cast<const void*>(cache->Q_buf)) + row : nullptr, (size_t)N * H * D,
                         cache->buf_dtype, done, B * H};
  rc = gate_call(ctx, stream, nullptr, cache->sum_q, B, H, D, 1.0f / (float)N, params, N, nullptr, t, g_out, nullptr, gate_ws,
                 gate_bytes, false, first ? nullptr : &tok);
  if (rc != SPECTRE_OK) return rc;
  // (a), (b), (e) one pass over the spectrum, ring buffers and running sum
  DecodeRows dr;
  for (int i = 0; i < SPECTRE_DECODE_MAX_ROWS; ++i) dr.r[i] = rows[i < nrows ? i : nrows - 1];
  const unsigned blocks_s = (unsigned)((size_t)B * H * nblk);
  const float2* g2 = reinterpret_cast<const float2*>(g_out);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks_s);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  SPECTRE_IO_DISPATCH(cache->buf_dtype, {
    auto kern = NR == 1 ? decode_spectrum_kernel<T, 1, true> : (NR == 2 ? decode_spectrum_kernel<T, 2, true> : decode_spectrum_kernel<T, SPECTRE_DECODE_MAX_ROWS, true>);
    if (first) kern = NR == 1 ? decode_spectrum_kernel<T, 1, false> : (NR == 2 ? decode_spectrum_kernel<T, 2, false> : decode_spectrum_kernel<T, SPECTRE_DECODE_MAX_ROWS, false>);
    SPECTRE_CUDA_OK(launch_kernel(&cfg, kern, cache->prefix_fft, reinterpret_cast<T*>(cache->V_buf), reinterpret_cast<T*>(cache->Q_buf),
                                       cache->sum_q, reinterpret_cast<const T*>(q_t), reinterpret_cast<const T*>(v_t), slot, evict, g2, partial,
                                       done, reinterpret_cast<T*>(y_rows), H, D, N, K, (unsigned)slot, dr, (int)nrows, nblk));
  });
  return SPECTRE_OK;
}

extern "C" size_t spectre_readout_workspace_bytes(const spectre_ctx* ctx, int32_t B, int32_t H, int32_t D, int32_t N_max) {
  if (!ctx || B < 1 || H < 1 || D < 8 || !transform_supported(ctx, N_max)) return 0;
  return inverse_workspace_bytes(ctx, N_max, D, B * H);
}

extern "C" int spectre_prefix_cache_readout(spectre_ctx* ctx, void* stream, const spectre_cache* cache, const float* g,
                                            const spectre_act* y, void* workspace, size_t workspace_bytes) {
  if (!ctx) return fail(SPECTRE_ERR_INVALID_ARG, "ctx is NULL");
  int rc = check_cache(cache);
  if (rc != SPECTRE_OK) return rc;
  rc = check_act(y, "y");
  if (rc != SPECTRE_OK) return rc;
  if (!g || (reinterpret_cast<uintptr_t>(g) & 7)) return fail(SPECTRE_ERR_INVALID_ARG, "g is NULL or not 8-byte aligned");
  const int N = cache->N_max;
  if (y->B != cache->B || y->H != cache->H || y->D != cache->D || y->L > N || y->L < 1)
    return fail(SPECTRE_ERR_INVALID_ARG, "y shape differs from the cache (rows 0..L-1 of the window, L <= N_max)");
  if (!transform_supported(ctx, N)) return fail(SPECTRE_ERR_UNSUPPORTED, "N_max outside the supported transform lengths");
  SPECTRE_CUDA_OK(cudaSetDevice(ctx->device));
  return inverse_from_spectrum(ctx, reinterpret_cast<cudaStream_t>(stream), cache->prefix_fft, g, y, N, workspace,
                               workspace_bytes);
}
