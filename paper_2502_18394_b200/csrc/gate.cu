// Content-adaptive spectral gate (Sec. 3.2 step 3; Sec. 3.3.2 steps c-d).
//   pool_kernel      sum of the query tokens over the sequence (bandwidth-bound)
//   gate_hidden_kernel LayerNorm + hidden layer once per (head, batch group), long transforms only
//   gate_out_kernel    LayerNorm + hidden layer (per CTA, short transforms) and the output layer as a
//                      stream over W2, 1-8 batch entries per pass; with the Toeplitz update off it also applies modReLU and
//                      the positional phase
//   gate_mma_kernel    the same on the tensor cores, several batch entries with bf16 weights
//   gate_short_kernel  the same for few bins and several batch entries, all weights staged
//   gate_split_kernel  the same for one batch entry and few bins, several threads per bin
//   gate_post_kernel Toeplitz update, modReLU, phase (only when r > 0)
#include "tc_common.cuh"

#include <atomic>
#include <string>
#include <type_traits>

namespace spectre {

// ---- pooled sum over the sequence --------------------------------------------
// Grid (groups of 32 vectors, slices of the sequence, B).  A lane owns one 8-channel vector of the
// [H*D] row, so a warp reads 512 contiguous bytes of a row; the CTA's 8 warps take rows 8 apart with
// up to 8 rows per thread in flight and four CTAs per SM.  The warps' partial sums meet in shared memory, and the CTA adds
// one value per channel with float atomics into copy (slice mod ncopy) of sums[ncopy][B,H,D] (zeroed
// by the caller on the same stream), which keeps the contention per address low; where there are as many copies
// as slices it stores its sums instead.
template <typename T> struct vec8;
template <> struct vec8<bf16> {
  typedef uint4 raw;
  static constexpr int kRows = 8;
  static __device__ __forceinline__ raw load(const bf16* p) { return *reinterpret_cast<const uint4*>(p); }
  static __device__ __forceinline__ raw zero() { return make_uint4(0u, 0u, 0u, 0u); }
  static __device__ __forceinline__ void add(const raw& r, float (&a)[8]) {
    const uint32_t u[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      a[2 * i] += __uint_as_float(u[i] << 16);
      a[2 * i + 1] += __uint_as_float(u[i] & 0xffff0000u);
    }
  }
};
template <> struct vec8<f16> {
  typedef uint4 raw;
  static constexpr int kRows = 8;
  static __device__ __forceinline__ raw load(const f16* p) { return *reinterpret_cast<const uint4*>(p); }
  static __device__ __forceinline__ raw zero() { return make_uint4(0u, 0u, 0u, 0u); }
  static __device__ __forceinline__ void add(const raw& r, float (&a)[8]) {
    const uint32_t u[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 v = __half22float2(*reinterpret_cast<const __half2*>(&u[i]));
      a[2 * i] += v.x;
      a[2 * i + 1] += v.y;
    }
  }
};
template <> struct vec8<float> {
  struct raw { float4 lo, hi; };
  static constexpr int kRows = 4;
  static __device__ __forceinline__ raw load(const float* p) {
    raw r;
    r.lo = *reinterpret_cast<const float4*>(p);
    r.hi = *(reinterpret_cast<const float4*>(p) + 1);
    return r;
  }
  static __device__ __forceinline__ raw zero() {
    raw r;
    r.lo = make_float4(0.f, 0.f, 0.f, 0.f);
    r.hi = r.lo;
    return r;
  }
  static __device__ __forceinline__ void add(const raw& r, float (&a)[8]) {
    a[0] += r.lo.x; a[1] += r.lo.y; a[2] += r.lo.z; a[3] += r.lo.w;
    a[4] += r.hi.x; a[5] += r.hi.y; a[6] += r.hi.z; a[7] += r.hi.w;
  }
};

// RING: the rows also go, as loaded, into the dense copy ring[B][N][H][D]; rows L..N-1 of it are zeroed
// (the ring buffer of the Prefix-FFT cache, Alg. 1 PreFill), and the slices cover N rows instead of L.
template <typename T, bool RING>
__global__ void __launch_bounds__(256, 4) pool_kernel(const T* q, int64_t sb, int64_t sl, int64_t sh, int L,
                                                   int H, int D, int rows_per, int ncopy, size_t copy_stride,
                                                   float* sums, T* ring, int N,
                                                   const char* warm, unsigned warm_per, size_t warm_bytes) {
  __shared__ float red[8][8][32];                              // [warp][channel][lane]
  const bool own = (int)gridDim.y <= ncopy;                    // a copy of the sums per slice: stored, nothing was cleared
  if (own) after_previous();
  // the gate kernels behind this one may start early: they stream weights before they need the sums
  asm volatile("griddepcontrol.launch_dependents;");
  constexpr int R = vec8<T>::kRows;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b = blockIdx.z;
  if (warm_per && threadIdx.x == 0) {                          // this CTA's part of the weights that the gate kernel reads next
    const size_t at = (size_t)((b * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) * warm_per;
    if (at < warm_bytes)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" :: "l"(warm + at), "r"((unsigned)min((size_t)warm_per, warm_bytes - at)) : "memory");
  }
  const int vec_per_head = D / 8, nvec = H * vec_per_head;
  const int vi = blockIdx.x * 32 + lane;
  const bool live = vi < nvec;
  const int h = live ? vi / vec_per_head : 0, c = live ? (vi - h * vec_per_head) * 8 : 0;
  const T* base = q + b * sb + h * sh + c;
  const int r0 = blockIdx.y * rows_per, r1 = min(L, r0 + rows_per), r2 = RING ? min(N, r0 + rows_per) : r1;
  float acc[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] = 0.f;
  if (live) {
    T* out = RING ? ring + ((size_t)b * N * H + h) * D + c : nullptr;
    for (int r = r0 + warp; r < r2; r += 8 * R) {
      typename vec8<T>::raw v[R];
#pragma unroll
      for (int u = 0; u < R; ++u) v[u] = (r + 8 * u < r1) ? vec8<T>::load(base + (int64_t)(r + 8 * u) * sl) : vec8<T>::zero();
#pragma unroll
      for (int u = 0; u < R; ++u) {
        vec8<T>::add(v[u], acc);
        if (RING && r + 8 * u < r2) *reinterpret_cast<typename vec8<T>::raw*>(out + (size_t)(r + 8 * u) * H * D) = v[u];
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) red[warp][i][lane] = acc[i];
  __syncthreads();
  float s = 0.f;                                               // thread (channel = warp, lane) adds up the 8 warps
#pragma unroll
  for (int w = 0; w < 8; ++w) s += red[w][warp][lane];
  // with more slices than copies the kernel runs as the programmatic dependent of the kernel that clears the sums:
  // everything above overlaps it, the additions wait for it (no effect in an ordinary launch)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (live) {
    float* dst = sums + (size_t)(blockIdx.y % ncopy) * copy_stride + ((size_t)b * H + h) * D + c + warp;
    if (own) *dst = s;
    else atomicAdd(dst, s);
  }
}

// Clears the partial sums ahead of a pooling pass with several slices; lets that pass start at once.
__global__ void __launch_bounds__(256) pool_clear_kernel(float4* sums, size_t n4) {
  after_previous();                                            // the pass behind reads its rows without a wait of its own
  asm volatile("griddepcontrol.launch_dependents;");
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n4) sums[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// Sums of q over the sequence into *ncopy_used <= ncopy_max partial copies (the consumer adds them up);
// with `ring`, also the copy of q into ring[B][N][H][D] (zero rows from L on).
static int pool_launch(const spectre_ctx* ctx, cudaStream_t st, const spectre_act* q, float* sums, int ncopy_max,
                       int* ncopy_used, void* ring, int N, const void* warm, size_t warm_bytes) {
  const int rows = ring ? N : q->L;
  const size_t copy_stride = (size_t)q->B * q->H * q->D;
  const int groups = (q->H * (q->D / 8) + 31) / 32;
  if (q->B > 65535) return fail(SPECTRE_ERR_UNSUPPORTED, "B exceeds 65535");
  // one resident wave (four CTAs per SM) of equal slices, never a few CTAs more than fit at once;
  // at least 8 rows (one per warp) per CTA
  const long long per_slice = (long long)groups * q->B;
  long long slices = (4LL * ctx->sm_count) / per_slice;
  if (slices < 1) slices = 1;
  int rows_per = (int)((rows + slices - 1) / slices);
  if (rows_per < 8) rows_per = 8;
  int nslice = (rows + rows_per - 1) / rows_per;
  // Sequences of up to 1024 rows: a slice per copy instead, stored without a kernel that clears them (2 us of host time, and
  // the second's launch; one warp's 16 rows take 2 or 4 rounds of loads).  Gate call alone, many slices -> 8: at 1024 rows it gains
  // throughout (1 x 8 heads bf16 7.9 -> 6.8 us, 8 x 8 13.9 -> 12.5, fp32 1 x 32 13.2 -> 11.8), at 2048 in bf16 only (10.9 -> 9.1,
  // 15.1 -> 14.9; fp32 14.5 -> 15.3, 4 x 4 13.2 -> 14.1), at 4096 hardly anywhere (12.0 -> 13.5, 19.4 -> 21.5, 18.5 -> 23.1).  With
  // the mixer behind it 2048 rows gain nothing on the whole (bf16 4 x 4 30.5 -> 31.0, 8 x 8 48.7 -> 49.2, fp32 4 x 4 31.9 -> 34.3).
  if (nslice > 8 && ncopy_max >= 8 && rows <= 1024) {
    rows_per = (rows + 7) / 8;
    nslice = (rows + rows_per - 1) / rows_per;
  }
  const bool own = nslice <= ncopy_max && nslice <= 8;
  int ncopy = own ? nslice : (nslice + 15) / 16;               // <= 16 CTAs add into one address
  if (ncopy > 8) ncopy = 8;                                    // one batch of loads for the consumer
  if (ncopy > ncopy_max) ncopy = ncopy_max;
  if (ncopy < 1) ncopy = 1;
  *ncopy_used = ncopy;
  // Several slices add into the same words: a small kernel clears them (D is a multiple of 8 and the sums are
  // 16-byte aligned: whole float4) and the pooling kernel, its programmatic dependent, reads its rows meanwhile.
  // A memset node in the stream instead costs the step 3.6 us at L = 8192.
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)groups, (unsigned)nslice, (unsigned)q->B);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (!own) {
    const size_t n4 = copy_stride * ncopy / 4;
    if ((reinterpret_cast<uintptr_t>(sums) & 15) || (copy_stride * ncopy) % 4) {
      SPECTRE_CUDA_OK(cudaMemsetAsync(sums, 0, copy_stride * ncopy * sizeof(float), st));
      cfg.numAttrs = 0;
    } else {
      SPECTRE_CUDA_OK(launch_after(pool_clear_kernel, (unsigned)((n4 + 255) / 256), 256, 0, st, reinterpret_cast<float4*>(sums), n4));
    }
  }
  // Whole 16-byte pieces of `warm` per CTA into L2 on the side
  const char* w0 = reinterpret_cast<const char*>((reinterpret_cast<uintptr_t>(warm) + 15) & ~(uintptr_t)15);
  size_t wb = 0;
  if (warm && warm_bytes >= 32) wb = (warm_bytes - (size_t)(w0 - reinterpret_cast<const char*>(warm))) & ~(size_t)15;
  const size_t ctas = (size_t)groups * nslice * q->B;
  const unsigned wper = (unsigned)(wb ? ((wb + ctas - 1) / ctas + 15) & ~(size_t)15 : 0);
  SPECTRE_IO_DISPATCH(q->dtype, {
    if (ring)
      SPECTRE_CUDA_OK(launch_kernel(&cfg, pool_kernel<T, true>, reinterpret_cast<const T*>(q->ptr), (int64_t)q->stride_b,
                                         (int64_t)q->stride_l, (int64_t)q->stride_h, (int)q->L, (int)q->H, (int)q->D, rows_per,
                                         ncopy, copy_stride, sums, reinterpret_cast<T*>(ring), N, w0, wper, wb));
    else
      SPECTRE_CUDA_OK(launch_kernel(&cfg, pool_kernel<T, false>, reinterpret_cast<const T*>(q->ptr), (int64_t)q->stride_b,
                                         (int64_t)q->stride_l, (int64_t)q->stride_h, (int)q->L, (int)q->H, (int)q->D, rows_per,
                                         ncopy, copy_stride, sums, static_cast<T*>(nullptr), 0, w0, wper, wb));
  });
  SPECTRE_LAUNCH_OK("pool_kernel");
  return SPECTRE_OK;
}

int pool_sum(const spectre_ctx* ctx, cudaStream_t st, const spectre_act* q, float* sums, int ncopy_max, int* ncopy_used,
             const void* warm, size_t warm_bytes) {
  return pool_launch(ctx, st, q, sums, ncopy_max, ncopy_used, nullptr, 0, warm, warm_bytes);
}

// Prefill of the cache's query side in one pass over q: sum over the sequence into sums[B,H,D] and the ring copy.
int pool_sum_ring(const spectre_ctx* ctx, cudaStream_t st, const spectre_act* q, float* sums, void* ring, int N) {
  int used = 1;
  return pool_launch(ctx, st, q, sums, 1, &used, ring, N, nullptr, 0);
}

__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// ---- MLP ---------------------------------------------------------------------
template <typename WT> __device__ __forceinline__ float wload(const WT* p);
template <> __device__ __forceinline__ float wload<float>(const float* p) { return *p; }
template <> __device__ __forceinline__ float wload<bf16>(const bf16* p) {
  return __uint_as_float((uint32_t)*reinterpret_cast<const unsigned short*>(p) << 16);
}

// q_bar = LN(inv_count * sum) into shared memory (Sec. 3.2 step 3a), then the hidden layer
// u = GELU(q_bar W1 + b1), for nb <= NB batch entries of one head at once: the means are spread over
// the CTA, a warp normalises one entry, then a thread takes one hidden unit for every g-th batch
// entry (g = threads / hidden groups), so a weight column is fetched once per group, not per entry.
// sums points at the first entry's [D] row, bstride is the distance between batch entries;
// u is written as [hidden][ustride] (batch entry fastest).
// STAGED: W1, gamma, beta and b1 point at copies in shared memory, requested ahead of the sums (ahead of the wait for them
// where the weights may be read then), so the hidden layer adds no memory round trip behind the sums.
template <typename WT> __device__ __forceinline__ float wvalue(WT x);
template <> __device__ __forceinline__ float wvalue<float>(float x) { return x; }
template <> __device__ __forceinline__ float wvalue<bf16>(bf16 x) { return __bfloat162float(x); }
template <typename WT, bool STAGED> __device__ __forceinline__ float wget(const WT* p) {
  if constexpr (STAGED) return wvalue<WT>(*p);
  else return wload<WT>(p);
}

// The means of a decode step, with its token in them; every load of a round in flight together
template <typename T>
__device__ __forceinline__ void token_means(const GateToken& t, int b0, int h, int H, const float* sums, int nb, float inv_count, int D, float* qbar) {
  const T *q = static_cast<const T*>(t.q) + ((size_t)b0 * H + h) * D, *o = static_cast<const T*>(t.old) + (size_t)b0 * t.old_stride + (size_t)h * D;
#pragma unroll 1
  for (int e0 = threadIdx.x; e0 < nb * D; e0 += 2 * blockDim.x) {
    float s[2];
    T a[2], b[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int e = min(e0 + u * (int)blockDim.x, nb * D - 1), bb = e / D, c = e - bb * D;
      const size_t at = (size_t)bb * H * D + c;
      s[u] = sums[at];
      a[u] = q[at];
      b[u] = t.old ? o[(size_t)bb * t.old_stride + c] : T(0.f);
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int e = e0 + u * (int)blockDim.x;
      if (e < nb * D) qbar[e] = (s[u] + ((float)a[u] - (float)b[u])) * inv_count;
    }
  }
}
__device__ __forceinline__ void token_means(const GateToken& t, int b0, int h, int H, const float* sums, int nb, float inv_count, int D, float* qbar) {
  if (t.dtype == SPECTRE_F32) token_means<float>(t, b0, h, H, sums, nb, inv_count, D, qbar);
  else if (t.dtype == SPECTRE_BF16) token_means<bf16>(t, b0, h, H, sums, nb, inv_count, D, qbar);
  else token_means<f16>(t, b0, h, H, sums, nb, inv_count, D, qbar);
}

// Activations in front of a gate kernel's shared memory: hidden [hidden][entries], then q_bar [entries][D].  The hidden layer of several entries
// reads q_bar 16 bytes at a time: 4 and 8 end there by themselves, two of an odd width 8 bytes off.  Only these are rounded up: with the
// rounding, one entry's kernel spilled 112 bytes (decode step of 1 x 12 x 4096, fp32 weights 13.9 -> 16.4 us).
__host__ __device__ __forceinline__ int qbar_at(int entries, int hidden) { return entries == 2 ? (2 * hidden + 3) & ~3 : entries * hidden; }
__host__ __device__ __forceinline__ int act_floats(int entries, int hidden, int D) { return (qbar_at(entries, hidden) + entries * D + 3) & ~3; }

// one hidden unit's sums over D inputs for N entries (rows of q; absent ones hold whatever is there, never used), two inputs per packed sum; ALIGNED: the rows
// start on 16 bytes, one load takes four inputs
template <typename WT, int N, bool ALIGNED>
__device__ __forceinline__ void hidden_unit(const WT* w, int hidden, int D, const float* q, float (&acc)[N]) {
  uint64_t a2[N];
#pragma unroll
  for (int s = 0; s < N; ++s) a2[s] = pk2(acc[s], 0.f);
  auto block = [&](auto size, int c) {
    constexpr int kLoads = decltype(size)::value;
    float wv[kLoads];
#pragma unroll
    for (int i = 0; i < kLoads; ++i) wv[i] = wload<WT>(w + (size_t)(c + i) * hidden);
#pragma unroll
    for (int i = 0; i < kLoads; i += 4) {
      const uint64_t w01 = pk2(wv[i], wv[i + 1]), w23 = pk2(wv[i + 2], wv[i + 3]);
#pragma unroll
      for (int s = 0; s < N; ++s) {
        const float* p = q + s * D + c + i;
        ulonglong2 t;
        if constexpr (ALIGNED) t = *reinterpret_cast<const ulonglong2*>(p);
        else t = make_ulonglong2(pk2(p[0], p[1]), pk2(p[2], p[3]));
        a2[s] = fma2(t.x, w01, a2[s]);
        a2[s] = fma2(t.y, w23, a2[s]);
      }
    }
  };
  int c = 0;
#pragma unroll 1
  for (; c + 32 <= D; c += 32) block(std::integral_constant<int, 32>(), c);
#pragma unroll 1
  for (; c + 4 <= D; c += 4) block(std::integral_constant<int, 4>(), c);
#pragma unroll
  for (int s = 0; s < N; ++s) {
    float lo, hi;
    upk2(a2[s], lo, hi);
    acc[s] = lo + hi;
  }
#pragma unroll 1
  for (; c < D; ++c) {
    const float wv = wload<WT>(w + (size_t)c * hidden);
#pragma unroll
    for (int s = 0; s < N; ++s) acc[s] = fmaf(q[s * D + c], wv, acc[s]);
  }
}

// TOK: the sums may be a decode step's
// DEEP: several entries, W1 from L2, D >= 32.  SHORT: blocks may have few threads
template <typename WT, int NB, bool STAGED, bool TOK = true, bool DEEP = false, bool SHORT = false>
__device__ __forceinline__ void descriptor_and_hidden(const GateToken& tok, int b0, int h, int H, const float* sums, size_t bstride, int nb, int ncopy,
                                                      size_t copy_stride, float inv_count, int D, int hidden,
                                                      const float* gamma, const float* beta,
                                                      float eps, const WT* W1, const float* b1,
                                                      float* qbar, float* u, int ustride) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
  if (TOK && tok.q) {                                        // a decode step: one copy, and the token
    token_means(tok, b0, h, H, sums, nb, inv_count, D, qbar);
  } else if (NB > 1 && ncopy == 1) {                         // means, one copy: up to 4 channels per thread in flight
    for (int e0 = threadIdx.x; e0 < nb * D; e0 += 4 * blockDim.x) {
      float v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = e0 + u * (int)blockDim.x, bb = e / D, c = e - bb * D;
        v[u] = e < nb * D ? sums[(size_t)bb * bstride + c] : 0.f;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = e0 + u * (int)blockDim.x;
        if (e < nb * D) qbar[e] = v[u] * inv_count;
      }
    }
  } else if (SHORT && NB == 8 && 2 * nb * D > 5 * (int)blockDim.x) {
    // means, up to 8 copies, more than two channels per thread: four in flight, every load of a round (layers of 8 x 100 x 12 heads fp32 17.9 -> 17.2 us,
    // 64 x 64 x 12 bf16 28.5 -> 27.5; with two channels a thread, 16 x 400 x 8, or 4 entries, 4 x 400 x 8, it loses 2 %)
#pragma unroll 1
    for (int e0 = threadIdx.x; e0 < nb * D; e0 += 4 * blockDim.x) {
      float v[4][8];
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const int e = e0 + x * (int)blockDim.x, bb = e / D, c = e - bb * D;
        const float* sb = sums + (size_t)bb * bstride + c;
#pragma unroll
        for (int k = 0; k < 8; ++k) v[x][k] = e < nb * D && k < ncopy ? sb[(size_t)k * copy_stride] : 0.f;
      }
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const int e = e0 + x * (int)blockDim.x;
        float m = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) m += v[x][k];
        if (e < nb * D) qbar[e] = m * inv_count;
      }
    }
  } else {
    for (int e = threadIdx.x; e < nb * D; e += blockDim.x) {   // means: the whole CTA, one channel per thread
      const int bb = e / D, c = e - bb * D;
      const float* sb = sums + (size_t)bb * bstride + c;
      float m = 0.f;
      for (int k0 = 0; k0 < ncopy; k0 += 8) {                   // eight copies in flight at once
        float v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = (k0 + k < ncopy) ? sb[(size_t)(k0 + k) * copy_stride] : 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) m += v[k];
      }
      qbar[e] = m * inv_count;
    }
  }
  if (STAGED) asm volatile("cp.async.wait_all;" ::: "memory");   // this thread's copies of the weights; the barrier makes them the CTA's
  __syncthreads();
  const int lw = NB > 1 && nb > nw ? 16 : 32, per = 32 / lw;   // statistics: a warp per batch entry, half a one where warps are fewer
  const int sl = lane & (lw - 1);
  for (int b0 = 0; b0 < nb; b0 += per * nw) {                  // every lane takes part in the shuffles
    const int bb = b0 + per * warp + lane / lw;
    float* qb = qbar + (bb < nb ? bb : 0) * D;
    float part = 0.f;
    for (int c = sl; c < D; c += lw) part += qb[c];
    for (int o = lw / 2; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    const float mean = part / (float)D;
    part = 0.f;
    for (int c = sl; c < D; c += lw) {
      float dlt = qb[c] - mean;
      part += dlt * dlt;
    }
    for (int o = lw / 2; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    const float rstd = 1.0f / sqrtf(part / (float)D + eps);
    if (bb < nb)
      for (int c = sl; c < D; c += lw) qb[c] = gamma[c] * (qb[c] - mean) * rstd + beta[c];
  }
  __syncthreads();
  if constexpr (NB == 1) {
    for (int jj = threadIdx.x; jj < hidden; jj += blockDim.x) {
      float acc = b1[jj];
      int c = 0;
      for (; c + 32 <= D; c += 32) {                // 32 independent loads in flight
        float wv[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) wv[i] = wget<WT, STAGED>(W1 + (size_t)(c + i) * hidden + jj);
#pragma unroll
        for (int i = 0; i < 32; ++i) acc = fmaf(qbar[c + i], wv[i], acc);
      }
      for (; c < D; ++c) acc = fmaf(qbar[c], wget<WT, STAGED>(W1 + (size_t)c * hidden + jj), acc);
      u[jj * ustride] = gelu_erf(acc);
    }
    __syncthreads();
    return;
  }
  if constexpr (DEEP) {
    // 32 loads of W1 in flight, each for all entries (gate of 2 x 4 x 32768, 256 hidden units, fp32 weights 40.2 -> 29.5 us,
    // 64 x 12 x 196 18.9 -> 16.8, against the loop below)
    for (int jj = threadIdx.x; jj < hidden; jj += blockDim.x) {
      float acc[NB];
#pragma unroll
      for (int s = 0; s < NB; ++s) acc[s] = b1[jj];
      if (D % 4 == 0) hidden_unit<WT, NB, true>(W1 + jj, hidden, D, qbar, acc);
      else hidden_unit<WT, NB, false>(W1 + jj, hidden, D, qbar, acc);
#pragma unroll
      for (int s = 0; s < NB; ++s)
        if (s < nb) u[jj * ustride + s] = gelu_erf(acc[s]);
    }
    __syncthreads();
    return;
  }
  // A thread takes one hidden unit of up to 4 entries, in loops of few instructions: they run once per launch, and straight-line code waits
  // for itself (layer of 16 x 1024 x 12 heads fp32 58.4 -> 57.0 us).
  constexpr int kE = NB < 4 ? NB : 4;
  for (int item = threadIdx.x; item < hidden * ((nb + kE - 1) / kE); item += blockDim.x) {
    const int e0 = item / hidden * kE, jj = item - item / hidden * hidden;
    const WT* w = W1 + jj;
    const float* q = qbar + e0 * D;                 // entries beyond nb: whatever is there, never used
    float acc[kE];
#pragma unroll
    for (int s = 0; s < kE; ++s) acc[s] = b1[jj];
    int c = 0;
    if (D % 4 == 0) {                               // rows of q_bar start on 16 bytes: four inputs per broadcast, two per packed sum
      uint64_t a2[kE];
#pragma unroll
      for (int s = 0; s < kE; ++s) a2[s] = pk2(acc[s], 0.f);
#pragma unroll 2
      for (; c < D; c += 4) {
        float wv[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) wv[i] = wget<WT, STAGED>(w + (size_t)(c + i) * hidden);
        const uint64_t w01 = pk2(wv[0], wv[1]), w23 = pk2(wv[2], wv[3]);
#pragma unroll
        for (int s = 0; s < kE; ++s) {
          const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(q + s * D + c);
          a2[s] = fma2(t.x, w01, a2[s]);
          a2[s] = fma2(t.y, w23, a2[s]);
        }
      }
#pragma unroll
      for (int s = 0; s < kE; ++s) {
        float lo, hi;
        upk2(a2[s], lo, hi);
        acc[s] = lo + hi;
      }
    }
#pragma unroll 1
    for (; c < D; ++c) {
      const float wv = wget<WT, STAGED>(w + (size_t)c * hidden);
#pragma unroll
      for (int s = 0; s < kE; ++s) acc[s] = fmaf(q[s * D + c], wv, acc[s]);
    }
#pragma unroll
    for (int s = 0; s < kE; ++s)
      if (e0 + s < nb) u[jj * ustride + e0 + s] = gelu_erf(acc[s]);   // [hidden][ustride]: one row = all batch entries
  }
  __syncthreads();
}

// 16-byte asynchronous copies into shared memory; the caller waits
__device__ __forceinline__ void copy_async16(const void* src, void* dst, int bytes) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  for (int i = 16 * (int)threadIdx.x; i < bytes; i += 16 * (int)blockDim.x)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(d + i), "l"(reinterpret_cast<const char*>(src) + i) : "memory");
}
__device__ __forceinline__ void stage_vectors(const float* gamma, const float* beta, const float* b1, int D, int hidden, float* vec) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(vec);
  for (int i = threadIdx.x; i < 2 * D + hidden; i += blockDim.x) {
    const float* src = i < D ? gamma + i : (i < 2 * D ? beta + (i - D) : b1 + (i - 2 * D));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" :: "r"(d + 4 * i), "l"(src) : "memory");
  }
}
// A head's W1, LayerNorm weights and hidden bias into shared memory: W1, then gamma, beta, b1.  Asynchronous, so that what the
// caller asks for next - the sums, where the wait came first - is on its way beside them (prompt of 1 x 1500 of 2048 x 4 heads, fp32:
// 60.8 -> 60.0 us against loads and stores, 1 x 6000 of 8192 x 16, fp16: 103.2 -> 101.6); descriptor_and_hidden waits for them.
template <typename WT>
__device__ __forceinline__ void stage_mlp(const WT* W1, const float* gamma, const float* beta, const float* b1, int D, int hidden, WT* w1s) {
  copy_async16(W1, w1s, D * hidden * (int)sizeof(WT));
  stage_vectors(gamma, beta, b1, D, hidden, reinterpret_cast<float*>(w1s + D * hidden));
}

// modReLU: max(|z| + b, 0) z / |z| = max(1 + b / |z|, 0) z   (0 at z = 0)
__device__ __forceinline__ float2 modrelu(float2 gk, float bias) {
  const float m2 = fmaf(gk.x, gk.x, gk.y * gk.y);
  const float sc = m2 > 0.f ? fmaxf(fmaf(bias, rsqrtf(m2), 1.0f), 0.f) : 0.f;
  return cscale(gk, sc);
}
// positional phase exp(+j 2 pi k p / n), angle reduced in integers
// pm = shift mod n in [0, n)
__device__ __forceinline__ float2 phase_reduced(int k, int n, unsigned pm) {
  if (pm == 0u) return make_float2(1.f, 0.f);
  // a power of two: the product's low bits are the remainder, and wrap-around does not touch them
  const unsigned kp = (n & (n - 1)) == 0 ? ((unsigned)k * pm) & (unsigned)(n - 1)
                                         : (unsigned)(((unsigned long long)k * (unsigned long long)pm) % (unsigned)n);
  const float2 w = twiddle_fwd(kp, (unsigned)n);  // exp(-j ...)
  return make_float2(w.x, -w.y);
}
__device__ __forceinline__ float2 phase_factor(int k, int n, long long shift) {
  long long pm = shift % n;
  if (pm < 0) pm += n;
  return phase_reduced(k, n, (unsigned)pm);
}
__device__ __forceinline__ float2 modrelu_phase(float2 gk, float bias, int k, int n, unsigned pm) {
  gk = modrelu(gk, bias);
  if (pm != 0u) gk = cmul(gk, phase_factor(k, n, (long long)pm));
  return gk;
}

struct GateMlpParams {
  const float* sums;      // [ncopy][B,H,D]
  int ncopy; size_t copy_stride;
  float inv_count;
  int B, H, D, hidden, n, K;
  size_t hs_ln, hs_w1, hs_b1, hs_w2, hs_b2, hs_mb;   // per-head strides (0 when shared)
  const float* gamma; const float* beta; float eps;
  const void* W1; const float* b1; const void* W2; const float* b2;
  const float* modrelu_bias;
  const long long* shift; long long shift_all;
  unsigned pm_all;        // shift_all mod n in [0, n), reduced on the host
  float2* g_out;          // final gate, or the raw MLP output when post != 0
  float* qbar_out;
  float* u_ws;            // [B,H,hidden] hidden activations (workspace)
  int post;               // 1: Toeplitz follows, skip modReLU/phase here
  int stage_w1;           // W1, gamma, beta and b1 of a head are copied to shared memory before the wait (size and alignment allow)
  GateToken tok;
  int early;              // the kernel in front is of the same call and has waited for the caller's work: the weights, which the caller's
                          // last kernel may have written, are read ahead of the wait.  Otherwise the wait comes first
};
// In front of the trigger: what triggers before it has waited lets its dependents start beside the caller's kernel too
template <bool TRIGGER = true, bool TOK = true>
__device__ __forceinline__ void gate_start(const GateMlpParams& p) {
  if (!p.early) after_previous();
  if (TRIGGER) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (TOK)
    for (int i = (blockIdx.y * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x; i < p.tok.nclear; i += gridDim.x * gridDim.y * blockDim.x)
      p.tok.clear[i] = 0;
}

// raw (re, im) weight pair of one bin in one hidden row
template <typename WT> struct wraw;
template <> struct wraw<bf16> {
  typedef unsigned type;
  static __device__ __forceinline__ type load(const bf16* p) { return *reinterpret_cast<const unsigned*>(p); }
  static __device__ __forceinline__ float2 cvt(type r) { return make_float2(__uint_as_float(r << 16), __uint_as_float(r & 0xffff0000u)); }
  static constexpr int kRows = 32;
};
template <> struct wraw<float> {
  typedef float2 type;
  static __device__ __forceinline__ type load(const float* p) { return *reinterpret_cast<const float2*>(p); }
  static __device__ __forceinline__ float2 cvt(type r) { return r; }
  static constexpr int kRows = 16;
};

// Output layer: grid (ceil(K / threads), H * ceil(B / BB)), one bin per thread for BB batch
// entries of one head: W2 is shared by the batch, so a column fetched once serves all of them.
// A thread issues the loads of kRows hidden rows of its W2 column before it uses any of them
// (32 rows in bf16: two round trips for the usual 64-wide hidden layer) and needs few enough
// registers for four CTAs per SM, so that the grid of an 8k-token transform is resident at once;
// the kernel is a pure stream over W2.
// Hidden activations of BB batch entries of one head, once: grid H * ceil(B / BB).  With the 48 registers of the compiler's own choice few of its loads were in
// flight (gate of 8 x 8 x 32768 fp32 19.7 -> 18.5 us).
template <typename WT, int BB, bool DEEP>
__global__ void __launch_bounds__(256, 2) gate_hidden_kernel(const GateMlpParams p) {
  extern __shared__ __align__(16) float u[];       // [hidden][BB], then q_bar [BB][D]
  const int nbg = (p.B + BB - 1) / BB;
  const int h = blockIdx.x / nbg, b0 = (blockIdx.x - h * nbg) * BB;
  const int nb = min(BB, p.B - b0);
  gate_start(p);
  float* qbar = u + qbar_at(BB, p.hidden);
  const WT* W1 = reinterpret_cast<const WT*>(p.W1) + h * p.hs_w1;
  WT* w1s = reinterpret_cast<WT*>(u + act_floats(BB, p.hidden, p.D));
  const float* vec = reinterpret_cast<const float*>(w1s + p.D * p.hidden);
  if (p.stage_w1) stage_mlp(W1, p.gamma + h * p.hs_ln, p.beta + h * p.hs_ln, p.b1 + h * p.hs_b1, p.D, p.hidden, w1s);
  asm volatile("griddepcontrol.wait;" ::: "memory");        // the sums come from the kernel before
  if constexpr (DEEP)
    descriptor_and_hidden<WT, BB, false, true, true>(p.tok, b0, h, p.H, p.sums + ((size_t)b0 * p.H + h) * p.D, (size_t)p.H * p.D, nb, p.ncopy, p.copy_stride,
                                                     p.inv_count, p.D, p.hidden, p.gamma + h * p.hs_ln, p.beta + h * p.hs_ln, p.eps, W1,
                                                     p.b1 + h * p.hs_b1, qbar, u, BB);
  else if (p.stage_w1)
    descriptor_and_hidden<WT, BB, true>(p.tok, b0, h, p.H, p.sums + ((size_t)b0 * p.H + h) * p.D, (size_t)p.H * p.D, nb, p.ncopy, p.copy_stride,
                                        p.inv_count, p.D, p.hidden, vec, vec + p.D, p.eps, w1s, vec + 2 * p.D, qbar, u, BB);
  else
    descriptor_and_hidden<WT, BB, false>(p.tok, b0, h, p.H, p.sums + ((size_t)b0 * p.H + h) * p.D, (size_t)p.H * p.D, nb, p.ncopy, p.copy_stride,
                                         p.inv_count, p.D, p.hidden, p.gamma + h * p.hs_ln, p.beta + h * p.hs_ln, p.eps, W1,
                                         p.b1 + h * p.hs_b1, qbar, u, BB);
  for (int e = threadIdx.x; e < nb * p.hidden; e += blockDim.x) {
    const int bb = e / p.hidden, jj = e - bb * p.hidden;
    p.u_ws[((size_t)(b0 + bb) * p.H + h) * p.hidden + jj] = u[jj * BB + bb];
  }
  if (p.qbar_out)
    for (int e = threadIdx.x; e < nb * p.D; e += blockDim.x) {
      const int bb = e / p.D, c = e - bb * p.D;
      p.qbar_out[((size_t)(b0 + bb) * p.H + h) * p.D + c] = qbar[e];
    }
}

// ---- the output layer's stream over W2: blocks of rows of one column (bin) per thread ----
// rows j .. j + N - 1 (all present when FULL) held in wc[o .. o + N - 1], added to the sums of BB batch entries
template <typename WT, int BB, bool FULL, int N>
__device__ __forceinline__ void gate_use_rows(const typename wraw<WT>::type (&wc)[wraw<WT>::kRows], int o, int j, int hidden,
                                              const float* __restrict__ u, float2 (&acc)[BB],
                                              uint64_t (&ax)[BB >= 4 ? BB / 2 : 1], uint64_t (&ay)[BB >= 4 ? BB / 2 : 1]) {
  const int nr = FULL ? N : min(N, hidden - j);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    if (FULL || i < nr) {
      const float2 wv = wraw<WT>::cvt(wc[o + i]);
      const float* ur = u + (j + i) * BB;                 // entries of absent batch rows hold stale values, never stored
      if (BB >= 4) {
        const uint64_t wx = pk2(wv.x, wv.x), wy = pk2(wv.y, wv.y);
#pragma unroll
        for (int v = 0; v < BB / 4; ++v) {
          const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(ur + 4 * v);   // entries 4v .. 4v + 3
          ax[2 * v] = fma2(t.x, wx, ax[2 * v]);         ay[2 * v] = fma2(t.x, wy, ay[2 * v]);
          ax[2 * v + 1] = fma2(t.y, wx, ax[2 * v + 1]); ay[2 * v + 1] = fma2(t.y, wy, ay[2 * v + 1]);
        }
      } else {
#pragma unroll
        for (int bb = 0; bb < BB; ++bb) {
          acc[bb].x = fmaf(ur[bb], wv.x, acc[bb].x);
          acc[bb].y = fmaf(ur[bb], wv.y, acc[bb].y);
        }
      }
    }
  }
}
template <typename WT, bool FULL, int N>
__device__ __forceinline__ void gate_fetch_rows(typename wraw<WT>::type (&wc)[wraw<WT>::kRows], int o, const WT* col,
                                                size_t ld, int j, int hidden) {
  const int nr = FULL ? N : min(N, hidden - j);
#pragma unroll
  for (int i = 0; i < N; ++i)
    if (FULL || i < nr) wc[o + i] = wraw<WT>::load(col + (size_t)(j + i) * ld);
}
// w holds rows 0 .. R - 1 on entry.  One batch entry per pass: a block of R rows is requested when the
// one before it has been used.  Several entries per pass (a thread then spends long enough on a row for
// the latency of a whole block to show): the two halves of w alternate, each refilled with the rows R
// further on as soon as it has been used, so R / 2 to R rows are in flight throughout.
template <typename WT, int BB, bool FULL>
__device__ __forceinline__ void gate_stream(typename wraw<WT>::type (&w)[wraw<WT>::kRows], const WT* col, size_t ld,
                                            int hidden, const float* __restrict__ u, float2 (&acc)[BB],
                                            uint64_t (&ax)[BB >= 4 ? BB / 2 : 1], uint64_t (&ay)[BB >= 4 ? BB / 2 : 1]) {
  constexpr int R = wraw<WT>::kRows, Hf = R / 2;
  if (BB >= 4) {
    for (int j = 0; j < hidden; j += R) {
      gate_use_rows<WT, BB, FULL, Hf>(w, 0, j, hidden, u, acc, ax, ay);
      if (j + R < hidden) gate_fetch_rows<WT, FULL, Hf>(w, 0, col, ld, j + R, hidden);
      if (j + Hf < hidden) gate_use_rows<WT, BB, FULL, Hf>(w, Hf, j + Hf, hidden, u, acc, ax, ay);
      if (j + R + Hf < hidden) gate_fetch_rows<WT, FULL, Hf>(w, Hf, col, ld, j + R + Hf, hidden);
    }
  } else {
    for (int j = 0; j < hidden; j += R) {
      if (j > 0) gate_fetch_rows<WT, FULL, R>(w, 0, col, ld, j, hidden);
      gate_use_rows<WT, BB, FULL, R>(w, 0, j, hidden, u, acc, ax, ay);
    }
  }
}

// PRE: the hidden activations were computed once per (head, batch entry) by gate_hidden_kernel
// (long transforms: hundreds of CTAs per head would otherwise repeat that work).
// TOK: for a decode step; without its loads the other calls' form spills nothing (28 bytes cost the layer of 8192 points 1.3 us of 63.2).
template <typename WT, int BB, bool PRE, bool TOK, bool DEEP>
__global__ void __launch_bounds__(256, BB == 1 ? 4 : 2) gate_out_kernel(const GateMlpParams p) {
  extern __shared__ __align__(16) float u[];       // [hidden][BB], then q_bar [BB][D]
  gate_start(p);                                   // a kernel launched behind this one as a programmatic dependent may do its set-up meanwhile
  constexpr int R = wraw<WT>::kRows;
  const int nbg = (p.B + BB - 1) / BB;
  const int h = blockIdx.y / nbg, b0 = (blockIdx.y - h * nbg) * BB;
  const int nb = min(BB, p.B - b0);
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  const bool live = k < p.K;
  const WT* col = reinterpret_cast<const WT*>(p.W2) + h * p.hs_w2 + 2 * (size_t)(live ? k : 0);
  const size_t ld = 2 * (size_t)p.K;
  WT* w1s = reinterpret_cast<WT*>(u + act_floats(BB, p.hidden, p.D));
  const float* vec = reinterpret_cast<const float*>(w1s + p.D * p.hidden);
  typename wraw<WT>::type w[R];
  const int n0 = min(R, p.hidden);
  if (live) {
#pragma unroll
    for (int i = 0; i < R; ++i)
      if (i < n0) w[i] = wraw<WT>::load(col + (size_t)i * ld);
  }
  const int kc = live ? k : 0;
  const float2 b2 = make_float2(p.b2[h * p.hs_b2 + 2 * kc], p.b2[h * p.hs_b2 + 2 * kc + 1]);
  const float bias = (!p.post && p.modrelu_bias) ? p.modrelu_bias[h * p.hs_mb + kc] : 0.f;
  if (!PRE && p.stage_w1)
    stage_mlp(reinterpret_cast<const WT*>(p.W1) + h * p.hs_w1, p.gamma + h * p.hs_ln, p.beta + h * p.hs_ln, p.b1 + h * p.hs_b1, p.D,
              p.hidden, w1s);
  // everything above reads only weights; the sums / hidden activations come from the kernel before
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (PRE) {
    for (int e = threadIdx.x; e < nb * p.hidden; e += blockDim.x) {
      const int bb = e / p.hidden, jj = e - bb * p.hidden;
      u[jj * BB + bb] = p.u_ws[((size_t)(b0 + bb) * p.H + h) * p.hidden + jj];
    }
    __syncthreads();
  } else {
    // LayerNorm + hidden layer, repeated by every CTA of the head (a few thousand FLOPs per batch
    // entry, two short round trips) while this thread's W2 column is already on its way
    float* qbar = u + qbar_at(BB, p.hidden);   // [BB][D]
    const WT* W1 = reinterpret_cast<const WT*>(p.W1) + h * p.hs_w1;
    if constexpr (DEEP)
      descriptor_and_hidden<WT, BB, false, TOK, true>(p.tok, b0, h, p.H, p.sums + ((size_t)b0 * p.H + h) * p.D, (size_t)p.H * p.D, nb, p.ncopy, p.copy_stride,
                                                      p.inv_count, p.D, p.hidden, p.gamma + h * p.hs_ln, p.beta + h * p.hs_ln, p.eps, W1,
                                                      p.b1 + h * p.hs_b1, qbar, u, BB);
    else if (p.stage_w1)
      descriptor_and_hidden<WT, BB, true, TOK>(p.tok, b0, h, p.H, p.sums + ((size_t)b0 * p.H + h) * p.D, (size_t)p.H * p.D, nb, p.ncopy, p.copy_stride,
                                          p.inv_count, p.D, p.hidden, vec, vec + p.D, p.eps, w1s, vec + 2 * p.D, qbar, u, BB);
    else
      descriptor_and_hidden<WT, BB, false, TOK>(p.tok, b0, h, p.H, p.sums + ((size_t)b0 * p.H + h) * p.D, (size_t)p.H * p.D, nb, p.ncopy, p.copy_stride,
                                           p.inv_count, p.D, p.hidden, p.gamma + h * p.hs_ln, p.beta + h * p.hs_ln, p.eps, W1,
                                           p.b1 + h * p.hs_b1, qbar, u, BB);
    if (p.qbar_out && blockIdx.x == 0)
      for (int e = threadIdx.x; e < nb * p.D; e += blockDim.x) {
        const int bb = e / p.D, c = e - bb * p.D;
        p.qbar_out[((size_t)(b0 + bb) * p.H + h) * p.D + c] = qbar[e];
      }
  }
  if (!live) return;
  float2 acc[BB];
#pragma unroll
  for (int bb = 0; bb < BB; ++bb) acc[bb] = b2;
  // BB >= 4: the sums of two batch entries share a packed fp32 pair (one instruction per pair and
  // component; each half rounds like a scalar fmaf, so the results do not change)
  constexpr int NP = BB >= 4 ? BB / 2 : 1;
  uint64_t ax[NP], ay[NP];
#pragma unroll
  for (int pp = 0; pp < NP; ++pp) { ax[pp] = pk2(acc[0].x, acc[0].x); ay[pp] = pk2(acc[0].y, acc[0].y); }
  if (p.hidden % R == 0) gate_stream<WT, BB, true>(w, col, ld, p.hidden, u, acc, ax, ay);
  else gate_stream<WT, BB, false>(w, col, ld, p.hidden, u, acc, ax, ay);
  if (BB >= 4) {
#pragma unroll
    for (int pp = 0; pp < NP; ++pp) {
      upk2(ax[pp], acc[2 * pp].x, acc[2 * pp + 1].x);
      upk2(ay[pp], acc[2 * pp].y, acc[2 * pp + 1].y);
    }
  }
  // one positional phase for the whole batch unless per-entry shifts are given
  float2 ph = make_float2(1.f, 0.f);
  if (!p.post && !p.shift) ph = phase_reduced(k, p.n, p.pm_all);
#pragma unroll
  for (int bb = 0; bb < BB; ++bb) {
    if (bb < nb) {
      const int b = b0 + bb;
      float2 a = acc[bb];
      if (!p.post) {
        if (p.modrelu_bias) a = modrelu(a, bias);         // without a bias modReLU is the identity (|z| z / |z| = z, exactly, in this arithmetic too)
        a = cmul(a, p.shift ? phase_factor(k, p.n, p.shift_all + p.shift[b]) : ph);
      }
      p.g_out[((size_t)b * p.H + h) * p.K + k] = a;
    }
  }
}

// ---- the whole gate of one batch entry in few CTAs ----
// kParts threads share a bin, each with kRows rows of W2: with the usual 64 hidden units every weight is requested ahead of the
// wait for the sums, where gate_out_kernel's thread takes 2 (bf16) or 4 (fp32) dependent rounds of loads.  The chain behind the wait is
// all that is left.
// TOK: for a decode step.  Calls that read W1 in place gain by a form without its loads (gate of 1 x 2 x 1024, 256 hidden units, fp32 8.6 -> 8.1 us); those
// that stage it are no faster in it (layer of 1 x 1024 x 2 heads, 64 units, 12.37 -> 12.43).
template <typename WT, bool TOK>
__global__ void __launch_bounds__(256, 4) gate_split_kernel(const GateMlpParams p) {
  constexpr int R = wraw<WT>::kRows, kParts = 64 / R, kBins = 256 / kParts;
  extern __shared__ __align__(16) float u[];       // [hidden], q_bar [D], W1, gamma, beta, b1
  __shared__ float2 part[kParts][kBins];
  gate_start<true, TOK>(p);
  const int h = blockIdx.y % p.H, b = blockIdx.y / p.H;
  const int q = threadIdx.x / kBins, t = threadIdx.x % kBins, k = blockIdx.x * kBins + t, kc = min(k, p.K - 1);
  const WT* W1 = reinterpret_cast<const WT*>(p.W1) + h * p.hs_w1;
  const WT* col = reinterpret_cast<const WT*>(p.W2) + h * p.hs_w2 + 2 * (size_t)kc;
  const size_t ld = 2 * (size_t)p.K;
  WT* w1s = reinterpret_cast<WT*>(u + act_floats(1, p.hidden, p.D));
  const float* vec = reinterpret_cast<const float*>(w1s + p.D * p.hidden);
  typename wraw<WT>::type w[R];
#pragma unroll
  for (int i = 0; i < R; ++i) w[i] = wraw<WT>::load(col + (size_t)min(q * R + i, p.hidden - 1) * ld);
  const float2 b2 = make_float2(p.b2[h * p.hs_b2 + 2 * kc], p.b2[h * p.hs_b2 + 2 * kc + 1]);
  const float bias = (!p.post && p.modrelu_bias) ? p.modrelu_bias[h * p.hs_mb + kc] : 0.f;
  if (p.stage_w1) stage_mlp(W1, p.gamma + h * p.hs_ln, p.beta + h * p.hs_ln, p.b1 + h * p.hs_b1, p.D, p.hidden, w1s);
  asm volatile("griddepcontrol.wait;" ::: "memory");         // the sums come from the kernel before
  float* qbar = u + qbar_at(1, p.hidden);
  const float* sums = p.sums + ((size_t)b * p.H + h) * p.D;
  if (p.stage_w1)
    descriptor_and_hidden<WT, 1, true, TOK>(p.tok, b, h, p.H, sums, (size_t)p.H * p.D, 1, p.ncopy, p.copy_stride, p.inv_count, p.D, p.hidden, vec, vec + p.D,
                                       p.eps, w1s, vec + 2 * p.D, qbar, u, 1);
  else
    descriptor_and_hidden<WT, 1, false, TOK>(p.tok, b, h, p.H, sums, (size_t)p.H * p.D, 1, p.ncopy, p.copy_stride, p.inv_count, p.D, p.hidden,
                                        p.gamma + h * p.hs_ln, p.beta + h * p.hs_ln, p.eps, W1, p.b1 + h * p.hs_b1, qbar, u, 1);
  if (p.qbar_out && blockIdx.x == 0)
    for (int c = threadIdx.x; c < p.D; c += blockDim.x) p.qbar_out[((size_t)b * p.H + h) * p.D + c] = qbar[c];
  float2 acc = make_float2(0.f, 0.f);
  for (int j0 = q * R; j0 < p.hidden; j0 += kParts * R) {
    if (j0 != q * R) {                                       // more than 64 hidden units
#pragma unroll
      for (int i = 0; i < R; ++i) w[i] = wraw<WT>::load(col + (size_t)min(j0 + i, p.hidden - 1) * ld);
    }
#pragma unroll
    for (int i = 0; i < R; ++i) {
      if (j0 + i < p.hidden) {
        const float2 wv = wraw<WT>::cvt(w[i]);
        const float uv = u[j0 + i];
        acc.x = fmaf(uv, wv.x, acc.x);
        acc.y = fmaf(uv, wv.y, acc.y);
      }
    }
  }
  part[q][t] = acc;
  __syncthreads();
  if (q > 0 || k >= p.K) return;
  acc = b2;
#pragma unroll
  for (int i = 0; i < kParts; ++i) acc = cadd(acc, part[i][t]);
  if (!p.post) {
    if (p.modrelu_bias) acc = modrelu(acc, bias);
    acc = cmul(acc, p.shift ? phase_factor(k, p.n, p.shift_all + p.shift[b]) : phase_reduced(k, p.n, p.pm_all));
  }
  p.g_out[((size_t)b * p.H + h) * p.K + k] = acc;
}

// ---- the whole gate of a short transform, several batch entries ----
// One CTA per head and BB entries, one bin per thread.  All of a head's weights go to shared memory (cp.async) ahead of the wait
// for the sums.  What bounds it is the chain of short phases behind that wait, and in a chain of kernels the first pass over
// their code: fetched once per SM and launch, so the loops here are rolled up (gate_out_kernel's 32 rows per thread are 600 instructions).
// FULL: with phases per entry or a decode step's token, whose code the usual call would have to step over.
template <typename WT, int BB, bool FULL>
__global__ void __launch_bounds__(256, 2) gate_short_kernel(const GateMlpParams p) {
  extern __shared__ __align__(16) float u[];       // [hidden][BB], q_bar [BB][D], W1, gamma, beta, b1, W2
  // no trigger: CTAs of the kernel behind would sit beside these and keep the one after it off the SM (layer of 256 x 196 x 12 heads
  // with refinement 144.5 us with a trigger, 135.8 without; 16 x 400 x 8 20.4, 16.8)
  gate_start<false>(p);
  const int nbg = (p.B + BB - 1) / BB;
  const int h = blockIdx.x / nbg, b0 = (blockIdx.x - h * nbg) * BB;
  const int nb = min(BB, p.B - b0), k = threadIdx.x;
  const bool live = k < p.K;
  WT* w1s = reinterpret_cast<WT*>(u + act_floats(BB, p.hidden, p.D));
  float* vec = reinterpret_cast<float*>(w1s + p.D * p.hidden);
  WT* w2s = reinterpret_cast<WT*>(vec + ((2 * p.D + p.hidden + 3) & ~3));
  copy_async16(reinterpret_cast<const WT*>(p.W1) + h * p.hs_w1, w1s, p.D * p.hidden * (int)sizeof(WT));
  copy_async16(reinterpret_cast<const WT*>(p.W2) + h * p.hs_w2, w2s, p.hidden * 2 * p.K * (int)sizeof(WT));
  stage_vectors(p.gamma + h * p.hs_ln, p.beta + h * p.hs_ln, p.b1 + h * p.hs_b1, p.D, p.hidden, vec);
  const int kc = live ? k : 0;
  const float2 b2 = make_float2(p.b2[h * p.hs_b2 + 2 * kc], p.b2[h * p.hs_b2 + 2 * kc + 1]);
  const float bias = (!p.post && p.modrelu_bias) ? p.modrelu_bias[h * p.hs_mb + kc] : 0.f;
  asm volatile("griddepcontrol.wait;" ::: "memory");         // the sums come from the kernel before
  float* qbar = u + qbar_at(BB, p.hidden);
  descriptor_and_hidden<WT, BB, true, FULL, false, true>(p.tok, b0, h, p.H, p.sums + ((size_t)b0 * p.H + h) * p.D, (size_t)p.H * p.D, nb, p.ncopy, p.copy_stride,
                                      p.inv_count, p.D, p.hidden, vec, vec + p.D, p.eps, w1s, vec + 2 * p.D, qbar, u, BB);
  if (p.qbar_out)
    for (int e = threadIdx.x; e < nb * p.D; e += blockDim.x) {
      const int bb = e / p.D, c = e - bb * p.D;
      p.qbar_out[((size_t)(b0 + bb) * p.H + h) * p.D + c] = qbar[e];
    }
  if (!live) return;
  uint64_t ax[BB / 2], ay[BB / 2];                           // two entries per packed fp32 pair
#pragma unroll
  for (int i = 0; i < BB / 2; ++i) { ax[i] = pk2(b2.x, b2.x); ay[i] = pk2(b2.y, b2.y); }
  const typename wraw<WT>::type* wk = reinterpret_cast<const typename wraw<WT>::type*>(w2s) + k;
#pragma unroll 4
  for (int j = 0; j < p.hidden; ++j) {
    const float2 wv = wraw<WT>::cvt(wk[j * p.K]);
    const uint64_t wx = pk2(wv.x, wv.x), wy = pk2(wv.y, wv.y);
#pragma unroll
    for (int v = 0; v < BB / 4; ++v) {
      const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(u + j * BB + 4 * v);   // entries 4v .. 4v + 3 (absent ones: stale, never stored)
      ax[2 * v] = fma2(t.x, wx, ax[2 * v]);         ay[2 * v] = fma2(t.x, wy, ay[2 * v]);
      ax[2 * v + 1] = fma2(t.y, wx, ax[2 * v + 1]); ay[2 * v + 1] = fma2(t.y, wy, ay[2 * v + 1]);
    }
  }
  float2 ph = make_float2(1.f, 0.f);                         // one positional phase for the whole batch unless per-entry shifts are given
  if (!p.post && !(FULL && p.shift)) ph = phase_reduced(k, p.n, p.pm_all);
#pragma unroll
  for (int bb = 0; bb < BB; ++bb) {
    if (bb < nb) {
      const int b = b0 + bb;
      float x0, x1, y0, y1;
      upk2(ax[bb / 2], x0, x1);
      upk2(ay[bb / 2], y0, y1);
      float2 a = bb & 1 ? make_float2(x1, y1) : make_float2(x0, y0);
      if (!p.post) {
        if (p.modrelu_bias) a = modrelu(a, bias);
        if (FULL && p.shift) ph = phase_factor(k, p.n, p.shift_all + p.shift[b]);
        a = cmul(a, ph);
      }
      p.g_out[((size_t)b * p.H + h) * p.K + k] = a;
    }
  }
}

// ---- output layer for several batch entries on the tensor cores ----
// o[b][col] = sum_j u[b][j] W2[j][col] for up to NB entries of one head is a [NB x hidden] x [hidden x 2K] contraction.
// With one bin per thread it took 15 instructions per weight word of 8 entries and 71 us at B = 8, H = 32, n = 32768, where
// W2 and the gate take 27.  Here: mma.m16n8k16 with the bf16 weights as they are and the fp32 activations split into three
// bf16 parts (hi + mid + lo, 24 bits), fp32 accumulation.  The 16 rows of A are, NB = 8: hi of the entries over mid, and
// lo over zeros in a second product; NB = 4: hi, mid, lo, zeros in one.
// A weight word is one (re, im) pair and W2 rows start on 4-byte boundaries only (2K values of 2 bytes, K odd), so a lane
// loads the words of its bin in rows 2q, 2q + 1, 2q + 8, 2q + 9 of every 16 (q = lane % 4), and two byte permutations make them
// the B fragments of the real and of the imaginary columns.  A warp walks a contiguous range of chunks of 16 bins (the second
// half of a line is still in L1 then), the next chunk's 32 words per lane in flight under the products of the current one.
// 71 -> 45 us; B = 2: 43 -> 37.  Bringing the words in by 4-byte asynchronous copies (61 us) or by a bulk copy per row and
// block (88 us: its producer and the barriers around it) was slower.
template <int NB> struct MmaRows { static constexpr int kSets = NB == 8 ? 2 : 1; };

__device__ __forceinline__ void split3(float x, float (&p)[3]) {
  p[0] = __bfloat162float(__float2bfloat16_rn(x));
  p[1] = __bfloat162float(__float2bfloat16_rn(x - p[0]));
  p[2] = x - p[0] - p[1];
}
// part of row `row` of A in set `set`: which entry, which part (3: zero)
template <int NB> __device__ __forceinline__ int mma_row_part(int set, int row) {
  if (NB == 8) return set == 0 ? (row >> 3) : (row < 8 ? 2 : 3);
  return row >> 2;
}

struct GateChunk {
  unsigned w[2][16];      // [group of 8 bins][row slot s]: row 16 (s / 4) + 8 (s / 2 % 2) + 2 q + s % 2
  float2 b2;              // of bin lane % 16
  float mb;
};
// A chunk's first bin: the last chunk ends at bin K - 1, so that none needs predicates (the bins it shares with the one
// before it get the same values twice).
__device__ __forceinline__ int gate_chunk_bin(int chunk, int K) { return min(16 * chunk, K - 16); }
// src: W2 of the head at row 2 q, bin i8
__device__ __forceinline__ void gate_fetch_chunk(GateChunk& x, const unsigned* src, const float2* b2, const float* mb, int K, int chunk, int lane) {
  const int k0 = gate_chunk_bin(chunk, K);
  const unsigned* r = src + k0;
  const size_t far = 7 * (size_t)K;
#pragma unroll
  for (int s = 0; s < 16; ++s) {
    x.w[0][s] = r[0];
    x.w[1][s] = r[8];
    r += (s & 1) ? far : (size_t)K;
  }
  x.b2 = b2[k0 + (lane & 15)];
  x.mb = mb ? mb[k0 + (lane & 15)] : 0.f;
}
// out: g_out of the lane's entry (i8) at bin 2 q; pm: the positional phase (per lane where entries differ)
template <int NB, bool SHIFTS>
__device__ __forceinline__ void gate_use_chunk(const GateChunk& x, const uint32_t (&A)[4][MmaRows<NB>::kSets][4], float2* out,
                                               int n, int k0, bool write, bool relu, unsigned pm, int q, int lane) {
  // the phase of bin k0 + lane % 16, handed round below (per-entry shifts: evaluated where they are used)
  float2 ph = make_float2(1.f, 0.f);
  if (!SHIFTS && pm) ph = phase_reduced(k0 + (lane & 15), n, pm);
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    float re[4] = {0.f, 0.f, 0.f, 0.f}, im[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
      const unsigned a = x.w[g][4 * ks], b = x.w[g][4 * ks + 1], c = x.w[g][4 * ks + 2], d = x.w[g][4 * ks + 3];
      const uint32_t r0 = __byte_perm(a, b, 0x5410), r1 = __byte_perm(c, d, 0x5410);
      const uint32_t m0 = __byte_perm(a, b, 0x7632), m1 = __byte_perm(c, d, 0x7632);
#pragma unroll
      for (int set = 0; set < MmaRows<NB>::kSets; ++set) {
        mma_16816(re, A[ks][set], r0, r1);
        mma_16816(im, A[ks][set], m0, m1);
      }
    }
    // C fragment: rows i8 and i8 + 8 (the entry's parts), columns = bins 8 g + 2 q + {0, 1}
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      float2 o = make_float2(re[c] + re[2 + c], im[c] + im[2 + c]);
      if (NB == 4) {                               // hi and lo here, mid 4 rows (16 lanes) further on
        o.x += __shfl_down_sync(0xffffffffu, re[c], 16);
        o.y += __shfl_down_sync(0xffffffffu, im[c], 16);
      }
      const int src = 8 * g + 2 * q + c;
      o.x += __shfl_sync(0xffffffffu, x.b2.x, src);
      o.y += __shfl_sync(0xffffffffu, x.b2.y, src);
      if (relu) o = modrelu(o, __shfl_sync(0xffffffffu, x.mb, src));
      if (SHIFTS) o = cmul(o, phase_reduced(k0 + src, n, pm));
      else if (pm) o = cmul(o, make_float2(__shfl_sync(0xffffffffu, ph.x, src), __shfl_sync(0xffffffffu, ph.y, src)));
      if (write) out[k0 + 8 * g + c] = o;
    }
  }
}

// q_bar and the hidden layer for gate_mma_kernel (64 hidden units, 256 threads, NB = 4 or 8 entries), the activations' three bf16
// parts left in As[part * NB + entry][unit] for the fragments of A.  The sums are descriptor_and_hidden's; its packed pair is
// added up after every 32 inputs, there once over all of D, so an entry's rounding differs with the route that the batch takes.  Its loops
// are rolled up: one pass over them per launch is all there is, and straight-line code of a few thousand instructions spent more
// time waiting for itself than for the data (four of thirteen cycles per instruction at 16 x 12 heads x 513 bins).  Forward and backward of
// 16 x 1024 x 12 heads 105.7 -> 98.9 us, projected layer of 4 x 4096 x 16 73.5 -> 63.5.
constexpr int kMmaPitch = 72;                      // bf16 elements between rows of As: the fragments' loads meet no bank twice
template <int NB, bool STAGED, bool TOK>
__device__ __forceinline__ void mma_hidden(const GateMlpParams& p, int b0, int h, const float* sums, int nb, const float* gamma, const float* beta,
                                           const float* b1, const bf16* W1, float* qbar, bf16* As) {
  constexpr int kSlots = NB / 4;                   // entries per thread: 4 groups of 64 threads
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, D = p.D;
  const size_t bstride = (size_t)p.H * D;
  if (TOK) token_means(p.tok, b0, h, p.H, sums, nb, p.inv_count, D, qbar);
  else
#pragma unroll 1
  for (int e0 = tid; e0 < nb * D; e0 += 512) {     // means: two channels per thread, all copies in flight at once
    const int e1 = e0 + 256, bb0 = e0 / D, bb1 = e1 / D;
    const float *s0 = sums + (size_t)bb0 * bstride + (e0 - bb0 * D), *s1 = sums + (size_t)bb1 * bstride + (e1 - bb1 * D);
    float m0 = 0.f, m1 = 0.f;
#pragma unroll 1
    for (int k0 = 0; k0 < p.ncopy; k0 += 8) {
      float v0[8], v1[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        v0[k] = k0 + k < p.ncopy ? s0[(size_t)(k0 + k) * p.copy_stride] : 0.f;
        v1[k] = k0 + k < p.ncopy && e1 < nb * D ? s1[(size_t)(k0 + k) * p.copy_stride] : 0.f;
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) { m0 += v0[k]; m1 += v1[k]; }
    }
    qbar[e0] = m0 * p.inv_count;
    if (e1 < nb * D) qbar[e1] = m1 * p.inv_count;
  }
  if (STAGED) asm volatile("cp.async.wait_all;" ::: "memory");   // this thread's copies of the weights; the barrier makes them the CTA's
  __syncthreads();
  if (warp < nb) {                                 // statistics: a warp per batch entry
    float* qb = qbar + warp * D;
    float part = 0.f;
#pragma unroll 2
    for (int c = lane; c < D; c += 32) part += qb[c];
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    const float mean = part / (float)D;
    part = 0.f;
#pragma unroll 2
    for (int c = lane; c < D; c += 32) {
      const float dlt = qb[c] - mean;
      part += dlt * dlt;
    }
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    const float rstd = 1.0f / sqrtf(part / (float)D + p.eps);
#pragma unroll 2
    for (int c = lane; c < D; c += 32) qb[c] = gamma[c] * (qb[c] - mean) * rstd + beta[c];
  }
  __syncthreads();
  const int jj = tid & 63, gi = tid >> 6;
  float acc[kSlots];
#pragma unroll
  for (int sl = 0; sl < kSlots; ++sl) acc[sl] = b1[jj];
  int c = 0;
  if (D % 4 == 0) {                                // rows of q_bar start on 16 bytes: four inputs per broadcast, two per packed sum
#pragma unroll 1
    for (; c + 32 <= D; c += 32) {
      uint64_t a2[kSlots];
#pragma unroll
      for (int sl = 0; sl < kSlots; ++sl) a2[sl] = pk2(acc[sl], 0.f);
      constexpr int kLoads = STAGED ? 4 : 32;      // from L2: all in flight at once (gate of 4 x 4 x 16384, 512 channels, 28.3 -> 26.5 us)
#pragma unroll 4
      for (int i = c; i < c + 32; i += kLoads) {
        float wv[kLoads];
#pragma unroll
        for (int x = 0; x < kLoads; ++x) wv[x] = wget<bf16, STAGED>(W1 + (i + x) * 64 + jj);
#pragma unroll
        for (int x = 0; x < kLoads; x += 4) {
          const uint64_t w01 = pk2(wv[x], wv[x + 1]), w23 = pk2(wv[x + 2], wv[x + 3]);
#pragma unroll
          for (int sl = 0; sl < kSlots; ++sl) {    // absent entries: whatever is there, never used
            const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(qbar + (gi + 4 * sl) * D + i + x);
            a2[sl] = fma2(t.x, w01, a2[sl]);
            a2[sl] = fma2(t.y, w23, a2[sl]);
          }
        }
      }
#pragma unroll
      for (int sl = 0; sl < kSlots; ++sl) {
        float lo, hi;
        upk2(a2[sl], lo, hi);
        acc[sl] = lo + hi;
      }
    }
  }
#pragma unroll 1
  for (; c < D; ++c) {
    const float wv = wget<bf16, STAGED>(W1 + c * 64 + jj);
#pragma unroll
    for (int sl = 0; sl < kSlots; ++sl) acc[sl] = fmaf(qbar[(gi + 4 * sl) * D + c], wv, acc[sl]);
  }
#pragma unroll
  for (int sl = 0; sl < kSlots; ++sl) {
    const int bb = gi + 4 * sl;
    float x[3] = {0.f, 0.f, 0.f};
    if (bb < nb) split3(gelu_erf(acc[sl]), x);
#pragma unroll
    for (int part = 0; part < 3; ++part) As[(part * NB + bb) * kMmaPitch + jj] = __float2bfloat16_rn(x[part]);
  }
  __syncthreads();
}

// SHIFTS: the entries' phases differ.  Every CTA computes the hidden layer of its head and entries itself, under the first
// chunks' loads: a kernel in front of this one for it takes longer than all of them (49 us in all against 45).
// TOK: for a decode step; its loads in the other calls' form are code to step over (projected layer of 4 x 4096 x 16 heads 63.5 -> 70.1 us).
template <int NB, bool SHIFTS, bool TOK, bool STAGED>
__global__ void __launch_bounds__(256, 2) gate_mma_kernel(const GateMlpParams p) {
  extern __shared__ __align__(16) float qbar[];    // [NB][D], then W1
  __shared__ __align__(16) bf16 As[3 * NB * kMmaPitch];
  gate_start<true, TOK>(p);
  constexpr int kSets = MmaRows<NB>::kSets;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = lane & 3, i8 = lane >> 2, nw = blockDim.x >> 5;
  const int nbg = (p.B + NB - 1) / NB;
  const int h = blockIdx.y / nbg, b0 = (blockIdx.y - h * nbg) * NB, nb = min(NB, p.B - b0);
  const unsigned* src = reinterpret_cast<const unsigned*>(reinterpret_cast<const bf16*>(p.W2) + h * p.hs_w2) + (size_t)(2 * q) * p.K + i8;
  const float2* b2 = reinterpret_cast<const float2*>(p.b2 + h * p.hs_b2);
  const float* mb = !p.post && p.modrelu_bias ? p.modrelu_bias + h * p.hs_mb : nullptr;
  bf16* w1s = reinterpret_cast<bf16*>(qbar + ((NB * p.D + 3) & ~3));
  const float* vec = reinterpret_cast<const float*>(w1s + p.D * p.hidden);
  const float *gamma = p.gamma + h * p.hs_ln, *beta = p.beta + h * p.hs_ln, *b1 = p.b1 + h * p.hs_b1;
  if constexpr (STAGED) stage_mlp(reinterpret_cast<const bf16*>(p.W1) + h * p.hs_w1, gamma, beta, b1, p.D, p.hidden, w1s);
  // a CTA's chunks are contiguous, its warps take neighbouring ones
  const int nchunk = (p.K + 15) / 16, per = (nchunk + (int)gridDim.x - 1) / (int)gridDim.x;
  const int c0 = blockIdx.x * per + warp, c1 = min(nchunk, (int)(blockIdx.x + 1) * per);
  GateChunk x;
  gate_fetch_chunk(x, src, b2, mb, p.K, min(c0, nchunk - 1), lane);
  // everything above reads only weights; the sums / hidden activations come from the kernel before
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const float* sums = p.sums + ((size_t)b0 * p.H + h) * p.D;
  if constexpr (STAGED) mma_hidden<NB, true, TOK>(p, b0, h, sums, nb, vec, vec + p.D, vec + 2 * p.D, w1s, qbar, As);
  else mma_hidden<NB, false, TOK>(p, b0, h, sums, nb, gamma, beta, b1, reinterpret_cast<const bf16*>(p.W1) + h * p.hs_w1, qbar, As);
  if (p.qbar_out && blockIdx.x == 0)
    for (int e = threadIdx.x; e < nb * p.D; e += blockDim.x) {
      const int bb = e / p.D, c = e - bb * p.D;
      p.qbar_out[((size_t)(b0 + bb) * p.H + h) * p.D + c] = qbar[e];
    }
  // A fragments: rows i8 and i8 + 8, columns 2q, 2q + 1 and + 8 of every 16 hidden units
  uint32_t A[4][kSets][4];
#pragma unroll
  for (int set = 0; set < kSets; ++set)
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int part = mma_row_part<NB>(set, i8 + 8 * r);
      const bf16* row = As + ((part < 3 ? part : 0) * NB + i8 % NB) * kMmaPitch + 2 * q;
#pragma unroll
      for (int ks = 0; ks < 4; ++ks)
#pragma unroll
        for (int c = 0; c < 2; ++c) A[ks][set][2 * c + r] = part < 3 ? *reinterpret_cast<const uint32_t*>(row + 16 * ks + 8 * c) : 0u;
    }
  const bool write = i8 < nb;
  float2* out = p.g_out + ((size_t)(b0 + (write ? i8 : 0)) * p.H + h) * p.K + 2 * q;
  unsigned pm = p.post ? 0u : p.pm_all;
  if (SHIFTS) {
    long long s = (p.shift_all + p.shift[b0 + (write ? i8 : 0)]) % p.n;
    pm = (unsigned)(s < 0 ? s + p.n : s);
  }
#pragma unroll 1
  for (int c = c0; c < c1; c += nw) {              // the next chunk's words are on their way under this one's products
    GateChunk y = x;
    if (c + nw < c1) gate_fetch_chunk(y, src, b2, mb, p.K, c + nw, lane);
    gate_use_chunk<NB, SHIFTS>(x, A, out, p.n, gate_chunk_bin(c, p.K), write, mb != nullptr, pm, q, lane);
    x = y;
  }
}

struct GatePostParams {
  const float2* g_raw; float2* g_out;
  const float* taps; size_t hs_t; int r;          // (re, im) pairs, read as single floats: the array may start at an odd one
  const float* modrelu_bias; size_t hs_mb;
  const long long* shift; long long shift_all;
  int H, K, n;
};

// Toeplitz update along the bin axis ('same' window, zero boundary, reads the
// pre-update gate), then modReLU and phase (Sec. 3.2 steps 3b-3c).
__global__ void __launch_bounds__(256) gate_post_kernel(const GatePostParams p) {
  after_previous();
  asm volatile("griddepcontrol.launch_dependents;");
  const int bh = blockIdx.y, b = bh / p.H, h = bh - b * p.H;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= p.K) return;
  const float2* g = p.g_raw + (size_t)bh * p.K;
  const float* t = p.taps + 2 * (h * p.hs_t + p.r);
  float2 acc = g[k];
  for (int m = -p.r; m <= p.r; ++m) {
    int src = k - m;
    if (src >= 0 && src < p.K) acc = cadd(acc, cmul(make_float2(t[2 * m], t[2 * m + 1]), g[src]));
  }
  long long sh = p.shift_all + (p.shift ? p.shift[b] : 0);
  long long pm = sh % p.n; if (pm < 0) pm += p.n;
  float bias = p.modrelu_bias ? p.modrelu_bias[h * p.hs_mb + k] : 0.f;
  p.g_out[(size_t)bh * p.K + k] = modrelu_phase(acc, bias, k, p.n, (unsigned)pm);
}

constexpr int kPoolCopies = 16;      // partial copies of the pooled sum in a full-size workspace

// Layout: [raw gate (Toeplitz only)] [hidden activations] [ncopy x pooled sums].  ncopy = 1 is the minimum.
static size_t gate_ws_layout(int B, int H, int D, int n_fft, int r, int hidden, int ncopy, size_t* u_off,
                             size_t* sums_off) {
  size_t raw = r > 0 ? align_up((size_t)B * H * (n_fft / 2 + 1) * sizeof(float2), 256) : 0;
  *u_off = raw;
  *sums_off = raw + align_up((size_t)B * H * hidden * sizeof(float), 256);
  return *sums_off + align_up((size_t)ncopy * B * H * D * sizeof(float), 256);
}

}  // namespace spectre

using namespace spectre;

namespace spectre {
// Smallest gate scratch (one copy of the sums, any hidden width); used by the decode step.
size_t gate_min_workspace(int B, int H, int D, int n_fft, int r) {
  size_t off, off2;
  return gate_ws_layout(B, H, D, n_fft, r, 1024, 1, &off, &off2);
}
}  // namespace spectre

extern "C" size_t spectre_gate_workspace_bytes(const spectre_ctx* ctx, int32_t B, int32_t H, int32_t D, int32_t n_fft,
                                               int32_t toeplitz_r) {
  (void)ctx;
  if (B < 1 || H < 1 || D < 1 || n_fft < 1 || toeplitz_r < 0) return 0;
  size_t off, off2;
  return gate_ws_layout(B, H, D, n_fft, toeplitz_r, 1024, kPoolCopies, &off, &off2);   // any hidden width
}

namespace spectre {
// Tensor cores for bf16 weights and 64 hidden units, the width of every workload here: the kernel's loops over the hidden units
// are written for it, and the fragments of A fill the registers then.  Narrower widths stay on the other kernels, which at 32 are
// no slower than this one would be at 64 (8 entries x 32 heads x 32768: 43.8 us against 54.0; 8 x 8 x 1024 9.7 : 9.8), but at 48 are
// (65.6 against 54.0): a form for multiples of 16 would gain there.  4 or 8 entries (5 ... 7 would need two passes over W2 with
// 4).  Under 256 bins it is the faster one while its CTAs are resident at once (two per SM): layers of 196 points, 12 heads,
// 37 entries 34.8 -> 26.7 us, 64 57.4 -> 45.8, 190 88.2 -> 83.3, of 256 points 7 x 32 heads 19.9 -> 15.5, of 128 points 24 x 4 19.6 -> 13.3; beyond that the narrower CTAs of the other kernels, more of them per SM, are (256
// entries with refinement 136.8 against 144.5).  Under 64 bins most of its warps have no chunk.  It reads a bin's two output biases as one 8-byte word: an array that
// starts at an odd float (part of a flat parameter buffer) goes to the kernels that read single floats.
// Entries per CTA: 8, or 4 (a shorter hidden layer, the weights read more often) while that makes at most a CTA per SM: layers of
// 256 points, 7 x 32 heads 15.5 -> 15.0 us, 1024 points, 9 x 8 19.7 -> 18.9; against it 64 x 12 heads of 196 points on 192 CTAs 45.8 -> 50.2.
static int mma_entries(const spectre_ctx* ctx, int B, int H, int K) {
  return B <= 4 || (long long)H * ((B + 3) / 4) * ((K + 127) / 128) <= ctx->sm_count ? 4 : 8;
}
static bool gate_on_mma(const spectre_ctx* ctx, const spectre_gate_params* gp, int B, int H, int K) {
  const int nb = mma_entries(ctx, B, H, K);
  const long long ctas = (long long)H * ((B + nb - 1) / nb);
  return gp->wdtype == SPECTRE_BF16 && gp->hidden == 64 && (K >= 256 || (K >= 64 && ctas <= 2 * ctx->sm_count)) && B >= 2 &&
         !(reinterpret_cast<uintptr_t>(gp->b2) & 7);
}
// batch entries per CTA: the weights of a head are fetched once for all of them
static int gate_entries(const spectre_ctx* ctx, const spectre_gate_params* gp, int B, int H, int K) {
  if (gate_on_mma(ctx, gp, B, H, K)) return mma_entries(ctx, B, H, K);
  return (gp->hidden > 256 || B < 2) ? 1 : (B < 4 ? 2 : (B < 8 ? 4 : 8));
}

// Everything that spectre_gate refuses, so that the decode step can ask before it changes the cache.
int gate_check(const spectre_ctx* ctx, const spectre_act* q, const float* sum_q, int B, int H, int D, float inv_count,
               const spectre_gate_params* gp, int n_fft, const float* g_out, const void* workspace, size_t workspace_bytes) {
  if (!ctx) return fail(SPECTRE_ERR_INVALID_ARG, "ctx is NULL");
  if (!gp) return fail(SPECTRE_ERR_INVALID_ARG, "gate parameters are NULL");
  if ((q != nullptr) == (sum_q != nullptr)) return fail(SPECTRE_ERR_INVALID_ARG, "give exactly one of q and sum_q");
  if (!g_out || (reinterpret_cast<uintptr_t>(g_out) & 7)) return fail(SPECTRE_ERR_INVALID_ARG, "g_out is NULL or misaligned");
  if (B < 1 || H < 1 || D < 1 || D > 1024) return fail(SPECTRE_ERR_INVALID_ARG, "B, H, D must be positive (D <= 1024)");
  if (n_fft < 1 || n_fft > (1 << 24)) return fail(SPECTRE_ERR_INVALID_ARG, "n_fft out of range");
  if (gp->hidden < 1 || gp->hidden > 1024) return fail(SPECTRE_ERR_UNSUPPORTED, "hidden width must be in 1..1024");
  if (gp->toeplitz_r < 0 || gp->toeplitz_r > 64) return fail(SPECTRE_ERR_UNSUPPORTED, "toeplitz_r must be in 0..64");
  if (gp->wdtype != SPECTRE_F32 && gp->wdtype != SPECTRE_BF16) return fail(SPECTRE_ERR_INVALID_ARG, "unknown weight dtype");
  if (!gp->ln_gamma || !gp->ln_beta || !gp->W1 || !gp->b1 || !gp->W2 || !gp->b2)
    return fail(SPECTRE_ERR_INVALID_ARG, "a gate parameter array is NULL");
  if (gp->toeplitz_r > 0 && !gp->toeplitz) return fail(SPECTRE_ERR_INVALID_ARG, "toeplitz taps are NULL");
  if (reinterpret_cast<uintptr_t>(gp->W2) & 7) return fail(SPECTRE_ERR_INVALID_ARG, "W2 not 8-byte aligned");
  if (!(gp->ln_eps >= 0.f)) return fail(SPECTRE_ERR_INVALID_ARG, "ln_eps must be >= 0");
  if (q) {
    int rc = check_act(q, "q");
    if (rc != SPECTRE_OK) return rc;
    if (q->B != B || q->H != H || q->D != D) return fail(SPECTRE_ERR_INVALID_ARG, "q shape differs from B, H, D");
  } else if (!(inv_count > 0.f)) {
    return fail(SPECTRE_ERR_INVALID_ARG, "inv_count must be positive with sum_q");
  }
  const int K = n_fft / 2 + 1, BB = gate_entries(ctx, gp, B, H, K);
  if ((long long)H * ((B + BB - 1) / BB) > 65535) return fail(SPECTRE_ERR_UNSUPPORTED, "H * ceil(B / 8) exceeds 65535");
  if (gp->toeplitz_r > 0 && (long long)B * H > 65535) return fail(SPECTRE_ERR_UNSUPPORTED, "B*H exceeds 65535");
  size_t sums_off, u_off;
  const size_t need = gate_ws_layout(B, H, D, n_fft, gp->toeplitz_r, gp->hidden, 1, &u_off, &sums_off);   // one copy is enough
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 15))
    return fail(SPECTRE_ERR_WORKSPACE, "workspace is NULL or not 16-byte aligned");
  if (workspace_bytes < need) return fail(SPECTRE_ERR_WORKSPACE, "gate workspace too small");
  return SPECTRE_OK;
}

// spectre_gate; `early`: see GateMlpParams
int gate_call(spectre_ctx* ctx, void* stream, const spectre_act* q, const float* sum_q, int B, int H, int D, float inv_count,
              const spectre_gate_params* gp, int n_fft, const int64_t* shift, int64_t shift_all, float* g_out, float* qbar_out,
              void* workspace, size_t workspace_bytes, bool early, const GateToken* tok) {
  int rc = gate_check(ctx, q, sum_q, B, H, D, inv_count, gp, n_fft, g_out, workspace, workspace_bytes);
  if (rc != SPECTRE_OK) return rc;
  if (q && !(inv_count > 0.f)) inv_count = 1.0f / (float)q->L;
  const int K = n_fft / 2 + 1;
  const int r = gp->toeplitz_r;
  size_t sums_off, u_off;
  gate_ws_layout(B, H, D, n_fft, r, gp->hidden, 1, &u_off, &sums_off);
  SPECTRE_CUDA_OK(cudaSetDevice(ctx->device));
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const float* sums = sum_q;
  int ncopy = 1;
  if (q) {
    float* pooled = reinterpret_cast<float*>(reinterpret_cast<char*>(workspace) + sums_off);
    const size_t one_copy = (size_t)B * H * D * sizeof(float);
    size_t fit = (workspace_bytes - sums_off) / one_copy;
    const size_t w2 = (size_t)(gp->shared_across_heads ? 1 : H) * gp->hidden * 2 * K * (gp->wdtype == SPECTRE_BF16 ? 2 : 4);
    // Small weights are brought into L2 by the pooling pass: the gate kernel's chain of loads is latency then (2 heads, n = 1024:
    // gate call 16.6 -> 15.4 us; 8 heads, n = 4096: 16.8 -> 16.2).  Larger ones take the pass's own bandwidth for no gain
    // (8k: 21.9 -> 23.6 us).
    rc = pool_sum(ctx, st, q, pooled, fit > (size_t)kPoolCopies ? kPoolCopies : (int)fit, &ncopy, gp->W2, w2 <= ((size_t)4 << 20) ? w2 : 0);
    if (rc != SPECTRE_OK) return rc;
    sums = pooled;
  }
  const size_t one = gp->shared_across_heads ? 0 : 1;
  GateMlpParams mp = {};
  mp.sums = sums; mp.ncopy = ncopy; mp.copy_stride = (size_t)B * H * D; mp.inv_count = inv_count;
  mp.B = B; mp.H = H; mp.D = D; mp.hidden = gp->hidden; mp.n = n_fft; mp.K = K;
  mp.hs_ln = one * D; mp.hs_w1 = one * (size_t)D * gp->hidden; mp.hs_b1 = one * gp->hidden;
  mp.hs_w2 = one * (size_t)gp->hidden * 2 * K; mp.hs_b2 = one * 2 * (size_t)K; mp.hs_mb = one * K;
  mp.gamma = gp->ln_gamma; mp.beta = gp->ln_beta; mp.eps = gp->ln_eps;
  mp.W1 = gp->W1; mp.b1 = gp->b1; mp.W2 = gp->W2; mp.b2 = gp->b2;
  mp.modrelu_bias = gp->modrelu_bias;
  mp.shift = reinterpret_cast<const long long*>(shift); mp.shift_all = shift_all;
  {
    long long pm = shift_all % n_fft;
    if (pm < 0) pm += n_fft;
    mp.pm_all = (unsigned)pm;
  }
  mp.qbar_out = qbar_out;
  mp.u_ws = reinterpret_cast<float*>(reinterpret_cast<char*>(workspace) + u_off);
  mp.post = r > 0;
  mp.early = early;
  if (tok) mp.tok = *tok;
  float2* raw = r > 0 ? reinterpret_cast<float2*>(workspace) : nullptr;
  mp.g_out = r > 0 ? raw : reinterpret_cast<float2*>(g_out);
  // block sized to the bin count for short transforms (K = 99 does not need 256 threads)
  const int thr_out = K >= 256 ? 256 : ((K + 31) / 32 * 32 < 64 ? 64 : (K + 31) / 32 * 32);
  const bool mma = gate_on_mma(ctx, gp, B, H, K);
  const int BB = gate_entries(ctx, gp, B, H, K);
  dim3 grid_out((K + thr_out - 1) / thr_out, (unsigned)(H * ((B + BB - 1) / BB)));
  const bool wb = gp->wdtype == SPECTRE_BF16;
  const size_t w1_bytes = (size_t)D * gp->hidden * (wb ? 2 : 4);
  const size_t act_bytes = act_floats(BB, gp->hidden, D) * sizeof(float);
  const size_t staged_bytes = w1_bytes + (2 * (size_t)D + gp->hidden) * sizeof(float);
  mp.stage_w1 = w1_bytes <= 16384 && w1_bytes % 16 == 0 && !(reinterpret_cast<uintptr_t>(gp->W1) & 15) && act_bytes + staged_bytes <= 49152;
  const size_t smem = act_bytes + (mp.stage_w1 ? staged_bytes : 0);
  // One CTA holds all bins and a head's weights fit beside its activations: all of them staged, one short kernel
  const size_t w2_bytes = (size_t)gp->hidden * 2 * K * (wb ? 2 : 4);
  const size_t short_bytes = act_bytes + w1_bytes + ((2 * (size_t)D + gp->hidden + 3) & ~(size_t)3) * sizeof(float) + w2_bytes;
  const bool all_staged = BB >= 4 && !mma && grid_out.x == 1 && w1_bytes % 16 == 0 && w2_bytes % 16 == 0 && short_bytes <= 49152 &&
                          !((reinterpret_cast<uintptr_t>(gp->W1) | reinterpret_cast<uintptr_t>(gp->W2)) & 15);
  // Several entries and W1 not staged: the hidden layer with its loads of 32 inputs in flight (in a kernel of its own: its registers cost the staged
  // form 2 ... 4 % in one kernel with it)
  const bool deep = BB > 1 && !mp.stage_w1 && D >= 32;
  const bool pre = grid_out.x >= 32;               // many CTAs per head: compute the hidden layer once
  // Programmatic dependent launch: the weight stream of the output layer overlaps the kernel before it where that is one of
  // this call (the pooling pass); each kernel waits for its predecessor
  // (griddepcontrol.wait) before it touches the sums, and first of all where the caller's own kernel precedes it.
  cudaLaunchAttribute pdl[1];
  pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  pdl[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg_out = {}, cfg_hid = {};
  cfg_out.gridDim = grid_out; cfg_out.blockDim = dim3(thr_out, 1, 1); cfg_out.dynamicSmemBytes = smem; cfg_out.stream = st;
  cfg_out.attrs = pdl; cfg_out.numAttrs = 1;
  cfg_hid = cfg_out;
  cfg_hid.gridDim = dim3(grid_out.y, 1, 1); cfg_hid.blockDim = dim3(256, 1, 1);
  // the tensor-core kernel: at most the two CTAs per SM that are resident, never a second wave of a few
  cudaLaunchConfig_t cfg_mma = cfg_out;
  if (mma) {
    const int blocks = ((K + 15) / 16 + 7) / 8, fit = 2 * ctx->sm_count / (int)grid_out.y;
    cfg_mma.gridDim = dim3((unsigned)(fit < 1 ? 1 : (blocks < fit ? blocks : fit)), grid_out.y, 1);
    cfg_mma.blockDim = dim3(256, 1, 1);
  }
  // One entry and 2 (bf16) or 4 (fp32) threads per bin where its CTAs are few: a quarter of the SMs in bf16, three eighths in fp32.
  // The gate by itself gains beyond that (fp32, 14 heads x 1024: 10.4 -> 9.2 us), but the kernel behind starts beside these CTAs
  // and shares SMs that it would have had to itself.  Gate and mixer together, one sequence of 512 ... 8192 points: every number of
  // heads below the line gains, 0.25 ... 2.1 us (bf16 4 x 2048 23.1 -> 22.0, fp32 4 x 1024 17.7 -> 16.0); between it and one CTA per SM
  // it is -2.4 ... +6.7 (bf16 8 x 4096 27.9 -> 34.6, fp32 12 x 1024 21.2 -> 26.0).  A decode step gains 0.1 ... 1.6 us below the line and
  // loses up to 1.7 with more CTAs than SMs (bf16 12 x 4096 15.3 -> 17.0).
  const int split_bins = wb ? 128 : 64;
  const long long split_ctas = (long long)((K + split_bins - 1) / split_bins) * B * H;
  const bool split = BB == 1 && !pre && 8 * split_ctas <= (wb ? 2 : 3) * (long long)ctx->sm_count;
  cudaLaunchConfig_t cfg_split = cfg_out;
  cfg_split.gridDim = dim3((unsigned)((K + split_bins - 1) / split_bins), (unsigned)(B * H), 1); cfg_split.blockDim = dim3(256, 1, 1);
  cudaLaunchConfig_t cfg_short = cfg_out;
  cfg_short.gridDim = dim3(grid_out.y, 1, 1); cfg_short.dynamicSmemBytes = short_bytes;
#define SPECTRE_GATE_LAUNCH_AS(WT, NB, DEEP)                                                     \
  do {                                                                                           \
    if (pre) {                                                                                   \
      SPECTRE_CUDA_OK(launch_kernel(&cfg_hid, gate_hidden_kernel<WT, NB, DEEP>, mp));            \
      mp.early = 1;                                                                              \
      mp.tok.nclear = 0;                                                                         \
      SPECTRE_CUDA_OK(launch_kernel(&cfg_out, gate_out_kernel<WT, NB, true, false, false>, mp)); \
    } else {                                                                                     \
      if (mp.tok.q) SPECTRE_CUDA_OK(launch_kernel(&cfg_out, gate_out_kernel<WT, NB, false, true, DEEP>, mp)); \
      else SPECTRE_CUDA_OK(launch_kernel(&cfg_out, gate_out_kernel<WT, NB, false, false, DEEP>, mp)); \
    }                                                                                            \
  } while (0)
#define SPECTRE_GATE_LAUNCH(WT, NB)                                                              \
  do {                                                                                           \
    if (deep) SPECTRE_GATE_LAUNCH_AS(WT, NB, true); else SPECTRE_GATE_LAUNCH_AS(WT, NB, false);  \
  } while (0)
#define SPECTRE_GATE_SPLIT(WT)                                                                   \
  SPECTRE_CUDA_OK(launch_kernel(&cfg_split, mp.tok.q || mp.stage_w1 ? gate_split_kernel<WT, true> : gate_split_kernel<WT, false>, mp))
#define SPECTRE_GATE_SHORT(WT, FULL)                                                             \
  SPECTRE_CUDA_OK(BB == 8 ? launch_kernel(&cfg_short, gate_short_kernel<WT, 8, FULL>, mp)        \
                          : launch_kernel(&cfg_short, gate_short_kernel<WT, 4, FULL>, mp))
#define SPECTRE_GATE_MMA_FORM(NB, SHIFTS, TOK)                                                   \
  SPECTRE_CUDA_OK(launch_kernel(&cfg_mma, mp.stage_w1 ? gate_mma_kernel<NB, SHIFTS, TOK, true> : gate_mma_kernel<NB, SHIFTS, TOK, false>, mp))
#define SPECTRE_GATE_MMA(NB)                                                                     \
  do {                                                                                           \
    if (mp.tok.q) SPECTRE_GATE_MMA_FORM(NB, false, true); /* one phase for all entries */        \
    else if (mp.shift && !mp.post) SPECTRE_GATE_MMA_FORM(NB, true, false);                       \
    else SPECTRE_GATE_MMA_FORM(NB, false, false);                                                \
  } while (0)
  if (mma) {
    if (BB == 8) SPECTRE_GATE_MMA(8); else SPECTRE_GATE_MMA(4);
  } else if (all_staged) {
    if (mp.tok.q || (mp.shift && !mp.post)) {
      if (wb) SPECTRE_GATE_SHORT(bf16, true); else SPECTRE_GATE_SHORT(float, true);
    } else {
      if (wb) SPECTRE_GATE_SHORT(bf16, false); else SPECTRE_GATE_SHORT(float, false);
    }
  } else if (split) {
    if (wb) SPECTRE_GATE_SPLIT(bf16); else SPECTRE_GATE_SPLIT(float);
  } else switch (BB) {
    case 8: if (wb) SPECTRE_GATE_LAUNCH(bf16, 8); else SPECTRE_GATE_LAUNCH(float, 8); break;
    case 4: if (wb) SPECTRE_GATE_LAUNCH(bf16, 4); else SPECTRE_GATE_LAUNCH(float, 4); break;
    case 2: if (wb) SPECTRE_GATE_LAUNCH(bf16, 2); else SPECTRE_GATE_LAUNCH(float, 2); break;
    default: if (wb) SPECTRE_GATE_LAUNCH_AS(bf16, 1, false); else SPECTRE_GATE_LAUNCH_AS(float, 1, false); break;
  }
#undef SPECTRE_GATE_LAUNCH
#undef SPECTRE_GATE_LAUNCH_AS
#undef SPECTRE_GATE_MMA
#undef SPECTRE_GATE_MMA_FORM
#undef SPECTRE_GATE_SPLIT
#undef SPECTRE_GATE_SHORT
  SPECTRE_LAUNCH_OK("gate_out_kernel");
  if (r > 0) {
    GatePostParams pp = {};
    pp.g_raw = raw; pp.g_out = reinterpret_cast<float2*>(g_out);
    pp.taps = gp->toeplitz; pp.hs_t = one * (2 * r + 1); pp.r = r;
    pp.modrelu_bias = gp->modrelu_bias; pp.hs_mb = one * K;
    pp.shift = mp.shift; pp.shift_all = shift_all;
    pp.H = H; pp.K = K; pp.n = n_fft;
    dim3 grid((K + 255) / 256, B * H);
    SPECTRE_CUDA_OK(launch_after(gate_post_kernel, grid, 256, 0, st, pp));
    SPECTRE_LAUNCH_OK("gate_post_kernel");
  }
  return SPECTRE_OK;
}
}  // namespace spectre

// With q the pooling pass is in front of the gate kernels; with sum_q whatever the caller launched last is.
extern "C" int spectre_gate(spectre_ctx* ctx, void* stream, const spectre_act* q, const float* sum_q, int32_t B,
                            int32_t H, int32_t D, float inv_count, const spectre_gate_params* gp, int32_t n_fft,
                            const int64_t* shift, int64_t shift_all, float* g_out, float* qbar_out, void* workspace,
                            size_t workspace_bytes) {
  return gate_call(ctx, stream, q, sum_q, B, H, D, inv_count, gp, n_fft, shift, shift_all, g_out, qbar_out, workspace, workspace_bytes,
                   q != nullptr, nullptr);
}

// ---- gate without any caller- or library-side allocation -----------------------
// Scratch of spectre_gate_static: one fixed array per GPU that loads this library,
// resident until the process exits.  Host code must not hand this name to a kernel
// (on the host it is only a stand-in for the symbol); the device address is looked
// up once per device below.
#define SPECTRE_GATE_STATIC_BYTES (1u << 20)
static __device__ __align__(256) unsigned char g_gate_static_scratch[SPECTRE_GATE_STATIC_BYTES];

namespace spectre {
static const int kMaxDevices = 64;
static std::atomic<void*> g_static_ptr[kMaxDevices];     // device address of the array, per device ordinal

// With `device` current: resolves (once) the device address of the static scratch.  Host threads
// that race on the first call of a device each look the address up and store the same value.
static int static_scratch_address(int device, void** out) {
  if (device < 0 || device >= kMaxDevices) return fail(SPECTRE_ERR_UNSUPPORTED, "device ordinal beyond 63");
  void* p = g_static_ptr[device].load(std::memory_order_acquire);
  if (!p) {
    cudaError_t e = cudaGetSymbolAddress(&p, g_gate_static_scratch);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(gate static scratch)");
    if (!p) return fail(SPECTRE_ERR_CUDA, "static scratch has no device address");
    g_static_ptr[device].store(p, std::memory_order_release);
  }
  *out = p;
  return SPECTRE_OK;
}
}  // namespace spectre

extern "C" size_t spectre_gate_static_max_bytes(void) { return SPECTRE_GATE_STATIC_BYTES; }

extern "C" int spectre_gate_static(spectre_ctx* ctx, void* stream, const spectre_act* q, const float* sum_q, int32_t B,
                                   int32_t H, int32_t D, float inv_count, const spectre_gate_params* gp, int32_t n_fft,
                                   const int64_t* shift, int64_t shift_all, float* g_out, float* qbar_out) {
  if (!ctx) return fail(SPECTRE_ERR_INVALID_ARG, "ctx is NULL");
  if (!gp) return fail(SPECTRE_ERR_INVALID_ARG, "gate parameters are NULL");
  if (B < 1 || H < 1 || D < 1 || D > 1024) return fail(SPECTRE_ERR_INVALID_ARG, "B, H, D must be positive (D <= 1024)");
  if (n_fft < 1 || n_fft > (1 << 24)) return fail(SPECTRE_ERR_INVALID_ARG, "n_fft out of range");
  // the widths that size the scratch are range-checked before the size is computed from them
  if (gp->hidden < 1 || gp->hidden > 1024) return fail(SPECTRE_ERR_UNSUPPORTED, "hidden width must be in 1..1024");
  if (gp->toeplitz_r < 0 || gp->toeplitz_r > 64) return fail(SPECTRE_ERR_UNSUPPORTED, "toeplitz_r must be in 0..64");
  size_t off_a, off_b;
  const size_t need = gate_ws_layout(B, H, D, n_fft, gp->toeplitz_r, gp->hidden, 1, &off_a, &off_b);   // one copy of the sums
  if (need > SPECTRE_GATE_STATIC_BYTES)
    return fail(SPECTRE_ERR_UNSUPPORTED,
                "spectre_gate_static: this shape needs " + std::to_string(need) + " bytes of scratch, the built-in array holds " +
                    std::to_string((size_t)SPECTRE_GATE_STATIC_BYTES) + "; use spectre_gate with a workspace");
  SPECTRE_CUDA_OK(cudaSetDevice(ctx->device));
  void* scratch = nullptr;
  int rc = static_scratch_address(ctx->device, &scratch);
  if (rc != SPECTRE_OK) return rc;
  // Same kernels as spectre_gate; the pooled sum is cleared inside (on the caller's stream), so what an
  // earlier call left in the array does not matter.
  return spectre_gate(ctx, stream, q, sum_q, B, H, D, inv_count, gp, n_fft, shift, shift_all, g_out, qbar_out, scratch,
                      SPECTRE_GATE_STATIC_BYTES);
}
