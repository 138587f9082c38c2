// Tensor-core spectral mixer for n = 4096, bf16 or fp16 I/O (Sec. 3.2 steps 2 and 4), one kernel, for few tiles and for lengths with
// a long partial block; the other calls take mixer_tc64.cu, where the rule stands (launch_mixer_tc4096).
//
// One CTA = one (batch, head, 4 column pairs) = a 16-byte piece of every row, two CTAs per SM.  The length-4096 transform
// of a pair is 64 x 64: the same stages, DFT matrix and dense operand images as a unit of the staged core (tc_stage.cuh,
// mixer_tc4k.cu), but the rows arrive and leave by TMA through a map that splits the row index t = 64 t1 + t2 into its
// digits, so nothing is written between the transform's passes: a box of 4 t1 x 64 t2 lands as one K group of the first
// operand and is converted (four rows x four pairs transposed) in place, and the last epilogue stages whole 16-byte pieces
// of 8 t1 x 32 t2 rows per warp, which that warp alone hands to the TMA engine.
//
// Why: the staged path spends three kernels and two fp16 intermediates on it (100 us at B = 4, H = 16, D = 64, rotating buffers;
// this kernel: 46 us, 48 with cold caches).  What bounds it is the latency of the epilogues: the 16-byte row requests (4096 in and 4096 out per CTA,
// about 1.2 cycles each on the SM's request path, 3.5 CTAs per SM) are 17 us of it, the rest is TMEM and twiddle loads in front
// of their use with only the other CTA of the SM to hide them, and 512 CTAs are 1.73 waves of the 296 that are resident.
//
// Rows beyond L are zero: the map ends at the last whole block of 64, TMA fills and clips the rest, and the L % 64 rows of
// a partial block are read by the conversion and written by the last epilogue with plain 16-byte accesses.
#include <cuda.h>

#include <string>

#include "tc_stage.cuh"

namespace spectre {

constexpr int k40Lbo = 4096, k40Sbo = 128;       // dense operand images: 4096 bytes between K groups, 128 between 8-column groups
constexpr int k40FBytes = 128 * 128 * 2, k40BBytes = 16 * k40Lbo, k40GBytes = 4096 * 4;
constexpr int k40EpiWarps = 8, k40EpiThreads = 32 * k40EpiWarps, k40Threads = k40EpiThreads + 32;
constexpr int k40Smem = k40FBytes + k40BBytes + k40GBytes + 128;   // + barriers, TMEM address, the warps' maxima
static_assert(2 * (k40Smem + 1024) <= 233472, "two CTAs per SM");

struct Tc4096Params {
  const float2* g;        // [B*H][2049]
  const __half* F;        // 64-point DFT matrix, canonical smem layout
  const float2* tw64;     // stage twiddles W_4096^{row d} (even d) in epilogue order
  const void* src;        // rows of the partial block (L % 64 of them)
  void* dst;
  int64_t s_sb, s_sl, s_sh, d_sb, d_sl, d_sh;
  int H, ntile, L;
  int* status;
};

__device__ __forceinline__ float2 gate4096(const float2* g, int k) {
  const int kk = k <= 2048 ? k : 4096 - k;
  float2 v = g[kk];
  if (kk != k) v.y = -v.y;
  if (k == 0 || k == 2048) v.y = 0.f;
  return v;
}

template <bool F16>
__global__ void __launch_bounds__(k40Threads, 2) mixer_tc4096_kernel(const __grid_constant__ CUtensorMap tm_in,
                                                                     const __grid_constant__ CUtensorMap tm_out,
                                                                     const Tc4096Params p) {
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* Fsm = smem;
  unsigned char* Bsm = smem + k40FBytes;
  uint32_t* Gsm = reinterpret_cast<uint32_t*>(smem + k40FBytes + k40BBytes);
  // 0, 1 halves of the rows landed; 2 F landed; 3 accumulator ready; 4 operand ready
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + k40FBytes + k40BBytes + k40GBytes);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 6);
  float* red = reinterpret_cast<float*>(bars + 8);
  const int tid = threadIdx.x, warp = tid >> 5, T = tid & 31;
  const int tile = blockIdx.x % p.ntile, slab = blockIdx.x / p.ntile;
  const int b = slab / p.H, h = slab - b * p.H;
  const int col0 = tile * 8;
  const uint32_t barF = smem_u32(&bars[2]), barD = smem_u32(&bars[3]), barB = smem_u32(&bars[4]);

  if (warp == k40EpiWarps) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(smem_u32(tmem_slot)), "r"(256));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int i = 0; i < 4; ++i) mbar_init(smem_u32(&bars[i]), 1);
    mbar_init(barB, k40EpiThreads);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  // programmatic dependent: nothing of V or g is read before the kernel in front of this one is complete
  asm volatile("griddepcontrol.wait;" ::: "memory");
  bool ok = true;

  if (warp == k40EpiWarps) {
    if (T == 0) {
      for (int half = 0; half < 2; ++half) {
        const uint32_t bar = smem_u32(&bars[half]);
        mbar_expect_tx(bar, 8 * 4096);
        for (int a = 8 * half; a < 8 * half + 8; ++a) tma_load_5d(smem_u32(Bsm) + 4096 * a, &tm_in, col0, 0, 4 * a, h, b, bar);
      }
      mbar_expect_tx(barF, k40FBytes);
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                   :: "r"(smem_u32(Fsm)), "l"(p.F), "r"(k40FBytes), "r"(barF) : "memory");
    }
    __syncwarp();
    const uint32_t idesc = umma_idesc_128x256();
    ok = mbar_wait(barF, 0);
    for (int stage = 0; stage < 4 && ok; ++stage) {
      ok = mbar_wait(barB, stage & 1);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (T == 0) {
        const uint32_t a0 = smem_u32(Fsm), b0 = smem_u32(Bsm);
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
          const uint64_t da = umma_desc(a0 + ks * 256, 128, 2048);
          const uint64_t db = umma_desc(b0 + ks * 2 * k40Lbo, k40Lbo, k40Sbo);
          const uint32_t acc = ks > 0;
          asm volatile(
              "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
              :: "r"(tmem), "l"(da), "l"(db), "r"(idesc), "r"(acc) : "memory");
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" :: "r"(barD) : "memory");
      }
      __syncwarp();
    }
    if (!ok) {                                   // do not leave with copies into this CTA still in flight (bounded again)
      mbar_wait(smem_u32(&bars[0]), 0);
      mbar_wait(smem_u32(&bars[1]), 0);
      mbar_wait(barF, 0);
    }
  } else {
    // ---- gate table while the rows are in flight: Hermitian extension, normalised by a bound on max |g| ----
    const float2* g = p.g + (size_t)slab * 2049;
    constexpr int kG = 4096 / k40EpiThreads;
    float2 gv[kG];
    float gmax = 0.f;
#pragma unroll
    for (int i = 0; i < kG; ++i) gv[i] = gate4096(g, tid + i * k40EpiThreads);
#pragma unroll
    for (int i = 0; i < kG; ++i) gmax = fmaxf(gmax, fmaxf(fabsf(gv[i].x), fabsf(gv[i].y)));
    for (int o = 16; o > 0; o >>= 1) gmax = fmaxf(gmax, __shfl_xor_sync(0xffffffffu, gmax, o));
    if (T == 0) red[warp] = gmax;
    asm volatile("bar.sync 1, %0;" :: "r"(k40EpiThreads) : "memory");
    gmax = red[0];
    for (int i = 1; i < k40EpiWarps; ++i) gmax = fmaxf(gmax, red[i]);
    gmax *= 1.41421356f;
    const float ginv = gmax > 0.f ? 1.0f / gmax : 0.f;
#pragma unroll
    for (int i = 0; i < kG; ++i) {               // bin k1 + 64 k2 at 64 k2 + (k1 ^ 8 (k2 % 4))
      const int k = tid + i * k40EpiThreads, k1 = k & 63, k2 = k >> 6;
      Gsm[64 * k2 + (k1 ^ (8 * (k2 & 3)))] = pack_h2(gv[i].x * ginv, gv[i].y * ginv);
    }

    // ---- rows -> first operand, in place: t1 = 4a .. 4a + 3 at one t2, four 16-byte rows in, four 16-byte K groups out ----
    const int t2 = tid & 63, lb = p.L >> 6, lr = p.L & 63;
#pragma unroll 1
    for (int i = 0; i < 4 && ok; ++i) {
      if ((i & 1) == 0) ok = mbar_wait(smem_u32(&bars[i >> 1]), 0);
      if (!ok) break;
      const int a = 4 * i + (tid >> 6);
      unsigned char* p0 = Bsm + 4096 * a + 16 * t2;
      uint4 r[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) r[u] = *reinterpret_cast<const uint4*>(p0 + 1024 * u);
      if (lr && (lb >> 2) == a && t2 < lr) {     // the partial block's rows
        const uint4 v = *reinterpret_cast<const uint4*>(reinterpret_cast<const __half*>(p.src) + b * p.s_sb + (int64_t)(64 * lb + t2) * p.s_sl +
                                                        h * p.s_sh + col0);
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (u == (lb & 3)) r[u] = v;
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint32_t e[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const uint32_t w = c == 0 ? r[u].x : (c == 1 ? r[u].y : (c == 2 ? r[u].z : r[u].w));
          if (F16) {
            e[u] = w;
          } else {
            const float2 f = unpack_bf2(w);
            e[u] = pack_h2(f.x, f.y);
          }
        }
        *reinterpret_cast<uint4*>(p0 + 1024 * c) = make_uint4(e[0], e[1], e[2], e[3]);
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    mbar_arrive(barB);

    const int q = warp & 3, wh = warp >> 2;
    const float2 wr0 = twiddle_fwd((unsigned)(16 * q + (T >> 2)), 4096u), wr1 = twiddle_fwd((unsigned)(16 * q + 8 + (T >> 2)), 4096u);
    asm volatile("bar.sync 1, %0;" :: "r"(k40EpiThreads) : "memory");        // the gate table is complete
#pragma unroll 1
    for (int stage = 0; stage < 3 && ok; ++stage) {
      ok = mbar_wait(barD, stage & 1);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (stage == 0) epilogue_twiddle2<k40Lbo, k40Sbo, 1>(tmem, Bsm, q, 2 * wh, T, p.tw64, wr0, wr1);
      else if (stage == 2) epilogue_twiddle2<k40Lbo, k40Sbo, 2>(tmem, Bsm, q, 2 * wh, T, p.tw64, wr0, wr1);
      else {
#pragma unroll 1
        for (int cc = 0; cc < 2; ++cc) epilogue_gate_t<k40Lbo, k40Sbo, 64, true>(tmem, Bsm, q, 2 * wh + cc, T, Gsm);
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_arrive(barB);
    }
    // ---- y[64 row + s1] = gmax conj(D).  A thread holds all four pairs of its rows (columns 16 (s1 / 4) + 8 (c / 2) +
    //      2 (s1 % 4) + c % 2); the warp's 8 t1 x 32 s1 rows are one box ----
    if (ok) ok = mbar_wait(barD, 1);
    if (ok) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int i = T >> 2, tq = T & 3;
      const uint32_t taddr0 = tmem + ((uint32_t)(32 * q) << 16) + 128 * wh;
      uint32_t r[2][16];
      bool bad = false;
      tmem_ld_16x256b_x4(taddr0, r[0]);
#pragma unroll
      for (int step = 0; step < 8; ++step) {     // step = 4 j + chunk, 32 columns = 8 s1 per chunk
        const int j = step >> 2, chunk = step & 3;
        tmem_ld_wait();
        if (step < 7) {
          const int ns = step + 1;
          tmem_ld_16x256b_x4(taddr0 + ((uint32_t)(16 * (ns >> 2)) << 16) + 32 * (ns & 3), r[ns & 1]);
        }
        const uint32_t (&x)[16] = r[step & 1];
        const int t1 = 8 * (2 * q + j) + i;
        unsigned char* box = Bsm + ((2 * q + j) * 2 + wh) * 4096 + i * 512;
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          uint32_t o[4];
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const int k = 4 * (2 * s + (c >> 1)) + (c & 1);
            const float re = gmax * __uint_as_float(x[k]), im = -gmax * __uint_as_float(x[k + 2]);
            o[c] = F16 ? pack_h2(re, im) : pack_bf2(re, im);
          }
          const uint4 row = make_uint4(o[0], o[1], o[2], o[3]);
          const int s1l = 8 * chunk + 4 * s + tq;
          // an overflow anywhere in a column makes every row of it non-finite: one row per thread is enough
          if (step == 0 && s == 0)
            bad = nonfinite16x2<F16>(o[0]) | nonfinite16x2<F16>(o[1]) | nonfinite16x2<F16>(o[2]) | nonfinite16x2<F16>(o[3]);
          *reinterpret_cast<uint4*>(box + 16 * s1l) = row;
          if (lr && t1 == lb && 32 * wh + s1l < lr)
            *reinterpret_cast<uint4*>(reinterpret_cast<__half*>(p.dst) + b * p.d_sb + (int64_t)(64 * lb + 32 * wh + s1l) * p.d_sl + h * p.d_sh +
                                      col0) = row;
        }
        if (chunk == 3) {
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (T == 0) {
            tma_store_5d(&tm_out, col0, 32 * wh, 8 * (2 * q + j), h, b, smem_u32(Bsm) + ((2 * q + j) * 2 + wh) * 4096);
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
          }
        }
      }
      if (T == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
      if (__any_sync(0xffffffffu, bad) && T == 0) report_range(p.status);
    }
  }
  if (!ok && T == 0) report_timeout(p.status);
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == k40EpiWarps) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(256));
  }
}

// ---- host side ----
// dims (column, t2, t1, head, batch)
static int make_map4096(CUtensorMap* tm, const spectre_act* a, unsigned box_t2, unsigned box_t1) {
  const cuuint64_t sl = (cuuint64_t)a->stride_l * 2, sh = (cuuint64_t)a->stride_h * 2, sb = (cuuint64_t)a->stride_b * 2;
  const cuuint64_t dims[5] = {(cuuint64_t)a->D, 64, (cuuint64_t)(a->L / 64), (cuuint64_t)a->H, (cuuint64_t)a->B};
  const cuuint64_t strides[4] = {sl, 64 * sl, sh, sb};
  const cuuint32_t box[5] = {8, box_t2, box_t1, 1, 1}, es[5] = {1, 1, 1, 1, 1};
  const CUresult r = tensor_map_encoder()(
      tm, a->dtype == SPECTRE_F16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, a->ptr, dims, strides, box, es,
      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(SPECTRE_ERR_CUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
  return SPECTRE_OK;
}

int launch_mixer_pairs4096(const spectre_ctx* ctx, cudaStream_t st, const spectre_act* v, const float* g, const spectre_act* y) {
  CUtensorMap tm_in, tm_out;
  int rc = make_map4096(&tm_in, v, 64, 4);
  if (rc == SPECTRE_OK) rc = make_map4096(&tm_out, y, 32, 8);
  if (rc != SPECTRE_OK) return rc;
  Tc4096Params p = {};
  p.g = reinterpret_cast<const float2*>(g);
  p.F = reinterpret_cast<const __half*>(ctx->dft64);
  p.tw64 = reinterpret_cast<const float2*>(ctx->tw64x64);
  p.src = v->ptr; p.s_sb = v->stride_b; p.s_sl = v->stride_l; p.s_sh = v->stride_h;
  p.dst = y->ptr; p.d_sb = y->stride_b; p.d_sl = y->stride_l; p.d_sh = y->stride_h;
  p.H = v->H; p.ntile = v->D / 8; p.L = v->L;
  p.status = ctx->status_dev;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((size_t)v->B * v->H * p.ntile));
  cfg.blockDim = dim3(k40Threads);
  cfg.dynamicSmemBytes = k40Smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  auto kern = v->dtype == SPECTRE_F16 ? mixer_tc4096_kernel<true> : mixer_tc4096_kernel<false>;
  SPECTRE_CUDA_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, k40Smem));
  SPECTRE_CUDA_OK(launch_kernel(&cfg, kern, tm_in, tm_out, p));
  return SPECTRE_OK;
}

}  // namespace spectre
