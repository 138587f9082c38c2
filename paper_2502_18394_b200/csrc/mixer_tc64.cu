// Tensor-core spectral mixer for n = 4096 and n = 8192, bf16 or fp16 I/O (Sec. 3.2 steps 2 and 4), one persistent kernel, which also
// transforms the 4096-point units of longer sequences (HALVES = 0).
//
// A tile is eight 4096-point problems that share a 32-byte piece of every row: n = 4096 the eight column pairs of one piece,
// n = 8192 the even and the odd output bins of four column pairs (radix-2 step on the ALUs; HALVES = 2), units two adjacent ones
// of a (head, k1), whose chunks land as operands from their images in the workspace and whose results return there.  A 4096-point problem
// is 64 x 64: four contractions with the 64-point DFT matrix F (128 x 128 in real form, scaled by 1/8, rows ordered so that Re
// and Im of a bin sit 8 TMEM lanes apart), the inverse as conj(FFT(conj(.))).  Row index t = 64 t1 + t2, bin k1 + 64 k2:
//
//   stage 0  contracts t1.  A = F, B = landed rows (shared memory): D has lanes (k1, part), columns (t2, problem)
//            epilogue: times W_4096^{k1 t2}, fp16, back to TMEM as an A operand with lanes (k1, b) and K along the columns
//   stage 1  contracts t2.  A = that operand (TMEM), B = F: D has lanes (k1, b), columns (k2, part)
//            epilogue: gate, conjugate, fp16, in place as the next A operand
//   stage 2  contracts k2.  A (TMEM), B = F: D has lanes (k1, b), columns (s2, part)
//            epilogue: times W_4096^{k1 s2}, fp16, to shared memory as a B operand (128-byte swizzle) with K = k1
//   stage 3  contracts k1.  A = F, B = that operand: D has lanes (s1, part), columns (s2, problem): rows 64 s1 + s2
//
// so between stages 0 and 2 nothing leaves TMEM but through registers of the lane that owns it, and shared memory holds one
// operand only: the rows go through a small ring, 8 values of t2 (512 pieces) at a time, each chunk converted in place and
// contracted as it lands, and the results leave through the last operand's own space, 8 values of s2 at a time.  Hence the
// next tile's rows are fetched and contracted under the last stage of the current one and under its stores.
//
// Work is cut into jobs of 8 MMAs: per tile 8 chunks of stage 0 and of stage 3 (64 accumulator columns, four in rotation) and 4
// groups of stages 1 and 2 (128 columns, two in rotation).  16 epilogue warps in two sets of 8 (a set: 4 TMEM lane quadrants x 2)
// take the chunks in turn and one half each of a group's columns; warp 16 issues the MMAs, warp 17 moves the rows.
//   problem = 4 b + G: b = lane half (0, 1) and G = group (0..3) in stages 1 and 2
//   TMEM columns: 32 (k >> 3) + 8 G + (k & 7) the A operands (k = t2, then k2), 256 ... accumulators
//
// Two more warps build the next tile's gate table under the current tile.
//
// Why: an SM moves one 32-byte piece of a row per 1.3 cycles (loads from L2; stores 1.4) and a 16-byte piece per 1.1 (1.4), so
// 32-byte pieces halve the time in the request path, and only the rows of 8 problems x 64 t2 steps that are in flight need shared
// memory besides the one operand.  The kernels before this one (mixer_tc4096.cu is one of them, still the better for few tiles) kept 4
// column pairs per CTA in 16-byte pieces and ran rows in, four stages and rows out one after the other.  Public calls, us: 4 x 4096 x 16 heads with projection 89.5 -> 74.7 (this kernel 47 -> 31),
// 1 x 8192 x 32 heads 70.8 -> 63.4 (51 -> 40), its backward included 200.2 -> 182.9.
// What bounds it now is the epilogues' latency: a tile of n = 4096 takes 13 k cycles to land and pass stage 0, 7.5 k in stages 1 and 2
// (MMAs 4.1 k, arithmetic 3 k) and 16 k in stage 3 side by side with the next tile's stage 0, of which the pieces are 11 k; a step of an
// epilogue is some 300 cycles of waits and fences around 200 of arithmetic, with four warps per scheduler to overlap them.
// A set waits for a job only when the job before it in the same accumulator is known to be complete (its own last job was a later one):
// a wait for a phase whose predecessor is still under way would be answered by the phase before that.
// Measured and not kept: chunks of 16 t2 with accumulators of 128 columns in stages 0 and 3, too (n = 4096 31 -> 33), four sets of
// four warps (31 -> 33), F in TMEM for stages 0 and 3, too (31 -> 33), the first gate table by the epilogue warps (31 -> 33),
// accumulators read one group ahead into registers (31 -> 33), two chunks of lookahead instead of three (31 -> 43).
#include <cuda.h>

#include <string>

#include "tc_common.cuh"

namespace spectre {

constexpr int k64Warps = 16, k64Epi = 32 * k64Warps, k64Threads = k64Epi + 128;
// registers a thread: 96 at launch; the epilogue warpgroups take 112 and the last one keeps 32 (4 x 112 + 32 = 5 x 96)
constexpr int k64Regs = 96, k64EpiRegs = 112, k64IoRegs = 32;
static_assert(4 * k64EpiRegs + k64IoRegs <= 5 * k64Regs && k64Threads * k64Regs <= 65536, "register split");
constexpr int k64Chunk = 16384, k64Op = 8 * k64Chunk, k64F = 128 * 128 * 2;
constexpr int k64TmAcc = 256;
constexpr int k64Rows = 33;                      // gate table: rows k2 = 0 ... 31 and, for k1 = 0, 32
template <int HALVES> struct Tc64 {
  static constexpr bool kUnits = HALVES == 0;
  static constexpr int n = 4096 * HALVES, kRing = HALVES == 1 ? 3 : 2;
  static constexpr int kGate = kUnits ? 16384 : HALVES * k64Rows * 256, kRowTw = kUnits ? 2048 : 0;
  static constexpr int kFOff = k64Op + kRing * k64Chunk, kGateOff = kFOff + k64F, kTwOff = kGateOff + kGate;
  static constexpr int kBarOff = kTwOff + 8192 + 64 + kRowTw, kSmem = kBarOff + 512;
  static_assert(kSmem <= 232448 && kBarOff % 8 == 0, "shared memory");
  // Where chunk c of a tile's rows lands, in chunks: the first ones behind the operand space, the others in the part of it that
  // the last tile's chunk c - kRing left through
  static __device__ __forceinline__ int land_slot(int c) { return c < kRing ? 8 + c : c - kRing; }
  // order of the groups in stages 1 and 2; n = 8192: those of the even bins, then those of the odd ones
  static __device__ __forceinline__ int group(int e) { return HALVES == 2 ? 2 * (e & 1) + (e >> 1) : e; }
};
struct Tc64Params {
  const float2* g;        // [B*H][n/2 + 1]
  const __half* F;        // 64-point DFT matrix, canonical K-major layout
  const void* src;        // rows of the partial block (L % 64 of them, n = 4096)
  void* dst;
  int64_t s_sb, s_sl, s_sh, d_sb, d_sl, d_sh;
  int H, ntile, L, D, total;
  int* status;
  // units of a longer transform
  const unsigned char* gimg;   // gate tables [head, k1][16 KB]
  const float* gscale;         // and their bounds
  const float2* twr;           // [R][128]: W_n^{64 k1 t1}, W_n^{k1 t2}
  float out_scale;
  int R;
};

#define SPECTRE_R16(r) "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), \
  "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
#define SPECTRE_R32(r) SPECTRE_R16(r), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), \
  "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
// 16 lanes x 64 columns (thread T: lanes T/4 and T/4 + 8, as tmem_ld_16x256b_x4)
__device__ __forceinline__ void tmem_ld_16x256b_x8(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,"
               "%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];" : SPECTRE_R32(r) : "r"(taddr));
}
// 32 lanes x 16 columns (thread T: lane T)
__device__ __forceinline__ void tmem_ld_32x32b_x16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];" : SPECTRE_R16(r) : "r"(taddr));
}
#undef SPECTRE_R32
#undef SPECTRE_R16
__device__ __forceinline__ void tmem_st_32x32b_x8(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
               :: "r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
}
#define SPECTRE_ST16(shape, taddr, r)                                                                                                    \
  asm volatile("tcgen05.st.sync.aligned." shape ".b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"                   \
               :: "r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), \
                  "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory")
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// A in TMEM, B by descriptor; issued by the one lane whose `one` is set.  The whole warp runs the code around it, so that
// addresses and descriptors stay in uniform registers: with the branch on the lane around the loop instead, an MMA took the
// issuing lane 80 cycles.
__device__ __forceinline__ void mma_ts(uint32_t one, uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile("{\n.reg .pred p, q;\nsetp.ne.b32 p, %4, 0;\nsetp.ne.b32 q, %5, 0;\n@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}"
               :: "r"(d), "r"(a), "l"(b), "r"(idesc), "r"(acc), "r"(one) : "memory");
}
// both operands by descriptor
__device__ __forceinline__ void mma_ss(uint32_t one, uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile("{\n.reg .pred p, q;\nsetp.ne.b32 p, %4, 0;\nsetp.ne.b32 q, %5, 0;\n@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
               :: "r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc), "r"(one) : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t one, uint32_t bar) {
  asm volatile("{\n.reg .pred q;\nsetp.ne.b32 q, %1, 0;\n@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}" :: "r"(bar), "r"(one) : "memory");
}
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t one;
  asm volatile("{\n.reg .pred q;\nelect.sync _|q, 0xffffffff;\nselp.u32 %0, 1, 0, q;\n}" : "=r"(one));
  return one;
}
__device__ __forceinline__ constexpr uint32_t idesc_f16(uint32_t N) { return (1u << 4) | ((N >> 3) << 17) | ((128u >> 4) << 24); }
// Bounded wait.  A first poll for what is already there; the others sleep up to 20 us each (the hint), so that waiting warps leave
// the issue slots to the rest; 2^16 of them are a little over a second.
__device__ __forceinline__ void warp_wait(bool& ok, uint32_t bar, uint32_t parity) {
  if (!ok) return;
  uint32_t done;
  asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
               : "=r"(done) : "r"(bar), "r"(parity) : "memory");
  if (done) return;
#pragma unroll 1
  for (uint32_t it = 0; it < (1u << 16); ++it) {
    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\nselp.u32 %0, 1, 0, p;\n}"
                 : "=r"(done) : "r"(bar), "r"(parity), "r"(20000u) : "memory");
    if (done) return;
  }
  ok = false;
}
// products of two packed values with two packed factors: X = re wx - im wy, Y = re wy + im wx
__device__ __forceinline__ void cmul2(uint64_t RE, uint64_t IM, uint64_t WX, uint64_t WY, uint64_t NWY, float (&x)[2], float (&y)[2]) {
  upk2(fma2(IM, NWY, mul2(RE, WX)), x[0], x[1]);
  upk2(fma2(IM, WX, mul2(RE, WY)), y[0], y[1]);
}

template <bool F16, int HALVES>
__global__ void __launch_bounds__(k64Threads, 1) mixer_tc64_kernel(const __grid_constant__ CUtensorMap tm_in, const __grid_constant__ CUtensorMap tm_out,
                                                                   const Tc64Params p) {
  typedef Tc64<HALVES> C;
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char *Op = smem, *Fsm = smem + C::kFOff;
  uint32_t* Gsm = reinterpret_cast<uint32_t*>(smem + C::kGateOff);
  float2* T8 = reinterpret_cast<float2*>(smem + C::kTwOff);      // W_4096^{8 c k1} at [c (8)][k1 (64)]
  float2* T1 = T8 + 512;                                         // W_4096^{r k1} at [r (8)][k1 (64)]
  float2* W8 = T8 + 1024;                                        // W_8192^{8 c}
  const float2* Rtw = T8 + 1032;                                 // units: the 128 factors of even and odd tiles' k1
  const uint32_t bars = smem_u32(smem + C::kBarOff);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::kBarOff + 424);
  float* gmax = reinterpret_cast<float*>(smem + C::kBarOff + 432);   // bound of the gates of even and odd tiles, the two warps' maxima
  auto landFull = [&](int c) { return bars + 8u * c; };          // rows of a chunk landed (transaction count)
  auto convFull = [&](int c) { return bars + 64u + 8u * c; };    // and are an operand (8 warps)
  auto stFull = [&](int c) { return bars + 128u + 8u * c; };     // results of a chunk staged (8 warps)
  auto accFull = [&](int i) { return bars + 192u + 8u * i; };    // accumulator of a chunk complete
  auto accFree = [&](int i) { return bars + 224u + 8u * i; };    // and read (8 warps)
  auto a2Full = [&](int G) { return bars + 256u + 8u * G; };     // a group's stage-2 operand complete (16 warps)
  auto yFull = [&](int i) { return bars + 288u + 8u * i; };      // accumulator of a group complete
  auto yFree = [&](int i) { return bars + 304u + 8u * i; };      // and read (16 warps)
  auto landFree = [&](int c) { return bars + 320u + 8u * c; };   // the MMAs of the first kRing chunks completed
  const uint32_t aFull = bars + 344;                             // stage 1's operand complete (8 chunks x 8 warps)
  const uint32_t opFull = bars + 352;                            // stage 3's operand complete (16 warps)
  const uint32_t opFree = bars + 360;                            // a tile's results have left the operand space
  const uint32_t fFull = bars + 368;                             // F landed
  const uint32_t gFull = bars + 376, gFree = bars + 384;         // gate table written (2 warps), read (16 warps)
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), T = tid & 31;    // the shuffle tells the compiler that the roles are uniform over a warp

  if (warp == k64Warps) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(smem_u32(tmem_slot)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int i = 0; i < 8; ++i) { mbar_init(landFull(i), 1); mbar_init(convFull(i), 8); mbar_init(stFull(i), 8); }
    for (int i = 0; i < 4; ++i) { mbar_init(accFull(i), 1); mbar_init(accFree(i), 8); mbar_init(a2Full(i), 16); }
    for (int i = 0; i < 2; ++i) { mbar_init(yFull(i), 1); mbar_init(yFree(i), 16); }
    for (int i = 0; i < 3; ++i) mbar_init(landFree(i), 1);
    mbar_init(gFull, C::kUnits ? 1 : 2);
    mbar_init(gFree, 16);
    mbar_init(aFull, 64);
    mbar_init(opFull, 16);
    mbar_init(opFree, 1);
    mbar_init(fFull, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = tid; i < 1024; i += k64Threads) T8[i] = twiddle_fwd((unsigned)((i < 512 ? 8 : 1) * ((i >> 6) & 7) * (i & 63)), 4096u);
  if (tid < 8) W8[tid] = twiddle_fwd((unsigned)tid, 1024u);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  if (tid == 0) {                                                // a table of the context: not behind the wait
    mbar_expect_tx(fFull, k64F);
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(smem_u32(Fsm)), "l"(p.F), "r"(k64F), "r"(fFull) : "memory");
  }
  // programmatic dependent: nothing of V or g is read before the kernel in front of this one is complete
  asm volatile("griddepcontrol.wait;" ::: "memory");
  bool ok = (smem_u32(smem) & 1023u) == 0;                       // the swizzled operand needs 1024-byte aligned rows

  if (warp >= k64Warps) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" :: "n"(k64IoRegs));
  if (warp == k64Warps + 1) {
    // ---- rows in and out.  Chunk c of a tile: 8 values of t2 of all t1 ----
    auto load = [&](int tile, int c) {
      mbar_expect_tx(landFull(c), k64Chunk);
      if constexpr (C::kUnits) {                                 // both units' columns of these t2, all K groups: an operand as it lands
        tma_load_5d(smem_u32(smem) + C::land_slot(c) * k64Chunk, &tm_in, 0, 0, 2 * tile, 0, c, landFull(c));
      } else {
        const int slab = tile / p.ntile, b = slab / p.H, h = slab - b * p.H, col0 = (tile - slab * p.ntile) * (16 / (HALVES ? HALVES : 1));
        for (int half = 0; half < HALVES; ++half)
          tma_load_5d(smem_u32(smem) + C::land_slot(c) * k64Chunk + half * 8192, &tm_in, col0, 8 * c, 64 * half, h, b, landFull(c));
      }
    };
    auto load_gate = [&](int tile, int it) {                     // units: gate table and row factors of (head, k1)
      const int gi = tile / p.ntile;
      mbar_expect_tx(gFull, 16384 + 1024);
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                   :: "r"(smem_u32(Gsm)), "l"(p.gimg + (size_t)gi * 16384), "r"(16384), "r"(gFull) : "memory");
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                   :: "r"(smem_u32(Rtw) + 1024 * (it & 1)), "l"(p.twr + 128 * (gi % p.R)), "r"(1024), "r"(gFull) : "memory");
    };
    int gates = 0;                                               // units: gate tables asked for
    int it = 0, loaded = 0;                                      // loaded: chunks asked for so far
    if ((int)blockIdx.x < p.total && ok)
      for (int c = 0; c < 8; ++c, ++loaded)
        if (T == 0) load(blockIdx.x, c);
    if (C::kUnits && (int)blockIdx.x < p.total && ok) {
      if (T == 0) load_gate(blockIdx.x, 0);
      ++gates;
    }
    for (int tile = blockIdx.x; tile < p.total; tile += gridDim.x, ++it) {
      const int next = tile + (int)gridDim.x;
      const bool more = next < p.total;
      for (int c = 0; c < C::kRing && more; ++c) {
        warp_wait(ok, landFree(c), it & 1);
        if (ok) {
          if (T == 0) load(next, c);
          ++loaded;
        }
      }
      if (C::kUnits && more) {
        warp_wait(ok, gFree, it & 1);
        if (ok) {
          if (T == 0) load_gate(next, it + 1);
          ++gates;
        }
      }
      for (int c = 0; c < 8; ++c) {
        warp_wait(ok, stFull(c), it & 1);
        if (!ok) break;
        if (T == 0) {
          if constexpr (C::kUnits) {                             // 8 KB of each unit's result
            for (int u = 0; u < 2; ++u)
              asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
                           :: "l"(&tm_out), "r"(0), "r"((2 * tile + u) * 1024 + 128 * c), "r"(smem_u32(Op) + c * k64Chunk + u * 8192) : "memory");
          } else {
            const int slab = tile / p.ntile, b = slab / p.H, h = slab - b * p.H, col0 = (tile - slab * p.ntile) * (16 / (HALVES ? HALVES : 1));
            for (int half = 0; half < HALVES; ++half) tma_store_5d(&tm_out, col0, 64 * half, 8 * c, h, b, smem_u32(Op) + c * k64Chunk + half * 8192);
          }
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
          if (c < 7) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
          else asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        }
        if (more && c >= 1 && c <= 8 - C::kRing) {               // chunk c - 1 has been read: rows may land there
          if (T == 0) load(next, c - 1 + C::kRing);
          ++loaded;
        }
        __syncwarp();
      }
      if (ok && T == 0) mbar_arrive(opFree);
    }
    if (T == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    if (!ok)                                                     // do not leave with copies in flight (bounded again)
    {
      for (int i = loaded > 8 ? loaded - 8 : 0; i < loaded; ++i) mbar_wait(landFull(i & 7), (i >> 3) & 1);
      if (gates) mbar_wait(gFull, (gates - 1) & 1);
    }
  } else if (warp == k64Warps) {
    // ---- MMAs, in the order of the jobs ----
    const uint32_t one = elect_one();
    const uint32_t f0 = smem_u32(Fsm), op0 = smem_u32(Op);
    int job = 0, buf = 0, y = 0;
    uint32_t jpar = 1;                                           // parity of the accumulators' last round
    auto begin = [&]() {                                         // the accumulator of the next job is free
      if (job >= 4) warp_wait(ok, accFree(buf), jpar);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      return tmem + k64TmAcc + 64 * buf;
    };
    auto finish = [&]() {
      if (ok) mma_commit(one, accFull(buf));
      ++job;
      if (++buf == 4) { buf = 0; jpar ^= 1; }
    };
    auto stage0 = [&](int c, int it) {
      warp_wait(ok, C::kUnits ? landFull(c) : convFull(c), it & 1);
      const uint32_t d = begin(), b0 = op0 + C::land_slot(c) * k64Chunk;
      if (ok) {
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
          if (HALVES != 2) {
            mma_ss(one, d, umma_desc(f0 + ks * 256, 128, 2048), umma_desc(b0 + ks * 2048, 1024, 128), idesc_f16(64), ks > 0);
          } else {
            mma_ss(one, d, umma_desc(f0 + ks * 256, 128, 2048), umma_desc(b0 + ks * 1024, 512, 128), idesc_f16(32), ks > 0);
            mma_ss(one, d + 32, umma_desc(f0 + ks * 256, 128, 2048), umma_desc(b0 + 8192 + ks * 1024, 512, 128), idesc_f16(32), ks > 0);
          }
        }
      }
      finish();
      if (ok && c < C::kRing) mma_commit(one, landFree(c));
    };
    auto stage12 = [&](int G) {
      if (y >= 2) warp_wait(ok, yFree(y & 1), ((y >> 1) - 1) & 1);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t d = tmem + k64TmAcc + 128 * (y & 1);
      if (ok) {
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) mma_ts(one, d, tmem + 32 * ks + 8 * G, umma_desc(f0 + ks * 256, 128, 2048), idesc_f16(128), ks > 0);
        mma_commit(one, yFull(y & 1));
      }
      ++y;
    };
    auto stage3 = [&](int c) {
      const uint32_t d = begin(), b0 = op0 + c * k64Chunk;
      if (ok) {
#pragma unroll
        for (int ks = 0; ks < 8; ++ks)
          mma_ss(one, d, umma_desc(f0 + ks * 256, 128, 2048), umma_desc_k_sw128(b0 + (ks >> 2) * 8192 + (ks & 3) * 32, 1024), idesc_f16(64), ks > 0);
      }
      finish();
    };
    warp_wait(ok, fFull, 0);
    int it = 0;
    for (int tile = blockIdx.x; tile < p.total && ok; tile += gridDim.x, ++it) {
      if (it == 0)
        for (int c = 0; c < 8; ++c) stage0(c, 0);
      warp_wait(ok, aFull, it & 1);
      for (int e = 0; e < 4; ++e) stage12(C::group(e));
      for (int e = 0; e < 4; ++e) {
        warp_wait(ok, a2Full(C::group(e)), it & 1);
        stage12(C::group(e));
      }
      warp_wait(ok, opFull, it & 1);
      const bool more = tile + (int)gridDim.x < p.total;
      for (int k = -4; k < 8; ++k) {                             // the last stage runs four chunks ahead of the next tile's first one
        if (k + 4 < 8) stage3(k + 4);
        if (more && k >= 0) stage0(k, it + 1);
      }
    }
  } else if (warp > k64Warps) {
    // ---- gates of a tile (two warps), normalised by a bound on max |g|, as fp16 (Re, Im) of bin k1 + 64 k2 < n/2 at [k2 (32)][k1];
    //      the other bins are their mirrors (row 32 holds the Nyquist bin for k1 = 0).  n = 8192: two tables, of the even and of the odd bins ----
    const int id = tid - k64Threads + 64;
    int it = 0;
    for (int tile = blockIdx.x; !C::kUnits && tile < p.total; tile += gridDim.x, ++it) {
      const float2* g = p.g + (size_t)(tile / p.ntile) * (C::n / 2 + 1);
      float m = id == 0 ? fabsf(g[C::n / 2].x) : 0.f;
#pragma unroll 1
      for (int k = id; k < C::n / 2; k += 8 * 64) {
        float2 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = g[k + 64 * u];
        if (k == 0) v[0].y = 0.f;
#pragma unroll
        for (int u = 0; u < 8; ++u) m = fmaxf(m, fmaxf(fabsf(v[u].x), fabsf(v[u].y)));
      }
      for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      if (T == 0) gmax[2 + (id >> 5)] = m;
      asm volatile("bar.sync 1, 64;" ::: "memory");
      m = 1.41421356f * fmaxf(gmax[2], gmax[3]);
      const float inv = m > 0.f ? 1.0f / m : 0.f;
      if (it > 0) warp_wait(ok, gFree, (it - 1) & 1);
#pragma unroll 1
      for (int k = id; k < C::n / 2; k += 8 * 64) {
        float2 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = g[k + 64 * u];
        if (k == 0) v[0].y = 0.f;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int kk = k + 64 * u;
          Gsm[HALVES == 2 ? (kk & 1) * k64Rows * 64 + (kk >> 1) : kk] = pack_h2(v[u].x * inv, v[u].y * inv);
        }
      }
      if (id == 0) {
        Gsm[2048] = pack_h2(g[C::n / 2].x * inv, 0.f);
        gmax[it & 1] = m;
      }
      asm volatile("bar.sync 1, 64;" ::: "memory");
      if (T == 0 && ok) mbar_arrive(gFull);
    }
  } else if (warp < k64Warps) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" :: "n"(k64EpiRegs));
    // ---- epilogue warps: set = chunk / group parity, TMEM lane quadrant q, j = lane half (stages 0, 3) or column half (1, 2) ----
    const int set = warp >> 3, w8 = warp & 7, q = w8 & 3, j = w8 >> 2;
    const int i = T >> 2, tq = T & 3;
    const uint32_t lane0 = (uint32_t)(32 * q) << 16, lane16 = lane0 + ((uint32_t)(16 * j) << 16);
    const int kr = 8 * (2 * q + j) + i;                          // stages 0, 3: this thread's row digit
    const int kl = 16 * q + 8 * (T >> 4) + (T & 7), bl = (T >> 3) & 1;   // stages 1, 2: this thread's lane (k1, b)
    const float2 wconv = twiddle_fwd((unsigned)(256 * (2 * w8 + (T >> 4)) + (T & 7)), 8192u);   // n = 8192: W_8192^{256 a + t2}
    const float2 wout = twiddle_fwd((unsigned)kr, 128u);                                        // and W_8192^{64 s1}
    auto acc = [&](int job) { return tmem + k64TmAcc + 64 * (job & 3); };
    auto wait_acc = [&](int job) {
      warp_wait(ok, accFull(job & 3), (job >> 2) & 1);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    };
    auto free_acc = [&](int job) {                               // after tcgen05.wait::ld
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (T == 0) mbar_arrive(accFree(job & 3));
    };
    auto to_h2 = [](uint32_t w) {
      if (F16) return w;
      const float2 f = unpack_bf2(w);
      return pack_h2(f.x, f.y);
    };
    auto at = [](const uint4& v, int e) { return e == 0 ? v.x : (e == 1 ? v.y : (e == 2 ? v.z : v.w)); };
    // rows of a chunk -> stage 0's operand, in place: four rows t1 = 4 a .. 4 a + 3 at one t2 in, four K groups out
    auto convert = [&](int tile, int c, int it) {
      if constexpr (C::kUnits) return;
      const int t2l = T & 7, a = 2 * w8 + (T >> 4);
      warp_wait(ok, landFull(c), it & 1);
      unsigned char* ring = smem + C::land_slot(c) * k64Chunk;
      if (HALVES == 1) {
        // 16-byte half of the 32-byte piece; the lanes of a phase alternate between the halves, which keeps them off each other's banks
        const int hf = ((T >> 3) & 1) ^ (t2l >> 2);
        unsigned char* p0 = ring + a * 1024 + t2l * 32 + hf * 16;
        uint4 r[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) r[u] = *reinterpret_cast<const uint4*>(p0 + 256 * u);
        const int lb = p.L >> 6, lr = p.L & 63;
        const int slab = tile / p.ntile, col = (tile - slab * p.ntile) * 16 + 8 * hf;
        if ((lb >> 2) == a && 8 * c + t2l < lr && col < p.D) {   // a row of the partial block
          const int b = slab / p.H, h = slab - b * p.H;
          const uint4 v = *reinterpret_cast<const uint4*>(reinterpret_cast<const __half*>(p.src) + b * p.s_sb +
                                                          (int64_t)(64 * lb + 8 * c + t2l) * p.s_sl + h * p.s_sh + col);
          if ((lb & 3) == 0) r[0] = v;
          else if ((lb & 3) == 1) r[1] = v;
          else if ((lb & 3) == 2) r[2] = v;
          else r[3] = v;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e)
          *reinterpret_cast<uint4*>(p0 + 256 * e) = make_uint4(to_h2(at(r[0], e)), to_h2(at(r[1], e)), to_h2(at(r[2], e)), to_h2(at(r[3], e)));
      } else {
        // radix-2 step: a lane takes two of the four pairs, the even bins' inputs into the lower half, the odd ones' into the upper
        const int hp = (T >> 3) & 1;
        unsigned char* p0 = ring + a * 512 + t2l * 16;
        uint2 lo[4], hi[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          lo[u] = *reinterpret_cast<const uint2*>(p0 + 128 * u + 8 * hp);
          hi[u] = *reinterpret_cast<const uint2*>(p0 + 8192 + 128 * u + 8 * hp);
        }
        const float2 w0 = cmul(wconv, W8[c]);
        const float2 w64[4] = {make_float2(1.f, 0.f), make_float2(0.998795456f, -0.049067674f),
                               make_float2(0.995184727f, -0.098017140f), make_float2(0.989176510f, -0.146730474f)};
        float2 w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) w[u] = cmul(w0, w64[u]);
        __syncwarp();                                            // every lane has read: the slots may be written
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          uint32_t ev[4], od[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const uint32_t ua = e ? lo[u].y : lo[u].x, ub = e ? hi[u].y : hi[u].x;
            const float2 va = F16 ? unpack_h2(ua) : unpack_bf2(ua), vb = F16 ? unpack_h2(ub) : unpack_bf2(ub);
            const float2 s = cadd(va, vb), d = cmul(csub(va, vb), w[u]);
            ev[u] = pack_h2(s.x, s.y);
            od[u] = pack_h2(d.x, d.y);
          }
          unsigned char* out = p0 + 128 * (2 * hp + e);
          *reinterpret_cast<uint4*>(out) = make_uint4(ev[0], ev[1], ev[2], ev[3]);
          *reinterpret_cast<uint4*>(out + 8192) = make_uint4(od[0], od[1], od[2], od[3]);
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (T == 0 && ok) mbar_arrive(convFull(c));
    };
    // stage 0's result of chunk c, times W_4096^{k1 t2}, to the A operand
    auto epilogue0 = [&](int c, int job) {
      float2 w[2];
      const float2 w8c = T8[c * 64 + kr];
#pragma unroll
      for (int e = 0; e < 2; ++e) w[e] = cmul(w8c, T1[(HALVES == 1 ? 4 * e + tq : 2 * tq + e) * 64 + kr]);     // t2 = 8 c + ...
      wait_acc(job);
      uint32_t r[32], o[16];
      tmem_ld_16x256b_x8(acc(job) + lane16, r);
      tmem_ld_wait();
      free_acc(job);
#pragma unroll
      for (int x = 0; x < 8; ++x) {
        const uint64_t RE = pk2u(r[4 * x], r[4 * x + 1]), IM = pk2u(r[4 * x + 2], r[4 * x + 3]);
        float X[2], Y[2];
        if (HALVES == 1) {                                       // column group x = (G, t2 / 4): registers (b), one t2
          const float2 v = w[x & 1];
          cmul2(RE, IM, pk2(v.x, v.x), pk2(v.y, v.y), pk2(-v.y, -v.y), X, Y);
          o[2 * x] = pack_h2(X[0], Y[0]);
          o[2 * x + 1] = pack_h2(X[1], Y[1]);
        } else {                                                 // column group x = (half, pair): registers two t2
          const int pr = x & 3, G = 2 * (pr & 1) + (x >> 2);
          cmul2(RE, IM, pk2(w[0].x, w[1].x), pk2(w[0].y, w[1].y), pk2(-w[0].y, -w[1].y), X, Y);
          o[4 * G + 2 * (pr >> 1)] = pack_h2(X[0], Y[0]);
          o[4 * G + 2 * (pr >> 1) + 1] = pack_h2(X[1], Y[1]);
        }
      }
      const uint32_t ta = tmem + 32 * c + lane16;
      if (HALVES == 1) SPECTRE_ST16("16x128b.x8", ta, o);
      else SPECTRE_ST16("16x256b.x4", ta, o);
      tmem_st_wait();
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (T == 0 && ok) mbar_arrive(aFull);
    };
    // Stages 1 and 2: the set takes its half of every group, so that a thread's gates and twiddles (16 digits) stay in registers.
    // Stage 1's result: times the gate; (-Re, Im) = - the conjugate goes on as the next A operand, in place
    auto yacc = [&](int y) { return tmem + k64TmAcc + 128 * (y & 1) + 64 * set + 32 * j + lane0; };
    // A group's accumulator is given back as soon as it is in registers, so that the MMAs are a group ahead of the arithmetic.
    auto take_y = [&](int y, uint32_t (&r)[2][16]) {
      warp_wait(ok, yFull(y & 1), (y >> 1) & 1);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      tmem_ld_32x32b_x16(yacc(y), r[0]);
      tmem_ld_32x32b_x16(yacc(y) + 16, r[1]);
      tmem_ld_wait();
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (T == 0) mbar_arrive(yFree(y & 1));
    };
    auto epilogue1 = [&](int it) {
      uint64_t GX[8], GY[8];
      uint32_t r[2][16];
      warp_wait(ok, gFull, it & 1);
#pragma unroll 1
      for (int e = 0; e < 4; ++e) {
        const int G = C::group(e);
        if (e == 0 || (HALVES == 2 && e == 2)) {
          if constexpr (C::kUnits) {                             // the image's order: bin k1 + 64 k2 at 64 k2 + (k1 ^ 8 (k2 % 4))
            const uint32_t* tab = Gsm + 64 * (32 * set + 16 * j);
#pragma unroll
            for (int m = 0; m < 8; ++m) {
              const float2 a = unpack_h2(tab[128 * m + (kl ^ (8 * ((2 * m) & 3)))]), b = unpack_h2(tab[128 * m + 64 + (kl ^ (8 * ((2 * m + 1) & 3)))]);
              GX[m] = pk2(a.x, b.x);
              GY[m] = pk2(a.y, b.y);
            }
          } else {
            // set 1 holds the upper half of the digits: mirrored bins
            const int half = HALVES == 2 ? G & 1 : 0;
            const int col = set ? (half ? 63 - kl : (64 - kl) & 63) : kl, row0 = set ? 31 - 16 * j + (half == 0 && kl == 0) : 16 * j;
            const uint32_t* tab = Gsm + half * k64Rows * 64 + col;
            const float sg = set ? -1.f : 1.f;
#pragma unroll
            for (int m = 0; m < 8; ++m) {
              const float2 a = unpack_h2(tab[(row0 + (set ? -2 * m : 2 * m)) * 64]), b = unpack_h2(tab[(row0 + (set ? -2 * m - 1 : 2 * m + 1)) * 64]);
              GX[m] = pk2(a.x, b.x);
              GY[m] = pk2(sg * a.y, sg * b.y);
            }
          }
        }
        take_y(8 * it + e, r);                                   // the job is done: its operand may be overwritten, too
        const uint32_t ta = tmem + 32 * (4 * set + 2 * j) + 8 * G + lane0;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          uint32_t o[8];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int m = 4 * half + u;
            const uint64_t RE = pk2u(r[half][2 * u], r[half][2 * u + 1]), IM = pk2u(r[half][8 + 2 * u], r[half][9 + 2 * u]);
            float X[2], Y[2];
            upk2(sub2(mul2(IM, GY[m]), mul2(RE, GX[m])), X[0], X[1]);
            upk2(fma2(IM, GX[m], mul2(RE, GY[m])), Y[0], Y[1]);
            o[2 * u] = pack_h2(X[0], Y[0]);
            o[2 * u + 1] = pack_h2(X[1], Y[1]);
          }
          tmem_st_32x32b_x8(ta + 32 * half, o);
        }
        tmem_st_wait();
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (T == 0 && ok) mbar_arrive(a2Full(G));
      }
      if (T == 0 && ok) mbar_arrive(gFree);
    };
    // stage 2's result, times W_4096^{k1 s2}: stage 3's operand, row 8 (s2 % 8) + problem of chunk s2 / 8, K = k1
    auto epilogue2 = [&](int it) {
      uint64_t WX[8], WY[8];
      uint32_t r[2][16];
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const float2 w8c = T8[(4 * set + 2 * j + half) * 64 + kl];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float2 a = cmul(w8c, T1[2 * u * 64 + kl]), b = cmul(w8c, T1[(2 * u + 1) * 64 + kl]);
          WX[4 * half + u] = pk2(a.x, b.x);
          WY[4 * half + u] = pk2(a.y, b.y);
        }
      }
      if (it > 0) warp_wait(ok, opFree, (it - 1) & 1);           // the last tile's results have left
#pragma unroll 1
      for (int e = 0; e < 4; ++e) {
        const int row = 4 * bl + C::group(e);
        unsigned char* base = Op + (4 * set + 2 * j) * k64Chunk + (kl >> 5) * 8192 + row * 128 + ((((kl & 31) >> 2) ^ row) << 4) + (kl & 3) * 4;
        take_y(8 * it + 4 + e, r);
#pragma unroll
        for (int half = 0; half < 2; ++half) {
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int m = 4 * half + u;
            const uint64_t RE = pk2u(r[half][2 * u], r[half][2 * u + 1]), IM = pk2u(r[half][8 + 2 * u], r[half][9 + 2 * u]);
            float X[2], Y[2];
            upk2(sub2(mul2(RE, WX[m]), mul2(IM, WY[m])), X[0], X[1]);
            upk2(fma2(IM, WX[m], mul2(RE, WY[m])), Y[0], Y[1]);
            unsigned char* out = base + half * k64Chunk + 2 * u * 1024;
            *reinterpret_cast<uint32_t*>(out) = pack_h2(X[0], Y[0]);
            *reinterpret_cast<uint32_t*>(out + 1024) = pack_h2(X[1], Y[1]);
          }
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    };
    bool bad = false;
    // stage 3's result of chunk c: rows 64 s1 + 8 c + x, conjugated and scaled, staged in the chunk's own space and stored
    auto epilogue3 = [&](int tile, int c, int job, float gs) {
      if constexpr (C::kUnits) return;
      float2 w[2];
      if (HALVES == 2) {
        w[0] = cscale(cmul(wout, W8[c]), gs);                    // W_8192^{64 s1 + 8 c}
        w[1] = cmul(w[0], make_float2(0.99999529380957617f, -0.0030679567629659761f));
      }
      wait_acc(job);
      uint32_t r[32];
      tmem_ld_16x256b_x8(acc(job) + lane16, r);
      tmem_ld_wait();
      free_acc(job);
      unsigned char* stg = Op + c * k64Chunk;
      const int lb = p.L >> 6, lr = (p.L & 63) - 8 * c;
      const bool part = HALVES == 1 && kr == lb && lr > 0;      // a row of the partial block
      constexpr float kStepX = 0.9999997058628822f, kStepY = -0.0007669903187427045f;     // W_8192
#pragma unroll
      for (int x = 0; x < 8; ++x) {
        float re[2] = {__uint_as_float(r[4 * x]), __uint_as_float(r[4 * x + 1])};
        float im[2] = {__uint_as_float(r[4 * x + 2]), __uint_as_float(r[4 * x + 3])};
        uint32_t o[2];
        if (HALVES == 2) {                                       // (even, odd) -> rows t and t + 4096
          const float2 v = cmul(make_float2(re[1], im[1]), w[x >> 2]);      // scaled with w
          if (x != 3 && x != 7) w[x >> 2] = cmul(w[x >> 2], make_float2(kStepX, kStepY));
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const float a = fmaf(gs, re[0], e ? -v.x : v.x), b = fmaf(-gs, im[0], e ? v.y : -v.y);
            o[e] = F16 ? pack_h2(a, b) : pack_bf2(a, b);
          }
        } else {
#pragma unroll
          for (int e = 0; e < 2; ++e) o[e] = F16 ? pack_h2(gs * re[e], -gs * im[e]) : pack_bf2(gs * re[e], -gs * im[e]);
        }
        // an overflow anywhere in a column makes every row of it non-finite: one row per thread is enough
        if (x == 0) bad |= nonfinite16x2<F16>(o[0]) | nonfinite16x2<F16>(o[1]);
        if (HALVES == 1) {                                       // [s2 % 8][s1][32 bytes]
          *reinterpret_cast<uint2*>(stg + x * 2048 + kr * 32 + tq * 8) = make_uint2(o[0], o[1]);
          if (part && x < lr) {
            const int slab = tile / p.ntile, b = slab / p.H, h = slab - b * p.H, col = (tile - slab * p.ntile) * 16 + 4 * tq;
            if (col < p.D)
              *reinterpret_cast<uint2*>(reinterpret_cast<__half*>(p.dst) + b * p.d_sb + (int64_t)(64 * lb + 8 * c + x) * p.d_sl + h * p.d_sh + col) =
                  make_uint2(o[0], o[1]);
          }
        } else {                                                 // [half of the rows][s2 % 8][s1][16 bytes]
          *reinterpret_cast<uint32_t*>(stg + x * 1024 + kr * 16 + tq * 4) = o[0];
          *reinterpret_cast<uint32_t*>(stg + 8192 + x * 1024 + kr * 16 + tq * 4) = o[1];
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (T == 0 && ok) mbar_arrive(stFull(c));
    };

    // Units: times W_n^{k1 t'}, conjugated and scaled, as fp16 rows of 4 pairs in unit_row_slot's order (mixer_tc4k.cu): 64 bytes hold
    // s2 % 4 = 0 ... 3 of a (s2 / 4, s1), swizzled as the tensor map unswizzles them
    auto epilogue3_units = [&](int c, int job, float gs, const float2* rtw) {
      const float2 fa = cscale(rtw[kr], gs);
      float2 fb[8];
#pragma unroll
      for (int x = 0; x < 8; ++x) fb[x] = rtw[64 + 8 * c + x];
      wait_acc(job);
      uint32_t r[32];
      tmem_ld_16x256b_x8(acc(job) + lane16, r);
      tmem_ld_wait();
      free_acc(job);
      unsigned char* stg = Op + c * k64Chunk + kr * 64 + tq * 4;
#pragma unroll
      for (int x = 0; x < 8; ++x) {                              // registers: pair tq of the two units
        const float2 w = cmul(fa, fb[x]);
        const uint64_t RE = pk2u(r[4 * x], r[4 * x + 1]), IM = pk2u(r[4 * x + 2], r[4 * x + 3]);
        const uint64_t WX = pk2(w.x, w.x), NWY = pk2(-w.y, -w.y);
        float X[2], Y[2];
        upk2(fma2(IM, NWY, mul2(RE, WX)), X[0], X[1]);
        upk2(sub2(mul2(RE, NWY), mul2(IM, WX)), Y[0], Y[1]);
        unsigned char* out = stg + (x >> 2) * 4096 + (((x & 3) ^ ((kr >> 1) & 3)) << 4);
        *reinterpret_cast<uint32_t*>(out) = pack_h2(X[0], Y[0]);
        *reinterpret_cast<uint32_t*>(out + 8192) = pack_h2(X[1], Y[1]);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (T == 0 && ok) mbar_arrive(stFull(c));
    };

    // Last stage of tile `tile` side by side with the first one of `next`, then the middle stages of `next`.  The job numbers
    // follow the MMA warp's order.
    int job = 0, it = 0, tile = -1, next = blockIdx.x;
    float gunit = 0.f;
#pragma unroll 1
    while (tile >= 0 || next < p.total) {
      const bool last = tile >= 0, first = next < p.total;
      const float gs = !last ? 0.f : C::kUnits ? gunit : (HALVES == 2 ? -0.5f : -1.f) * gmax[(it - 1) & 1];     // the sign of epilogue 1
#pragma unroll 1
      for (int k = set - (last ? 4 : 2); k < 8; k += 2) {       // rows are converted one of the set's chunks ahead
        if (last && k + 4 < 8) {
          const int jb = !first ? job + k + 4 : (k < 0 ? job + k + 4 : job + 2 * k + 4);
          if constexpr (C::kUnits) epilogue3_units(k + 4, jb, gs, Rtw + 128 * ((it - 1) & 1));
          else epilogue3(tile, k + 4, jb, gs);
        }
        if (!first) continue;
        if (k + 2 >= 0 && k + 2 < 8) convert(next, k + 2, it);
        if (k >= 0) epilogue0(k, !last ? job + k : (k < 4 ? job + 5 + 2 * k : job + 8 + k));
      }
      if (!first) break;
      job += last ? 16 : 8;
      if constexpr (C::kUnits) gunit = -p.out_scale * p.gscale[next / p.ntile];      // for the tile's last stage
      epilogue1(it);
      epilogue2(it);
      __syncwarp();
      if (T == 0 && ok) mbar_arrive(opFull);
      ++it;
      tile = next;
      next += gridDim.x;
    }
    if (__any_sync(0xffffffffu, bad) && T == 0) report_range(p.status);
  }
  if (!ok && T == 0) report_timeout(p.status);
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == k64Warps) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(512));
  }
}

// ---- host side ----
// The tensor maps need 16-byte aligned bases and strides; n = 4096 at least one whole block of 64 rows, n = 8192 whole blocks only.
static bool tc64_act_ok(const spectre_act* a) {
  return (reinterpret_cast<uintptr_t>(a->ptr) & 15) == 0 && a->stride_l % 8 == 0 && a->stride_h % 8 == 0 && a->stride_b % 8 == 0 &&
         a->stride_l > 0 && a->stride_h > 0 && a->stride_b > 0;
}
bool tc4096_supported(const spectre_act* v, const spectre_act* y) {
  return v->L >= 64 && v->D % 8 == 0 && tc64_act_ok(v) && tc64_act_ok(y) && tensor_map_encoder() != nullptr;
}
bool tc8192_supported(const spectre_act* v, const spectre_act* y) {
  return v->L % 64 == 0 && v->D % 8 == 0 && tc64_act_ok(v) && tc64_act_ok(y) && tensor_map_encoder() != nullptr;
}

// dims (column, row digits, head, batch) of the whole 64-row blocks, the digits as (t2, t1) for loads and (t1, t2) for stores:
// a box lands as [t1][t2][piece] and leaves as [t2][t1][piece]
static int make_map64(CUtensorMap* tm, const spectre_act* a, bool out, unsigned cols) {
  const cuuint64_t sl = (cuuint64_t)a->stride_l * 2, sh = (cuuint64_t)a->stride_h * 2, sb = (cuuint64_t)a->stride_b * 2;
  const cuuint64_t nb = (cuuint64_t)(a->L / 64);
  const cuuint64_t dims[5] = {(cuuint64_t)a->D, out ? nb : 64, out ? 64 : nb, (cuuint64_t)a->H, (cuuint64_t)a->B};
  const cuuint64_t strides[4] = {out ? 64 * sl : sl, out ? sl : 64 * sl, sh, sb};
  const cuuint32_t box[5] = {cols, out ? 64u : 8u, out ? 8u : 64u, 1, 1}, es[5] = {1, 1, 1, 1, 1};
  const CUresult r = tensor_map_encoder()(
      tm, a->dtype == SPECTRE_F16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, a->ptr, dims, strides, box, es,
      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(SPECTRE_ERR_CUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
  return SPECTRE_OK;
}

template <bool F16, int HALVES>
static int launch_tc64(const spectre_ctx* ctx, cudaStream_t st, const spectre_act* v, const float* g, const spectre_act* y) {
  constexpr int kCols = 16 / HALVES;
  CUtensorMap tm_in, tm_out;
  int rc = make_map64(&tm_in, v, false, kCols);
  if (rc == SPECTRE_OK) rc = make_map64(&tm_out, y, true, kCols);
  if (rc != SPECTRE_OK) return rc;
  Tc64Params p = {};
  p.g = reinterpret_cast<const float2*>(g);
  p.F = reinterpret_cast<const __half*>(ctx->dft64);
  p.src = v->ptr; p.s_sb = v->stride_b; p.s_sl = v->stride_l; p.s_sh = v->stride_h;
  p.dst = y->ptr; p.d_sb = y->stride_b; p.d_sl = y->stride_l; p.d_sh = y->stride_h;
  p.H = v->H; p.ntile = (v->D + kCols - 1) / kCols; p.L = v->L; p.D = v->D;
  p.total = v->B * v->H * p.ntile;
  p.status = ctx->status_dev;
  auto kern = mixer_tc64_kernel<F16, HALVES>;
  SPECTRE_CUDA_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Tc64<HALVES>::kSmem));
  SPECTRE_CUDA_OK(launch_after(kern, p.total < ctx->sm_count ? p.total : ctx->sm_count, k64Threads, Tc64<HALVES>::kSmem, st, tm_in, tm_out, p));
  return SPECTRE_OK;
}
int launch_mixer_pairs4096(const spectre_ctx* ctx, cudaStream_t st, const spectre_act* v, const float* g, const spectre_act* y);   // mixer_tc4096.cu
// Half-width tiles (4 column pairs, mixer_tc4096.cu) or whole ones, whichever the counts of both let expect to be done first.  An SM holds two
// half tiles at once and takes 21 us for a pair, 13.5 for one that is left alone; it takes 13 for a whole tile, 0.75 more for each
// chunk of 8 rows of a partial block (the whole tile fetches them one by one) and 0.5 more for tiles that reach beyond D.  The numbers are
// fitted, in quarters of a microsecond, to 1294 mixer calls of 4 ... 600 heads of 8 ... 128 channels, 1024 ... 4096 rows: the choice costs 0.16 per
// cent of the better kernel's time on average and 7 at most (fewer rows go the same way but for calls of 8 heads and 64 ... 100 rows, 21.0 | 16.0 ...
// 21.0, where 2 and 18 heads take 16.0 and 15.3).  Some of them, us, half | whole: 64 channels, whole blocks, 18 heads 15.3 | 16.1,
// 19 heads 20.8 | 16.2, 38 heads 34.7 | 29.2, 64 heads 40.9 | 30.0; 20 rows beyond, 16 heads 15.6 | 18.9, 24 heads 22.0 | 19.2, 48 heads 36.4 | 35.2, 64 heads
// 42.0 | 35.6; 40 rows, 24 heads 22.1 | 22.3, 48 heads 36.5 | 41.0, 256 heads 161.8 | 138.2; 63 rows, 64 heads 42.4 | 45.9, 256 heads 161.8 | 145.5;
// 8 channels (a whole tile is half empty), 149 heads 20.7 | 30.5.
int launch_mixer_tc4096(const spectre_ctx* ctx, cudaStream_t st, const spectre_act* v, const float* g, const spectre_act* y) {
  const long long slabs = (long long)v->B * v->H, sms = ctx->sm_count;
  const long long half = (slabs * (v->D / 8) + sms - 1) / sms, whole = (slabs * ((v->D + 15) / 16) + sms - 1) / sms;      // the fullest SM's share
  const int chunks = (v->L % 64 + 7) / 8;
  if (42 * half + 12 * (half & 1) <= 16 + whole * (52 + 3 * chunks + (v->D % 16 ? 2 : 0))) return launch_mixer_pairs4096(ctx, st, v, g, y);
  return v->dtype == SPECTRE_F16 ? launch_tc64<true, 1>(ctx, st, v, g, y) : launch_tc64<false, 1>(ctx, st, v, g, y);
}
int launch_mixer_tc8192(const spectre_ctx* ctx, cudaStream_t st, const spectre_act* v, const float* g, const spectre_act* y) {
  return v->dtype == SPECTRE_F16 ? launch_tc64<true, 2>(ctx, st, v, g, y) : launch_tc64<false, 2>(ctx, st, v, g, y);
}

// The 4096-point units of a longer transform (mixer_tc4k.cu), two adjacent ones (eight column pairs of one head and k1) a tile: first
// operands from the images that the radix-R step wrote, results in their place in the workspace.
int launch_units_tc64(const spectre_ctx* ctx, cudaStream_t st, const unsigned char* ws_in, const unsigned char* gimg, const float* gscale,
                      unsigned char* ws_out, int nunits, int ntile, int R, float out_scale) {
  // an image is [K group a (16)][pair (4)][t2 (64)][16 bytes]; a chunk takes 8 t2 of both units
  const cuuint64_t dims[5] = {64, 4, (cuuint64_t)nunits, 16, 8}, strides[4] = {1024, 65536, 4096, 128};
  const cuuint32_t box[5] = {64, 4, 2, 16, 1}, es[5] = {1, 1, 1, 1, 1};
  const cuuint64_t odims[2] = {32, (cuuint64_t)nunits * 1024}, ostrides[1] = {64};
  const cuuint32_t obox[2] = {32, 128};
  CUtensorMap tm_in, tm_out;
  CUresult r = tensor_map_encoder()(&tm_in, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 5, const_cast<unsigned char*>(ws_in), dims, strides, box, es,
                                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r == CUDA_SUCCESS)
    r = tensor_map_encoder()(&tm_out, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, ws_out, odims, ostrides, obox, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                             CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(SPECTRE_ERR_CUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
  Tc64Params p = {};
  p.F = reinterpret_cast<const __half*>(ctx->dft64);
  p.ntile = ntile / 2;
  p.total = nunits / 2;
  p.status = ctx->status_dev;
  p.gimg = gimg; p.gscale = gscale; p.R = R; p.out_scale = out_scale;
  p.twr = reinterpret_cast<const float2*>(ctx->tw_staged) + (size_t)(R - 1) * 128;
  auto kern = mixer_tc64_kernel<true, 0>;
  SPECTRE_CUDA_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Tc64<0>::kSmem));
  SPECTRE_CUDA_OK(launch_after(kern, p.total < ctx->sm_count ? p.total : ctx->sm_count, k64Threads, Tc64<0>::kSmem, st, tm_in, tm_out, p));
  return SPECTRE_OK;
}

}  // namespace spectre
