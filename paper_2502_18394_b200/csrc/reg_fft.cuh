// Transforms of up to 2048 points per CTA with the points in registers (fp32): decompositions, parameters and
// the kernel.  Instantiated per activation type in reg_*.cu, launched through the functions of reg_fft.h.
//
// A thread holds 32 points of one column pair (see mixer.cu for the pair packing).  A 1024-point transform is a 32-point
// DFT in registers, one exchange through shared memory and a second 32-point DFT; the spectrum is then still in
// registers, where the gate is applied, and the inverse runs the same steps backwards, so that a point crosses shared
// memory twice in all and global rows move straight from and to registers.  Bound by instruction issue (about 2700 per
// thread and tile, half of them floating point); two CTAs per SM overlap one another's loads and barriers.
// Measured, mixer call at B = 16, H = 12, D = 64, bf16, n = 1024: 86 us on the shared-memory kernel (eleven passes over the
// tile, run-time radices) -> 30 us = 1.7 TB/s of its rows; its backward 287 us (four transforms and a reduction) -> 57 us;
// n = 2048 86 -> 43 us at the same size.
#pragma once
#include <type_traits>

#include "fft_reg.cuh"
#include "reg_fft.h"

namespace spectre {

// Twiddle loads.  Volatile, so that the forward transform's factors are not kept in registers (and spilled) for the
// inverse's use of the same ones.
__device__ __forceinline__ float4 tw_load4(const float4* p) {
  float4 v;
  asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ float2 tw_load2(const float2* p) {
  float2 v;
  asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}
struct TwGlobal {
  const float4* p;
  __device__ __forceinline__ float4 load4(int i) const { return tw_load4(p + i); }
  __device__ __forceinline__ float2 load2(int i) const { return tw_load2(reinterpret_cast<const float2*>(p) + i); }
};
// The same from a copy of the table in shared memory
struct TwShared {
  uint32_t p;
  __device__ __forceinline__ float4 load4(int i) const {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(p + 16u * (uint32_t)i));
    return v;
  }
  __device__ __forceinline__ float2 load2(int i) const {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(p + 8u * (uint32_t)i));
    return v;
  }
};

// Keeps the work in front of this point in front of it: without it the compiler interleaves the end of the forward
// transform with the start of the inverse one and runs out of registers.
template <int E> __device__ __forceinline__ void settle(float2 (&x)[E]) {
#pragma unroll
  for (int i = 0; i < E; ++i) asm volatile("" : "+f"(x[i].x), "+f"(x[i].y));
}
template <int E> __device__ __forceinline__ void settle(cx2 (&x)[E]) {
#pragma unroll
  for (int i = 0; i < E; ++i) asm volatile("" : "+l"(x[i].x), "+l"(x[i].y));
}

enum RegMode { kRegMix = 0, kRegForward = 1, kRegInverse = 2, kRegGrad = 3 };

// n = R1 R2 in two steps (R1 a multiple of R2): j = j1 R2 + j2, k = k1 + R1 k2.  Thread (pair p, m): the R1-point DFT
// over j1 at j2 = m, then R1 / R2 DFTs of R2 points at k1 = m + R2 u.  Rows of the exchange buffer (k1, j2) lie
// R2 + 1 apart per k1: an odd pitch keeps the side whose lanes differ in k1 free of bank conflicts.
// PP: column pairs per thread, neighbours in a row.  Two of them, packed (cx2), take 28 % fewer instructions and half the threads at the
// registers of nearly two.  Forward transforms of 16-bit tokens of 1024 points gain by it with three CTAs of 128 threads at 168 registers
// on an SM (1024 tiles 28.0 -> 25.1 us; prompt of 2 x 20011 of 32768 x 32 heads 928 -> 896, forward and backward of 1 x 8192 x 32
// 183 -> 178), if the exchange buffer is halved: with three whole ones no L1 is left for the loads in flight (40 us).  Mixer and gradient lose
// the latency that twice the warps hide (16 x 1024 x 12 bf16 30.1 -> 32.8 and 57.6 -> 64.1 us), and so do fp32 tokens (prompt of
// 2 x 6000 of 8192 x 8 114 -> 120).
template <int R1, int R2, int C_, int PP_ = 1>
struct TwoStep {
  static constexpr int PP = PP_, C = C_, G = C / PP, M = R1 * R2, E = R1, S = R2, U = R1 / R2;
  typedef typename PointOf<PP>::type V;
  // mix() runs the steps as a loop over one copy of the DFT.  From 32 points on, straight-line code (four DFTs) waits for
  // instructions: 1024 = 32 x 32 at 12.6 M elements takes 35.9 us in the loop against 38.6 (fp32), 27.3 against 30.1 (bf16).
  // 28 x 28 and smaller ones lose 1 - 10 % to its extra barrier and moves, and so does the gradient (55 -> 58 us), whose loop over
  // three transforms carries more state; the forward transform alone gains nothing.
  static constexpr bool kLoop = R1 == R2 && R1 >= 32;
  static constexpr int kActive = S * G, kThreads = (kActive + 31) / 32 * 32;
  static constexpr int kExch = R1 * (R2 + 1) * C;                   // elements of the exchange buffer
  static constexpr int kGate = M, kTw = 0;                       // twiddles in shared memory: none
  static constexpr int kParts = 1, kRed = C, kRedShift = 0;         // pairs side by side in a warp after the transform
  int p, m;
  __device__ __forceinline__ explicit TwoStep(int tid) : p(tid % G), m(tid / G) {}
  __device__ __forceinline__ int pair_in() const { return PP * p; }
  __device__ __forceinline__ int pair_out() const { return PP * p; }
  __device__ __forceinline__ int part() const { return 0; }
  __device__ __forceinline__ int bin(int i) const { return m + S * (i / R2) + R1 * (i % R2); }
  static __device__ __forceinline__ int gate_slot(int k) { return k; }

  // before: called in front of the exchange's (first) barrier
  struct Nothing { __device__ __forceinline__ void operator()() const {} };
  template <bool HALF, class Before = Nothing>
  __device__ __forceinline__ void forward(V (&x)[E], void* buf, const float4* __restrict__ tw, bool act, Before before = Before()) const {
    RegDft<R1, false>::run(x);
    turn<HALF>(x, buf, tw, act, before);
#pragma unroll
    for (int u = 0; u < U; ++u) sub<false>(x, u);
  }
  static __device__ __forceinline__ void swap_parts(V (&x)[E]) {
#pragma unroll
    for (int i = 0; i < E; ++i) x[i] = V{x[i].y, x[i].x};
  }
  // kLoop: forward transform, gate(x), inverse transform.  The inverse is the forward one of the values with real and
  // imaginary parts swapped, its exchange the same one, so all four DFTs are one piece of code.
  template <class Before, class Gate>
  __device__ __forceinline__ void mix(V (&x)[E], void* buf, const float4* __restrict__ tw, bool act, Before before, Gate gate) const {
#pragma unroll 1
    for (int step = 0; step < 4; ++step) {
      RegDft<R1, false>::run(x);
      settle(x);
      if (!(step & 1)) {
        turn<false>(x, buf, tw, act, [&] { if (step == 0) before(); });
      } else if (step == 1) {
        gate(x);
        swap_parts(x);
        __syncthreads();                                   // every thread has read the exchange buffer: it may be written again
      }
    }
    swap_parts(x);
  }
  template <bool HALF>
  __device__ __forceinline__ void inverse(V (&x)[E], void* buf, const float4* __restrict__ tw, bool act) const {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      sub<true>(x, u);
#pragma unroll
      for (int a = 0; a < R2 / 2; ++a) {
        const float4 w = tw_load4(tw + a * R1 + m + S * u);
        if (a > 0) x[u * R2 + 2 * a] = cmulc(x[u * R2 + 2 * a], make_float2(w.x, w.y));
        x[u * R2 + 2 * a + 1] = cmulc(x[u * R2 + 2 * a + 1], make_float2(w.z, w.w));
      }
    }
    exchange<HALF, false>(x, buf, act, Nothing());
    RegDft<R1, true>::run(x);
  }

 private:
  // between the steps: twiddles and exchange
  template <bool HALF, class Before>
  __device__ __forceinline__ void turn(V (&x)[E], void* buf, const float4* __restrict__ tw, bool act, Before before) const {
#pragma unroll
    for (int a = 0; a < R1 / 2; ++a) {
      const float4 w = tw_load4(tw + a * R1 + m);
      if (a > 0) x[2 * a] = cmul(x[2 * a], make_float2(w.x, w.y));
      x[2 * a + 1] = cmul(x[2 * a + 1], make_float2(w.z, w.w));
    }
    exchange<HALF, true>(x, buf, act, before);
  }
  template <bool INV>
  __device__ __forceinline__ void sub(V (&x)[E], int u) const {
    V y[R2];
#pragma unroll
    for (int i = 0; i < R2; ++i) y[i] = x[u * R2 + i];
    RegDft<R2, INV>::run(y);
#pragma unroll
    for (int i = 0; i < R2; ++i) x[u * R2 + i] = y[i];
  }
  // element i of the first step's side is (k1 = i, j2 = m), of the second step's (k1 = m + S u, j2 = i % R2)
  __device__ __forceinline__ int at(bool first, int i) const {
    return first ? (i * (R2 + 1) + m) * G + p : ((m + S * (i / R2)) * (R2 + 1) + i % R2) * G + p;
  }
  // FWD: first step's order -> second step's.  The inverse writes the positions this thread read last, so it needs no
  // barrier in front.  HALF: real and imaginary parts one after the other through half the space.
  template <bool HALF, bool FWD, class Before>
  __device__ __forceinline__ void exchange(V (&x)[E], void* buf, bool act, Before before) const {
    if constexpr (!HALF) {
      V* b = reinterpret_cast<V*>(buf);
      if (act) {
#pragma unroll
        for (int i = 0; i < E; ++i) b[at(FWD, i)] = x[i];
      }
      before();
      __syncthreads();

#pragma unroll
      for (int i = 0; i < E; ++i) x[i] = b[at(!FWD, i)];
    } else {
      decltype(V::x)* b = reinterpret_cast<decltype(V::x)*>(buf);
      if (act) {
#pragma unroll
        for (int i = 0; i < E; ++i) b[at(FWD, i)] = x[i].x;
      }
      __syncthreads();

#pragma unroll
      for (int i = 0; i < E; ++i) x[i].x = b[at(!FWD, i)];
      __syncthreads();

      if (act) {
#pragma unroll
        for (int i = 0; i < E; ++i) b[at(FWD, i)] = x[i].y;
      }
      __syncthreads();

#pragma unroll
      for (int i = 0; i < E; ++i) x[i].y = b[at(!FWD, i)];
    }
  }
};

// n = 2048 = 32 x (8 x 8).  Step one as above with j2 = 8 ja + jb in 0..63.  The 64-point DFT over j2 is two steps of 8
// points whose exchange stays inside a warp: after the first exchange lane l serves jb (later ka) = l % 8 and pair
// l / 8 (+ 4 per further warp), the warp index the group of k1, so a __syncwarp is enough.
//   k = k1 + 32 (ka + 8 kb),  k1 = kg + 8 u for u < 4
// Row (k1, j2) of the exchange buffer sits at row + row / 8, its C slots permuted by bits of the row (an exclusive or
// with f(jb) and f(ja)), so that all four access patterns are free of bank conflicts.
template <int C_>
struct ThreeStep2048 {
  typedef float2 V;
  static constexpr int PP = 1, C = C_, M = 2048, E = 32, S = 64, PW = C / 4;
  static constexpr bool kLoop = false;
  static constexpr int kActive = S * C, kThreads = kActive;
  static constexpr int kExch = (2048 + 256) * C;
  static constexpr int kGate = 2048 + 64;
  // Mixer and gradient take the twiddles from a copy in shared memory: the one CTA of an SM leaves room for it, and its loads take no 64-bit addresses, with
  // which the mixer spilled 300 bytes a thread (public calls, us: layer of 8 x 2048 x 8 heads fp32 60.1 -> 56.0, of 16 x 2048 x 12 fp16
  // 116.3 -> 109.3, forward and backward of 4 x 2048 x 8 bf16 62.6 -> 58.5).  The other modes spill nothing and lose by the copy
  // (prompt of 4 x 1800 x 16 102.9 -> 103.5), and so do the two-step plans, whose exchanges take the same path (forward and backward
  // of 16 x 1024 x 12 105 -> 117).
  static constexpr int kTw = 16 * 64 + 32;
  static constexpr int kParts = PW, kRed = 4, kRedShift = 3;
  int p, m, p2, kg, l8;
  int o1, ojb, oka, q;                                    // offsets of the three access patterns, slot of row digit 0
  static __device__ __forceinline__ int f(int digit) { return C == 8 ? digit : 2 * (digit >> 2); }
  __device__ __forceinline__ explicit ThreeStep2048(int tid) : p(tid % C), m(tid / C) {
    const int warp = tid >> 5, lane = tid & 31;
    l8 = lane & 7;
    p2 = (lane >> 3) + 4 * (warp % PW);
    kg = warp / PW;
    o1 = (m + (m >> 3)) * C + (p ^ f(m & 7) ^ f(m >> 3));
    ojb = (72 * kg + l8) * C;
    oka = (72 * kg + 9 * l8) * C;
    q = p2 ^ f(l8);
  }
  __device__ __forceinline__ int pair_in() const { return p; }
  __device__ __forceinline__ int pair_out() const { return p2; }
  __device__ __forceinline__ int part() const { return p2 >> 2; }
  __device__ __forceinline__ int bin(int i) const { return kg + 8 * (i >> 3) + 32 * l8 + 256 * (i & 7); }
  static __device__ __forceinline__ int gate_slot(int k) { return k + (k >> 5); }

  template <bool HALF, class TW>
  __device__ __forceinline__ void forward(float2 (&x)[E], void* buf, const TW& tw, bool) const {
    RegDft<32, false>::run(x);
#pragma unroll
    for (int a = 0; a < 16; ++a) {
      const float4 w = tw.load4(a * 64 + m);
      if (a > 0) x[2 * a] = cmul(x[2 * a], make_float2(w.x, w.y));
      x[2 * a + 1] = cmul(x[2 * a + 1], make_float2(w.z, w.w));
    }
    move<HALF, 0, 1>(x, buf);
#pragma unroll
    for (int u = 0; u < 4; ++u) sub<false>(x, u);
#pragma unroll
    for (int a = 1; a < 8; ++a) {
      const float2 w = tw.load2(2 * 16 * 64 + 8 * a + l8);
#pragma unroll
      for (int u = 0; u < 4; ++u) x[8 * u + a] = cmul(x[8 * u + a], w);
    }
    move<HALF, 1, 2>(x, buf);
#pragma unroll
    for (int u = 0; u < 4; ++u) sub<false>(x, u);
  }
  template <bool HALF, class TW>
  __device__ __forceinline__ void inverse(float2 (&x)[E], void* buf, const TW& tw, bool) const {
#pragma unroll
    for (int u = 0; u < 4; ++u) sub<true>(x, u);
    move<HALF, 2, 1>(x, buf);
#pragma unroll
    for (int a = 1; a < 8; ++a) {
      const float2 w = tw.load2(2 * 16 * 64 + 8 * a + l8);
#pragma unroll
      for (int u = 0; u < 4; ++u) x[8 * u + a] = cmulc(x[8 * u + a], w);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) sub<true>(x, u);
    move<HALF, 1, 0>(x, buf);
#pragma unroll
    for (int a = 0; a < 16; ++a) {
      const float4 w = tw.load4(a * 64 + m);
      if (a > 0) x[2 * a] = cmulc(x[2 * a], make_float2(w.x, w.y));
      x[2 * a + 1] = cmulc(x[2 * a + 1], make_float2(w.z, w.w));
    }
    RegDft<32, true>::run(x);
  }

 private:
  template <bool INV>
  __device__ __forceinline__ void sub(float2 (&x)[E], int u) const {
    float2 y[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) y[i] = x[u * 8 + i];
    RegDft<8, INV>::run(y);
#pragma unroll
    for (int i = 0; i < 8; ++i) x[u * 8 + i] = y[i];
  }
  // position of element i: 0 = (k1 = i, j2 = m); 1 = (k1 = kg + 8 u, ja or ka = i % 8, jb = l8); 2 = (k1, ka = l8, jb = i % 8)
  template <int KIND>
  __device__ __forceinline__ int at(int i) const {
    if (KIND == 0) return o1 + i * 72 * C;
    const int u = i >> 3, a = i & 7;
    return (KIND == 1 ? ojb + (u * 576 + a * 9) * C : oka + (u * 576 + a) * C) + (q ^ f(a));
  }
  // between kinds 0 and 1 across the CTA, between 1 and 2 inside the warp, over positions that only it uses meanwhile
  template <bool HALF, int FROM, int TO>
  __device__ __forceinline__ void move(float2 (&x)[E], void* buf) const {
    auto sync = [] { if (FROM == 0 || TO == 0) __syncthreads(); else __syncwarp(); };
    if constexpr (!HALF) {
      float2* b = reinterpret_cast<float2*>(buf);
#pragma unroll
      for (int i = 0; i < E; ++i) b[at<FROM>(i)] = x[i];
      sync();
#pragma unroll
      for (int i = 0; i < E; ++i) x[i] = b[at<TO>(i)];
    } else {
      float* b = reinterpret_cast<float*>(buf);
#pragma unroll
      for (int i = 0; i < E; ++i) b[at<FROM>(i)] = x[i].x;
      sync();
#pragma unroll
      for (int i = 0; i < E; ++i) x[i].x = b[at<TO>(i)];
      sync();
#pragma unroll
      for (int i = 0; i < E; ++i) b[at<FROM>(i)] = x[i].y;
      sync();
#pragma unroll
      for (int i = 0; i < E; ++i) x[i].y = b[at<TO>(i)];
    }
  }
};

// how many of the rows m, m + step, ... lie below `rows` (0 for an idle thread)
__device__ __forceinline__ int rows_below(int rows, int m, int step, bool live) { return live && rows > m ? (rows - m + step - 1) / step : 0; }

// Rows m, m + S, ... of the CTA's sequence at this thread's column pairs, all loads in flight before the first
// conversion.  Tokens beyond L are the zero padding; `ring`: they also go, as loaded, into the cache's buffer.
// The base of every row is uniform over the CTA and the thread's part one 32-bit offset, so that a load takes no
// address arithmetic of its own; whole tiles take no predicates either.
template <typename T, class P, int MODE>
__device__ __forceinline__ void reg_load_tokens(typename P::V (&x)[P::E], const void* src, int64_t sb, int64_t sl, int64_t sh,
                                                const RegParams& p, int b, int h, int k1, int col, int m, bool live) {
  typedef ColumnGroup<T, P::PP> IO;
  typedef typename IO::raw raw;
  const int step = MODE == kRegForward && p.decim ? p.N1 : 1, off = MODE == kRegForward && p.decim ? k1 : 0;
  const char* base = reinterpret_cast<const char*>(reinterpret_cast<const T*>(src) + b * sb + (int64_t)off * sl + h * sh);
  const int64_t ds = (int64_t)(P::S * step) * sl * (int64_t)sizeof(T);
  const uint32_t mine = (uint32_t)((int64_t)m * step * sl + col) * (uint32_t)sizeof(T);
  const int count = rows_below(p.L, m * step + off, P::S * step, live);
  raw v[P::E];
  if (count >= P::E) {
#pragma unroll
    for (int i = 0; i < P::E; ++i) v[i] = *reinterpret_cast<const raw*>(base + i * ds + mine);
  } else {
#pragma unroll
    for (int i = 0; i < P::E; ++i) {
      v[i] = IO::zero();
      if (i < count) v[i] = *reinterpret_cast<const raw*>(base + i * ds + mine);
    }
  }
  if (MODE == kRegForward && p.ring && live) {
    T* out = reinterpret_cast<T*>(p.ring) + (((size_t)b * p.n + (m * step + off)) * p.H + h) * p.D + col;
    const size_t dr = (size_t)(P::S * step) * p.H * p.D;
#pragma unroll
    for (int i = 0; i < P::E; ++i) __stcs(reinterpret_cast<raw*>(out + i * dr), v[i]);
  }
#pragma unroll
  for (int i = 0; i < P::E; ++i) {
    float2 t[P::PP];
    IO::cvt(v[i], t);
    x[i] = PointOf<P::PP>::from(t);
  }
}

template <class P>
__device__ __forceinline__ void reg_load_ws(float2 (&x)[P::E], const float2* row, int w) {
#pragma unroll
  for (int i = 0; i < P::E; ++i) x[i] = row[P::S * i * w];
}

// the rows back, those below L
template <typename T, class P>
__device__ __forceinline__ void reg_store_tokens(const float2 (&x)[P::E], const RegParams& p, int b, int h, int col, int m, bool live) {
  typedef typename PairIo<T>::raw raw;
  char* base = reinterpret_cast<char*>(reinterpret_cast<T*>(p.dst) + b * p.d_sb + h * p.d_sh);
  const int64_t ds = (int64_t)P::S * p.d_sl * (int64_t)sizeof(T);
  const uint32_t mine = (uint32_t)((int64_t)m * p.d_sl + col) * (uint32_t)sizeof(T);
  const int count = rows_below(p.L, m, P::S, live);
  if (count >= P::E) {
#pragma unroll
    for (int i = 0; i < P::E; ++i) *reinterpret_cast<raw*>(base + i * ds + mine) = PairIo<T>::pack(x[i]);
  } else {
#pragma unroll
    for (int i = 0; i < P::E; ++i)
      if (i < count) *reinterpret_cast<raw*>(base + i * ds + mine) = PairIo<T>::pack(x[i]);
  }
}

// Sum over the RL pairs that sit side by side in the warp (lane bits SHIFT ...) of RL values each; the lane whose pair
// is s keeps the sum of value s.
template <int RL, int SHIFT>
__device__ __forceinline__ float2 reduce_scatter(float2 (&q)[RL], int s) {
#pragma unroll
  for (int h = RL / 2; h >= 1; h >>= 1) {
    const bool up = s & h;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const float2 send = up ? q[i] : q[i + h], keep = up ? q[i + h] : q[i];
      const float rx = __shfl_xor_sync(0xffffffffu, send.x, h << SHIFT), ry = __shfl_xor_sync(0xffffffffu, send.y, h << SHIFT);
      q[i] = make_float2(keep.x + rx, keep.y + ry);
    }
  }
  return q[0];
}

// 128 registers a thread for 20 and more points (168 for twice 32); fewer points leave room for more CTAs
template <class P> constexpr int reg_min_blocks() {
  constexpr int r = P::PP == 2 ? 384 : (P::E > 16 ? 512 : 768), b = r / P::kThreads;
  return b < 1 ? 1 : (b > 16 ? 16 : b);
}
// real and imaginary parts one after the other through half the exchange buffer
template <class P, int MODE> __host__ __device__ constexpr bool reg_half() { return MODE == kRegGrad || P::PP == 2; }
template <class P, int MODE> __host__ __device__ constexpr size_t reg_exch_bytes() { return ((size_t)P::kExch * (reg_half<P, MODE>() ? 4 : 8) + 15) / 16 * 16; }
template <class P, int MODE> __host__ __device__ constexpr bool reg_tw_shared() { return P::kTw != 0 && (MODE == kRegMix || MODE == kRegGrad); }
template <class P, int MODE> __host__ __device__ constexpr size_t reg_smem_bytes() {
  return reg_exch_bytes<P, MODE>() + (MODE == kRegGrad ? (size_t)P::E * P::kThreads * 8 : 0) + (MODE == kRegMix ? (size_t)P::kGate * 8 : 0) +
         (reg_tw_shared<P, MODE>() ? (size_t)P::kTw * 16 : 0);
}

// MODE kRegMix      rows -> forward, gate, inverse -> rows
//      kRegForward  rows -> spectrum rows in ws
//      kRegInverse  gated half spectra -> inverse -> rows
//      kRegGrad     two tensors' rows: the sum over the pairs of conj(Vhat) Ghat for every bin (sums), and the inverse
//                   transform of conj(gate) Ghat (dst).  Vhat waits in shared memory, one slot per thread and
//                   element; exchanging real and imaginary parts in turn keeps two CTAs on an SM (one at M = 2048).
// WS: rows of the complex workspace instead of tokens.
template <typename T, class P, int MODE, bool WS>
__global__ void __launch_bounds__(P::kThreads, reg_min_blocks<P>()) reg_kernel(const __grid_constant__ RegParams p) {
  extern __shared__ __align__(16) unsigned char reg_smem[];
  constexpr int E = P::E;
  constexpr bool HALF = reg_half<P, MODE>();
  static_assert(P::PP == 1 || (MODE == kRegForward && !WS), "two pairs a thread: forward transforms of tokens");
  void* buf = reg_smem;
  float2* extra = reinterpret_cast<float2*>(reg_smem + reg_exch_bytes<P, MODE>());     // gate table, or the parked spectrum
  const bool act = threadIdx.x < P::kActive;
  const P pl(act ? (int)threadIdx.x : 0);
  int u = blockIdx.x;
  const int tile = u % p.ntile; u /= p.ntile;
  const int k1 = u % p.N1; u /= p.N1;
  const bool second = MODE == kRegForward && p.src2 && u >= p.nslab;              // uniform over the CTA
  if (second) u -= p.nslab;
  const int slab_local = u, slab = p.slab0 + u;
  const int b = slab / p.H, h = slab - b * p.H;
  const int half = p.D / 2;
  const int pin = tile * P::C + pl.pair_in(), pout = tile * P::C + pl.pair_out();
  const bool live = act && pin < half, live_out = act && pout < half;
  const size_t seq = (size_t)slab_local * p.N1 + k1;
  const float2* g = p.g + (size_t)slab * p.K;
  typename std::conditional<P::kTw == 0, const float4*, typename std::conditional<reg_tw_shared<P, MODE>(), TwShared, TwGlobal>::type>::type tw;
  if constexpr (reg_tw_shared<P, MODE>()) {                // the table is the context's: not behind the wait
    const float4* tab = p.tw;
    float4* dst = reinterpret_cast<float4*>(reg_smem + reg_smem_bytes<P, MODE>() - P::kTw * 16);
    for (int i = threadIdx.x; i < P::kTw; i += P::kThreads) dst[i] = __ldg(tab + i);
    tw.p = smem_u32(dst);
    __syncthreads();
  } else if constexpr (P::kTw != 0) {
    tw.p = p.tw;
  } else {
    tw = p.tw;
  }
  // a programmatic dependent of the kernel before it: the set-up overlaps that kernel's end, nothing is read earlier
  asm volatile("griddepcontrol.wait;" ::: "memory");

  typename P::V x[E];
  if constexpr (MODE != kRegInverse) {
    // an idle thread reads the row of pair 0 like the others and stores nothing
    if constexpr (WS) reg_load_ws<P>(x, p.ws + ws_at(half, P::M, seq, pl.m, live ? pin : 0), ws_width(half, live ? pin : 0));
    else reg_load_tokens<T, P, MODE>(x, second ? p.src2 : p.src, second ? p.s2_sb : p.s_sb, second ? p.s2_sl : p.s_sl,
                                     second ? p.s2_sh : p.s_sh, p, b, h, k1, 2 * pin, pl.m, live);
  }
  if constexpr (MODE == kRegMix) {
    for (int i = threadIdx.x; i < P::M; i += P::kThreads) {
      const int k = k1 + p.N1 * i, kk = 2 * k <= p.n ? k : p.n - k;
      float2 v = cscale(g[kk], p.scale);
      if (kk != k) v.y = -v.y;
      if (k == 0 || 2 * k == p.n) v.y = 0.f;
      extra[P::gate_slot(i)] = v;
    }
  }
  auto gate = [&](typename P::V (&z)[E]) {                 // the gate table is complete: the exchange had a barrier
#pragma unroll
    for (int i = 0; i < E; ++i) {
      z[i] = cmul(z[i], extra[P::gate_slot(pl.bin(i))]);
      if (i % 4 == 3) asm volatile("" ::: "memory");        // four gates at a time: there are no registers for more
    }
  };
  constexpr bool kRolled = MODE == kRegMix && P::kLoop;
  if constexpr (kRolled) {
    pl.mix(x, buf, tw, act, [] {}, gate);
  } else if constexpr (MODE != kRegInverse) {
    pl.template forward<HALF>(x, buf, tw, act);
    settle(x);
    if constexpr (MODE == kRegMix) gate(x);
  }
  if constexpr (MODE == kRegForward) {
    float2* out = (second ? p.ws2 : p.ws) + ws_at(half, P::M, seq, 0, pout);
    const int w = ws_width(half, pout);
    if (live_out) {
#pragma unroll
      for (int i = 0; i < E; ++i) {
        float2 t[P::PP];
        PointOf<P::PP>::to(x[i], t);
        ColumnGroup<float, P::PP>::store(reinterpret_cast<float*>(out + pl.bin(i) * w), t);
      }
    }
    return;
  }
  if constexpr (MODE == kRegInverse) {
    const float2* spec = p.spec + (size_t)slab * p.K * p.D + 2 * pout;
#pragma unroll
    for (int i = 0; i < E; ++i) {
      const int k = k1 + p.N1 * pl.bin(i), kk = 2 * k <= p.n ? k : p.n - k;
      x[i] = make_float2(0.f, 0.f);
      if (live_out) {
        const float4 ab = *reinterpret_cast<const float4*>(spec + (size_t)kk * p.D);
        x[i] = pair_from_half(cscale(g[kk], p.scale), ab, k, kk, p.n);
      }
    }
  }
  if constexpr (MODE == kRegGrad) {
#pragma unroll
    for (int i = 0; i < E; ++i) extra[i * P::kThreads + threadIdx.x] = x[i];
    reg_load_tokens<T, P, MODE>(x, p.src2, p.s2_sb, p.s2_sl, p.s2_sh, p, b, h, k1, 2 * pin, pl.m, live);
    __syncthreads();
    pl.template forward<HALF>(x, buf, tw, act);
    if (p.sums) {
      constexpr int RL = P::kRed;
      const int s = (threadIdx.x >> P::kRedShift) % RL;
      float2* out = p.sums + (((size_t)slab_local * p.ntile + tile) * P::kParts + pl.part()) * p.n;
#pragma unroll
      for (int i0 = 0; i0 < E; i0 += RL) {
        float2 q[RL];
#pragma unroll
        for (int i = 0; i < RL; ++i)
          q[i] = i0 + i < E && act ? cmulc(x[(i0 + i) % E], extra[((i0 + i) % E) * P::kThreads + threadIdx.x]) : make_float2(0.f, 0.f);
        const float2 r = reduce_scatter<RL, P::kRedShift>(q, s);
        if (act && i0 + s < E) out[pl.bin(i0 + s)] = r;
      }
    }
    if (!p.dst) return;
#pragma unroll
    for (int i = 0; i < E; ++i) {
      const int k = pl.bin(i), kk = 2 * k <= p.n ? k : p.n - k;
      float2 v = cscale(g[kk], p.scale);
      if (kk == k) v.y = -v.y;
      if (k == 0 || 2 * k == p.n) v.y = 0.f;
      x[i] = cmul(x[i], v);
    }
  }

  if constexpr (!kRolled) {
    settle(x);
    pl.template inverse<HALF>(x, buf, tw, act);
  }
  if (!live) return;
  if constexpr (MODE == kRegForward) {                     // stored above
  } else if constexpr (WS) {
    float2* row = p.ws + ws_at(half, P::M, seq, pl.m, pin);
    const int w = ws_width(half, pin);
#pragma unroll
    for (int i = 0; i < E; ++i) row[P::S * i * w] = x[i];
  } else {
    reg_store_tokens<T, P>(x, p, b, h, 2 * pin, pl.m, live);
  }
}

// kRegMix of the two-step plans for 16-bit tokens and more tiles than are resident: persistent CTAs, the next tile's rows on
// their way by TMA under this one's arithmetic.  Measured at 12.6 M elements: n = 1024 32.0 -> 29.6 us, 784 29.9 -> 26.7,
// 576 28.6 -> 25.9, 512 23.4 -> 21.2, 256 20.7 -> 19.6.  The forward-only mode lost by it (prefill of 2 x 32 x 32k 513 -> 620 us:
// rows N1 tokens apart).
//   map   dims (column, row, head, batch) of the tokens; boxes of 16 columns x reg_box_rows() rows land as [row][8 pairs],
//         from which the threads of a warp read 128 contiguous bytes; rows and columns beyond the tensor are zeros
template <class P> __host__ __device__ constexpr int reg_box_rows() {                  // the most that divide M: at most 256, whole 128-byte pieces
  int r = 256;
  while (P::M % r || r % 4) --r;
  return r;
}
template <class P> __host__ __device__ constexpr size_t reg_stream_bytes() {            // rows, exchange, gate table, barrier
  return (size_t)P::M * P::C * 4 + reg_exch_bytes<P, kRegMix>() + (size_t)P::kGate * 8 + 16;
}

template <typename T, class P>
__global__ void __launch_bounds__(P::kThreads, reg_min_blocks<P>()) reg_stream_kernel(const __grid_constant__ CUtensorMap map,
                                                                                      const __grid_constant__ RegParams p, int ntotal) {
  extern __shared__ __align__(1024) unsigned char reg_stream_smem[];               // all of it dynamic: TMA needs the base 128-byte aligned
  constexpr int E = P::E;
  typedef typename PairIo<T>::raw raw;
  constexpr int kRaw = P::M * P::C * 4, kRows = reg_box_rows<P>(), kGv = (P::M + P::kThreads - 1) / P::kThreads;
  static_assert(P::M % kRows == 0 && kRows * 32 % 128 == 0 && P::C == 8, "whole boxes, 128-byte aligned");
  raw* rows = reinterpret_cast<raw*>(reg_stream_smem);                             // [M][8]
  void* buf = reg_stream_smem + kRaw;
  float2* gs = reinterpret_cast<float2*>(reg_stream_smem + kRaw + reg_exch_bytes<P, kRegMix>());
  const uint32_t bar = smem_u32(reg_stream_smem + reg_stream_bytes<P>() - 16);
  const bool act = threadIdx.x < P::kActive;
  const P pl(act ? (int)threadIdx.x : 0);
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  asm volatile("griddepcontrol.wait;" ::: "memory");
  auto fetch = [&](int w) {                                                        // one thread
    const int slab = p.slab0 + w / p.ntile, b = slab / p.H;
    mbar_expect_tx(bar, kRaw);
#pragma unroll 1
    for (int r = 0; r < P::M; r += kRows) tma_load_4d(smem_u32(rows) + r * 32, &map, 16 * (w % p.ntile), r, slab - b * p.H, b, bar);
  };
  if (threadIdx.x == 0) fetch(blockIdx.x);
  uint32_t par = 0;
  bool ok = true;
#pragma unroll 1
  for (int w = blockIdx.x; w < ntotal; w += gridDim.x, par ^= 1) {
    const int slab = p.slab0 + w / p.ntile, b = slab / p.H, h = slab - b * p.H;
    const int pair = (w % p.ntile) * P::C + pl.p;
    float2 gv[kGv];                                                                // the tile's gates wait in registers for the table
    const float2* g = p.g + (size_t)slab * p.K;
#pragma unroll
    for (int i = 0; i < kGv; ++i) {
      const int k = threadIdx.x + i * P::kThreads;
      gv[i] = k < P::M ? g[2 * k <= P::M ? k : P::M - k] : make_float2(0.f, 0.f);
    }
    ok = mbar_wait(bar, par);
    float2 x[E];
#pragma unroll
    for (int i = 0; i < E; ++i) x[i] = PairIo<T>::cvt(rows[(pl.m + P::S * i) * 8 + pl.p]);
    if (__syncthreads_or(!ok)) break;
    if (threadIdx.x == 0 && w + (int)gridDim.x < ntotal) fetch(w + gridDim.x);     // every thread has its rows: the buffer is free
    auto fill = [&] {
#pragma unroll
      for (int i = 0; i < kGv; ++i) {
        const int k = threadIdx.x + i * P::kThreads;
        float2 v = cscale(gv[i], p.scale);
        if (2 * k > P::M) v.y = -v.y;
        if (k == 0 || 2 * k == P::M) v.y = 0.f;
        if (k < P::M) gs[P::gate_slot(k)] = v;
      }
    };
    auto gate = [&](float2 (&z)[E]) {
#pragma unroll
      for (int i = 0; i < E; ++i) {
        z[i] = cmul(z[i], gs[P::gate_slot(pl.bin(i))]);
        if (i % 4 == 3) asm volatile("" ::: "memory");
      }
    };
    if constexpr (P::kLoop) {
      pl.mix(x, buf, p.tw, act, fill, gate);
    } else {
      pl.template forward<false>(x, buf, p.tw, act, fill);
      settle(x);
      gate(x);
      settle(x);
      pl.template inverse<false>(x, buf, p.tw, act);
    }
    reg_store_tokens<T, P>(x, p, b, h, 2 * pair, pl.m, act && pair < p.D / 2);
  }
  if (!ok) {                                       // do not leave with copies in flight (bounded again)
    report_timeout(p.status);
    mbar_wait(bar, par);
  }
}

template <typename T, class P, int MODE, bool WS>
static int reg_launch(RegParams p, int nslab, cudaStream_t st) {
  auto kern = reg_kernel<T, P, MODE, WS>;
  constexpr size_t smem = reg_smem_bytes<P, MODE>();
  if (smem > 48 * 1024) SPECTRE_CUDA_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  p.ntile = (p.D / 2 + P::C - 1) / P::C;
  cfg.gridDim = dim3((unsigned)((size_t)nslab * p.N1 * p.ntile));
  cfg.blockDim = dim3(P::kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  SPECTRE_CUDA_OK(launch_kernel(&cfg, kern, p));
  return SPECTRE_OK;
}

template <typename T, class P>
static int reg_launch_stream(RegParams p, int nslab, cudaStream_t st, int sm_count, bool* done) {
  constexpr size_t smem = reg_stream_bytes<P>();
  constexpr int fit = (int)(233472 / (smem + 1024)), resident = fit < reg_min_blocks<P>() ? fit : reg_min_blocks<P>();
  p.ntile = (p.D / 2 + P::C - 1) / P::C;
  const long long total = (long long)nslab * p.ntile;
  *done = false;
  if (total <= (long long)resident * sm_count || total > 0x7fffffff || !tensor_map_encoder()) return SPECTRE_OK;
  const cuuint64_t sl = (cuuint64_t)p.s_sl * 2, sh = (cuuint64_t)p.s_sh * 2, sb = (cuuint64_t)p.s_sb * 2;
  const cuuint64_t dims[4] = {(cuuint64_t)p.D, (cuuint64_t)p.L, (cuuint64_t)p.H, (cuuint64_t)p.batch}, strides[3] = {sl, sh, sb};
  const cuuint32_t box[4] = {16, (cuuint32_t)reg_box_rows<P>(), 1, 1}, es[4] = {1, 1, 1, 1};
  CUtensorMap map;
  const CUresult r = tensor_map_encoder()(
      &map, std::is_same<T, f16>::value ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(p.src), dims,
      strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return SPECTRE_OK;                         // strides that a map cannot describe (a broadcast view)
  auto kern = reg_stream_kernel<T, P>;
  SPECTRE_CUDA_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(resident * sm_count));
  cfg.blockDim = dim3(P::kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  SPECTRE_CUDA_OK(launch_kernel(&cfg, kern, map, p, (int)total));
  *done = true;
  return SPECTRE_OK;
}

// Pairs per CTA: 32-byte pieces of a 16-bit row (a whole sector), 64 bytes of an fp32 or workspace row.  With 4 pairs the
// same tiles are 20 % slower (batch of 16 x 12 heads, n = 1024: fp32 45 us against 38, workspace rows 35 against 32): a
// request covers more rows, and each row costs the load/store unit a cycle.
constexpr int kRegPairs = 8;
// The mixer of 1024 and 2048 points with tiles for at most half the SMs: 4 pairs per CTA, so that the few warps there are have
// twice the SMs (up to 16 heads of one sequence: n = 1024 7.5 -> 6.1 us, 2048 15.0 -> 10.1; 512 and less are slower, 5.2 -> 5.4,
// and with 2 pairs 1024 is too, 8.0).

// Column pairs per thread (see TwoStep).  Two where the tiles are more than two per SM, the number of CTAs with one pair a thread that are resident
// at once: up to there every tile is on the chip either way, and one pair brings twice the warps (prompt of 1 x 1000 x 12 heads 26.7 -> 23.7 us, 64 heads
// 25.9 -> 23.2, 1 x 6000 of 8192 x 8 42.8 -> 40.4; against it 1 x 1000 x 80 26.3 -> 25.1 and 1 x 6000 x 10 39.2 -> 37.8 with two).
template <typename T, int MODE, int M> constexpr int reg_pp() { return sizeof(T) == 2 && MODE == kRegForward && M == 1024 ? 2 : 1; }

template <typename T, int MODE>
static int reg_launch_tokens(const spectre_ctx* ctx, const RegParams& q, int M, int nslab, cudaStream_t st) {
  constexpr int C = kRegPairs;
  RegParams p = q;
  p.tw = reg_table(ctx, M);
  p.status = ctx->status_dev;
  constexpr bool kStream = sizeof(T) == 2 && MODE == kRegMix;      // rows by TMA ahead of their tile where CTAs have more than one
#define SPECTRE_REG_CASE(R1, R2)                                                                     \
  case R1 * R2:                                                                                      \
    if constexpr (kStream) {                                                                         \
      bool done = false;                                                                             \
      const int rc = reg_launch_stream<T, TwoStep<R1, R2, C>>(p, nslab, st, ctx->sm_count, &done); \
      if (rc != SPECTRE_OK || done) return rc;                                                       \
    }                                                                                                \
    if constexpr (MODE == kRegMix && R1 == 32 && R2 == 32) {                                         \
      if (2 * tiles <= ctx->sm_count) return reg_launch<T, TwoStep<R1, R2, 4>, MODE, false>(p, nslab, st); \
    }                                                                                                \
    if constexpr (reg_pp<T, MODE, R1 * R2>() == 2) {                                                 \
      if (whole > 2 * ctx->sm_count) return reg_launch<T, TwoStep<R1, R2, C, 2>, MODE, false>(p, nslab, st); \
    }                                                                                                \
    return reg_launch<T, TwoStep<R1, R2, C>, MODE, false>(p, nslab, st);
  const long long tiles = (long long)nslab * ((p.D / 2 + C - 1) / C);
  // of the call, which a small workspace splits into several launches: the choice, and with it the rounding, is one for all of them
  const long long whole = (long long)p.batch * p.H * (p.src2 ? 2 : 1) * p.N1 * ((p.D / 2 + C - 1) / C);
  switch (M) {
    SPECTRE_REG_TWO_STEP(SPECTRE_REG_CASE)
    case 2048:
      if constexpr (MODE == kRegMix) {
        if (2 * tiles <= ctx->sm_count) return reg_launch<T, ThreeStep2048<4>, MODE, false>(p, nslab, st);
      }
      return reg_launch<T, ThreeStep2048<C>, MODE, false>(p, nslab, st);
    default: return fail(SPECTRE_ERR_UNSUPPORTED, "transform length not supported");
  }
#undef SPECTRE_REG_CASE
}
template <int MODE>
static int reg_launch_ws(const spectre_ctx* ctx, const RegParams& q, int M, int nslab, cudaStream_t st) {
  if (M != kRegWsM) return fail(SPECTRE_ERR_UNSUPPORTED, "transform length not supported");
  RegParams p = q;
  p.tw = reg_table(ctx, M);
  return reg_launch<float, TwoStep<32, 32, kRegPairs>, MODE, true>(p, nslab, st);
}

}  // namespace spectre
