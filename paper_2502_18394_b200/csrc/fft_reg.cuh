// DFTs of 2 ... 32 points held in one thread's registers, with every root of unity a compile-time
// literal and the additions of complex values issued as packed fp32 pairs.
#pragma once
#include <utility>

#include "tc_common.cuh"

namespace spectre {

// cos / sin of 2 pi J / R at compile time: the angle is reduced to [0, pi / 4] in integers, where the
// Taylor series reaches double precision.
__host__ __device__ constexpr double cx_series(double x, bool sine) {
  double t = sine ? x : 1.0, s = t;
  for (int k = sine ? 2 : 1; k < 26; k += 2) {
    t = -t * x * x / (double)(k * (k + 1));
    s += t;
  }
  return s;
}
__host__ __device__ constexpr double cx_root(int J, int R, bool sine) {
  const double kTwoPi = 6.283185307179586476925286766559;
  J = ((J % R) + R) % R;
  double sign = 1.0;
  if (2 * J > R) { J = R - J; if (sine) sign = -sign; }                   // mirror: lower half plane
  bool cosine = !sine;
  int num = 2 * J, den = 2 * R;                                           // angle 2 pi num / den, at most pi
  if (4 * num > den) { num = den / 2 - num; if (cosine) sign = -sign; }   // second quadrant
  if (8 * num > den) { num = den - 4 * num; den *= 4; cosine = !cosine; } // pi / 2 - angle
  return sign * cx_series(kTwoPi * (double)num / (double)den, !cosine);
}

// loop whose index is a compile-time constant (decltype(i)::v)
template <int I> struct Index { static constexpr int v = I; };
template <class F, int... I>
__device__ __forceinline__ void static_for_impl(F&& f, std::integer_sequence<int, I...>) {
  (f(Index<I>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void static_for(F&& f) { static_for_impl(f, std::make_integer_sequence<int, N>{}); }

__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float2 padd(float2 a, float2 b) {
  float2 r;
  upk2(add2(pk2(a.x, a.y), pk2(b.x, b.y)), r.x, r.y);
  return r;
}
__device__ __forceinline__ float2 psub(float2 a, float2 b) {
  float2 r;
  upk2(sub2(pk2(a.x, a.y), pk2(b.x, b.y)), r.x, r.y);
  return r;
}

// x exp(-j 2 pi J / R); INV conjugates the root
template <int J, int R, bool INV>
__device__ __forceinline__ float2 rot(float2 x) {
  constexpr int j = ((J % R) + R) % R;
  if constexpr (j == 0) return x;
  else if constexpr (2 * j == R) return make_float2(-x.x, -x.y);
  else if constexpr (4 * j == R || 4 * j == 3 * R) {
    if constexpr ((4 * j == R) != INV) return make_float2(x.y, -x.x);
    else return make_float2(-x.y, x.x);
  } else if constexpr ((8 * j) % R == 0) {
    constexpr float h = 0.70710678118654752440f;
    constexpr int e = INV ? 8 - 8 * j / R : 8 * j / R;
    if constexpr (e == 1) return make_float2((x.x + x.y) * h, (x.y - x.x) * h);
    else if constexpr (e == 3) return make_float2((x.y - x.x) * h, -(x.x + x.y) * h);
    else if constexpr (e == 5) return make_float2(-(x.x + x.y) * h, (x.x - x.y) * h);
    else return make_float2((x.x - x.y) * h, (x.x + x.y) * h);
  } else {
    constexpr float c = (float)cx_root(j, R, false), s = (float)cx_root(INV ? -j : j, R, true);
    return make_float2(fmaf(x.x, c, x.y * s), fmaf(x.y, c, -x.x * s));
  }
}

// Natural order in and out: X_k = sum_t x_t exp(-j 2 pi k t / R); INV takes the conjugate kernel, no scaling.
template <int R, bool INV> struct RegDft;

template <int R1, int R2, bool INV>
__device__ __forceinline__ void reg_ct(float2 (&x)[R1 * R2]) {
  constexpr int R = R1 * R2;
  float2 a[R1][R2];
  static_for<R2>([&](auto i2) {
    constexpr int n2 = decltype(i2)::v;
    float2 t[R1];
#pragma unroll
    for (int n1 = 0; n1 < R1; ++n1) t[n1] = x[n1 * R2 + n2];
    RegDft<R1, INV>::run(t);
    static_for<R1>([&](auto i1) {
      constexpr int k1 = decltype(i1)::v;
      a[k1][n2] = rot<k1 * n2, R, INV>(t[k1]);
    });
  });
#pragma unroll
  for (int k1 = 0; k1 < R1; ++k1) {
    float2 u[R2];
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) u[n2] = a[k1][n2];
    RegDft<R2, INV>::run(u);
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) x[k1 + R1 * k2] = u[k2];
  }
}

// Odd R: sums and differences of mirrored inputs halve the multiplications.
template <int R, bool INV>
__device__ __forceinline__ void reg_odd(float2 (&x)[R]) {
  constexpr int P = (R - 1) / 2;
  float2 t[P], d[P], sum = x[0];
#pragma unroll
  for (int i = 0; i < P; ++i) {
    t[i] = padd(x[i + 1], x[R - 1 - i]);
    d[i] = psub(x[i + 1], x[R - 1 - i]);
    sum = padd(sum, t[i]);
  }
  float2 y[R];
  y[0] = sum;
  static_for<P>([&](auto ik) {
    constexpr int k = decltype(ik)::v + 1;
    float2 e = x[0], o = make_float2(0.f, 0.f);
    static_for<P>([&](auto ii) {
      constexpr int i = decltype(ii)::v;
      constexpr float c = (float)cx_root(k * (i + 1), R, false), s = (float)cx_root(k * (i + 1), R, true);
      e = make_float2(fmaf(t[i].x, c, e.x), fmaf(t[i].y, c, e.y));
      o = make_float2(fmaf(d[i].x, s, o.x), fmaf(d[i].y, s, o.y));
    });
    const float2 jo = make_float2(-o.y, o.x);
    y[k] = INV ? padd(e, jo) : psub(e, jo);
    y[R - k] = INV ? psub(e, jo) : padd(e, jo);
  });
#pragma unroll
  for (int k = 0; k < R; ++k) x[k] = y[k];
}

template <bool INV> struct RegDft<1, INV> { static __device__ __forceinline__ void run(float2 (&)[1]) {} };
template <bool INV> struct RegDft<2, INV> {
  static __device__ __forceinline__ void run(float2 (&x)[2]) {
    const float2 a = x[0], b = x[1];
    x[0] = padd(a, b);
    x[1] = psub(a, b);
  }
};
template <bool INV> struct RegDft<4, INV> {
  static __device__ __forceinline__ void run(float2 (&x)[4]) {
    const float2 t0 = padd(x[0], x[2]), t1 = psub(x[0], x[2]), t2 = padd(x[1], x[3]), t3 = psub(x[1], x[3]);
    x[0] = padd(t0, t2);
    x[2] = psub(t0, t2);
    const float2 lo = make_float2(t1.x + t3.y, t1.y - t3.x), hi = make_float2(t1.x - t3.y, t1.y + t3.x);   // t1 -+ j t3
    x[1] = INV ? hi : lo;
    x[3] = INV ? lo : hi;
  }
};
#define SPECTRE_REG_ODD(R) \
  template <bool INV> struct RegDft<R, INV> { static __device__ __forceinline__ void run(float2 (&x)[R]) { reg_odd<R, INV>(x); } };
#define SPECTRE_REG_CT(R, A, B) \
  template <bool INV> struct RegDft<R, INV> { static __device__ __forceinline__ void run(float2 (&x)[R]) { reg_ct<A, B, INV>(x); } };
SPECTRE_REG_ODD(3)
SPECTRE_REG_ODD(5)
SPECTRE_REG_ODD(7)
SPECTRE_REG_CT(6, 2, 3)
SPECTRE_REG_CT(8, 2, 4)
SPECTRE_REG_CT(9, 3, 3)
SPECTRE_REG_CT(10, 2, 5)
SPECTRE_REG_CT(12, 3, 4)
SPECTRE_REG_CT(14, 2, 7)
SPECTRE_REG_CT(16, 4, 4)
SPECTRE_REG_CT(18, 2, 9)
SPECTRE_REG_CT(20, 4, 5)
SPECTRE_REG_CT(24, 3, 8)
SPECTRE_REG_CT(28, 4, 7)
SPECTRE_REG_CT(30, 5, 6)
SPECTRE_REG_CT(32, 4, 8)
#undef SPECTRE_REG_ODD
#undef SPECTRE_REG_CT

// ---- one column pair of a token row in each activation type ----
template <typename T> struct PairIo;
template <> struct PairIo<float> {
  typedef float2 raw;
  static __device__ __forceinline__ float2 cvt(raw r) { return r; }
  static __device__ __forceinline__ raw pack(float2 v) { return v; }
  static __device__ __forceinline__ raw zero() { return make_float2(0.f, 0.f); }
};
template <> struct PairIo<bf16> {
  typedef uint32_t raw;
  static __device__ __forceinline__ float2 cvt(raw r) { return unpack_bf2(r); }
  static __device__ __forceinline__ raw pack(float2 v) { return pack_bf2(v.x, v.y); }
  static __device__ __forceinline__ raw zero() { return 0u; }
};
template <> struct PairIo<f16> {
  typedef uint32_t raw;
  static __device__ __forceinline__ float2 cvt(raw r) { return unpack_h2(r); }
  static __device__ __forceinline__ raw pack(float2 v) { return pack_h2(v.x, v.y); }
  static __device__ __forceinline__ raw zero() { return 0u; }
};

// PP = 1 or 2 adjacent column pairs of a row
template <typename T, int PP> struct ColumnGroup;
template <typename T> struct ColumnGroup<T, 1> {
  typedef typename PairIo<T>::raw raw;
  static __device__ __forceinline__ raw zero() { return PairIo<T>::zero(); }
  static __device__ __forceinline__ raw load(const T* p) { return *reinterpret_cast<const raw*>(p); }
  static __device__ __forceinline__ void cvt(raw r, float2 (&x)[1]) { x[0] = PairIo<T>::cvt(r); }
  static __device__ __forceinline__ void store(T* p, const float2 (&x)[1]) { *reinterpret_cast<raw*>(p) = PairIo<T>::pack(x[0]); }
};
template <typename T> struct ColumnGroup<T, 2> {
  typedef uint2 raw;
  static __device__ __forceinline__ raw zero() { return make_uint2(0u, 0u); }
  static __device__ __forceinline__ raw load(const T* p) { return *reinterpret_cast<const uint2*>(p); }
  static __device__ __forceinline__ void cvt(raw r, float2 (&x)[2]) { x[0] = PairIo<T>::cvt(r.x); x[1] = PairIo<T>::cvt(r.y); }
  static __device__ __forceinline__ void store(T* p, const float2 (&x)[2]) {
    *reinterpret_cast<uint2*>(p) = make_uint2(PairIo<T>::pack(x[0]), PairIo<T>::pack(x[1]));
  }
};
template <> struct ColumnGroup<float, 2> {
  typedef float4 raw;
  static __device__ __forceinline__ raw zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
  static __device__ __forceinline__ raw load(const float* p) { return *reinterpret_cast<const float4*>(p); }
  static __device__ __forceinline__ void cvt(raw r, float2 (&x)[2]) { x[0] = make_float2(r.x, r.y); x[1] = make_float2(r.z, r.w); }
  static __device__ __forceinline__ void store(float* p, const float2 (&x)[2]) {
    *reinterpret_cast<float4*>(p) = make_float4(x[0].x, x[0].y, x[1].x, x[1].y);
  }
};

}  // namespace spectre
