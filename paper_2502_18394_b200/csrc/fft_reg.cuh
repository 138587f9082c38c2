// DFTs of 2 ... 32 points held in one thread's registers, with every root of unity a compile-time
// literal and the additions of complex values issued as packed fp32 pairs.  A point is one complex value (float2) or those
// of two independent columns (cx2), whose multiplications are packed as well.
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

// The same point of two columns: real parts and imaginary parts each a packed pair.  The FMA pipe takes two cycles for a packed
// instruction and 1.28 for a scalar one (measured, four warps a scheduler), so products cost 1.28 times less per column than
// those of a float2 (4 cycles against 5.1), and a swap of real and imaginary parts is a renaming.
struct __align__(16) cx2 { uint64_t x, y; };
__device__ __forceinline__ cx2 padd(cx2 a, cx2 b) { return {add2(a.x, b.x), add2(a.y, b.y)}; }
__device__ __forceinline__ cx2 psub(cx2 a, cx2 b) { return {sub2(a.x, b.x), sub2(a.y, b.y)}; }
__device__ __forceinline__ cx2 cmul(cx2 a, float2 w) {
  const uint64_t wx = pk2(w.x, w.x), wy = pk2(w.y, w.y), ny = pk2(-w.y, -w.y);
  return {fma2(a.y, ny, mul2(a.x, wx)), fma2(a.x, wy, mul2(a.y, wx))};
}
__device__ __forceinline__ cx2 cmulc(cx2 a, float2 w) { return cmul(a, make_float2(w.x, -w.y)); }

// real arithmetic on a component of a point: one value or a packed pair
__device__ __forceinline__ float radd(float a, float b) { return a + b; }
__device__ __forceinline__ float rsub(float a, float b) { return a - b; }
__device__ __forceinline__ float rneg(float a) { return -a; }
__device__ __forceinline__ float rmul(float a, float c) { return a * c; }
__device__ __forceinline__ float rfma(float a, float c, float b) { return fmaf(a, c, b); }
__device__ __forceinline__ uint64_t radd(uint64_t a, uint64_t b) { return add2(a, b); }
__device__ __forceinline__ uint64_t rsub(uint64_t a, uint64_t b) { return sub2(a, b); }
__device__ __forceinline__ uint64_t rneg(uint64_t a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ uint64_t rmul(uint64_t a, float c) { return mul2(a, pk2(c, c)); }
__device__ __forceinline__ uint64_t rfma(uint64_t a, float c, uint64_t b) { return fma2(a, pk2(c, c), b); }

// x exp(-j 2 pi J / R); INV conjugates the root
template <int J, int R, bool INV, class V>
__device__ __forceinline__ V rot(V x) {
  constexpr int j = ((J % R) + R) % R;
  if constexpr (j == 0) return x;
  else if constexpr (2 * j == R) return V{rneg(x.x), rneg(x.y)};
  else if constexpr (4 * j == R || 4 * j == 3 * R) {
    if constexpr ((4 * j == R) != INV) return V{x.y, rneg(x.x)};
    else return V{rneg(x.y), x.x};
  } else if constexpr ((8 * j) % R == 0) {
    constexpr float h = 0.70710678118654752440f;
    constexpr int e = INV ? 8 - 8 * j / R : 8 * j / R;
    if constexpr (e == 1) return V{rmul(radd(x.x, x.y), h), rmul(rsub(x.y, x.x), h)};
    else if constexpr (e == 3) return V{rmul(rsub(x.y, x.x), h), rmul(radd(x.x, x.y), -h)};
    else if constexpr (e == 5) return V{rmul(radd(x.x, x.y), -h), rmul(rsub(x.x, x.y), h)};
    else return V{rmul(rsub(x.x, x.y), h), rmul(radd(x.x, x.y), h)};
  } else {
    constexpr float c = (float)cx_root(j, R, false), s = (float)cx_root(INV ? -j : j, R, true);
    return V{rfma(x.x, c, rmul(x.y, s)), rfma(x.y, c, rmul(x.x, -s))};
  }
}

// Natural order in and out: X_k = sum_t x_t exp(-j 2 pi k t / R); INV takes the conjugate kernel, no scaling.
template <int R, bool INV> struct RegDft;

template <int R1, int R2, bool INV, class V>
__device__ __forceinline__ void reg_ct(V (&x)[R1 * R2]) {
  constexpr int R = R1 * R2;
  V a[R1][R2];
  static_for<R2>([&](auto i2) {
    constexpr int n2 = decltype(i2)::v;
    V t[R1];
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
    V u[R2];
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) u[n2] = a[k1][n2];
    RegDft<R2, INV>::run(u);
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) x[k1 + R1 * k2] = u[k2];
  }
}

// Odd R: sums and differences of mirrored inputs halve the multiplications.
template <int R, bool INV, class V>
__device__ __forceinline__ void reg_odd(V (&x)[R]) {
  constexpr int P = (R - 1) / 2;
  V t[P], d[P], sum = x[0];
#pragma unroll
  for (int i = 0; i < P; ++i) {
    t[i] = padd(x[i + 1], x[R - 1 - i]);
    d[i] = psub(x[i + 1], x[R - 1 - i]);
    sum = padd(sum, t[i]);
  }
  V y[R];
  y[0] = sum;
  static_for<P>([&](auto ik) {
    constexpr int k = decltype(ik)::v + 1;
    V e = x[0], o;
    static_for<P>([&](auto ii) {
      constexpr int i = decltype(ii)::v;
      constexpr float c = (float)cx_root(k * (i + 1), R, false), s = (float)cx_root(k * (i + 1), R, true);
      e = V{rfma(t[i].x, c, e.x), rfma(t[i].y, c, e.y)};
      if constexpr (i == 0) o = V{rmul(d[i].x, s), rmul(d[i].y, s)};
      else o = V{rfma(d[i].x, s, o.x), rfma(d[i].y, s, o.y)};
    });
    const V jo{rneg(o.y), o.x};
    y[k] = INV ? padd(e, jo) : psub(e, jo);
    y[R - k] = INV ? psub(e, jo) : padd(e, jo);
  });
#pragma unroll
  for (int k = 0; k < R; ++k) x[k] = y[k];
}

template <bool INV> struct RegDft<1, INV> { template <class V> static __device__ __forceinline__ void run(V (&)[1]) {} };
template <bool INV> struct RegDft<2, INV> {
  template <class V> static __device__ __forceinline__ void run(V (&x)[2]) {
    const V a = x[0], b = x[1];
    x[0] = padd(a, b);
    x[1] = psub(a, b);
  }
};
template <bool INV> struct RegDft<4, INV> {
  template <class V> static __device__ __forceinline__ void run(V (&x)[4]) {
    const V t0 = padd(x[0], x[2]), t1 = psub(x[0], x[2]), t2 = padd(x[1], x[3]), t3 = psub(x[1], x[3]);
    x[0] = padd(t0, t2);
    x[2] = psub(t0, t2);
    const V lo{radd(t1.x, t3.y), rsub(t1.y, t3.x)}, hi{rsub(t1.x, t3.y), radd(t1.y, t3.x)};   // t1 -+ j t3
    x[1] = INV ? hi : lo;
    x[3] = INV ? lo : hi;
  }
};
#define SPECTRE_REG_ODD(R) \
  template <bool INV> struct RegDft<R, INV> { template <class V> static __device__ __forceinline__ void run(V (&x)[R]) { reg_odd<R, INV>(x); } };
#define SPECTRE_REG_CT(R, A, B) \
  template <bool INV> struct RegDft<R, INV> { template <class V> static __device__ __forceinline__ void run(V (&x)[R]) { reg_ct<A, B, INV>(x); } };
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

// a point of PP adjacent column pairs
template <int PP> struct PointOf;
template <> struct PointOf<1> {
  typedef float2 type;
  static __device__ __forceinline__ float2 from(const float2 (&a)[1]) { return a[0]; }
  static __device__ __forceinline__ void to(float2 v, float2 (&a)[1]) { a[0] = v; }
};
template <> struct PointOf<2> {
  typedef cx2 type;
  static __device__ __forceinline__ cx2 from(const float2 (&a)[2]) { return {pk2(a[0].x, a[1].x), pk2(a[0].y, a[1].y)}; }
  static __device__ __forceinline__ void to(cx2 v, float2 (&a)[2]) {
    upk2(v.x, a[0].x, a[1].x);
    upk2(v.y, a[0].y, a[1].y);
  }
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
