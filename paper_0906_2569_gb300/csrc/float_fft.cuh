// Float32 DFT codelets of sign e^{+2 pi i} for the line stages (line_stages.cuh): 2, 3, 4, 5 written out as fused
// multiply-adds, 6, 10, 12, 15 in the prime-factor form (no twiddles), 8, 9, 16 with constant rotations.
#pragma once

#include <cuda_runtime.h>

namespace hpsi {

// The arithmetic on a float2 or, on the host, a double2 (line_gain: the same constants without other rounding)
template <typename V> __host__ __device__ __forceinline__ V ff_make(decltype(V::x) x, decltype(V::x) y) {
  V v;
  v.x = x;
  v.y = y;
  return v;
}
__host__ __device__ __forceinline__ float ff_fma(float a, float b, float c) { return fmaf(a, b, c); }
__host__ __device__ __forceinline__ double ff_fma(double a, double b, double c) { return fma(a, b, c); }
template <typename V> __host__ __device__ __forceinline__ V ff_add(V a, V b) { return ff_make<V>(a.x + b.x, a.y + b.y); }
template <typename V> __host__ __device__ __forceinline__ V ff_sub(V a, V b) { return ff_make<V>(a.x - b.x, a.y - b.y); }
// a + i s b and a - i s b
template <typename V> __host__ __device__ __forceinline__ V ff_addi(V a, V b, decltype(V::x) s) {
  return ff_make<V>(ff_fma(-s, b.y, a.x), ff_fma(s, b.x, a.y));
}
template <typename V> __host__ __device__ __forceinline__ V ff_subi(V a, V b, decltype(V::x) s) {
  return ff_make<V>(ff_fma(s, b.y, a.x), ff_fma(-s, b.x, a.y));
}
template <typename V> __host__ __device__ __forceinline__ V ff_mul(V v, decltype(V::x) c, decltype(V::x) s) {   // v (c + i s)
  return ff_make<V>(ff_fma(v.x, c, -(v.y * s)), ff_fma(v.x, s, v.y * c));
}
// v e^{2 pi i E / R} for the rotations of the 8-, 9- and 16-point codelets
template <int R, int E, typename V>
__host__ __device__ __forceinline__ V ff_rot(V v) {
  constexpr int e = E % R;
  constexpr float h = 0.70710678118654752440f;
  if constexpr (e == 0) return v;
  else if constexpr (4 * e == R) return ff_make<V>(-v.y, v.x);
  else if constexpr (8 * e == R) return ff_make<V>((v.x - v.y) * h, (v.x + v.y) * h);
  else if constexpr (8 * e == 3 * R) return ff_make<V>(-(v.x + v.y) * h, (v.x - v.y) * h);
  else if constexpr (R == 9 && e == 1) return ff_mul(v, 0.76604444311897803520f, 0.64278760968653932632f);
  else if constexpr (R == 9 && e == 2) return ff_mul(v, 0.17364817766693034885f, 0.98480775301220805937f);
  else if constexpr (R == 9 && e == 4) return ff_mul(v, -0.93969262078590838405f, 0.34202014332566873304f);
  else if constexpr (R == 16 && e == 1) return ff_mul(v, 0.92387953251128675613f, 0.38268343236508977173f);
  else if constexpr (R == 16 && e == 3) return ff_mul(v, 0.38268343236508977173f, 0.92387953251128675613f);
  else {
    static_assert(R == 16 && e == 9, "rotation not tabulated");
    return ff_mul(v, -0.92387953251128675613f, -0.38268343236508977173f);
  }
}

template <int R> struct FfDft;
template <> struct FfDft<2> {
  template <typename V> static __host__ __device__ __forceinline__ void run(V* v) {
    const V a = v[0], b = v[1];
    v[0] = ff_add(a, b);
    v[1] = ff_sub(a, b);
  }
};
template <> struct FfDft<3> {
  template <typename V> static __host__ __device__ __forceinline__ void run(V* v) {
    const V t = ff_add(v[1], v[2]), d = ff_sub(v[1], v[2]);
    using T = decltype(V::x);
    const V m = ff_make<V>(ff_fma(T(-0.5), t.x, v[0].x), ff_fma(T(-0.5), t.y, v[0].y));
    v[0] = ff_add(v[0], t);
    v[1] = ff_addi(m, d, 0.86602540378443864676f);
    v[2] = ff_subi(m, d, 0.86602540378443864676f);
  }
};
template <> struct FfDft<4> {
  template <typename V> static __host__ __device__ __forceinline__ void run(V* v) {
    const V a = ff_add(v[0], v[2]), b = ff_sub(v[0], v[2]);
    const V c = ff_add(v[1], v[3]), d = ff_sub(v[1], v[3]);
    v[0] = ff_add(a, c);
    v[1] = ff_make<V>(b.x - d.y, b.y + d.x);
    v[2] = ff_sub(a, c);
    v[3] = ff_make<V>(b.x + d.y, b.y - d.x);
  }
};
template <> struct FfDft<5> {
  template <typename V> static __host__ __device__ __forceinline__ void run(V* v) {
    using T = decltype(V::x);
    constexpr T c1 = 0.30901699437494742410f, c2 = -0.80901699437494742410f;
    constexpr T s1 = 0.95105651629515357212f, s2 = 0.58778525229247312917f;
    const V a1 = ff_add(v[1], v[4]), a2 = ff_add(v[2], v[3]);
    const V b1 = ff_sub(v[1], v[4]), b2 = ff_sub(v[2], v[3]);
    const V p1 = ff_make<V>(ff_fma(c1, a1.x, ff_fma(c2, a2.x, v[0].x)), ff_fma(c1, a1.y, ff_fma(c2, a2.y, v[0].y)));
    const V p2 = ff_make<V>(ff_fma(c2, a1.x, ff_fma(c1, a2.x, v[0].x)), ff_fma(c2, a1.y, ff_fma(c1, a2.y, v[0].y)));
    const V q1 = ff_make<V>(ff_fma(s1, b1.x, s2 * b2.x), ff_fma(s1, b1.y, s2 * b2.y));
    const V q2 = ff_make<V>(ff_fma(s2, b1.x, -(s1 * b2.x)), ff_fma(s2, b1.y, -(s1 * b2.y)));
    v[0] = ff_add(v[0], ff_add(a1, a2));
    v[1] = ff_make<V>(p1.x - q1.y, p1.y + q1.x);
    v[4] = ff_make<V>(p1.x + q1.y, p1.y - q1.x);
    v[2] = ff_make<V>(p2.x - q2.y, p2.y + q2.x);
    v[3] = ff_make<V>(p2.x + q2.y, p2.y - q2.x);
  }
};
// R = A B with coprime A, B: input (B a + A b) mod R, output k with k = k1 mod A, k = k2 mod B
template <int A, int B> struct FfPfa {
  static constexpr int unit(int p, int q) {   // the k < p q that is 1 mod p and 0 mod q
    int k = 0;
    while (k % p != 1 || k % q != 0) ++k;
    return k;
  }
  static constexpr int EA = unit(A, B), EB = unit(B, A);
  template <typename V> static __host__ __device__ __forceinline__ void run(V* x) {
    V y[A * B];
#pragma unroll
    for (int b = 0; b < B; ++b) {
      V t[A];
#pragma unroll
      for (int a = 0; a < A; ++a) t[a] = x[(B * a + A * b) % (A * B)];
      FfDft<A>::run(t);
#pragma unroll
      for (int a = 0; a < A; ++a) y[a * B + b] = t[a];
    }
#pragma unroll
    for (int a = 0; a < A; ++a) {
      FfDft<B>::run(y + a * B);
#pragma unroll
      for (int b = 0; b < B; ++b) x[(EA * a + EB * b) % (A * B)] = y[a * B + b];
    }
  }
};
template <> struct FfDft<6> : FfPfa<2, 3> {};
template <> struct FfDft<10> : FfPfa<2, 5> {};
template <> struct FfDft<12> : FfPfa<4, 3> {};
template <> struct FfDft<15> : FfPfa<3, 5> {};
// R = A B with a common factor: rotations in between
template <int A, int B> struct FfCt {
  template <int K1, int N2, typename V>
  static __host__ __device__ __forceinline__ void rot(V (&y)[A][B]) {
    y[K1][N2] = ff_rot<A * B, K1 * N2>(y[K1][N2]);
    if constexpr (N2 + 1 < B) rot<K1, N2 + 1>(y);
    else if constexpr (K1 + 1 < A) rot<K1 + 1, 1>(y);
  }
  template <typename V> static __host__ __device__ __forceinline__ void run(V* x) {
    V y[A][B];
#pragma unroll
    for (int n = 0; n < B; ++n) {
      V t[A];
#pragma unroll
      for (int a = 0; a < A; ++a) t[a] = x[B * a + n];
      FfDft<A>::run(t);
#pragma unroll
      for (int a = 0; a < A; ++a) y[a][n] = t[a];
    }
    rot<1, 1>(y);
#pragma unroll
    for (int k = 0; k < A; ++k) {
      FfDft<B>::run(y[k]);
#pragma unroll
      for (int m = 0; m < B; ++m) x[k + A * m] = y[k][m];
    }
  }
};
template <> struct FfDft<8> : FfCt<2, 4> {};
template <> struct FfDft<9> : FfCt<3, 3> {};
template <> struct FfDft<16> : FfCt<4, 4> {};

}  // namespace hpsi
