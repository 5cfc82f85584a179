// Float32 DFT codelets of sign e^{+2 pi i} for the line stages (line_stages.cuh): 2, 3, 4, 5 written out as fused
// multiply-adds, 6, 10, 12, 15 in the prime-factor form (no twiddles), 8, 9, 16 with constant rotations.
#pragma once

#include <cuda_runtime.h>

namespace hpsi {

__device__ __forceinline__ float2 ff_add(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 ff_sub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
// a + i s b and a - i s b
__device__ __forceinline__ float2 ff_addi(float2 a, float2 b, float s) {
  return make_float2(fmaf(-s, b.y, a.x), fmaf(s, b.x, a.y));
}
__device__ __forceinline__ float2 ff_subi(float2 a, float2 b, float s) {
  return make_float2(fmaf(s, b.y, a.x), fmaf(-s, b.x, a.y));
}
__device__ __forceinline__ float2 ff_mul(float2 v, float c, float s) {   // v (c + i s)
  return make_float2(fmaf(v.x, c, -(v.y * s)), fmaf(v.x, s, v.y * c));
}
// v e^{2 pi i E / R} for the rotations of the 8-, 9- and 16-point codelets
template <int R, int E>
__device__ __forceinline__ float2 ff_rot(float2 v) {
  constexpr int e = E % R;
  constexpr float h = 0.70710678118654752440f;
  if constexpr (e == 0) return v;
  else if constexpr (4 * e == R) return make_float2(-v.y, v.x);
  else if constexpr (8 * e == R) return make_float2((v.x - v.y) * h, (v.x + v.y) * h);
  else if constexpr (8 * e == 3 * R) return make_float2(-(v.x + v.y) * h, (v.x - v.y) * h);
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
  static __device__ __forceinline__ void run(float2* v) {
    const float2 a = v[0], b = v[1];
    v[0] = ff_add(a, b);
    v[1] = ff_sub(a, b);
  }
};
template <> struct FfDft<3> {
  static __device__ __forceinline__ void run(float2* v) {
    const float2 t = ff_add(v[1], v[2]), d = ff_sub(v[1], v[2]);
    const float2 m = make_float2(fmaf(-0.5f, t.x, v[0].x), fmaf(-0.5f, t.y, v[0].y));
    v[0] = ff_add(v[0], t);
    v[1] = ff_addi(m, d, 0.86602540378443864676f);
    v[2] = ff_subi(m, d, 0.86602540378443864676f);
  }
};
template <> struct FfDft<4> {
  static __device__ __forceinline__ void run(float2* v) {
    const float2 a = ff_add(v[0], v[2]), b = ff_sub(v[0], v[2]);
    const float2 c = ff_add(v[1], v[3]), d = ff_sub(v[1], v[3]);
    v[0] = ff_add(a, c);
    v[1] = make_float2(b.x - d.y, b.y + d.x);
    v[2] = ff_sub(a, c);
    v[3] = make_float2(b.x + d.y, b.y - d.x);
  }
};
template <> struct FfDft<5> {
  static __device__ __forceinline__ void run(float2* v) {
    constexpr float c1 = 0.30901699437494742410f, c2 = -0.80901699437494742410f;
    constexpr float s1 = 0.95105651629515357212f, s2 = 0.58778525229247312917f;
    const float2 a1 = ff_add(v[1], v[4]), a2 = ff_add(v[2], v[3]);
    const float2 b1 = ff_sub(v[1], v[4]), b2 = ff_sub(v[2], v[3]);
    const float2 p1 = make_float2(fmaf(c1, a1.x, fmaf(c2, a2.x, v[0].x)), fmaf(c1, a1.y, fmaf(c2, a2.y, v[0].y)));
    const float2 p2 = make_float2(fmaf(c2, a1.x, fmaf(c1, a2.x, v[0].x)), fmaf(c2, a1.y, fmaf(c1, a2.y, v[0].y)));
    const float2 q1 = make_float2(fmaf(s1, b1.x, s2 * b2.x), fmaf(s1, b1.y, s2 * b2.y));
    const float2 q2 = make_float2(fmaf(s2, b1.x, -(s1 * b2.x)), fmaf(s2, b1.y, -(s1 * b2.y)));
    v[0] = ff_add(v[0], ff_add(a1, a2));
    v[1] = make_float2(p1.x - q1.y, p1.y + q1.x);
    v[4] = make_float2(p1.x + q1.y, p1.y - q1.x);
    v[2] = make_float2(p2.x - q2.y, p2.y + q2.x);
    v[3] = make_float2(p2.x + q2.y, p2.y - q2.x);
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
  static __device__ __forceinline__ void run(float2* x) {
    float2 y[A * B];
#pragma unroll
    for (int b = 0; b < B; ++b) {
      float2 t[A];
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
  template <int K1, int N2>
  static __device__ __forceinline__ void rot(float2 (&y)[A][B]) {
    y[K1][N2] = ff_rot<A * B, K1 * N2>(y[K1][N2]);
    if constexpr (N2 + 1 < B) rot<K1, N2 + 1>(y);
    else if constexpr (K1 + 1 < A) rot<K1 + 1, 1>(y);
  }
  static __device__ __forceinline__ void run(float2* x) {
    float2 y[A][B];
#pragma unroll
    for (int n = 0; n < B; ++n) {
      float2 t[A];
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
