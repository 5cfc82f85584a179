// Line FFTs on 64-bit fixed-point numbers: the arithmetic of the float64 local term.
//
// Why: GB300 issues one float64 instruction per scheduler in ~76 cycles (1.6 lanes per clock and SM, measured), while
// 64-bit integer adds run at 55 lanes per clock and a 64 x 64 -> high 64 multiplication by a constant (three 32 x 32 ->
// 64 multiply-adds) at ~5.  An FFT is adds and multiplications by constants of modulus 1, so a block-scaled
// fixed-point transform does the same work ~9 times faster than the float64 pipe, and with 63 bits it
// also rounds less: adds are exact, and a multiplication rounds at 2^-63 of the block's full scale.
//
// A complex value is q 2^e with one exponent e per block (local_fixed.cu keeps the blocks and chooses e so that no
// intermediate can reach 2^63).  Bound used there: every intermediate of a transform of x over L nonzero entries is
// a combination of the entries with complex coefficients of modulus <= kGain, so its parts stay below
// kGain sum |x_n|; the largest coefficient is sin 72 + sin 36 = 1.539 of the 5-point kernel.
//
// The transforms have the sign e^{+2 pi i}; the opposite sign is the same code with real and imaginary parts
// swapped on the way in and out.  A line of n = R1 R2 values lies in n cells and is transformed in place in two stages:
//   stage 1, item t < R2:   R1-point DFT over the cells  a R2 + t, a < R1
//   stage 2, item k1 < R1:  R2-point DFT over the cells  k1 R2 + b, b < R2
// Coprime R1, R2 use the prime-factor form: value n starts in cell a R2 + t with n = R2 a + R1 t (mod n), X[k] ends in cell
// (k mod R1) R2 + (k mod R2), and there are no twiddles.  Otherwise (Cooley-Tukey) values start in natural order, stage
// 1 multiplies its output k1 by e^{2 pi i t k1 / n}, and X[k] ends in cell (k mod R1) R2 + (k div R1).  The reversed
// sequence (stage 2, the twiddles, stage 1) goes from the last order to the first.
#pragma once

#include <cuda_runtime.h>

namespace hpsi {

constexpr double kFixGain = 1.54;

// a = hi 2^32 + lo with lo a signed 32-bit number
__host__ __device__ __forceinline__ int fx_lo(long long a) { return (int)(unsigned)(unsigned long long)a; }
__host__ __device__ __forceinline__ int fx_hi(long long a) {
  return (int)(a >> 32) + (int)((unsigned)fx_lo(a) >> 31);
}

// M a + a K / 2^64, rounded; |K| < 2^63 (the product of the two low halves, below a quarter, is left out)
template <long long K, int M = 0>
__host__ __device__ __forceinline__ long long fx_mulc(long long a) {
  constexpr int cl = (int)(unsigned)(unsigned long long)K;
  constexpr int ch = (int)(K >> 32) + (int)((unsigned)cl >> 31);
  const int al = fx_lo(a), ah = fx_hi(a);
  long long t = (long long)ah * cl + 0x80000000LL;
  t = (long long)al * ch + t;
  const long long r = (long long)ah * ch + (M == 0 ? 0LL : M == 1 ? a : 2 * a);
  return r + (t >> 32);
}
template <long long K, int M = 0>
__host__ __device__ __forceinline__ longlong2 fx_mulc(longlong2 v) {
  longlong2 r;
  r.x = fx_mulc<K, M>(v.x);
  r.y = fx_mulc<K, M>(v.y);
  return r;
}
// a b / 2^64 for run-time |b| <= 2^62
__host__ __device__ __forceinline__ long long fx_mulr(long long a, int bh, int bl) {
  const int al = fx_lo(a), ah = fx_hi(a);
  long long t = (long long)ah * bl + 0x80000000LL;
  t = (long long)al * bh + t;
  return (long long)ah * bh + (t >> 32);
}

__host__ __device__ __forceinline__ longlong2 fx_add(longlong2 a, longlong2 b) {
  longlong2 r;
  r.x = a.x + b.x;
  r.y = a.y + b.y;
  return r;
}
__host__ __device__ __forceinline__ longlong2 fx_sub(longlong2 a, longlong2 b) {
  longlong2 r;
  r.x = a.x - b.x;
  r.y = a.y - b.y;
  return r;
}
// a + i b and a - i b
__host__ __device__ __forceinline__ longlong2 fx_addi(longlong2 a, longlong2 b) {
  longlong2 r;
  r.x = a.x - b.y;
  r.y = a.y + b.x;
  return r;
}
__host__ __device__ __forceinline__ longlong2 fx_subi(longlong2 a, longlong2 b) {
  longlong2 r;
  r.x = a.x + b.y;
  r.y = a.y - b.x;
  return r;
}
__host__ __device__ __forceinline__ longlong2 fx_i(longlong2 a) {
  longlong2 r;
  r.x = -a.y;
  r.y = a.x;
  return r;
}

// Constants times 2^64 (those above one half less an integer, which fx_mulc's M adds back).
constexpr long long kS60m1 = -2471395088767036514LL;    // sin 60 - 1
constexpr long long kR5m1 = -8134700645620564469LL;     // sqrt(5)/4 - 1
constexpr long long kS72m1 = -902847917979075853LL;     // sin 72 - 1
constexpr long long kS72pm2 = -8506867872348575135LL;   // sin 72 + sin 36 - 2
constexpr long long kS72m = 6701172036390423429LL;      // sin 72 - sin 36
constexpr long long kR2m1 = -5402926248376769404LL;     // sqrt(1/2) - 1
constexpr long long kT20 = 6714065761956745581LL;       // tan 20
constexpr long long kS40m1 = -6589405544070453923LL;    // sin 40 - 1
constexpr long long kT5 = 1613880985413607648LL;        // tan 5
constexpr long long kS10 = 3203243492287910726LL;       // sin 10
constexpr long long kT10 = 3252658686418974684LL;       // tan 10
constexpr long long kS20 = 6309158051982071155LL;       // sin 20
constexpr long long kT11 = 3669285534148243471LL;       // tan 11.25
constexpr long long kS22 = 7059263338087549767LL;       // sin 22.5

// Rotation by a positive or negative angle as three shears: T = tan(angle/2), S = sin(angle).
template <long long T, long long S, int MS, int SIGN>
__host__ __device__ __forceinline__ longlong2 fx_shear(longlong2 v) {
  longlong2 r;
  const long long t0 = fx_mulc<T>(v.y);
  r.x = SIGN > 0 ? v.x - t0 : v.x + t0;
  const long long s0 = fx_mulc<S, MS>(r.x);
  r.y = SIGN > 0 ? v.y + s0 : v.y - s0;
  const long long t1 = fx_mulc<T>(r.y);
  r.x = SIGN > 0 ? r.x - t1 : r.x + t1;
  return r;
}
// v e^{2 pi i E / R}
template <int R, int E>
__host__ __device__ __forceinline__ longlong2 fx_rot(longlong2 v) {
  constexpr int e = E % R;
  if constexpr (e == 0) return v;
  else if constexpr (4 * e == R) return fx_i(v);
  else if constexpr (8 * e == R || 8 * e == 3 * R) {
    longlong2 r;
    r.x = fx_mulc<kR2m1, 1>(v.x - v.y);
    r.y = fx_mulc<kR2m1, 1>(v.x + v.y);
    if constexpr (8 * e == R) return r;
    else return fx_i(r);
  } else if constexpr (R == 9 && e == 1) return fx_shear<kT20, kS40m1, 1, 1>(v);
  else if constexpr (R == 9 && e == 2) return fx_i(fx_shear<kT5, kS10, 0, -1>(v));
  else if constexpr (R == 9 && e == 4) {
    const longlong2 r = fx_shear<kT10, kS20, 0, -1>(v);
    longlong2 o;
    o.x = -r.x;
    o.y = -r.y;
    return o;
  } else if constexpr (R == 16 && e == 1) return fx_shear<kT11, kS22, 0, 1>(v);
  else if constexpr (R == 16 && e == 3) return fx_i(fx_shear<kT11, kS22, 0, -1>(v));
  else {
    static_assert(R == 16 && e == 9, "rotation not tabulated");
    const longlong2 r = fx_shear<kT11, kS22, 0, 1>(v);
    longlong2 o;
    o.x = -r.x;
    o.y = -r.y;
    return o;
  }
}

template <int R> struct FxDft;
template <> struct FxDft<2> {
  static __host__ __device__ __forceinline__ void run(longlong2* v) {
    const longlong2 a = v[0], b = v[1];
    v[0] = fx_add(a, b);
    v[1] = fx_sub(a, b);
  }
};
template <> struct FxDft<3> {
  static __host__ __device__ __forceinline__ void run(longlong2* v) {
    const longlong2 t = fx_add(v[1], v[2]), s = fx_mulc<kS60m1, 1>(fx_sub(v[1], v[2]));
    longlong2 m;
    m.x = v[0].x - ((t.x + 1) >> 1);
    m.y = v[0].y - ((t.y + 1) >> 1);
    v[0] = fx_add(v[0], t);
    v[1] = fx_addi(m, s);
    v[2] = fx_subi(m, s);
  }
};
template <> struct FxDft<4> {
  static __host__ __device__ __forceinline__ void run(longlong2* v) {
    const longlong2 a = fx_add(v[0], v[2]), b = fx_sub(v[0], v[2]);
    const longlong2 c = fx_add(v[1], v[3]), d = fx_sub(v[1], v[3]);
    v[0] = fx_add(a, c);
    v[1] = fx_addi(b, d);
    v[2] = fx_sub(a, c);
    v[3] = fx_subi(b, d);
  }
};
// Winograd's 5-point form: four constants instead of eight
template <> struct FxDft<5> {
  static __host__ __device__ __forceinline__ void run(longlong2* v) {
    const longlong2 a1 = fx_add(v[1], v[4]), a2 = fx_add(v[2], v[3]);
    const longlong2 b1 = fx_sub(v[1], v[4]), b2 = fx_sub(v[2], v[3]);
    const longlong2 t = fx_add(a1, a2), d = fx_mulc<kR5m1, 1>(fx_sub(a1, a2));
    longlong2 m;
    m.x = v[0].x - ((t.x + 2) >> 2);
    m.y = v[0].y - ((t.y + 2) >> 2);
    const longlong2 u = fx_mulc<kS72m1, 1>(fx_add(b1, b2));
    const longlong2 q1 = fx_sub(u, fx_mulc<kS72m>(b2)), q2 = fx_sub(fx_mulc<kS72pm2, 2>(b1), u);
    const longlong2 p1 = fx_add(m, d), p2 = fx_sub(m, d);
    v[0] = fx_add(v[0], t);
    v[1] = fx_addi(p1, q1);
    v[4] = fx_subi(p1, q1);
    v[2] = fx_addi(p2, q2);
    v[3] = fx_subi(p2, q2);
  }
};
// R = A B with coprime A, B, no twiddles: input (B a + A b) mod R, output k with k = k1 mod A, k = k2 mod B
template <int A, int B> struct FxPfa {
  static constexpr int unit(int p, int q) {   // the k < p q that is 1 mod p and 0 mod q
    int k = 0;
    while (k % p != 1 || k % q != 0) ++k;
    return k;
  }
  static constexpr int EA = unit(A, B), EB = unit(B, A);
  static __host__ __device__ __forceinline__ void run(longlong2* x) {
    longlong2 y[A * B];
#pragma unroll
    for (int b = 0; b < B; ++b) {
      longlong2 t[A];
#pragma unroll
      for (int a = 0; a < A; ++a) t[a] = x[(B * a + A * b) % (A * B)];
      FxDft<A>::run(t);
#pragma unroll
      for (int a = 0; a < A; ++a) y[a * B + b] = t[a];
    }
#pragma unroll
    for (int a = 0; a < A; ++a) {
      FxDft<B>::run(y + a * B);
#pragma unroll
      for (int b = 0; b < B; ++b) x[(EA * a + EB * b) % (A * B)] = y[a * B + b];
    }
  }
};
template <> struct FxDft<6> : FxPfa<2, 3> {};
template <> struct FxDft<10> : FxPfa<2, 5> {};
template <> struct FxDft<12> : FxPfa<4, 3> {};
template <> struct FxDft<15> : FxPfa<3, 5> {};
template <> struct FxDft<8> {
  static __host__ __device__ __forceinline__ void run(longlong2* x) {
    longlong2 e[4], o[4];
#pragma unroll
    for (int n = 0; n < 4; ++n) {
      e[n] = fx_add(x[n], x[n + 4]);
      o[n] = fx_sub(x[n], x[n + 4]);
    }
    o[1] = fx_rot<8, 1>(o[1]);
    o[2] = fx_i(o[2]);
    o[3] = fx_rot<8, 3>(o[3]);
    FxDft<4>::run(e);
    FxDft<4>::run(o);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      x[2 * k] = e[k];
      x[2 * k + 1] = o[k];
    }
  }
};
template <> struct FxDft<9> {
  static __host__ __device__ __forceinline__ void run(longlong2* x) {
    longlong2 y[3][3];
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      longlong2 t[3] = {x[n], x[n + 3], x[n + 6]};
      FxDft<3>::run(t);
      y[0][n] = t[0];
      y[1][n] = t[1];
      y[2][n] = t[2];
    }
    y[1][1] = fx_rot<9, 1>(y[1][1]);
    y[1][2] = fx_rot<9, 2>(y[1][2]);
    y[2][1] = fx_rot<9, 2>(y[2][1]);
    y[2][2] = fx_rot<9, 4>(y[2][2]);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      FxDft<3>::run(y[k]);
      x[k] = y[k][0];
      x[k + 3] = y[k][1];
      x[k + 6] = y[k][2];
    }
  }
};
template <> struct FxDft<16> {
  static __host__ __device__ __forceinline__ void run(longlong2* x) {
    longlong2 y[4][4];
#pragma unroll
    for (int n = 0; n < 4; ++n) {
      longlong2 t[4] = {x[n], x[n + 4], x[n + 8], x[n + 12]};
      FxDft<4>::run(t);
      y[0][n] = t[0];
      y[1][n] = t[1];
      y[2][n] = t[2];
      y[3][n] = t[3];
    }
    y[1][1] = fx_rot<16, 1>(y[1][1]);
    y[1][2] = fx_rot<16, 2>(y[1][2]);
    y[1][3] = fx_rot<16, 3>(y[1][3]);
    y[2][1] = fx_rot<16, 2>(y[2][1]);
    y[2][2] = fx_rot<16, 4>(y[2][2]);
    y[2][3] = fx_rot<16, 6>(y[2][3]);
    y[3][1] = fx_rot<16, 3>(y[3][1]);
    y[3][2] = fx_rot<16, 6>(y[3][2]);
    y[3][3] = fx_rot<16, 9>(y[3][3]);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      FxDft<4>::run(y[k]);
#pragma unroll
      for (int m = 0; m < 4; ++m) x[k + 4 * m] = y[k][m];
    }
  }
};

// e^{2 pi i j / n} times 2^62 in balanced halves (cos = ch 2^32 + cl, sin = sh 2^32 + sl)
struct FxTw {
  int ch, cl, sh, sl;
};
__host__ __device__ __forceinline__ longlong2 fx_twiddle(longlong2 v, FxTw w) {
  const int xh = fx_hi(v.x), xl = fx_lo(v.x), yh = fx_hi(v.y), yl = fx_lo(v.y);
  long long p = (long long)xh * w.ch - (long long)yh * w.sh;
  long long t = (long long)xh * w.cl + (1LL << 29);
  t += (long long)xl * w.ch;
  t -= (long long)yh * w.sl;
  t -= (long long)yl * w.sh;
  longlong2 r;
  r.x = (long long)((unsigned long long)p << 2) + (t >> 30);
  p = (long long)xh * w.sh + (long long)yh * w.ch;
  t = (long long)xh * w.sl + (1LL << 29);
  t += (long long)xl * w.sh;
  t += (long long)yh * w.cl;
  t += (long long)yl * w.ch;
  r.y = (long long)((unsigned long long)p << 2) + (t >> 30);
  return r;
}

// q 2^d, rounded when d < 0 (|d| < 63), as a left and a right shift, one of them by zero: no selection per value
struct FxShift {
  int l, r;
  long long half;
  __host__ __device__ __forceinline__ explicit FxShift(int d)
      : l(d > 0 ? d : 0), r(d < 0 ? -d : 0), half(d < 0 ? 1LL << (-d - 1) : 0) {}
  __host__ __device__ __forceinline__ longlong2 operator()(longlong2 v) const {
    longlong2 o;
    o.x = ((long long)((unsigned long long)v.x << l) + half) >> r;
    o.y = ((long long)((unsigned long long)v.y << l) + half) >> r;
    return o;
  }
};

// A float64 from its bits as the integer m 2^(E - e0), E its exponent field (1 for a subnormal x) and m its significand
// (that is, x 2^(1075 - e0)), rounded.
__host__ __device__ __forceinline__ long long fx_from_bits(long long bits, int e0) {
  const int ex = (int)((bits >> 52) & 0x7ff);
  const long long m = (bits & 0xfffffffffffffLL) | (ex ? 0x10000000000000LL : 0LL);
  const int sh = (ex ? ex : 1) - e0;
  const long long q = sh >= 0 ? m << sh : (sh < -60 ? 0 : (m + (1LL << (-sh - 1))) >> -sh);
  return bits < 0 ? -q : q;
}

}  // namespace hpsi
