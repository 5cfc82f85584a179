// Local part of H|psi> in float64 contexts, in 64-bit fixed point (fixed_fft.cuh says why and how the line FFTs go).
//
// Three kernels per band block, the sphere-pruned order of the other local paths (App. A.1: V applied in real space
// between the two transforms), for any box whose edges are products of two of 2, 3, 4, 5, 6, 8, 9, 10, 12, 15, 16:
//   k_fx_zinv   per (chunk of sticks, band): psi(G) as integers with one exponent per chunk, inverse z-transform,
//               Zt[b][j3][stick] and the chunk's exponent.
//   k_fx_plane  per (z-plane, band): the plane [m1-plane][j2] in shared memory; inverse y, then in chunks of columns
//               inverse x, x V, forward x, then forward y; Y[b][j3][stick] and the plane's exponent.
//   k_fx_zfwd   per (chunk of sticks, band): forward z-transform, the sphere's values back to float64, 1/N_r,
//               plus the kinetic term in float64.
// Between the 1-D transforms a block is shifted so that its largest value (x: its largest column norm) and the
// transform's growth bound just stay below 2^63.  The exponents travel beside the rows: rows from different
// chunks or planes are aligned to the largest exponent of the block they meet in.  A non-finite psi makes its
// chunk's exponent kFxNan, which spreads to every value that the transform would have reached (NaN out).
//
// Work distribution: a stage's items (one R-point DFT each) are dealt over all threads of the CTA, so warps are full
// whatever R1 and R2 are, and the stages run in place in shared memory.  One kernel serves every box: the
// radices are run-time switches over the same codelets, since a codelet is hundreds of instructions.
//
// What bounds it: instruction issue and the latency of the multiplications (an add is 2 instructions, a 64-bit
// multiplication by a constant ~9); 27 bands of 90^3: 56% of issue cycles, ALU pipe 51%, DRAM 2%.  Measured on the 90^3
// box with 160 bands: plane kernel 19.35 -> 2.6 ms, z kernels 1.07 + 1.17 -> 0.28 + 0.30 ms against float64 register codelets; 32 cells of 25^3 to 50^3: 9.6 -> 1.41 ms
// (planes); 27 x 30 x 32: 428 -> 31 us against the float64 Stockham kernels.  Error of the local term against 128-bit
// arithmetic: below the float64 kernels' at every edge tried (16 to 135), by 5 to 40%.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "fixed_fft.cuh"
#include "hpsi_internal.h"

namespace hpsi {

namespace {

#include "line_stages.cuh"

// Fixed-point arithmetic for the line stages
struct FixArith {
  using V = longlong2;
  using Tw = FxTw;
  template <int R> using Dft = FxDft<R>;
  static __device__ __forceinline__ longlong2 twiddle(longlong2 v, FxTw w) { return fx_twiddle(v, w); }
};

constexpr int kFxNan = 1 << 28;      // exponent of a block that holds a non-finite value
constexpr int kFxZero = -(1 << 20);  // exponent of a block of zeros

struct FxItem {
  int nb, npw, npl, nst;
  int n1, n2, n3;
  LineAxis ax[3];
  int cw;                       // columns per x chunk
  int nch;                      // z chunks
  int hz, hy, hx, s3, hyf, hzf; // growth bounds of the transforms, in bits (FixedPlan)
  const int *soff, *zoff, *zbeg;   // Problem's lookup tables
  const int* xmap;
  const double2* psi;
  double2* hpsi;
  const double* kin;
  longlong2* Zt;                // [nb][n3][nst]
  longlong2* Yb;                // [nb][n3][nst]
  int* Ez;                      // [nb][nch]
  int* Ey;                      // [nb][n3]
  const long long* V;           // [n3][slot of j1][slot of j2], V 2^(62 - vexp)
  const int* vexp;
  double inv_nr;
};

struct FxBatch {
  int nitems;
  int off_z[kMaxLocalItems + 1];   // first z tile of each item (nch x nb tiles)
  int off_p[kMaxLocalItems + 1];   // first plane tile (n3 x nb tiles)
  FxItem item[kMaxLocalItems];
};

// Resident threads per SM the plane kernel's registers allow (80 and 128 a thread): more warps hide more of the
// multiplications' latency, but the 16-point codelet alone holds 64 registers of data.
template <int MAXR> constexpr int kFxThreads = MAXR > 10 ? 512 : 768;

__device__ __forceinline__ unsigned long long fx_mag(longlong2 v) {
  return (unsigned long long)((v.x ^ (v.x >> 63)) | (v.y ^ (v.y >> 63)));
}
// q >> d with rounding, d >= 0 (any size)
__device__ __forceinline__ longlong2 fx_align(longlong2 v, int d) {
  longlong2 r;
  if (d == 0) return v;
  if (d > 62) {
    r.x = r.y = 0;
    return r;
  }
  r.x = (v.x + (1LL << (d - 1))) >> d;
  r.y = (v.y + (1LL << (d - 1))) >> d;
  return r;
}

// Shared scratch of a tile's CTA-wide reductions.
struct FxShared {
  unsigned long long mag;
  int emax;
  float norm;
  int tile;
};

// One OR of every thread's bits (all threads call; sh->mag is cleared by the caller a barrier earlier).
__device__ __forceinline__ void fx_or(FxShared* sh, unsigned long long m) {
  const unsigned lo = __reduce_or_sync(0xffffffffu, (unsigned)m);
  const unsigned hi = __reduce_or_sync(0xffffffffu, (unsigned)(m >> 32));
  if ((threadIdx.x & 31) == 0) {
    unsigned* w = reinterpret_cast<unsigned*>(&sh->mag);
    if (lo) atomicOr(w, lo);
    if (hi) atomicOr(w + 1, hi);
  }
}
// Shift that brings values below 2^bits(m) up to (or down to) 2^(63 - head)
__device__ __forceinline__ int fx_headroom(unsigned long long m, int head) { return (int)__clzll((long long)m) - 1 - head; }

struct FxPlaced {   // a value and its place in the tile
  longlong2 v;
  int at;
};

// Inverse z-transform of one chunk of sticks of one band.
template <int MAXR>
__device__ __forceinline__ void fx_zinv_tile(const FxItem& a, int ch, int b, unsigned char* smem, FxShared* sh) {
  constexpr int SC = kStickChunk, ld = SC + 1;
  const int n = a.n3;
  FxTw* tw = reinterpret_cast<FxTw*>(smem);
  longlong2* L = reinterpret_cast<longlong2*>(smem + sizeof(FxTw) * n);   // [cell][stick], rows of SC + 1
  const int s0 = ch * SC, ns = min(SC, a.nst - s0);
  const int lane = threadIdx.x & 31;
  // the chunk's sticks are one contiguous range of G
  const int g0 = a.zbeg[ch], ng = a.zbeg[ch + 1] - g0;
  const longlong2* ps = reinterpret_cast<const longlong2*>(a.psi + (size_t)b * a.npw + g0);
  if (threadIdx.x == 0) sh->emax = 0;
  load_table(tw, a.ax[2].fxtw, a.ax[2]);
  for (int i = threadIdx.x; i < n * ld; i += blockDim.x) L[i] = {0, 0};
  __syncthreads();
  // float64 bits into their places, and the largest exponent field
  unsigned hi = 0, any = 0;
  staged_loop(ng, [&](int i) { return FxPlaced{ps[i], a.zoff[g0 + i]}; },
              [&](int, FxPlaced q) {
                hi = max(hi, max((unsigned)(q.v.x >> 32) & 0x7fffffffu, (unsigned)(q.v.y >> 32) & 0x7fffffffu));
                any |= (unsigned)q.v.x | (unsigned)q.v.y;
                L[q.at] = q.v;
              });
  hi = __reduce_max_sync(0xffffffffu, max(hi, any != 0 ? 1u : 0u));
  if (lane == 0) atomicMax(&sh->emax, (int)hi);
  __syncthreads();
  hi = (unsigned)sh->emax;
  const int emax = max(1, (int)(hi >> 20));   // subnormal numbers have exponent 1
  if (threadIdx.x == 0)
    a.Ez[(size_t)b * a.nch + ch] = emax == 0x7ff ? kFxNan : hi == 0 ? kFxZero : emax - 1022 - 63 + a.hz;
  if (emax == 0x7ff) return;   // (every thread) the plane kernel reads the exponent only
  // |x| < 2^(emax - 1022), so q = x 2^(63 - hz - (emax - 1022)) stays below 2^(63 - hz).  The bits become integers as the
  // first stage reads them (a cell without a G holds the bits of zero).
  const int e0 = emax - 10 + a.hz;
  auto to_fixed = [&](longlong2 w) {
    longlong2 v;
    v.x = fx_from_bits(w.x, e0);
    v.y = fx_from_bits(w.y, e0);
    return v;
  };
  const LineView<longlong2> lines{L, 1, ld};
  line_stage1<FixArith, MAXR, false>(a.ax[2], ns, tw, lines, to_fixed);
  __syncthreads();
  line_stage2<FixArith, MAXR, false>(a.ax[2], ns, tw, lines);
  __syncthreads();
  longlong2* Z = a.Zt + (size_t)b * n * a.nst + s0;
  const int per = blockDim.x / SC, r0 = threadIdx.x / SC, sl = threadIdx.x % SC;
  if (sl < ns)
    for (int j3 = r0; j3 < n; j3 += per) Z[(size_t)j3 * a.nst + sl] = L[a.ax[2].slot[j3] * ld + sl];
}

template <int MAXR>
__device__ __forceinline__ void fx_plane_tile(const FxItem& a, int j3, int b, unsigned char* smem, FxShared* sh) {
  const int n1 = a.n1, n2 = a.n2, npl = a.npl, PS = n2 | 1, cw = a.cw;
  FxTw* twx = reinterpret_cast<FxTw*>(smem);
  FxTw* twy = twx + (a.ax[0].twiddled ? n1 : 0);
  longlong2* P = reinterpret_cast<longlong2*>(twy + (a.ax[1].twiddled ? n2 : 0));  // [plane][cell of j2], a row of zeros
  longlong2* X = P + (size_t)(npl + 1) * PS;                                       // [cell of x][column of the chunk]
  int* xo = reinterpret_cast<int*>(X + (size_t)n1 * cw);
  float* cn = reinterpret_cast<float*>(X);                                         // column norms, before X is in use
  const int lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    sh->mag = 0;
    sh->emax = kFxZero;
    sh->norm = 0.f;
  }
  load_table(twx, a.ax[0].fxtw, a.ax[0]);
  load_table(twy, a.ax[1].fxtw, a.ax[1]);
  build_row_table(xo, a.ax[0], a.xmap, PS, npl * PS);
  for (int i = threadIdx.x; i < (npl + 1) * PS; i += blockDim.x) P[i] = {0, 0};
  __syncthreads();
  const int* ez = a.Ez + (size_t)b * a.nch;
  int em = kFxZero;
  for (int i = threadIdx.x; i < a.nch; i += blockDim.x) em = max(em, ez[i]);
  em = __reduce_max_sync(0xffffffffu, em);
  if (lane == 0 && em > kFxZero) atomicMax(&sh->emax, em);
  __syncthreads();
  int e = sh->emax;
  const int ve = *a.vexp;
  if (e >= kFxNan / 2 || ve >= kFxNan / 2) {
    if (threadIdx.x == 0) a.Ey[(size_t)b * a.n3 + j3] = kFxNan;
    return;
  }
  // the plane's sticks, aligned to the largest exponent
  const longlong2* zin = a.Zt + ((size_t)b * a.n3 + j3) * a.nst;
  struct In {
    longlong2 v;
    int at, e;
  };
  unsigned long long m = 0;
  staged_loop(a.nst, [&](int i) { return In{zin[i], a.soff[i], ez[i / kStickChunk]}; },
              [&](int, In q) {
                const longlong2 v = fx_align(q.v, e - q.e);
                m |= fx_mag(v);
                P[q.at] = v;
              });
  fx_or(sh, m);
  __syncthreads();
  m = sh->mag;
  if (m == 0) {   // a plane of zeros: zeros out
    longlong2* yo = a.Yb + ((size_t)b * a.n3 + j3) * a.nst;
    const longlong2 z = {0, 0};
    for (int i = threadIdx.x; i < a.nst; i += blockDim.x) yo[i] = z;
    if (threadIdx.x == 0) a.Ey[(size_t)b * a.n3 + j3] = kFxZero;
    return;
  }
  const LineView<longlong2> rows{P, PS, 1};
  {
    const int d = fx_headroom(m, a.hy);
    e -= d;
    line_stage1<FixArith, MAXR, false>(a.ax[1], npl, twy, rows, FxShift(d));
  }
  __syncthreads();
  line_stage2<FixArith, MAXR, false>(a.ax[1], npl, twy, rows);
  if (threadIdx.x == 0) sh->mag = 0;
  __syncthreads();
  // the largest column norm, in units of 2^32, rounded up (the +2 and the factor cover every rounding here)
  for (int i = threadIdx.x; i < 4 * n2; i += blockDim.x) {
    const int part = i / n2, c = i - part * n2;
    float s = 0.f;
    for (int p = part; p < npl; p += 4) {
      const longlong2 v = P[p * PS + c];
      const float x = (float)(abs((int)(v.x >> 32)) + 2), y = (float)(abs((int)(v.y >> 32)) + 2);
      s = fmaf(x, x, fmaf(y, y, s));
    }
    cn[i] = s;
  }
  __syncthreads();
  {
    float s = 0.f;
    for (int c = threadIdx.x; c < n2; c += blockDim.x) s = fmaxf(s, cn[c] + cn[n2 + c] + cn[2 * n2 + c] + cn[3 * n2 + c]);
    const unsigned u = __reduce_max_sync(0xffffffffu, __float_as_uint(s));
    if (lane == 0) atomicMax(reinterpret_cast<unsigned*>(&sh->norm), u);
  }
  __syncthreads();
  // norm < 2^bits: bits from the exponent of its square
  const float nrm = sh->norm * 1.001f;
  const int sq = (int)((__float_as_uint(nrm) >> 23) & 0xff) - 126;   // square < 2^sq (in units of 2^64)
  const int bits = 32 + ((sq + 1) >> 1);
  const int dx = 63 - bits - a.hx;
  const FxShift shx(dx);
  e += ve + 2 + a.s3 - dx;
  const long long* V = a.V + (size_t)j3 * n1 * n2;
  unsigned long long my = 0;
  const LineView<longlong2> cols{X, 1, cw};
  for (int c0 = 0; c0 < n2; c0 += cw) {
    const int nc = min(cw, n2 - c0);
    x_stage1<FixArith, MAXR>(a.ax[0], nc, twx, xo, P + c0, cols, shx);
    __syncthreads();
    radix_switch<MAXR>(a.ax[0].r2, [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      const LineAxis& ax = a.ax[0];
      const int items = nc * ax.r1;
      const float inv = 1.0f / (float)nc;
      for (int it = threadIdx.x; it < items; it += blockDim.x) {
        int k1, c;
        split_index(it, nc, inv, k1, c);
        longlong2* q = X + k1 * R * cw + c;
        const long long* vp = V + (size_t)(k1 * R) * n2 + c0 + c;
        longlong2 v[R];
#pragma unroll
        for (int i = 0; i < R; ++i) v[i] = q[i * cw];
        FxDft<R>::run(v);
#pragma unroll
        for (int i = 0; i < R; ++i) {
          const long long w = __ldg(vp + i * n2);
          const int wh = fx_hi(w), wl = fx_lo(w);
          const longlong2 u = {fx_mulr(v[i].y, wh, wl), fx_mulr(v[i].x, wh, wl)};   // swapped: the forward sign
          v[i] = u;
        }
        FxDft<R>::run(v);
        const int s3 = a.s3;
        const long long half = s3 ? 1LL << (s3 - 1) : 0;
#pragma unroll
        for (int i = 0; i < R; ++i) {
          longlong2 u = {(v[i].x + half) >> s3, (v[i].y + half) >> s3};
          if (i > 0 && ax.twiddled) u = fx_twiddle(u, twx[k1 * i]);
          q[i * cw] = u;
        }
      }
    });
    __syncthreads();
    x_stage1_rev<FixArith, MAXR>(a.ax[0], nc, xo, npl * PS, cols, P + c0, [&](longlong2 v) { my |= fx_mag(v); });
    __syncthreads();
  }
  fx_or(sh, my);
  __syncthreads();
  my = sh->mag;
  const int d = my ? fx_headroom(my, a.hyf) : 0;
  e -= d;
  line_stage2<FixArith, MAXR, true>(a.ax[1], npl, twy, rows, FxShift(d));
  __syncthreads();
  line_stage1<FixArith, MAXR, true>(a.ax[1], npl, twy, rows);
  __syncthreads();
  longlong2* yo = a.Yb + ((size_t)b * a.n3 + j3) * a.nst;
  // still swapped: the z kernel goes on with the forward sign
  staged_loop(a.nst, [&](int i) { return a.soff[i]; }, [&](int i, int at) { yo[i] = P[at]; });
  if (threadIdx.x == 0) a.Ey[(size_t)b * a.n3 + j3] = my ? e : kFxZero;
}

template <int MAXR>
__device__ __forceinline__ void fx_zfwd_tile(const FxItem& a, int ch, int b, unsigned char* smem, FxShared* sh) {
  constexpr int SC = kStickChunk, ld = SC + 1;
  const int n = a.n3;
  FxTw* tw = reinterpret_cast<FxTw*>(smem);
  longlong2* L = reinterpret_cast<longlong2*>(smem + sizeof(FxTw) * n);
  const int s0 = ch * SC, ns = min(SC, a.nst - s0);
  const int lane = threadIdx.x & 31;
  const int g0 = a.zbeg[ch], ng = a.zbeg[ch + 1] - g0;
  if (threadIdx.x == 0) {
    sh->emax = kFxZero;
    sh->mag = 0;
  }
  load_table(tw, a.ax[2].fxtw, a.ax[2]);
  __syncthreads();
  const int* ey = a.Ey + (size_t)b * n;
  int em = kFxZero;
  for (int i = threadIdx.x; i < n; i += blockDim.x) em = max(em, ey[i]);
  em = __reduce_max_sync(0xffffffffu, em);
  if (lane == 0 && em > kFxZero) atomicMax(&sh->emax, em);
  __syncthreads();
  int e = sh->emax;
  const bool bad = e >= kFxNan / 2;
  if (!bad) {
    const longlong2* Y = a.Yb + (size_t)b * n * a.nst + s0;
    struct In {
      longlong2 v;
      int e;
    };
    unsigned long long m = 0;
    staged_loop(
        n * SC,
        [&](int i) {
          In q{{0, 0}, e};
          if (i % SC < ns) q = In{Y[(size_t)(i / SC) * a.nst + i % SC], ey[i / SC]};
          return q;
        },
        [&](int i, In q) {
          const longlong2 v = fx_align(q.v, e - q.e);
          m |= fx_mag(v);
          L[a.ax[2].slot[i / SC] * ld + i % SC] = v;
        });
    fx_or(sh, m);
    __syncthreads();
    m = sh->mag;
    const int d = m ? fx_headroom(m, a.hzf) : 0;
    e -= d;
    const LineView<longlong2> lines{L, 1, ld};
    line_stage2<FixArith, MAXR, true>(a.ax[2], ns, tw, lines, FxShift(d));
    __syncthreads();
    line_stage1<FixArith, MAXR, true>(a.ax[2], ns, tw, lines);
    __syncthreads();
  }
  // f = 2^e / N_r by its exponent field; where that would leave the normal numbers, f g with g = 2^-+1000: the results,
  // 2^62 larger, may well be normal
  const int fe = (int)(__double_as_longlong(a.inv_nr) >> 52) + e;
  const int shift = fe <= 0 ? 1000 : fe >= 0x7ff ? -1000 : 0;
  const double f = bad                                    ? __longlong_as_double(0x7ff8000000000000LL)
                   : fe + shift > 0 && fe + shift < 0x7ff ? __longlong_as_double(__double_as_longlong(a.inv_nr) +
                                                                                 ((long long)(e + shift) << 52))
                   : fe > 0                               ? INFINITY
                                                          : 0.0;
  const double g = __longlong_as_double((long long)(1023 - shift) << 52);
  struct Out {
    double2 x;
    double kg;
    int at;
  };
  const double2* ps = a.psi + (size_t)b * a.npw + g0;
  double2* out = a.hpsi + (size_t)b * a.npw + g0;
  auto load = [&](int i) { return Out{ps[i], a.kin[g0 + i], a.zoff[g0 + i]}; };
  if (shift == 0 || bad)
    staged_loop(ng, load, [&](int i, Out q) {
      longlong2 v = {0, 0};
      if (!bad) v = L[q.at];   // swapped
      out[i] = make_double2(fma(q.kg, q.x.x, (double)v.y * f), fma(q.kg, q.x.y, (double)v.x * f));
    });
  else
    staged_loop(ng, load, [&](int i, Out q) {
      const longlong2 v = L[q.at];
      out[i] = make_double2(fma(q.kg, q.x.x, (double)v.y * f * g), fma(q.kg, q.x.y, (double)v.x * f * g));
    });
}

template <int MAXR>
__global__ void __launch_bounds__(256, MAXR > 10 ? 2 : 3) k_fx_zinv(const __grid_constant__ FxBatch bt) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ FxShared sh;
  const int i = tile_item(bt.off_z, bt.nitems, blockIdx.x), l = blockIdx.x - bt.off_z[i];
  fx_zinv_tile<MAXR>(bt.item[i], l % bt.item[i].nch, l / bt.item[i].nch, smem_raw, &sh);
}
template <int MAXR>
__global__ void __launch_bounds__(kFxThreads<MAXR>, 1) k_fx_plane(const __grid_constant__ FxBatch bt) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ FxShared sh;
  const int i = tile_item(bt.off_p, bt.nitems, blockIdx.x), l = blockIdx.x - bt.off_p[i];
  fx_plane_tile<MAXR>(bt.item[i], l % bt.item[i].n3, l / bt.item[i].n3, smem_raw, &sh);
}
template <int MAXR>
__global__ void __launch_bounds__(256, MAXR > 10 ? 2 : 3) k_fx_zfwd(const __grid_constant__ FxBatch bt) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ FxShared sh;
  const int i = tile_item(bt.off_z, bt.nitems, blockIdx.x), l = blockIdx.x - bt.off_z[i];
  fx_zfwd_tile<MAXR>(bt.item[i], l % bt.item[i].nch, l / bt.item[i].nch, smem_raw, &sh);
}

#include "nonlocal_tiles.cuh"

// The whole batch in one cooperative launch: the tiles of the three kernels above phase by phase, and, when
// nl.nitems > 0, the float64 nonlocal term of the items, with a bounded grid barrier between the phases.  CTAs
// take tiles from a phase's list one at a time through an atomic counter.
struct FxPersist {
  unsigned* bar;   // [0]: arrival counter; [1 + phase]: tile counters; zero at launch
  int* err;
};

template <int MAXR>
__global__ void __launch_bounds__(256, 2) k_fx_batch(const __grid_constant__ FxBatch bt,
                                                     const __grid_constant__ NlBatch nl, const FxPersist pc) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ FxShared sh;
  const unsigned G = gridDim.x;
  const int nz = bt.off_z[bt.nitems], np = bt.off_p[bt.nitems];
  for (int t = persist_next(pc.bar + 1); t < nz; t = persist_next(pc.bar + 1)) {
    const int i = tile_item(bt.off_z, bt.nitems, t), l = t - bt.off_z[i];
    fx_zinv_tile<MAXR>(bt.item[i], l % bt.item[i].nch, l / bt.item[i].nch, smem_raw, &sh);
  }
  if (!persist_sync(pc.bar, G, pc.err)) return;
  for (int t = persist_next(pc.bar + 2); t < np; t = persist_next(pc.bar + 2)) {
    const int i = tile_item(bt.off_p, bt.nitems, t), l = t - bt.off_p[i];
    fx_plane_tile<MAXR>(bt.item[i], l % bt.item[i].n3, l / bt.item[i].n3, smem_raw, &sh);
  }
  if (!persist_sync(pc.bar, 2 * G, pc.err)) return;
  for (int t = persist_next(pc.bar + 3); t < nz; t = persist_next(pc.bar + 3)) {
    const int i = tile_item(bt.off_z, bt.nitems, t), l = t - bt.off_z[i];
    fx_zfwd_tile<MAXR>(bt.item[i], l % bt.item[i].nch, l / bt.item[i].nch, smem_raw, &sh);
  }
  if (nl.nitems > 0) nonlocal_phases(nl, pc.bar, pc.err, G, 3, reinterpret_cast<double2*>(smem_raw));
}

// ---- setup ------------------------------------------------------------------------------------

constexpr int kRadices[] = {2, 3, 4, 5, 6, 8, 9, 10, 12, 15, 16};

int gcd(int a, int b) { return b ? gcd(b, a % b) : a; }
int ceil_log2(double x) { return std::max(0, (int)std::ceil(std::log2(x))); }

// The largest |V| bit pattern (NaN above infinity above every finite value)
__global__ void k_fx_vmax(size_t n, const double* __restrict__ v, unsigned long long* __restrict__ out) {
  unsigned long long m = 0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    m = max(m, (unsigned long long)__double_as_longlong(v[i]) & 0x7fffffffffffffffULL);
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}
// V[j3][j2][j1] -> [j3][slot of j1][slot of j2] as V 2^(62 - vexp), |V| < 2^vexp
__global__ void k_fx_v(LineAxis a1, LineAxis a2, int n3, const double* __restrict__ v,
                       const unsigned long long* __restrict__ vmax, long long* __restrict__ out, int* __restrict__ vexp) {
  const int emax = max(1, (int)(*vmax >> 52));
  const size_t n = (size_t)a1.n * a2.n * n3;
  if (blockIdx.x == 0 && threadIdx.x == 0) *vexp = emax == 0x7ff ? kFxNan : *vmax == 0 ? 0 : emax - 1022;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const int j1 = (int)(i % a1.n), j2 = (int)(i / a1.n % a2.n);
    const size_t j3 = i / ((size_t)a1.n * a2.n);
    out[(j3 * a1.n + a1.slot[j1]) * a2.n + a2.slot[j2]] = fx_from_bits(__double_as_longlong(v[i]), emax - 9);
  }
}

struct FxLaunch {
  FxBatch bt;
  size_t smem_z = 0, smem_p = 0;
  int maxr = 0, items = 0;   // largest radix, largest stage of a plane
  int block = 0;             // plane block of the item with the largest planes
  void add(Context& c, const Problem& p, const double2* psi, double2* hpsi, int nb, void* zt, void* yb) {
    const int i = bt.nitems++;
    FxItem& it = bt.item[i];
    const FixedPlan& f = p.fixed;
    it.nb = nb;
    it.npw = p.npw;
    it.npl = p.npl;
    it.nst = p.nst;
    it.n1 = p.n[0];
    it.n2 = p.n[1];
    it.n3 = p.n[2];
    for (int a = 0; a < 3; ++a) {
      it.ax[a] = f.ax[a];
      maxr = std::max(maxr, std::max(f.ax[a].r1, f.ax[a].r2));
    }
    items = std::max(items, std::max(it.npl * std::max(f.ax[1].r1, f.ax[1].r2), f.cw * std::max(f.ax[0].r1, f.ax[0].r2)) + 31);
    it.cw = f.cw;
    it.nch = f.nch;
    it.hz = f.hz;
    it.hy = f.hy;
    it.hx = f.hx;
    it.s3 = f.s3;
    it.hyf = f.hyf;
    it.hzf = f.hzf;
    it.soff = p.tab[HPSI_FP64].soff;
    it.zoff = p.tab[HPSI_FP64].zoff;
    it.zbeg = p.tab[HPSI_FP64].zbeg;
    it.xmap = p.d_xmap;
    it.psi = psi;
    it.hpsi = hpsi;
    it.kin = p.d_kin;
    const size_t rows = (size_t)nb * p.n[2] * p.nst;
    it.Zt = static_cast<longlong2*>(zt);
    it.Yb = static_cast<longlong2*>(yb);
    it.Ez = reinterpret_cast<int*>(it.Zt + rows);   // beside the rows (local_row_bytes)
    it.Ey = reinterpret_cast<int*>(it.Yb + rows);
    it.V = static_cast<const long long*>(c.vbufs[p.vslot + 2]);
    it.vexp = reinterpret_cast<const int*>(it.V + (size_t)p.n[0] * p.n[1] * p.n[2]) + 2;
    it.inv_nr = 1.0 / ((double)p.n[0] * p.n[1] * p.n[2]);
    bt.off_z[i + 1] = bt.off_z[i] + f.nch * nb;
    bt.off_p[i + 1] = bt.off_p[i] + p.n[2] * nb;
    smem_z = std::max(smem_z, f.smem_z);
    if (f.smem_p > smem_p) block = f.block;
    smem_p = std::max(smem_p, f.smem_p);
  }
  void reset() {
    bt.nitems = 0;
    bt.off_z[0] = bt.off_p[0] = 0;
    smem_z = smem_p = 0;
    maxr = items = 0;
  }
  template <int MAXR> int run_t(Context& c) {
    static std::atomic<unsigned long long> devices{0};
    cudaError_t e = allow_smem(c, devices, {(const void*)k_fx_zinv<MAXR>, (const void*)k_fx_plane<MAXR>, (const void*)k_fx_zfwd<MAXR>});
    if (e != cudaSuccess) return cuda_fail(c, e, "fixed-point local kernels");
    const int nz = bt.off_z[bt.nitems], np = bt.off_p[bt.nitems];
    // plane_shape's block, or one round of a stage's items where there is a CTA per SM at most; never more than this
    // instance's launch bound, which another item's radix may have set (any block size serves: items are dealt over it)
    const int want = np <= c.sm_count ? std::max(block, items / 32 * 32) : block;
    const int plane = std::min(kFxThreads<MAXR>, want);
    HPSI_LAUNCH(c, HPSI_K_INV_ZY, (k_fx_zinv<MAXR><<<nz, 256, smem_z, c.stream>>>(bt)));
    HPSI_LAUNCH(c, HPSI_K_XVX_Y, (k_fx_plane<MAXR><<<np, plane, smem_p, c.stream>>>(bt)));
    HPSI_LAUNCH(c, HPSI_K_FWD_Z, (k_fx_zfwd<MAXR><<<nz, 256, smem_z, c.stream>>>(bt)));
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(c, e, "fixed-point local kernels launch");
    return HPSI_OK;
  }
  int run(Context& c) { return maxr > 10 ? run_t<16>(c) : run_t<10>(c); }
  template <int MAXR> int persistent_t(Context& c, const NlBatch& nl, unsigned* bar, bool* done) {
    const void* kern = (const void*)k_fx_batch<MAXR>;
    size_t dyn = std::max(smem_z, smem_p);
    if (nl.nitems > 0) dyn = std::max(dyn, sizeof(double2) * (size_t)std::max(CB_SMEM, AV_SMEM));
    static std::atomic<unsigned long long> devices{0};
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, kern) != cudaSuccess || fa.sharedSizeBytes + dyn > c.smem_optin ||
        allow_smem(c, devices, {kern}) != cudaSuccess) {
      cudaGetLastError();
      return HPSI_OK;
    }
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, 256, dyn) != cudaSuccess || occ < 1) {
      cudaGetLastError();
      return HPSI_OK;
    }
    cudaError_t e = cudaMemsetAsync(bar, 0, 8 * sizeof(unsigned), c.stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "persistent batch barrier reset");
    FxPersist pc{bar, c.d_err};
    void* args[] = {(void*)&bt, (void*)&nl, (void*)&pc};
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(occ * c.sm_count);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = dyn;
    cfg.stream = c.stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    HPSI_LAUNCH(c, HPSI_K_BATCH, (e = cudaLaunchKernelExC(&cfg, kern, args)));
    if (e != cudaSuccess) return cuda_fail(c, e, "persistent batched H|psi> launch");
    *done = true;
    return HPSI_OK;
  }
  int persistent(Context& c, const NlBatch& nl, unsigned* bar, bool* done) {
    return maxr > 10 ? persistent_t<16>(c, nl, bar, done) : persistent_t<10>(c, nl, bar, done);
  }
};

}  // namespace

// Factors of an edge (0 if it has none), r1 >= r2: that gives the x stage between the transforms more items and a
// tighter bound.  Fixed point: coprime ones first (a twiddle costs as much as a third of a codelet), then the smaller larger one.
// Float32: factors up to 10, else up to 12 (the codelets' registers set how many threads an SM holds), and among
// those the same order.
static void line_factors(int n, int precision, int* r1, int* r2) {
  *r1 = *r2 = 0;
  int best = 0;
  for (int a : kRadices)
    for (int b : kRadices) {
      if (a * b != n || a < b) continue;
      const int size = precision == HPSI_FP64 ? 0 : a <= 10 ? 0 : a <= 12 ? 1 : 2;
      const int rank = 1000 * size + (gcd(a, b) == 1 ? 0 : 100) + a;
      if (*r1 == 0 || rank < best) {
        *r1 = a;
        *r2 = b;
        best = rank;
      }
    }
}

// The table of an edge (empty if it has no factors): in the Cooley-Tukey form the twiddles e^{2 pi i j / n} in fixed point
// and, from *ftw on, in float32; from *cells on the cell of every index before the inverse transform and after it.
void line_tables(int n, int precision, std::vector<int>& table, size_t* ftw, size_t* cells, LineAxis* ax) {
  int r1, r2;
  line_factors(n, precision, &r1, &r2);
  ax->n = n;
  ax->r1 = r1;
  ax->r2 = r2;
  table.clear();
  if (!r1) return;
  const bool pfa = gcd(r1, r2) == 1;
  ax->s2 = pfa ? r1 : 1;
  ax->twiddled = !pfa;
  std::vector<int> tw32;
  for (int j = 0; j < (pfa ? 0 : n); ++j) {
    // reduced to the first octant, so that long double keeps 62 bits
    const int o = 8 * j / n, r = 8 * j % n;
    const long double pi4 = 0.785398163397448309615660845819875721L;
    const long double th = pi4 * (long double)((o & 1) ? n - r : r) / (long double)n;
    const long double c0 = std::cos(th), s0 = std::sin(th);
    long double c = 0, s = 0;
    switch (o) {
      case 0: c = c0; s = s0; break;
      case 1: c = s0; s = c0; break;
      case 2: c = -s0; s = c0; break;
      case 3: c = -c0; s = s0; break;
      case 4: c = -c0; s = -s0; break;
      case 5: c = -s0; s = -c0; break;
      case 6: c = s0; s = -c0; break;
      default: c = c0; s = -s0; break;
    }
    for (const long double x : {c, s}) {
      const long long q = std::llround(x * 4611686018427387904.0L);
      table.push_back(fx_hi(q));
      table.push_back(fx_lo(q));
      const float f = (float)x;
      int bits = 0;
      std::memcpy(&bits, &f, sizeof(bits));
      tw32.push_back(bits);
    }
  }
  *ftw = table.size();
  table.insert(table.end(), tw32.begin(), tw32.end());
  *cells = table.size();
  std::vector<int> cell(n);
  for (int a = 0; a < r1; ++a)
    for (int t = 0; t < r2; ++t) cell[(r2 * a + ax->s2 * t) % n] = a * r2 + t;
  table.insert(table.end(), cell.begin(), cell.end());
  for (int k = 0; k < n; ++k) table.push_back((k % r1) * r2 + (pfa ? k % r2 : k / r1));
}

// The plan of a problem whose axes are filled in (ok = false: no factors, or a plane does not fit).
void fixed_plan(Problem& p, size_t smem_optin) {
  FixedPlan& f = p.fixed;
  f.ok = false;
  for (int a = 0; a < 3; ++a)
    if (!f.ax[a].r1) return;
  const int n1 = p.n[0], n2 = p.n[1], n3 = p.n[2];
  auto tws = [&](int a) { return f.ax[a].twiddled ? sizeof(FxTw) * (size_t)p.n[a] : 0; };
  f.nch = (p.nst + kStickChunk - 1) / kStickChunk;
  f.smem_z = sizeof(FxTw) * (size_t)n3 + sizeof(longlong2) * (size_t)n3 * (kStickChunk + 1);
  const size_t base = tws(0) + tws(1) + sizeof(longlong2) * (size_t)(p.npl + 1) * (n2 | 1) +
                      sizeof(int) * f.ax[0].r2 * (size_t)((f.ax[0].r1 + 3) & ~3);
  const size_t col = sizeof(longlong2) * (size_t)n1;
  int rmax = 0;
  for (int a = 0; a < 3; ++a) rmax = std::max(rmax, f.ax[a].r1);
  plane_shape(f.ax[0], f.ax[1], p.npl, base, col, smem_optin, rmax > 10 ? kFxThreads<16> : kFxThreads<10>, &f.cw, &f.block);
  if (f.cw == 0) return;
  f.smem_p = base + col * f.cw;
  if (col * f.cw < sizeof(float) * 4 * (size_t)n2 || f.smem_z > smem_optin - 1024) return;
  int zl = 1;
  for (const StickDev& s : p.sticks) zl = std::max(zl, s.len);
  // growth bounds: sum |x_n| <= L sqrt2 max for the stages scaled by their largest component ...
  const double r2 = std::sqrt(2.0);
  f.hz = ceil_log2(kFixGain * r2 * zl);
  f.hy = ceil_log2(kFixGain * r2 * p.ns_max);
  f.hyf = ceil_log2(kFixGain * r2 * n2);
  f.hzf = ceil_log2(kFixGain * r2 * n3);
  // ... and for the x stages, scaled by the largest column 2-norm B: sqrt(npl) B before V; behind V (scaled to 1/4)
  // sqrt(n1) B / 4 is the line's 2-norm, so sqrt(R2 n1) B / 4 after the first codelet and n1 B / 4 at the end, with
  // s3 further bits given up in between
  f.hx = ceil_log2(kFixGain * std::max(std::sqrt((double)p.npl), std::sqrt((double)f.ax[0].r2 * n1) / 4.0));
  f.s3 = std::max(0, ceil_log2(kFixGain * n1 / 4.0) - f.hx);
  f.ok = true;
}

// Fixed-point copy of V and its exponent (vbufs[slot + 2]) from the float64 one.
int fixed_potential(Context& c, int slot, const LineAxis ax[3], int kernel_class) {
  const size_t nr = (size_t)ax[0].n * ax[1].n * ax[2].n;
  unsigned long long* vm = static_cast<unsigned long long*>(c.vbufs[slot + 2]) + nr;
  const double* v = static_cast<const double*>(c.vbufs[slot]);
  const int grid = (int)std::min<size_t>(4 * c.sm_count, (nr + 255) / 256);
  cudaError_t e = cudaMemsetAsync(vm, 0, kFixedScaleBytes, c.stream);
  if (e != cudaSuccess) return cuda_fail(c, e, "fixed-point potential");
  HPSI_LAUNCH(c, kernel_class, (k_fx_vmax<<<grid, 256, 0, c.stream>>>(nr, v, vm)));
  HPSI_LAUNCH(c, kernel_class, (k_fx_v<<<grid, 256, 0, c.stream>>>(ax[0], ax[1], ax[2].n, v, vm,
                                                                   static_cast<long long*>(c.vbufs[slot + 2]),
                                                                   reinterpret_cast<int*>(vm) + 2)));
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(c, e, "fixed-point potential");
  return HPSI_OK;
}

int local_fixed_apply(Context& c, const Problem& p, const double2* psi, double2* hpsi, int nbnd, void* Zt, void* Yb,
                      int nbb) {
  static thread_local FxLaunch fl;   // host staging of the parameter block: threads use contexts of their own at the same time
  const int rv = ensure_fixed_potential(c, p.vslot, p.fixed.ax);
  if (rv) return rv;
  for (int b0 = 0; b0 < nbnd; b0 += nbb) {
    fl.reset();
    fl.add(c, p, psi + (size_t)b0 * p.npw, hpsi + (size_t)b0 * p.npw, std::min(nbb, nbnd - b0), Zt, Yb);
    const int rc = fl.run(c);
    if (rc) return rc;
  }
  return HPSI_OK;
}

int local_fixed_apply_multi(Context& c, int nitem, const int* prob, const int* nbnd, const double2* const* psi,
                            double2* const* hpsi, void* const* zt, void* const* yb) {
  static thread_local FxLaunch fl;
  for (int i0 = 0; i0 < nitem; i0 += kMaxLocalItems) {
    fl.reset();
    for (int i = i0; i < std::min(nitem, i0 + kMaxLocalItems); ++i)
      fl.add(c, c.probs[prob[i]], psi[i], hpsi[i], nbnd[i], zt[i], yb[i]);
    const int rc = fl.run(c);
    if (rc) return rc;
  }
  return HPSI_OK;
}

int local_fixed_persistent(Context& c, int nitem, const int* prob, const int* nbnd, const double2* const* psi,
                           double2* const* hpsi, void* const* zt, void* const* yb, bool with_nl, bool* done) {
  static thread_local FxLaunch fl;
  static thread_local NlBatch nl;
  fl.reset();
  for (int i = 0; i < nitem; ++i) fl.add(c, c.probs[prob[i]], psi[i], hpsi[i], nbnd[i], zt[i], yb[i]);
  nl.nitems = 0;
  if (with_nl) {
    const int rc = persistent_nl_batch(c, nitem, prob, nbnd, psi, hpsi, nl);
    if (rc) return rc;
  }
  int rc = ensure_buffer(c, &c.ws.pbar, &c.ws.pbarbytes, 256);
  if (rc) return rc;
  return fl.persistent(c, nl, static_cast<unsigned*>(c.ws.pbar), done);
}

}  // namespace hpsi
