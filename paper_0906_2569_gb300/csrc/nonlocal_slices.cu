// The float64 nonlocal contractions (paper Sec. 3: becp = <beta|psi>, hpsi += beta w) on the tensor cores.
//
// GB300's float64 pipe runs at ~1 TFLOP/s, its bf16 tensor cores at ~1900.  A float64 row scaled by a power of two
// is a 63-bit integer X = x 2^(62 - e), |x| < 2^e, and an integer has digits: X = sum_s v_s 256^(7-s) with eight
// balanced digits in [-128, 127], which bf16 holds exactly (the published error-free splitting of Ozaki et al., in
// fixed point).  A product of two digits has 14 bits, and sums of 1024 of them are integers below 2^24, which a float32
// accumulator adds without rounding.  So
//     sum_k a_k b_k = 2^(ea + eb - 124) sum_l 256^(14-l) sum_{i+j=l} sum_k v_i(a_k) v_j(b_k)
// is taken level by level (l = i + j <= 7: 36 of the 64 digit products) with one accumulator per level, emptied into 64-bit
// integers every 128 values of k (level 7 then holds 8 x 128 products, its limit).  The sums of the 36 products are exact.
// The 28 left out are at most 7 x 2^14 x 256^6, 2^-59 of 2^(ea + eb), for each k (random digits: 2^-62).  A K-split's total
// is rounded once, to float64.
//
// So the error is relative to the rows' largest entries, 2^-59 to 2^-62 of them a term, where a chain of float64 FMAs errs by
// 2^-53 of each term and partial sum.  An entry below 2^-10 of its row's largest has fewer than a float64's 53 bits, and one
// below 2^-62 none: for a projector that vanishes where psi is largest the chain may be the more accurate one.  On orbitals
// and projectors the digits are: a chain over tens of thousands of terms rounds more.  Against 128-bit arithmetic the nonlocal
// term of 256 projectors and 36785 plane waves errs by 1.49e-15 of its norm (the FMA kernels: 2.16e-15; Gamma form 2.23e-15
// and 2.49e-15), of which most is the final float64 sum.
//
// Measured on that case with 160 bands: calbec + add_vuspsi 20.0 -> 1.01 ms (0.86 PFLOP/s of digit products, 0.45 of
// the measured bf16 rate: the accumulators hold all of TMEM, so they are emptied while the tensor cores wait), the
// digits of psi and w 0.12 ms; real form, 75 bands: 3.16 -> 0.24 ms.
//
// Kernel: one CTA per 128 x 64 output tile (and K-split).  Warp 16 loads the eight digit planes of a 32-wide K step
// with two 3-D TMA copies (64-byte swizzle, two stages), warp 17 issues 72 tcgen05.mma a step (M = 128, N = 64,
// K = 16) into 8 x 64 TMEM columns, warps 0-15 empty the accumulators.  Every wait is bounded.
//
// Row orders: A is always the projectors.  calbec: A row p = beta_p as (re, im) pairs; B row 2b = psi_b as (re, im),
// row 2b + 1 as (im, -re); C[p][2b], C[p][2b+1] = Re, Im <beta_p|psi_b>.  add_vuspsi: A row G = (re, im) of beta_p(G)
// over p; B row 2b = (re, -im), 2b + 1 = (im, re) of w_b; C[G][2b], C[G][2b+1] = Re, Im of the sum.  Gamma form: the same
// with real rows.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "fixed_fft.cuh"
#include "hpsi_internal.h"
#include "tcgen05.cuh"

namespace hpsi {

namespace {

constexpr int kDigits = 8;
constexpr int SM_ = 128, SN = 64, SK = 32;            // tile and K step
constexpr int kChunkSteps = 4;                        // K steps per emptying of the accumulators (128 values of k)
constexpr int kABytes = kDigits * SM_ * SK * 2;       // 64 KB
constexpr int kBBytes = kDigits * SN * SK * 2;        // 32 KB
constexpr int kStages = 2;
constexpr int kSliceSmem = kStages * (kABytes + kBBytes) + 1024;
constexpr int kDrainWarps = 16;
constexpr int kThreads = 32 * (kDrainWarps + 2);
constexpr int kColsPerWarp = SN / (kDrainWarps / 4);  // 16
constexpr int kRowNan = 1 << 28;                      // exponent of a row with a non-finite entry

struct SliceArgs {
  int M, N;            // rows of A and of B
  int nsteps;          // K steps
  int split;           // K steps per split, a multiple of kChunkSteps
  int pairs;           // columns come in (re, im) pairs
  int add;             // 1: out += C, 0: out = C
  const int* ea;       // [M] row exponents
  const int* eb;       // [N]
  double* out;         // element (m, n): pairs: out[split][n/2][m] complex, else out[split][n][m]
  size_t split_stride; // doubles between the splits
  size_t ldn;          // row length of out (complex or real elements)
  int* err;
};

constexpr uint32_t kSliceIdesc =
    (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(SN >> 3) << 17) | ((uint32_t)(SM_ >> 4) << 24);

__device__ __forceinline__ void mma_slice(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(a), "l"(b), "r"(kSliceIdesc), "r"(accumulate)
      : "memory");
}

// (hi 2^32 + lo) 2^e as a float64 (a NaN for a row with a non-finite entry)
__device__ __forceinline__ double slice_value(long long hi, long long lo, int e) {
  hi += lo >> 32;
  const double d = fma((double)hi, 4294967296.0, (double)(unsigned)lo);
  if (e >= kRowNan / 2) return __longlong_as_double(0x7ff8000000000000LL);
  if (e > -1000 && e < 900) return d * __longlong_as_double((long long)(1023 + e) << 52);
  const int h = max(-1060, min(e, 1000)) / 2;
  return d * ldexp(1.0, h) * ldexp(1.0, max(-2200, min(e, 2100)) - h);
}

__global__ void __launch_bounds__(kThreads, 1)
    k_slice_gemm(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, SliceArgs a) {
  extern __shared__ __align__(1024) unsigned char smem_dyn[];
  __shared__ __align__(8) uint64_t full_bar[kStages], empty_bar[kStages], acc_full, acc_empty;
  __shared__ uint32_t tmem_base;
  __shared__ volatile int abort_flag;
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tile_n = blockIdx.x * SN, tile_m = blockIdx.y * SM_, split = blockIdx.z;
  const int kbeg = split * a.split, nk = min(a.nsteps, kbeg + a.split) - kbeg;
  const int nchunk = (nk + kChunkSteps - 1) / kChunkSteps;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&full_bar[s])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&empty_bar[s])));
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&acc_full)));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(&acc_empty)), "r"(kDrainWarps));
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    abort_flag = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(smem_u32(&tmem_base)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = tmem_base;
  int issued[kStages] = {0, 0};
  if (warp == kDrainWarps) {
    if (lane == 0) {
      for (int i = 0; i < nk; ++i) {
        const int s = i % kStages, round = i / kStages;
        if (round > 0 && !mbar_wait(smem_u32(&empty_bar[s]), (round - 1) & 1, &abort_flag)) break;
        const uint32_t fb = smem_u32(&full_bar[s]);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(fb), "r"(kABytes + kBBytes)
                     : "memory");
        unsigned char* st = smem + s * (kABytes + kBBytes);
        tma_load_3d(smem_u32(st), &mapA, (kbeg + i) * SK, tile_m, 0, fb);
        tma_load_3d(smem_u32(st + kABytes), &mapB, (kbeg + i) * SK, tile_n, 0, fb);
        issued[s] = round + 1;
      }
    }
    __syncwarp();
  } else if (warp == kDrainWarps + 1) {
    if (lane == 0) {
      int i = 0;
      for (int c = 0; c < nchunk; ++c) {
        if (c > 0 && !mbar_wait(smem_u32(&acc_empty), (c - 1) & 1, &abort_flag)) break;
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        bool ok = true;
        const int iend = min(nk, (c + 1) * kChunkSteps);
        for (uint32_t first = 0; i < iend; ++i, first = 1) {
          const int s = i % kStages;
          ok = mbar_wait(smem_u32(&full_bar[s]), (i / kStages) & 1, &abort_flag);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
          const uint32_t sa = smem_u32(smem + s * (kABytes + kBBytes)), sb = sa + kABytes;
#pragma unroll
          for (int l = 0; l < kDigits; ++l)
#pragma unroll
            for (int ia = 0; ia <= l; ++ia)
#pragma unroll
              for (int kk = 0; kk < SK / 16; ++kk)
                mma_slice(tmem + l * SN, sw64_desc(sa + ia * (SM_ * SK * 2) + kk * 32),
                          sw64_desc(sb + (l - ia) * (SN * SK * 2) + kk * 32), (ia == 0 && kk == 0) ? first : 1u);
          mma_commit(smem_u32(&empty_bar[s]));
        }
        if (!ok) break;
        mma_commit(smem_u32(&acc_full));
      }
    }
    __syncwarp();
  } else {
    // warp w empties TMEM lanes 32 (w % 4) .. and columns 16 (w / 4) .. of every level
    const uint32_t base = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (warp >> 2) * kColsPerWarp;
    long long hi[kColsPerWarp], lo[kColsPerWarp];
#pragma unroll
    for (int j = 0; j < kColsPerWarp; ++j) hi[j] = lo[j] = 0;
    bool ok = true;
    for (int c = 0; c < nchunk; ++c) {
      ok = mbar_wait(smem_u32(&acc_full), c & 1, &abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
#pragma unroll
      for (int j0 = 0; j0 < kColsPerWarp; j0 += 4) {
        uint32_t r[kDigits][4];
#pragma unroll
        for (int l = 0; l < kDigits; ++l)
          asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n"
                       : "=r"(r[l][0]), "=r"(r[l][1]), "=r"(r[l][2]), "=r"(r[l][3])
                       : "r"(base + (uint32_t)(l * SN + j0)));
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          auto at = [&](int l) { return (long long)__float2int_rn(__uint_as_float(r[l][j])); };
          hi[j0 + j] += (at(0) << 24) + (at(1) << 16) + (at(2) << 8) + at(3);
          lo[j0 + j] += (at(4) << 24) + (at(5) << 16) + (at(6) << 8) + at(7);
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(&acc_empty)) : "memory");
    }
    const int m = tile_m + (warp & 3) * 32 + lane;
    if (ok && m < a.M) {
      const int ea = a.ea[m];
      const int n0 = tile_n + (warp >> 2) * kColsPerWarp;
      double* out = a.out + (size_t)split * a.split_stride;
      // level 7 counts in units of 2^(ea + eb - 124 + 56): digits of x are those of x 2^(62 - e)
      if (a.pairs) {
        double2* o = reinterpret_cast<double2*>(out);
#pragma unroll
        for (int j = 0; j < kColsPerWarp; j += 2) {
          const int n = n0 + j;
          if (n >= a.N) break;
          const int e = ea + a.eb[n] - 68;
          const double x = slice_value(hi[j], lo[j], e), y = slice_value(hi[j + 1], lo[j + 1], e);
          double2* p = o + (size_t)(n >> 1) * a.ldn + m;
          *p = a.add ? make_double2(p->x + x, p->y + y) : make_double2(x, y);
        }
      } else {
#pragma unroll
        for (int j = 0; j < kColsPerWarp; ++j) {
          const int n = n0 + j;
          if (n >= a.N) break;
          const double x = slice_value(hi[j], lo[j], ea + a.eb[n] - 68);
          double* p = out + (size_t)n * a.ldn + m;
          *p = a.add ? *p + x : x;
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (abort_flag && threadIdx.x == 0) atomicExch(a.err, 1);
  // every TMA this CTA issued has landed before the CTA (and its shared memory) goes away
  if (warp == kDrainWarps && lane == 0) {
    volatile int never = 0;
    for (int s = 0; s < kStages; ++s)
      if (issued[s] > 0) mbar_wait(smem_u32(&full_bar[s]), (issued[s] - 1) & 1, &never);
  }
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem));
}

// ---- digits -----------------------------------------------------------------------------------

// exponent e of a row whose largest exponent field is f: |x| < 2^e (kRowNan: a non-finite entry)
__device__ __forceinline__ int row_exponent(int f) { return f == 0x7ff ? kRowNan : max(f, 1) - 1022; }

// The digits of x 2^(62 - e), e the row's exponent from field f, most significant in the top byte, the lower seven
// biased by 128 (so that all are plain bytes)
__device__ __forceinline__ unsigned long long digits_of(double x, int f) {
  const long long X = f == 0x7ff ? 0 : fx_from_bits(__double_as_longlong(x), max(f, 1) - 9);
  return (unsigned long long)X + 0x0080808080808080ULL;
}
// bf16 pattern of digit s, s > 0: byte - 128; s = 0: the signed top byte
__device__ __forceinline__ unsigned digit_bf16(unsigned long long y, int s) {
  const unsigned b = (unsigned)(y >> (8 * (7 - s))) & 0xff;
  // 2^23 + b as a float, minus 2^23 + 128 (or, for the signed top byte xor 0x80, the same)
  const float v = __uint_as_float(0x4b000000u | (s == 0 ? b ^ 0x80u : b)) - 8388736.0f;
  return __float_as_uint(v) >> 16;   // an integer below 256: exact in bf16
}

// Largest exponent field of each row of src (rows of `len` doubles); fields must start at zero.  scaled = 0 (Gamma
// coefficients): entries from the third on are multiplied by sqrt2.
constexpr double kSqrt2s = 1.4142135623730950488;
template <typename R>
__device__ __forceinline__ double slice_load(const R* row, int i, int scaled) {
  const double x = (double)row[i];
  return scaled || i < 2 ? x : x * kSqrt2s;
}
template <typename R>
__global__ void __launch_bounds__(256) k_row_field(int rows, int len, int scaled, const R* __restrict__ src,
                                                   int* __restrict__ field) {
  for (int r = blockIdx.y; r < rows; r += gridDim.y) {
    const R* row = src + (size_t)r * len;
    unsigned h = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < len; i += gridDim.x * blockDim.x)
      h = max(h, (unsigned)__double2hiint(slice_load(row, i, scaled)) & 0x7fffffffu);
    h = __reduce_max_sync(0xffffffffu, h);
    if ((threadIdx.x & 31) == 0) atomicMax(field + r, (int)(h >> 20));
  }
}

// Digit planes [8][rows][kpad] of rows of `len` doubles, two entries per thread.  dup = 0: row r from row r.
// dup = 1: rows 2r: as they are, 2r + 1: (im, -re) of each pair; dup = 2: 2r: (re, -im), 2r + 1: (im, re).
// exps: row exponents of the planes' rows.
template <typename R>
__global__ void __launch_bounds__(256) k_digits(int nrow, int len, int kpad, int dup, int scaled,
                                                const R* __restrict__ src, const int* __restrict__ field,
                                                __nv_bfloat16* __restrict__ out, int* __restrict__ exps) {
  const size_t rows = (size_t)nrow * (dup ? 2 : 1), half = kpad / 2;
  unsigned* o = reinterpret_cast<unsigned*>(out);
  for (int r = blockIdx.y; r < nrow; r += gridDim.y) {
  const int f = field[r];
  const R* row = src + (size_t)r * len;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    const int e = row_exponent(f);
    if (dup) exps[2 * r] = exps[2 * r + 1] = e;
    else exps[r] = e;
  }
  for (int h = blockIdx.x * blockDim.x + threadIdx.x; h < kpad / 2; h += gridDim.x * blockDim.x) {
    const int i = 2 * h;
    const unsigned long long x = i < len ? digits_of(slice_load(row, i, scaled), f) : 0x0080808080808080ULL;
    const unsigned long long y = i + 1 < len ? digits_of(slice_load(row, i + 1, scaled), f) : 0x0080808080808080ULL;
#pragma unroll
    for (int s = 0; s < kDigits; ++s) {
      const unsigned a = digit_bf16(x, s), b = digit_bf16(y, s);
      const size_t plane = (size_t)s * rows * half;
      if (dup == 0) {
        o[plane + (size_t)r * half + h] = a | b << 16;
      } else {
        o[plane + (size_t)(2 * r) * half + h] = dup == 1 ? a | b << 16 : a | (b ^ 0x8000u) << 16;
        o[plane + (size_t)(2 * r + 1) * half + h] = dup == 1 ? b | (a ^ 0x8000u) << 16 : b | a << 16;
      }
    }
  }
  }
}

// A of add_vuspsi: row g (of `cols` columns of beta, each CW doubles wide: 2 = complex, 1 = real), entries over p.
// One CTA per 32 rows; 16 projectors at a time through shared memory.
template <int CW>
__global__ void __launch_bounds__(256) k_digits_transposed(int P, int cols, int kpad, const double* __restrict__ beta,
                                                           __nv_bfloat16* __restrict__ out, int* __restrict__ exps) {
  __shared__ unsigned long long t[32][16 * CW + 1];
  __shared__ int field[32];
  const int g0 = blockIdx.x * 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  if (threadIdx.x < 32) field[threadIdx.x] = 0;
  __syncthreads();
  unsigned h = 0;
  if (g0 + tx < cols)
    for (int p = ty; p < P; p += 8)
#pragma unroll
      for (int c = 0; c < CW; ++c)
        h = max(h, (unsigned)__double2hiint(beta[((size_t)p * cols + g0 + tx) * CW + c]) & 0x7fffffffu);
  atomicMax(&field[tx], (int)(h >> 20));
  __syncthreads();
  if (threadIdx.x < 32 && g0 + tx < cols) exps[g0 + tx] = row_exponent(field[tx]);
  unsigned* o = reinterpret_cast<unsigned*>(out);
  const size_t half = kpad / 2, plane = (size_t)cols * half;
  const int words = 16 * CW / 2;   // bf16 pairs of a row in this step
  for (int p0 = 0; p0 * CW < kpad; p0 += 16) {
    for (int p = ty; p < 16; p += 8)
#pragma unroll
      for (int c = 0; c < CW; ++c)
        t[tx][p * CW + c] = p0 + p < P && g0 + tx < cols
                                ? digits_of(beta[((size_t)(p0 + p) * cols + g0 + tx) * CW + c], field[tx])
                                : 0x0080808080808080ULL;
    __syncthreads();
    for (int i = threadIdx.x; i < 32 * words; i += 256) {
      const int r = i / words, w = i - r * words;
      if (g0 + r < cols && p0 * CW / 2 + w < (int)half) {
        const unsigned long long x = t[r][2 * w], y = t[r][2 * w + 1];
#pragma unroll
        for (int s = 0; s < kDigits; ++s)
          o[s * plane + (size_t)(g0 + r) * half + p0 * CW / 2 + w] = digit_bf16(x, s) | digit_bf16(y, s) << 16;
      }
    }
    __syncthreads();
  }
}

// part[0][i] = sum over the K-splits of part[s][i], with the rounding errors of the sum added back (Knuth's TwoSum): the
// D-scale then reads each sum once per nonzero of D, and a split's only error is its own rounding to float64
__global__ void __launch_bounds__(256) k_sum_splits(size_t n, int nsplit, double* part) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    double s = part[i], c = 0.0;
    for (int k = 1; k < nsplit; ++k) {
      const double x = part[(size_t)k * n + i];
      const double t = __dadd_rn(s, x), z = __dadd_rn(t, -s);
      c = __dadd_rn(c, __dadd_rn(__dadd_rn(s, -__dadd_rn(t, -z)), __dadd_rn(x, -z)));
      s = t;
    }
    // an infinite or NaN sum keeps its value
    part[i] = fabs(s) <= 1.7976931348623157e308 ? __dadd_rn(s, c) : s;
  }
}

inline int pad32(int x) { return (x + SK - 1) / SK * SK; }
inline size_t al256(size_t x) { return (x + 255) & ~size_t(255); }

int slice_map(Context& c, CUtensorMap* m, const void* base, size_t rows, int kpad, int box_rows) {
  PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  int rc = tma_encoder(c, &encode);
  if (rc) return rc;
  cuuint64_t dims[3] = {(cuuint64_t)kpad, (cuuint64_t)rows, (cuuint64_t)kDigits};
  cuuint64_t strides[2] = {(cuuint64_t)kpad * 2, (cuuint64_t)kpad * 2 * rows};
  cuuint32_t box[3] = {(cuuint32_t)SK, (cuuint32_t)box_rows, (cuuint32_t)kDigits};
  cuuint32_t es[3] = {1, 1, 1};
  const CUresult r = encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, es,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(c, HPSI_ECUDA, "cuTensorMapEncodeTiled failed with code " + std::to_string((int)r));
  return HPSI_OK;
}

// Splits of K: one wave of CTAs where the tiles alone leave SMs idle
int slice_splits(const Context& c, int M, int N, int nsteps, int* per) {
  const int tiles = ((M + SM_ - 1) / SM_) * ((N + SN - 1) / SN);
  const int chunks = (nsteps + kChunkSteps - 1) / kChunkSteps;
  const int ns = std::max(1, std::min(chunks, c.sm_count / std::max(1, tiles)));
  const int cp = (chunks + ns - 1) / ns;
  *per = cp * kChunkSteps;
  return (chunks + cp - 1) / cp;
}

int slice_gemm(Context& c, const __nv_bfloat16* A, const int* ea, int M, const __nv_bfloat16* B, const int* eb, int N,
               int kpad, int nsplit, int per, bool pairs, bool add, double* out, size_t split_stride, size_t ldn,
               int kernel_class) {
  CUtensorMap ma, mb;
  int rc = slice_map(c, &ma, A, M, kpad, SM_);
  if (!rc) rc = slice_map(c, &mb, B, N, kpad, SN);
  if (rc) return rc;
  static std::atomic<unsigned long long> devices{0};
  const cudaError_t e = allow_smem(c, devices, {(const void*)k_slice_gemm});
  if (e != cudaSuccess) return cuda_fail(c, e, "digit products");
  SliceArgs a;
  a.M = M;
  a.N = N;
  a.nsteps = kpad / SK;
  a.split = per;
  a.pairs = pairs;
  a.add = add;
  a.ea = ea;
  a.eb = eb;
  a.out = out;
  a.split_stride = split_stride;
  a.ldn = ldn;
  a.err = c.d_err;
  const dim3 grid((N + SN - 1) / SN, (M + SM_ - 1) / SM_, nsplit);
  HPSI_LAUNCH(c, kernel_class, (k_slice_gemm<<<grid, kThreads, kSliceSmem, c.stream>>>(ma, mb, a)));
  return HPSI_OK;
}

}  // namespace

// Digit planes of the projectors, made on first use: which = 0: calbec's A, 1: add_vuspsi's A (complex form); 2, 3: the
// same of the Gamma form.  They take twice the projectors' memory each; a float64 context, which needs both, makes them
// together.  *ok = false, and nothing wrong, when the device has no room (the float64 CUDA-core kernels serve then, for the
// life of the context; the other planes of the pair are not kept either).
static int slice_planes(Context& c, const Problem& p, int which, bool* ok) {
  *ok = p.slices[which].digits != nullptr;
  const int first = which & ~1;
  if (*ok || p.slices[first].no_room) return HPSI_OK;
  const bool real = which >= 2, both = c.precision == HPSI_FP64;
  const int P = p.nproj, len = real ? 2 * ((p.npw + 1) / 2) : 2 * p.npw;   // doubles of a projector
  const int cols = real ? len : p.npw;
  size_t rows[2], at[2] = {0, 0}, ints[2], total = 0;
  int kpad[2];
  for (int i = 0; i < 2; ++i) {
    rows[i] = i ? cols : P;
    kpad[i] = pad32(i ? (real ? P : 2 * P) : len);
    ints[i] = al256(sizeof(__nv_bfloat16) * kDigits * rows[i] * kpad[i]);   // then row exponents, and room for the
    if (!both && first + i != which) continue;                              // rows' exponent fields
    at[i] = total;
    total += ints[i] + al256(sizeof(int) * (rows[i] + P));
  }
  void* mem = nullptr;
  if (cudaMalloc(&mem, total) != cudaSuccess) {
    cudaGetLastError();
    for (int i = 0; i < 2; ++i) {
      SlicePlanes& s = p.slices[first + i];
      if (s.owned) {
        cudaStreamSynchronize(c.stream);
        cudaFree(s.owned);
        c.ws.epoch++;   // captured batches refer to them
      }
      s = SlicePlanes();
      s.no_room = true;
    }
    return HPSI_OK;
  }
  p.slices[which].owned = mem;
  const double* beta = real ? p.d_betar : reinterpret_cast<const double*>(p.d_beta);
  for (int i = 0; i < 2; ++i) {
    if (!both && first + i != which) continue;
    SlicePlanes& s = p.slices[first + i];
    s.digits = static_cast<unsigned char*>(mem) + at[i];
    s.exps = reinterpret_cast<int*>(static_cast<unsigned char*>(s.digits) + ints[i]);
    s.kpad = kpad[i];
    __nv_bfloat16* d = static_cast<__nv_bfloat16*>(s.digits);
    if (i) {
      const int grid = (cols + 31) / 32;
      if (real) HPSI_LAUNCH(c, HPSI_K_SPLIT, (k_digits_transposed<1><<<grid, 256, 0, c.stream>>>(P, cols, kpad[i], beta, d, s.exps)));
      else HPSI_LAUNCH(c, HPSI_K_SPLIT, (k_digits_transposed<2><<<grid, 256, 0, c.stream>>>(P, cols, kpad[i], beta, d, s.exps)));
    } else {
      int* field = s.exps + rows[i];
      cudaError_t e = cudaMemsetAsync(field, 0, sizeof(int) * P, c.stream);
      if (e != cudaSuccess) return cuda_fail(c, e, "projector digit setup");
      const dim3 grid(std::max(1, std::min(64, kpad[i] / 512)), std::min(P, 65535));
      HPSI_LAUNCH(c, HPSI_K_SPLIT, (k_row_field<double><<<grid, 256, 0, c.stream>>>(P, len, 1, beta, field)));
      HPSI_LAUNCH(c, HPSI_K_SPLIT,
                  (k_digits<double><<<grid, 256, 0, c.stream>>>(P, len, kpad[i], 0, 1, beta, field, d, s.exps)));
    }
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(c, e, "projector digit setup");
  *ok = true;
  return HPSI_OK;
}

bool release_slices(Context& c) {
  bool any = false;
  for (Problem& p : c.probs)
    for (SlicePlanes& s : p.slices) any = any || s.owned;
  if (!any) return false;
  cudaStreamSynchronize(c.stream);
  for (Problem& p : c.probs)
    for (int first : {0, 2}) {
      bool had = false;
      for (int i = 0; i < 2; ++i) {
        had = had || p.slices[first + i].digits;
        cudaFree(p.slices[first + i].owned);
        p.slices[first + i] = SlicePlanes();
      }
      p.slices[first].no_room = p.slices[first + 1].no_room = had;
    }
  c.ws.epoch++;   // captured batches refer to them
  return true;
}

// Complex form: above 16 projectors.  Below, the CUDA-core kernels' float64 work is microseconds, they run over a whole
// batch in one launch, and the persistent batch and hpsi_apply give the same bits.  Measured (H|psi>, CUDA-core against
// this form): P = 32, 1503 plane waves, 4 bands 249 -> 94 us; P = 256, 6031, 64 bands 1982 -> 400 us.
bool nonlocal_slices_use(const Problem& p, int nbnd) {
  return p.nproj > 16 && nbnd > 0 && !p.slices[0].no_room;
}

// Items of a batch of nitem take this form one by one, about ten launches and 45 us each, where the tiles run over all items
// at once.  It is the faster one from about 6e6 multiply-adds an item, and for a few items of many projectors, where the
// tiles' chain over the projectors (1.7 us each for 16 bands and more) is longer.  Measured, tiles against this form, 16
// items: P = 17, 1503 plane waves, 8 bands 240 / 1123 us; P = 32, 1503, 24 bands 634 / 1411; P = 64, 3911, 24 bands 2115 /
// 2125; P = 128, 1503, 64 bands 3528 / 2229; 2 items: P = 32, 1503, 24 bands 180 / 189; P = 96, 1503, 24 bands 280 / 213.
bool batch_slices_use(const Problem& p, int nbnd, int nitem) {
  return nonlocal_slices_use(p, nbnd) &&
         ((double)p.nproj * p.npw * nbnd >= 6.0e6 || (nbnd >= 16 && p.nproj > 26 * nitem));
}

// Digit planes of `rows` rows of `len` doubles (src) in the workspace at `at`; returns the planes and row exponents.
template <typename R>
static int slice_rows(Context& c, const R* src, int rows, int len, int kpad, int dup, int scaled, unsigned char* at,
                      __nv_bfloat16** digits, int** exps) {
  const size_t planes = (size_t)rows * (dup ? 2 : 1);
  *digits = reinterpret_cast<__nv_bfloat16*>(at);
  int* field = reinterpret_cast<int*>(at + al256(sizeof(__nv_bfloat16) * kDigits * planes * kpad));
  *exps = field + rows;
  cudaError_t e = cudaMemsetAsync(field, 0, sizeof(int) * rows, c.stream);
  if (e != cudaSuccess) return cuda_fail(c, e, "digit workspace clear");
  const dim3 grid(std::max(1, std::min((8 * c.sm_count + rows - 1) / rows, (len + 1023) / 1024)), std::min(rows, 65535));
  HPSI_LAUNCH(c, HPSI_K_SPLIT, (k_row_field<R><<<grid, 256, 0, c.stream>>>(rows, len, scaled, src, field)));
  HPSI_LAUNCH(c, HPSI_K_SPLIT,
              (k_digits<R><<<grid, 256, 0, c.stream>>>(rows, len, kpad, dup, scaled, src, field, *digits, *exps)));
  return HPSI_OK;
}
static size_t slice_rows_bytes(int rows, int kpad, int dup) {
  const size_t planes = (size_t)rows * (dup ? 2 : 1);
  return al256(sizeof(__nv_bfloat16) * kDigits * planes * kpad) + al256(sizeof(int) * (rows + planes));
}

static int sum_splits(Context& c, size_t n, int nsplit) {
  if (nsplit > 1)
    HPSI_LAUNCH(c, HPSI_K_DSCALE, (k_sum_splits<<<(int)std::min<size_t>(8 * c.sm_count, (n + 255) / 256), 256, 0,
                                                  c.stream>>>(n, nsplit, static_cast<double*>(c.ws.part))));
  return HPSI_OK;
}

// Bands per pass: their digit planes stay near 1 GB
static int slice_band_block(int nbnd, size_t per_band) {
  const int nb = (int)std::max<size_t>(32, (size_t)(1u << 30) / std::max<size_t>(1, per_band));
  const int passes = (nbnd + nb - 1) / nb;
  return (nbnd + passes - 1) / passes;
}

// Workspaces of the projections: the digit planes of nbk bands and the K-splits' partial sums of every block (cw = 2: complex)
static bool slice_room(Context& c, int P, int nbnd, int nbk, int cw, int kpad, int dup) {
  size_t part = 0;
  for (int nb : {std::min(nbk, nbnd), nbnd % nbk}) {
    int per = 0;
    if (nb > 0) part = std::max(part, sizeof(double) * cw * (size_t)slice_splits(c, P, cw * nb, kpad / SK, &per) * nb * P);
  }
  return try_buffer(c, &c.ws.mixed, &c.ws.mixedbytes, slice_rows_bytes(nbk, kpad, dup)) &&
         try_buffer(c, &c.ws.part, &c.ws.partbytes, part);
}

// w = D <beta|psi> for nb bands (complex form) into w; *ok as slice_planes
int slices_w(Context& c, const Problem& p, const double2* psi, int nbnd, double2* w, bool* ok) {
  int rc = slice_planes(c, p, 0, ok);
  if (rc || !*ok) return rc;
  const SlicePlanes& s = p.slices[0];
  const int P = p.nproj, nbk = slice_band_block(nbnd, slice_rows_bytes(1, s.kpad, 1));
  *ok = slice_room(c, P, nbnd, nbk, 2, s.kpad, 1);
  if (!*ok) return HPSI_OK;
  for (int b0 = 0; b0 < nbnd; b0 += nbk) {
    const int nb = std::min(nbk, nbnd - b0);
    int per = 0;
    const int ns = slice_splits(c, P, 2 * nb, s.kpad / SK, &per);
    __nv_bfloat16* d = nullptr;
    int* e = nullptr;
    rc = slice_rows(c, reinterpret_cast<const double*>(psi + (size_t)b0 * p.npw), nb, 2 * p.npw, s.kpad, 1, 1,
                    static_cast<unsigned char*>(c.ws.mixed), &d, &e);
    if (rc) return rc;
    rc = slice_gemm(c, static_cast<const __nv_bfloat16*>(s.digits), s.exps, P, d, e, 2 * nb, s.kpad, ns, per, true, false,
                    static_cast<double*>(c.ws.part), 2 * (size_t)nb * P, P, HPSI_K_CALBEC);
    if (!rc) rc = sum_splits(c, 2 * (size_t)nb * P, ns);
    if (!rc) rc = dscale_fp64(c, p, nb, 1, static_cast<double2*>(c.ws.part), w + (size_t)b0 * P);
    if (rc) return rc;
  }
  return HPSI_OK;
}

// hpsi += beta w
int slices_add(Context& c, const Problem& p, const double2* w, double2* hpsi, int nbnd, bool* ok) {
  int rc = slice_planes(c, p, 1, ok);
  if (rc || !*ok) return rc;
  const SlicePlanes& s = p.slices[1];
  *ok = try_buffer(c, &c.ws.mixed, &c.ws.mixedbytes, slice_rows_bytes(nbnd, s.kpad, 1));
  if (!*ok) return HPSI_OK;
  __nv_bfloat16* d = nullptr;
  int* e = nullptr;
  rc = slice_rows(c, reinterpret_cast<const double*>(w), nbnd, 2 * p.nproj, s.kpad, 2, 1,
                  static_cast<unsigned char*>(c.ws.mixed), &d, &e);
  if (rc) return rc;
  return slice_gemm(c, static_cast<const __nv_bfloat16*>(s.digits), s.exps, p.npw, d, e, 2 * nbnd, s.kpad, 1,
                    (s.kpad / SK + kChunkSteps - 1) / kChunkSteps * kChunkSteps, true, true,
                    reinterpret_cast<double*>(hpsi), 0, p.npw, HPSI_K_ADDVUS);
}

// Gamma form: always (the smallest measured, P = 4, 1503 plane waves, 4 bands: 108 -> 97 us; P = 256, 30047, 64 bands:
// 2478 -> 860 us)
bool gamma_slices_use(const Problem& p, int nbnd) {
  return p.nproj > 0 && nbnd > 0 && !p.slices[2].no_room;
}

template <typename R>
static int gamma_slices_w_t(Context& c, const Problem& p, const R* x, int nbnd, bool scaled, double* w, bool* ok) {
  int rc = slice_planes(c, p, 2, ok);
  if (rc || !*ok) return rc;
  const SlicePlanes& s = p.slices[2];
  const int P = p.nproj, nr = 2 * ((p.npw + 1) / 2), nbk = slice_band_block(nbnd, slice_rows_bytes(1, s.kpad, 0));
  *ok = slice_room(c, P, nbnd, nbk, 1, s.kpad, 0);
  if (!*ok) return HPSI_OK;
  for (int b0 = 0; b0 < nbnd; b0 += nbk) {
    const int nb = std::min(nbk, nbnd - b0);
    int per = 0;
    const int ns = slice_splits(c, P, nb, s.kpad / SK, &per);
    __nv_bfloat16* d = nullptr;
    int* e = nullptr;
    rc = slice_rows(c, x + (size_t)b0 * nr, nb, nr, s.kpad, 0, scaled ? 1 : 0, static_cast<unsigned char*>(c.ws.mixed),
                    &d, &e);
    if (rc) return rc;
    rc = slice_gemm(c, static_cast<const __nv_bfloat16*>(s.digits), s.exps, P, d, e, nb, s.kpad, ns, per, false, false,
                    static_cast<double*>(c.ws.part), (size_t)nb * P, P, HPSI_K_CALBEC);
    if (!rc) rc = sum_splits(c, (size_t)nb * P, ns);
    if (!rc) rc = gamma_dscale_fp64(c, p, nb, 1, static_cast<const double*>(c.ws.part), w + (size_t)b0 * P);
    if (rc) return rc;
  }
  return HPSI_OK;
}
int gamma_slices_w(Context& c, const Problem& p, const void* x, bool x32, int nbnd, bool scaled, double* w, bool* ok) {
  return x32 ? gamma_slices_w_t(c, p, static_cast<const float*>(x), nbnd, scaled, w, ok)
             : gamma_slices_w_t(c, p, static_cast<const double*>(x), nbnd, scaled, w, ok);
}

// out[b] = sum_p betar_p w[b][p]
int gamma_slices_add(Context& c, const Problem& p, const double* w, double* out, int nbnd, bool* ok) {
  int rc = slice_planes(c, p, 3, ok);
  if (rc || !*ok) return rc;
  const SlicePlanes& s = p.slices[3];
  const int nr = 2 * ((p.npw + 1) / 2);
  *ok = try_buffer(c, &c.ws.mixed, &c.ws.mixedbytes, slice_rows_bytes(nbnd, s.kpad, 0));
  if (!*ok) return HPSI_OK;
  __nv_bfloat16* d = nullptr;
  int* e = nullptr;
  rc = slice_rows(c, w, nbnd, p.nproj, s.kpad, 0, 1, static_cast<unsigned char*>(c.ws.mixed), &d, &e);
  if (rc) return rc;
  return slice_gemm(c, static_cast<const __nv_bfloat16*>(s.digits), s.exps, nr, d, e, nbnd, s.kpad, 1,
                    (s.kpad / SK + kChunkSteps - 1) / kChunkSteps * kChunkSteps, false, false, out, 0, nr,
                    HPSI_K_ADDVUS);
}


// ---- subspace products (subspace_fp64.cu) -------------------------------------------------------

// out[i + j ldo] = src[j][i], rows of m
template <typename V>
static __global__ void __launch_bounds__(256) k_copy_cols(int m, int n, const V* __restrict__ src, V* __restrict__ out,
                                                          int ldo) {
  for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < (size_t)m * n; t += (size_t)gridDim.x * blockDim.x)
    out[t / m * ldo + t % m] = src[t];
}
// dst[j][i] = sign coef[i + j ldc], rows of k entries of CW doubles
template <int CW>
static __global__ void __launch_bounds__(256) k_pack_coef(int k, int n, double sign, const double* __restrict__ coef, int ldc,
                                                          double* __restrict__ dst) {
  const int kw = CW * k;
  for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < (size_t)kw * n; t += (size_t)gridDim.x * blockDim.x)
    dst[t] = sign * coef[t / kw * ldc * CW + t % kw];
}
static int few_ctas(const Context& c, size_t n) { return (int)std::min<size_t>(8 * c.sm_count, (n + 255) / 256); }

// out[i + j ldo] = <a_i|b_j> for complex (CW = 2) or real (1) rows of len entries; *ok = false: no room for the digit planes
// (out is to be written anew)
template <int CW>
static int slices_inner_t(Context& c, const double* a, int m, const double* b, int n, int len, double* out, int ldo,
                          bool* ok) {
  using V = typename std::conditional<CW == 2, double2, double>::type;
  constexpr int dup = CW == 2 ? 1 : 0;
  *ok = false;
  const int kpad = pad32(CW * len);
  const int nbk = slice_band_block(n, slice_rows_bytes(1, kpad, dup)), mbk = slice_band_block(m, slice_rows_bytes(1, kpad, 0));
  const size_t bb = slice_rows_bytes(nbk, kpad, dup), ab = slice_rows_bytes(mbk, kpad, 0);
  if (!try_buffer(c, &c.ws.mixed, &c.ws.mixedbytes, ab + bb)) return HPSI_OK;
  int rc = HPSI_OK;
  unsigned char* w0 = static_cast<unsigned char*>(c.ws.mixed);
  for (int j0 = 0; j0 < n; j0 += nbk) {
    const int nj = std::min(nbk, n - j0);
    __nv_bfloat16 *db = nullptr, *da = nullptr;
    int *eb = nullptr, *ea = nullptr;
    rc = slice_rows(c, b + (size_t)j0 * len * CW, nj, CW * len, kpad, dup, 1, w0, &db, &eb);
    if (rc) return rc;
    for (int i0 = 0; i0 < m; i0 += mbk) {
      const int mi = std::min(mbk, m - i0);
      rc = slice_rows(c, a + (size_t)i0 * len * CW, mi, CW * len, kpad, 0, 1, w0 + bb, &da, &ea);
      if (rc) return rc;
      int per = 0;
      const int ns = slice_splits(c, mi, CW * nj, kpad / SK, &per);
      if (!try_buffer(c, &c.ws.part, &c.ws.partbytes, sizeof(V) * (size_t)ns * mi * nj)) return HPSI_OK;
      double* part = static_cast<double*>(c.ws.part);
      rc = slice_gemm(c, da, ea, mi, db, eb, CW * nj, kpad, ns, per, CW == 2, false, part, CW * (size_t)mi * nj, mi,
                      HPSI_K_DAVIDSON);
      if (!rc) rc = sum_splits(c, CW * (size_t)mi * nj, ns);
      if (rc) return rc;
      HPSI_LAUNCH(c, HPSI_K_DAVIDSON, (k_copy_cols<V><<<few_ctas(c, (size_t)mi * nj), 256, 0, c.stream>>>(
                                          mi, nj, reinterpret_cast<const V*>(part),
                                          reinterpret_cast<V*>(out) + (size_t)j0 * ldo + i0, ldo)));
    }
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(c, e, "subspace inner products");
  *ok = true;
  return HPSI_OK;
}

// out_j = (accumulate ? out_j : 0) + sign sum_i coef[i + j ldc] a_i
template <int CW>
static int slices_outer_t(Context& c, const double* a, int k, const double* coef, int ldc, int n, int len, double sign,
                          bool accumulate, double* out, bool* ok) {
  constexpr int dup = CW == 2 ? 2 : 0;
  *ok = false;
  // the rows' digits [len][CW k] in blocks of k that stay near 2 GB
  const size_t per_k = sizeof(__nv_bfloat16) * kDigits * CW * (size_t)len;
  const int blocks = (int)std::max<size_t>(1, (per_k * k + (2ull << 30) - 1) / (2ull << 30));
  const int kbk = ((k + blocks - 1) / blocks + 15) / 16 * 16;
  const int kpad0 = pad32(CW * std::min(k, kbk));
  const size_t eb_ = al256(sizeof(int) * (size_t)len);
  const size_t ab = al256(sizeof(__nv_bfloat16) * kDigits * (size_t)len * kpad0) + eb_;
  const size_t bb = slice_rows_bytes(n, kpad0, dup), cb = al256(sizeof(double) * CW * (size_t)n * kbk);
  if (!try_buffer(c, &c.ws.mixed, &c.ws.mixedbytes, ab + bb + cb)) return HPSI_OK;
  int rc = HPSI_OK;
  unsigned char* w0 = static_cast<unsigned char*>(c.ws.mixed);
  __nv_bfloat16* da = reinterpret_cast<__nv_bfloat16*>(w0);
  int* ea = reinterpret_cast<int*>(w0 + ab - eb_);
  double* pack = reinterpret_cast<double*>(w0 + ab + bb);
  for (int k0 = 0; k0 < k; k0 += kbk) {
    const int nk = std::min(kbk, k - k0), kpad = pad32(CW * nk);
    HPSI_LAUNCH(c, HPSI_K_DAVIDSON, (k_pack_coef<CW><<<few_ctas(c, CW * (size_t)nk * n), 256, 0, c.stream>>>(
                                        nk, n, sign, coef + (size_t)k0 * CW, ldc, pack)));
    HPSI_LAUNCH(c, HPSI_K_SPLIT, (k_digits_transposed<CW><<<(len + 31) / 32, 256, 0, c.stream>>>(
                                     nk, len, kpad, a + (size_t)k0 * len * CW, da, ea)));
    __nv_bfloat16* db = nullptr;
    int* eb = nullptr;
    rc = slice_rows(c, static_cast<const double*>(pack), n, CW * nk, kpad, dup, 1, w0 + ab, &db, &eb);
    if (rc) return rc;
    rc = slice_gemm(c, da, ea, len, db, eb, CW * n, kpad, 1, (kpad / SK + kChunkSteps - 1) / kChunkSteps * kChunkSteps,
                    CW == 2, accumulate || k0 > 0, out, 0, len, HPSI_K_DAVIDSON);
    if (rc) return rc;
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(c, e, "subspace combinations");
  *ok = true;
  return HPSI_OK;
}

int slices_inner(Context& c, const double* a, int m, const double* b, int n, int len, bool real, double* out, int ldo,
                 bool* ok) {
  return real ? slices_inner_t<1>(c, a, m, b, n, len, out, ldo, ok) : slices_inner_t<2>(c, a, m, b, n, len, out, ldo, ok);
}
int slices_outer(Context& c, const double* a, int k, const double* coef, int ldc, int n, int len, bool real, double sign,
                 bool accumulate, double* out, bool* ok) {
  return real ? slices_outer_t<1>(c, a, k, coef, ldc, n, len, sign, accumulate, out, ok)
              : slices_outer_t<2>(c, a, k, coef, ldc, n, len, sign, accumulate, out, ok);
}

}  // namespace hpsi
