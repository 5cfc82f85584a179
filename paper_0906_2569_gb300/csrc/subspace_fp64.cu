// Float64 subspace products of the Davidson solvers: inner products A^H B of blocks of npw-long rows and linear combinations
// of rows.  The blocks are a few to a few hundred rows by thousands of plane waves, a shape on which the library
// GEMMs of float64 leave most of the chip idle (16 x 64 rows of 1503: 104 us where the FMAs are 12 us of
// the float64 pipe).  Two forms each:
//   small   CUDA-core FMAs: inner products with K split over CTAs, combinations with one output per thread;
//   large   exact digit products on the tensor cores (nonlocal_slices.cu).
// The line between them, kDigitMacs, is ~170 us of the float64 pipe and ~80 us as digits (their planes are made on each
// call).  davidson_solve in float64: 16 bands of 1503 plane waves 43 -> 25 ms; 160 bands of 36785, where every product is large,
// 6.5 -> 0.91 s.
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "hpsi_internal.h"

namespace hpsi {

namespace {

#include "nonlocal_tiles.cuh"

template <int TP>
__global__ void __launch_bounds__(256) k_sub_inner(int npw, int m, int n, int kchunk, const double2* __restrict__ a,
                                                   const double2* __restrict__ b, double2* __restrict__ part) {
  __shared__ double2 sm[CB_SMEM];
  calbec_tile_t<TP>(npw, m, n, kchunk, a, b, part, blockIdx.x, blockIdx.y, blockIdx.z, sm);
}

// out[i + j ldo] = sum of the splits of part[split][j][i]
__global__ void __launch_bounds__(128) k_sub_reduce(int m, int n, int nsplit, const double2* __restrict__ part,
                                                    double2* __restrict__ out, int ldo) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= m * n) return;
  double2 s = make_double2(0.0, 0.0);
  for (int k = 0; k < nsplit; ++k) {
    const double2 v = part[(size_t)k * m * n + t];
    s.x += v.x;
    s.y += v.y;
  }
  out[(size_t)(t / m) * ldo + t % m] = s;
}

constexpr int SO_G = 32, SO_B = 4, SO_K = 16;

// out[j][g] = (acc ? out[j][g] : 0) + sign sum_i a[i][g] c[i + j ldc]: one output per thread, so that a few thousand plane
// waves by a few rows still occupy every scheduler
__global__ void __launch_bounds__(SO_G* SO_B) k_sub_outer(int npw, int k, int n, double sign, int acc,
                                                          const double2* __restrict__ a, const double2* __restrict__ c,
                                                          int ldc, double2* __restrict__ out) {
  __shared__ double2 sa[SO_K][SO_G], sc[SO_B][SO_K];
  const int tx = threadIdx.x % SO_G, ty = threadIdx.x / SO_G;
  const int g = blockIdx.x * SO_G + tx, j = blockIdx.y * SO_B + ty;
  double2 s = make_double2(0.0, 0.0);
  for (int i0 = 0; i0 < k; i0 += SO_K) {
    const int ni = min(SO_K, k - i0);
    for (int i = ty; i < ni; i += SO_B) sa[i][tx] = g < npw ? a[(size_t)(i0 + i) * npw + g] : make_double2(0.0, 0.0);
    if (threadIdx.x < SO_B * SO_K) {
      const int jj = threadIdx.x / SO_K, i = threadIdx.x % SO_K;
      double2 v = make_double2(0.0, 0.0);
      if (i < ni && blockIdx.y * SO_B + jj < n) v = c[(size_t)(blockIdx.y * SO_B + jj) * ldc + i0 + i];
      sc[jj][i] = make_double2(sign * v.x, sign * v.y);
    }
    __syncthreads();
    if (j < n)
#pragma unroll 4
      for (int i = 0; i < ni; ++i) cmac(s, sc[ty][i], sa[i][tx]);
    __syncthreads();
  }
  if (g < npw && j < n) {
    double2* o = out + (size_t)j * npw + g;
    *o = acc ? make_double2(o->x + s.x, o->y + s.y) : s;
  }
}

}  // namespace

int fp64_inner(Context& c, const double2* a, int m, const double2* b, int n, int npw, double2* out, int ldo) {
  if (m < 1 || n < 1) return HPSI_OK;
  if ((double)m * n * npw >= kDigitMacs) {
    bool ok = false;
    const int rc = slices_inner(c, reinterpret_cast<const double*>(a), m, reinterpret_cast<const double*>(b), n, npw, false,
                                reinterpret_cast<double*>(out), ldo, &ok);
    if (rc || ok) return rc;
  }
  const int tp = (double)m * n * npw < 4.0e6 ? 8 : CB_TP;   // small: one output a thread, more CTAs
  const int tiles = ((m + tp - 1) / tp) * ((n + CB_TB - 1) / CB_TB);
  int ns = std::max(1, (4 * c.sm_count) / tiles);
  int kc = (npw + ns - 1) / ns;
  kc = std::max(2 * CB_TK, (kc + CB_TK - 1) / CB_TK * CB_TK);
  ns = (npw + kc - 1) / kc;
  int rc = ensure_buffer(c, &c.ws.part, &c.ws.partbytes, sizeof(double2) * (size_t)ns * m * n);
  if (rc) return rc;
  double2* part = static_cast<double2*>(c.ws.part);
  const dim3 grid((m + tp - 1) / tp, (n + CB_TB - 1) / CB_TB, ns);
  auto go = [&](auto k) { HPSI_LAUNCH(c, HPSI_K_DAVIDSON, (k<<<grid, 256, 0, c.stream>>>(npw, m, n, kc, a, b, part))); };
  if (tp == 8) go(k_sub_inner<8>);
  else go(k_sub_inner<CB_TP>);
  HPSI_LAUNCH(c, HPSI_K_DAVIDSON, (k_sub_reduce<<<(m * n + 127) / 128, 128, 0, c.stream>>>(m, n, ns, part, out, ldo)));
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(c, e, "subspace inner products");
  return HPSI_OK;
}

int fp64_outer(Context& c, const double2* a, int k, const double2* coef, int ldc, int n, int npw, double sign,
               bool accumulate, double2* out) {
  if (n < 1) return HPSI_OK;
  if ((double)k * n * npw >= kDigitMacs) {
    bool ok = false;
    const int rc = slices_outer(c, reinterpret_cast<const double*>(a), k, reinterpret_cast<const double*>(coef), ldc, n, npw,
                                false, sign, accumulate, reinterpret_cast<double*>(out), &ok);
    if (rc || ok) return rc;
  }
  HPSI_LAUNCH(c, HPSI_K_DAVIDSON,
              (k_sub_outer<<<dim3((npw + SO_G - 1) / SO_G, (n + SO_B - 1) / SO_B), SO_G * SO_B, 0, c.stream>>>(
                  npw, k, n, sign, accumulate ? 1 : 0, a, coef, ldc, out)));
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(c, e, "subspace combinations");
  return HPSI_OK;
}

}  // namespace hpsi
