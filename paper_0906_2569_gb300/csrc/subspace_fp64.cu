// Float64 subspace products of the Davidson solvers: inner products A^H B of blocks of npw-long rows and linear combinations
// of rows.  The blocks are a few to a few hundred rows by thousands of plane waves, a shape on which the library
// GEMMs of float64 leave most of the chip idle (16 x 64 rows of 1503: 104 us where the FMAs are 12 us of
// the float64 pipe).  Two forms each:
//   small   CUDA-core FMAs: inner products with K split over CTAs, combinations with one output per thread;
//   large   digit products on the tensor cores (nonlocal_slices.cu).
// The line between them, kDigitMacs, is ~170 us of the float64 pipe and ~80 us as digits (their planes are made on each
// call).  davidson_solve in float64: 16 bands of 1503 plane waves 43 -> 27 ms; 160 bands of 36785, where every product is large,
// 6.5 -> 0.91 s.
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "hpsi_internal.h"

namespace hpsi {

namespace {

#include "nonlocal_tiles.cuh"

template <int TP>
__global__ void __launch_bounds__(256) k_sub_inner(int npw, int ld, int m, int n, int kchunk, const double2* __restrict__ a,
                                                   const double2* __restrict__ b, double2* __restrict__ part) {
  __shared__ double2 sm[CB_SMEM];
  calbec_tile_t<TP>(npw, m, n, kchunk, a, b, part, blockIdx.x, blockIdx.y, blockIdx.z, sm, ld);
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
__global__ void __launch_bounds__(SO_G* SO_B) k_sub_outer(int npw, int ld, int k, int n, double sign, int acc,
                                                          const double2* __restrict__ a, const double2* __restrict__ c,
                                                          int ldc, double2* __restrict__ out) {
  __shared__ double2 sa[SO_K][SO_G], sc[SO_B][SO_K];
  const int tx = threadIdx.x % SO_G, ty = threadIdx.x / SO_G;
  const int g = blockIdx.x * SO_G + tx, j = blockIdx.y * SO_B + ty;
  double2 s = make_double2(0.0, 0.0);
  for (int i0 = 0; i0 < k; i0 += SO_K) {
    const int ni = min(SO_K, k - i0);
    for (int i = ty; i < ni; i += SO_B) sa[i][tx] = g < npw ? a[(size_t)(i0 + i) * ld + g] : make_double2(0.0, 0.0);
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
    double2* o = out + (size_t)j * ld + g;
    *o = acc ? make_double2(o->x + s.x, o->y + s.y) : s;
  }
}

// K[i + j n]: the anti-Hermitian generator of the mixing of x_i and x_j in the eigenvectors of (H, S), where H_ij =
// <x_i|H x_j> is nearly diagonal and S nearly the identity: the angle of each pair's own 2 x 2 problem, which is exact for a
// pair that is close and first order between others; zero where it would be above 0.03 (degenerate to
// float32 accuracy).  The Hermitian part of H alone: the rounding of h x in its float32 local term is not symmetric, and
// would come back as a lost orthogonality over the gap.
template <int CW>
__global__ void __launch_bounds__(256) k_ritz_mix(int n, const double* __restrict__ H, const double* __restrict__ S,
                                                  double* __restrict__ K) {
  const size_t t = (size_t)blockIdx.x * 256 + threadIdx.x;
  if (t >= (size_t)n * n) return;
  const int i = (int)(t % n), j = (int)(t / n);
  const size_t di = CW * (size_t)i * (n + 1), dj = CW * (size_t)j * (n + 1), u = CW * ((size_t)i * n + j);
  const double ei = H[di] / S[di], ej = H[dj] / S[dj], g = ej - ei, em = 0.5 * (ei + ej);
  double v[CW], a2 = 0.0;
  for (int k = 0; k < CW; ++k) {
    v[k] = 0.5 * (H[CW * t + k] + (k == 0 ? H[u] : -H[u + k])) - em * S[CW * t + k];
    a2 = fma(v[k], v[k], a2);
  }
  const double a = sqrt(a2);
  const bool apart = i != j && a > 0.0 && a <= 0.03 * fabs(g);
  const double f = apart ? 0.5 * atan(2.0 * a / g) / a : 0.0;
  for (int k = 0; k < CW; ++k) K[CW * t + k] = v[k] * f;
}
// out = one + alpha A (bone + bscale B) (n x n); orth: A stands for the first-order S^-1/2 of the overlaps S that it holds
template <int CW>
__global__ void __launch_bounds__(256) k_small_product(int n, double one, double alpha, const double* __restrict__ A,
                                                       bool orth, double bone, double bscale, const double* __restrict__ B,
                                                       double* __restrict__ out) {
  const size_t t = (size_t)blockIdx.x * 256 + threadIdx.x;
  if (t >= (size_t)n * n) return;
  const int i = (int)(t % n), j = (int)(t / n);
  double q[2] = {0.0, 0.0};
  for (int l = 0; l < n; ++l) {
    const size_t a = CW * ((size_t)l * n + i), b = CW * ((size_t)j * n + l);
    const double x = A[a], y = CW == 2 ? A[a + CW - 1] : 0.0;
    const double u = fma(bscale, B[b], l == j ? bone : 0.0);
    q[0] = fma(x, u, q[0]);
    if (CW == 2) {
      const double w = bscale * B[b + CW - 1];
      q[0] = fma(-y, w, q[0]);
      q[1] = fma(x, w, fma(y, u, q[1]));
    }
  }
  if (orth) {   // 1 / sqrt(S_ii) and -S_il / 2
    const double d = A[CW * (size_t)i * (n + 1)], f = 1.0 / sqrt(d) + 0.5 * d;
    for (int k = 0; k < CW; ++k)
      q[k] = fma(-0.5, q[k], f * fma(bscale, B[CW * t + k], i == j && k == 0 ? bone : 0.0));
  }
  for (int k = 0; k < CW; ++k) out[CW * t + k] = fma(alpha, q[k], i == j && k == 0 ? one : 0.0);
}

}  // namespace

// The vectors of a float32 basis carry rounding noise that the Rayleigh-Ritz step turns into mixing of neighbours, noise
// over their gap (1e-5 at a gap of 1e-3 Ha): most of the vectors' error, and the part that varies between equally accurate
// forms of H|psi>.  x and h x are at hand in float64 for the quotients, so the mixing inside the block is taken out: two N x N
// products, C = S^-1/2 exp(K) (S^-1/2 to first order, the exponential to fourth) and two rotations as digit products.
// small: 4 N^2, tx and thx: N rows of len (complex or real).  Without room for the digits x stays as it is.
int ritz_refine(Context& c, int n, int len, bool real, double* x, double* hx, double* small, double* tx, double* thx) {
  if (n < 2) return HPSI_OK;
  const size_t nn = (size_t)n * n * (real ? 1 : 2), bytes = sizeof(double) * (real ? 1 : 2) * (size_t)n * len;
  double *H = small, *S = small + nn, *K = S + nn, *T = K + nn;
  bool ok = false;
  int rc = slices_inner(c, x, n, hx, n, len, real, H, n, &ok);
  if (!rc && ok) rc = slices_inner(c, x, n, x, n, len, real, S, n, &ok);
  if (rc || !ok) return rc;
  const unsigned grid = (unsigned)(((size_t)n * n + 255) / 256);
  if (real) HPSI_LAUNCH(c, HPSI_K_DAVIDSON, (k_ritz_mix<1><<<grid, 256, 0, c.stream>>>(n, H, S, K)));
  else HPSI_LAUNCH(c, HPSI_K_DAVIDSON, (k_ritz_mix<2><<<grid, 256, 0, c.stream>>>(n, H, S, K)));
  auto product = [&](double one, double alpha, const double* A, bool orth, double bone, double bscale, const double* B,
                     double* out) {
    auto go = [&](auto k) { HPSI_LAUNCH(c, HPSI_K_DAVIDSON, (k<<<grid, 256, 0, c.stream>>>(n, one, alpha, A, orth, bone, bscale, B, out))); };
    if (real) go(k_small_product<1>);
    else go(k_small_product<2>);
  };
  // exp(K) = 1 + K (1 + K / 2 (1 + K / 3 (1 + K / 4))); H is free from here on
  product(1.0, 1.0 / 3.0, K, false, 1.0, 0.25, K, T);
  product(1.0, 0.5, K, false, 0.0, 1.0, T, H);
  product(1.0, 1.0, K, false, 0.0, 1.0, H, T);
  double* C = H;
  product(0.0, 1.0, S, true, 0.0, 1.0, T, C);
  rc = slices_outer(c, x, n, C, n, n, len, real, 1.0, false, tx, &ok);
  if (!rc && ok) rc = slices_outer(c, hx, n, C, n, n, len, real, 1.0, false, thx, &ok);
  if (rc || !ok) return rc;
  cudaError_t e = cudaMemcpyAsync(x, tx, bytes, cudaMemcpyDeviceToDevice, c.stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(hx, thx, bytes, cudaMemcpyDeviceToDevice, c.stream);
  if (e != cudaSuccess) return cuda_fail(c, e, "refinement of the Ritz vectors");
  return HPSI_OK;
}

int fp64_inner(Context& c, const double2* a, int m, const double2* b, int n, int npw, double2* out, int ldo, int ld) {
  if (m < 1 || n < 1) return HPSI_OK;
  if (ld == 0) ld = npw;
  if (ld == npw && (double)m * n * npw >= kDigitMacs) {
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
  auto go = [&](auto k) { HPSI_LAUNCH(c, HPSI_K_DAVIDSON, (k<<<grid, 256, 0, c.stream>>>(npw, ld, m, n, kc, a, b, part))); };
  if (tp == 8) go(k_sub_inner<8>);
  else go(k_sub_inner<CB_TP>);
  HPSI_LAUNCH(c, HPSI_K_DAVIDSON, (k_sub_reduce<<<(m * n + 127) / 128, 128, 0, c.stream>>>(m, n, ns, part, out, ldo)));
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(c, e, "subspace inner products");
  return HPSI_OK;
}

int fp64_outer(Context& c, const double2* a, int k, const double2* coef, int ldc, int n, int npw, double sign,
               bool accumulate, double2* out, int ld) {
  if (n < 1) return HPSI_OK;
  if (ld == 0) ld = npw;
  if (ld == npw && (double)k * n * npw >= kDigitMacs) {
    bool ok = false;
    const int rc = slices_outer(c, reinterpret_cast<const double*>(a), k, reinterpret_cast<const double*>(coef), ldc, n, npw,
                                false, sign, accumulate, reinterpret_cast<double*>(out), &ok);
    if (rc || ok) return rc;
  }
  HPSI_LAUNCH(c, HPSI_K_DAVIDSON,
              (k_sub_outer<<<dim3((npw + SO_G - 1) / SO_G, (n + SO_B - 1) / SO_B), SO_G * SO_B, 0, c.stream>>>(
                  npw, ld, k, n, sign, accumulate ? 1 : 0, a, coef, ldc, out)));
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(c, e, "subspace combinations");
  return HPSI_OK;
}

}  // namespace hpsi
