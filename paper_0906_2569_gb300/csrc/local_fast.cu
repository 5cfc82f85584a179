// Local part of H|psi> in float32 (mixed contexts), for any box whose edges are products of two of 2, 3, 4, 5, 6, 8, 9, 10,
// 12, 15, 16 (App. A.1: V applied in real space between the two transforms).  Three kernels per band block:
//   k_zinv   per (chunk of sticks, band): psi(G) to float32 into the z-sticks (zeros elsewhere), inverse z-transform,
//            Zt[b][j3][stick].
//   k_plane  per (z-plane, band): the plane [m1-plane][j2] in shared memory; inverse y, then in chunks of columns
//            inverse x, x V, forward x keeping the m1-planes, then forward y keeping the sticks -> Y[b][j3][stick].
//   k_zfwd   per (chunk of sticks, band): forward z-transform, keep the sphere, add the kinetic term |k+G|^2/2 psi(G)
//            in float64 (1/N_r is in the float32 copy of V but for a power of two, which would take values of small bands below
//            float32's range before the forward transform sums them).
// The transforms are the in-place two-stage form of line_stages.cuh: a stage's items are dealt over all threads of the CTA,
// coprime factors need no twiddles, and one kernel (run-time radix switch) serves every box, cubic or not.
// psi is read, and H psi written, by integer conversions (convert.cuh), since a cast costs as much as a float64 FMA.
//
// What bounds it: instruction issue (a codelet's ~10 float32 instructions a value and stage, a load, a store and their
// addresses) and the barriers between stages.  Measured with 160 bands on 90^3: planes 729 -> 594 us, z kernels 295 ->
// 240 us against register codelets with a fixed line group per warp (24 to 30 of 32 lanes busy, cubic boxes of
// 20 edges only; the others had the generic kernels).
//
// The raw form takes float32 psi and gives 2^sh times the local term alone in float32, [nb][npw] both: the Gamma form packs two
// real bands into one complex one in float32 and adds the kinetic term itself (gamma.cu).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <utility>
#include <vector>

#include "convert.cuh"
#include "float_fft.cuh"
#include "hpsi_internal.h"

namespace hpsi {

namespace {

#include "line_stages.cuh"

struct FloatArith {
  using V = float2;
  using Tw = float2;
  template <int R> using Dft = FfDft<R>;
  static __device__ __forceinline__ float2 twiddle(float2 v, float2 w) { return ff_mul(v, w.x, w.y); }
};

struct FastItem {
  int nb, npw, npl, nst;
  int n1, n2, n3;
  LineAxis ax[3];
  int cw, nch;                 // columns per x chunk, z chunks
  int raw;
  int sh;                      // V holds 2^sh / N_r: results times 2^-sh
  const int *soff, *zoff, *zbeg;   // Problem's lookup tables
  const int* xmap;             // [n1]: plane of ix or -1
  const void* psi;             // double2 (raw: float2) [nb][npw]
  void* hpsi;
  const double* kin;
  float2* Zt;                  // [nb][n3][nst]
  float2* Yb;
  const float* V;              // [n3][slot of j1][slot of j2], V 2^sh / N_r
};

// Every launch takes its items by value (the parameter block is 32 KB on sm_70 and later).
struct FastBatch {
  int nitems;
  int off_z[kMaxLocalItems + 1];
  int off_p[kMaxLocalItems + 1];
  FastItem item[kMaxLocalItems];
};

struct Placed {   // a value and its place in the tile
  float2 v;
  int at;
};

template <int MAXR>
__device__ __forceinline__ void zinv_tile(const FastItem& a, int ch, int b, unsigned char* smem) {
  constexpr int SC = kStickChunk, ld = SC + 1;
  const int n = a.n3;
  float2* tw = reinterpret_cast<float2*>(smem);
  float2* L = tw + n;                                   // [cell][stick], rows of SC + 1
  const int s0 = ch * SC, ns = min(SC, a.nst - s0);
  const int g0 = a.zbeg[ch], ng = a.zbeg[ch + 1] - g0;
  load_table(tw, a.ax[2].ftw, a.ax[2]);
  for (int i = threadIdx.x; i < n * ld; i += blockDim.x) L[i] = make_float2(0.f, 0.f);
  __syncthreads();
  const size_t row = (size_t)b * a.npw + g0;
  auto place = [&](int, Placed q) { L[q.at] = q.v; };
  if (a.raw) {
    const float2* ps = static_cast<const float2*>(a.psi) + row;
    staged_loop(ng, [&](int i) { return Placed{ps[i], a.zoff[g0 + i]}; }, place);
  } else {
    const double2* ps = static_cast<const double2*>(a.psi) + row;
    staged_loop(ng, [&](int i) { return Placed{f64_to_f32(ps[i]), a.zoff[g0 + i]}; }, place);
  }
  __syncthreads();
  const LineView<float2> lines{L, 1, ld};
  line_stage1<FloatArith, MAXR, false>(a.ax[2], ns, tw, lines);
  __syncthreads();
  line_stage2<FloatArith, MAXR, false>(a.ax[2], ns, tw, lines);
  __syncthreads();
  float2* Z = a.Zt + (size_t)b * n * a.nst + s0;
  const int per = blockDim.x / SC, r0 = threadIdx.x / SC, sl = threadIdx.x % SC;
  if (sl < ns)
    for (int j3 = r0; j3 < n; j3 += per) Z[(size_t)j3 * a.nst + sl] = L[a.ax[2].slot[j3] * ld + sl];
}

template <int MAXR>
__device__ __forceinline__ void plane_tile(const FastItem& a, int j3, int b, unsigned char* smem) {
  const int n1 = a.n1, n2 = a.n2, npl = a.npl, PS = n2 | 1, cw = a.cw;
  float2* twx = reinterpret_cast<float2*>(smem);
  float2* twy = twx + (a.ax[0].twiddled ? n1 : 0);
  float2* P = twy + (a.ax[1].twiddled ? n2 : 0);        // [plane][cell of j2], a row of zeros
  float2* X = P + (npl + 1) * PS;                       // [cell of x][column of the chunk]
  int* xo = reinterpret_cast<int*>(X + n1 * cw);
  xo += (4 - ((reinterpret_cast<uintptr_t>(xo) >> 2) & 3)) & 3;   // read as int4
  load_table(twx, a.ax[0].ftw, a.ax[0]);
  load_table(twy, a.ax[1].ftw, a.ax[1]);
  build_row_table(xo, a.ax[0], a.xmap, PS, npl * PS);
  for (int i = threadIdx.x; i < (npl + 1) * PS; i += blockDim.x) P[i] = make_float2(0.f, 0.f);
  __syncthreads();
  const float2* zin = a.Zt + ((size_t)b * a.n3 + j3) * a.nst;
  staged_loop(a.nst, [&](int i) { return Placed{zin[i], a.soff[i]}; }, [&](int, Placed q) { P[q.at] = q.v; });
  __syncthreads();
  const LineView<float2> rows{P, PS, 1}, cols{X, 1, cw};
  line_stage1<FloatArith, MAXR, false>(a.ax[1], npl, twy, rows);
  __syncthreads();
  line_stage2<FloatArith, MAXR, false>(a.ax[1], npl, twy, rows);
  __syncthreads();
  const float* V = a.V + (size_t)j3 * n1 * n2;
  for (int c0 = 0; c0 < n2; c0 += cw) {
    const int nc = min(cw, n2 - c0);
    x_stage1<FloatArith, MAXR>(a.ax[0], nc, twx, xo, P + c0, cols);
    __syncthreads();
    // the last inverse stage, x V, and the first forward one on the same registers; from here on real and imaginary
    // parts are swapped, which turns the codelets' sign into the forward one
    radix_switch<MAXR>(a.ax[0].r2, [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      const LineAxis& ax = a.ax[0];
      const int items = nc * ax.r1;
      const float inv = 1.0f / (float)nc;
      for (int it = threadIdx.x; it < items; it += blockDim.x) {
        int k1, c;
        split_index(it, nc, inv, k1, c);
        float2* q = X + k1 * R * cw + c;
        const float* vp = V + k1 * R * n2 + c0 + c;
        float2 v[R];
        float w[R];
#pragma unroll
        for (int i = 0; i < R; ++i) {
          v[i] = q[i * cw];
          w[i] = __ldg(vp + i * n2);
        }
        FfDft<R>::run(v);
#pragma unroll
        for (int i = 0; i < R; ++i) v[i] = make_float2(v[i].y * w[i], v[i].x * w[i]);
        FfDft<R>::run(v);
        if (ax.twiddled) {
#pragma unroll
          for (int i = 1; i < R; ++i) v[i] = FloatArith::twiddle(v[i], twx[k1 * i]);
        }
#pragma unroll
        for (int i = 0; i < R; ++i) q[i * cw] = v[i];
      }
    });
    __syncthreads();
    x_stage1_rev<FloatArith, MAXR>(a.ax[0], nc, xo, npl * PS, cols, P + c0, [](float2) {});
    __syncthreads();
  }
  line_stage2<FloatArith, MAXR, true>(a.ax[1], npl, twy, rows);
  __syncthreads();
  line_stage1<FloatArith, MAXR, true>(a.ax[1], npl, twy, rows);
  __syncthreads();
  float2* yo = a.Yb + ((size_t)b * a.n3 + j3) * a.nst;
  staged_loop(a.nst, [&](int i) { return a.soff[i]; }, [&](int i, int at) { yo[i] = P[at]; });
}

template <int MAXR>
__device__ __forceinline__ void zfwd_tile(const FastItem& a, int ch, int b, unsigned char* smem) {
  constexpr int SC = kStickChunk, ld = SC + 1;
  const int n = a.n3;
  float2* tw = reinterpret_cast<float2*>(smem);
  float2* L = tw + n;
  const int s0 = ch * SC, ns = min(SC, a.nst - s0);
  const int g0 = a.zbeg[ch], ng = a.zbeg[ch + 1] - g0;
  load_table(tw, a.ax[2].ftw, a.ax[2]);
  const float2* Y = a.Yb + (size_t)b * n * a.nst + s0;
  // (sticks past the last one are transformed with the others, from whatever the tile holds, and not read)
  staged_loop(
      n * SC, [&](int i) { return i % SC < ns ? Y[(size_t)(i / SC) * a.nst + i % SC] : make_float2(0.f, 0.f); },
      [&](int i, float2 v) { L[a.ax[2].slot[i / SC] * ld + i % SC] = v; });
  __syncthreads();
  const LineView<float2> lines{L, 1, ld};
  line_stage2<FloatArith, MAXR, true>(a.ax[2], ns, tw, lines);
  __syncthreads();
  line_stage1<FloatArith, MAXR, true>(a.ax[2], ns, tw, lines);
  __syncthreads();
  const size_t row = (size_t)b * a.npw + g0;
  if (a.raw) {
    float2* out = static_cast<float2*>(a.hpsi) + row;
    staged_loop(ng, [&](int i) { return a.zoff[g0 + i]; },
                [&](int i, int at) {
                  const float2 v = L[at];   // swapped
                  out[i] = make_float2(v.y, v.x);
                });
  } else {
    struct In {
      double2 x;
      double kg;
      int at;
    };
    const double2* ps = static_cast<const double2*>(a.psi) + row;
    double2* out = static_cast<double2*>(a.hpsi) + row;
    staged_loop(ng, [&](int i) { return In{ps[i], a.kin[g0 + i], a.zoff[g0 + i]}; },
                [&](int i, In q) {
                  const float2 v = L[q.at];   // swapped
                  out[i] = make_double2(fma(q.kg, q.x.x, f32_to_f64(v.y, a.sh)), fma(q.kg, q.x.y, f32_to_f64(v.x, a.sh)));
                });
  }
}

// Threads per SM that the kernels' registers allow
template <int MAXR> constexpr int kPlaneThreads = MAXR > 12 ? 768 : 1024;
inline int plane_threads(int rmax) { return rmax > 12 ? kPlaneThreads<16> : kPlaneThreads<10>; }

template <int MAXR>
__global__ void __launch_bounds__(512, MAXR > 12 ? 1 : 2) k_zinv(const __grid_constant__ FastBatch bt) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int i = tile_item(bt.off_z, bt.nitems, blockIdx.x), l = blockIdx.x - bt.off_z[i];
  zinv_tile<MAXR>(bt.item[i], l % bt.item[i].nch, l / bt.item[i].nch, smem_raw);
}
template <int MAXR>
__global__ void __launch_bounds__(kPlaneThreads<MAXR>, 1) k_plane(const __grid_constant__ FastBatch bt) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int i = tile_item(bt.off_p, bt.nitems, blockIdx.x), l = blockIdx.x - bt.off_p[i];
  plane_tile<MAXR>(bt.item[i], l % bt.item[i].n3, l / bt.item[i].n3, smem_raw);
}
template <int MAXR>
__global__ void __launch_bounds__(512, MAXR > 12 ? 1 : 2) k_zfwd(const __grid_constant__ FastBatch bt) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int i = tile_item(bt.off_z, bt.nitems, blockIdx.x), l = blockIdx.x - bt.off_z[i];
  zfwd_tile<MAXR>(bt.item[i], l % bt.item[i].nch, l / bt.item[i].nch, smem_raw);
}

#include "nonlocal_tiles.cuh"

// The whole batch in one cooperative launch: the tiles of the three kernels above phase by phase, and, when
// nl.nitems > 0, the float64 nonlocal term of the items, with a bounded grid barrier between the phases.
struct FastPersist {
  unsigned* bar;   // [0]: arrival counter; [1 + phase]: tile counters; zero at launch
  int* err;
};
template <int MAXR>
__global__ void __launch_bounds__(256) k_hpsi_batch(const __grid_constant__ FastBatch bt,
                                                    const __grid_constant__ NlBatch nl, const FastPersist pc) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const unsigned G = gridDim.x;
  const int nz = bt.off_z[bt.nitems], np = bt.off_p[bt.nitems];
  for (int t = persist_next(pc.bar + 1); t < nz; t = persist_next(pc.bar + 1)) {
    const int i = tile_item(bt.off_z, bt.nitems, t), l = t - bt.off_z[i];
    zinv_tile<MAXR>(bt.item[i], l % bt.item[i].nch, l / bt.item[i].nch, smem_raw);
  }
  if (!persist_sync(pc.bar, G, pc.err)) return;
  for (int t = persist_next(pc.bar + 2); t < np; t = persist_next(pc.bar + 2)) {
    const int i = tile_item(bt.off_p, bt.nitems, t), l = t - bt.off_p[i];
    plane_tile<MAXR>(bt.item[i], l % bt.item[i].n3, l / bt.item[i].n3, smem_raw);
  }
  if (!persist_sync(pc.bar, 2 * G, pc.err)) return;
  for (int t = persist_next(pc.bar + 3); t < nz; t = persist_next(pc.bar + 3)) {
    const int i = tile_item(bt.off_z, bt.nitems, t), l = t - bt.off_z[i];
    zfwd_tile<MAXR>(bt.item[i], l % bt.item[i].nch, l / bt.item[i].nch, smem_raw);
  }
  if (nl.nitems > 0) nonlocal_phases(nl, pc.bar, pc.err, G, 3, reinterpret_cast<double2*>(smem_raw));
}

// floor(log2 N_r)
inline int scale_bits(const int n[3]) { return std::ilogb((double)n[0] * n[1] * n[2]); }

// V[j3][j2][j1] -> [j3][slot of j1][slot of j2] in float32, times 2^scale_bits / N_r (and line_gain's correction)
__global__ void k_fast_v(LineAxis a1, LineAxis a2, int n3, double scale, const double* __restrict__ v,
                         float* __restrict__ out) {
  const size_t n = (size_t)a1.n * a2.n * n3;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const int j1 = (int)(i % a1.n), j2 = (int)(i / a1.n % a2.n);
    const size_t j3 = i / ((size_t)a1.n * a2.n);
    out[(j3 * a1.n + a1.slot[j1]) * a2.n + a2.slot[j2]] = (float)(v[i] * scale);
  }
}

struct FastLaunch {
  FastBatch bt;
  size_t smem_z = 0, smem_p = 0;
  int maxr = 0, items_z = 0, items_p = 0;   // largest radix, largest stages
  int block = 0;                            // plane block of the item with the largest planes
  void reset() {
    bt.nitems = 0;
    bt.off_z[0] = bt.off_p[0] = 0;
    smem_z = smem_p = 0;
    maxr = items_z = items_p = 0;
  }
  void add(Context& c, const Problem& p, const void* psi, void* hpsi, int nb, void* zt, void* yb, bool raw = false) {
    const int i = bt.nitems++;
    FastItem& it = bt.item[i];
    const FloatPlan& f = p.fast;
    it.nb = nb;
    it.npw = p.npw;
    it.npl = p.npl;
    it.nst = p.nst;
    it.n1 = p.n[0];
    it.n2 = p.n[1];
    it.n3 = p.n[2];
    for (int a = 0; a < 3; ++a) {
      it.ax[a] = p.fast.ax[a];
      maxr = std::max(maxr, std::max(it.ax[a].r1, it.ax[a].r2));
    }
    it.cw = f.cw;
    it.nch = f.nch;
    it.raw = raw;
    it.sh = f.sh;
    it.soff = p.tab[HPSI_MIXED].soff;
    it.zoff = p.tab[HPSI_MIXED].zoff;
    it.zbeg = p.tab[HPSI_MIXED].zbeg;
    it.xmap = p.d_xmap;
    it.psi = psi;
    it.hpsi = hpsi;
    it.kin = p.d_kin;
    it.Zt = static_cast<float2*>(zt);
    it.Yb = static_cast<float2*>(yb);
    it.V = static_cast<const float*>(c.vbufs[p.vslot + 3]);
    items_z = std::max(items_z, kStickChunk * std::max(it.ax[2].r1, it.ax[2].r2));
    items_p = std::max(items_p, std::max(it.npl * std::max(it.ax[1].r1, it.ax[1].r2),
                                         f.cw * std::max(it.ax[0].r1, it.ax[0].r2)));
    bt.off_z[i + 1] = bt.off_z[i] + f.nch * nb;
    bt.off_p[i + 1] = bt.off_p[i] + p.n[2] * nb;
    smem_z = std::max(smem_z, f.smem_z);
    if (f.smem_p > smem_p) block = f.block;
    smem_p = std::max(smem_p, f.smem_p);
  }
  template <int MAXR> int run_t(Context& c) {
    static std::atomic<unsigned long long> devices{0};
    cudaError_t e = allow_smem(c, devices, {(const void*)k_zinv<MAXR>, (const void*)k_plane<MAXR>, (const void*)k_zfwd<MAXR>});
    if (e != cudaSuccess) return cuda_fail(c, e, "fast local kernels");
    const int nz = bt.off_z[bt.nitems], np = bt.off_p[bt.nitems];
    auto warps = [](int items) { return (items + 31) / 32 * 32; };
    // z: one round of a stage's items; planes: plane_shape's block, or one round where there is a CTA per SM at most;
    // never more than this instance's launch bound, which another item's radix may have set (any block size serves)
    const int bz = std::max(128, std::min(512, warps(items_z)));
    const int bp = std::min(kPlaneThreads<MAXR>, np <= c.sm_count ? std::max(block, warps(items_p)) : block);
    HPSI_LAUNCH(c, HPSI_K_INV_ZY, (k_zinv<MAXR><<<nz, bz, smem_z, c.stream>>>(bt)));
    HPSI_LAUNCH(c, HPSI_K_XVX_Y, (k_plane<MAXR><<<np, bp, smem_p, c.stream>>>(bt)));
    HPSI_LAUNCH(c, HPSI_K_FWD_Z, (k_zfwd<MAXR><<<nz, bz, smem_z, c.stream>>>(bt)));
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(c, e, "fast local kernels launch");
    return HPSI_OK;
  }
  int run(Context& c) { return maxr > 12 ? run_t<16>(c) : maxr > 10 ? run_t<12>(c) : run_t<10>(c); }
  template <int MAXR> int persistent_t(Context& c, const NlBatch& nl, unsigned* bar, bool* done) {
    const void* kern = (const void*)k_hpsi_batch<MAXR>;
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
    FastPersist pc{bar, c.d_err};
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

// Tile sizes of a problem's float32 local term (ok = false: an edge without factors, or a plane that does not fit).
void float_plan(Problem& p, size_t smem_optin) {
  FloatPlan& f = p.fast;
  f.ok = false;
  for (int a = 0; a < 3; ++a)
    if (!p.fast.ax[a].r1) return;
  const int n1 = p.n[0], n2 = p.n[1], n3 = p.n[2];
  auto tws = [&](int a) { return p.fast.ax[a].twiddled ? sizeof(float2) * (size_t)p.n[a] : 0; };
  f.nch = (p.nst + kStickChunk - 1) / kStickChunk;
  f.smem_z = sizeof(float2) * (size_t)n3 * (kStickChunk + 2);
  const size_t base = tws(0) + tws(1) + sizeof(float2) * (size_t)(p.npl + 1) * (n2 | 1) +
                      sizeof(int) * (p.fast.ax[0].r2 * (size_t)((p.fast.ax[0].r1 + 3) & ~3) + 4);
  const size_t col = sizeof(float2) * (size_t)n1;
  int rmax = 0;
  for (int a = 0; a < 3; ++a) rmax = std::max(rmax, p.fast.ax[a].r1);
  plane_shape(p.fast.ax[0], p.fast.ax[1], p.npl, base, col, smem_optin, plane_threads(rmax),
              &f.cw, &f.block);
  if (f.cw == 0) return;
  f.smem_p = base + col * f.cw;
  f.sh = scale_bits(p.n);
  f.ok = f.smem_z <= smem_optin - 1024;
}

// The float32 constants of the codelets and twiddles are up to 2^-25 off, the same on every line, so the two transforms of a
// line make an operator that is not n times the identity but off by up to 6e-8 of it (81 points; the 9-point codelet's
// rotations): an error in <psi|V|psi> that does not average out as the other roundings do.  This is that operator's
// mean diagonal over n, with the same constants in double, by which V is divided: what stays is a tenth of it
// (eigenvalues on 36^3 and 45^3 boxes: 5.4e-8 and 5.9e-8 -> 6e-9 Ha from the constants; of mixed solves there in
// all 7.0e-8 and 1.1e-7 -> 1.7e-8 and 5.1e-8).
double line_gain(const LineAxis& ax, const float2* tw) {
  const int n = ax.n, r1 = ax.r1, r2 = ax.r2;
  std::vector<double2> w(n);
  // items from .. to - 1 of a stage, item i in the cells i first + a step
  auto stage = [&](int r, int from, int to, int first, int step, bool twiddled) {
    for (int i = from; i < to; ++i) {
      double2 v[16];
      for (int a = 0; a < r; ++a) v[a] = w[i * first + a * step];
      switch (r) {
        case 2: FfDft<2>::run(v); break;
        case 3: FfDft<3>::run(v); break;
        case 4: FfDft<4>::run(v); break;
        case 5: FfDft<5>::run(v); break;
        case 6: FfDft<6>::run(v); break;
        case 8: FfDft<8>::run(v); break;
        case 9: FfDft<9>::run(v); break;
        case 10: FfDft<10>::run(v); break;
        case 12: FfDft<12>::run(v); break;
        case 15: FfDft<15>::run(v); break;
        default: FfDft<16>::run(v);
      }
      for (int a = 0; a < r; ++a) {
        if (twiddled && a > 0) v[a] = ff_mul(v[a], tw[i * a].x, tw[i * a].y);
        w[i * first + a * step] = v[a];
      }
    }
  };
  double sum = 0.0;
  for (int a = 0; a < r1; ++a)
    for (int t = 0; t < r2; ++t) {
      std::fill(w.begin(), w.end(), make_double2(0.0, 0.0));
      w[a * r2 + t].x = 1.0;
      stage(r1, t, t + 1, 1, r2, ax.twiddled);   // the others are zero
      stage(r2, 0, r1, r2, 1, false);
      for (double2& v : w) std::swap(v.x, v.y);   // the opposite sign, as in plane_tile
      stage(r2, 0, r1, r2, 1, ax.twiddled);
      stage(r1, t, t + 1, 1, r2, false);          // the diagonal is in this one
      sum += w[a * r2 + t].y;
    }
  return sum / ((double)n * n);
}

// V 2^sh / N_r in float32 in slot order (vbufs[slot + 3]) from the float64 V.
int float_potential(Context& c, int slot, const LineAxis ax[3], int kernel_class) {
  const size_t nr = (size_t)ax[0].n * ax[1].n * ax[2].n;
  const int n[3] = {ax[0].n, ax[1].n, ax[2].n};
  const double scale = std::ldexp(1.0, scale_bits(n)) / ((double)nr * ax[0].gain * ax[1].gain * ax[2].gain);
  HPSI_LAUNCH(c, kernel_class, (k_fast_v<<<(int)std::min<size_t>(4 * c.sm_count, (nr + 255) / 256), 256, 0, c.stream>>>(
                                   ax[0], ax[1], ax[2].n, scale, static_cast<const double*>(c.vbufs[slot]),
                                   static_cast<float*>(c.vbufs[slot + 3]))));
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(c, e, "float32 potential");
  return HPSI_OK;
}

int local_fast_apply(Context& c, const Problem& p, const double2* psi, double2* hpsi, int nbnd, void* Zt, void* Yb,
                     int nbb) {
  if (cur_prec(c) == HPSI_FP64) return local_fixed_apply(c, p, psi, hpsi, nbnd, Zt, Yb, nbb);
  static thread_local FastLaunch fl;   // host staging of the parameter block: threads use contexts of their own at the same time
  for (int b0 = 0; b0 < nbnd; b0 += nbb) {
    fl.reset();
    fl.add(c, p, psi + (size_t)b0 * p.npw, hpsi + (size_t)b0 * p.npw, std::min(nbb, nbnd - b0), Zt, Yb);
    const int rc = fl.run(c);
    if (rc) return rc;
  }
  return HPSI_OK;
}

int local_fast_apply_raw(Context& c, const Problem& p, const float2* f, float2* F, int nbnd, void* Zt, void* Yb, int nbb) {
  static thread_local FastLaunch fl;
  for (int b0 = 0; b0 < nbnd; b0 += nbb) {
    fl.reset();
    fl.add(c, p, f + (size_t)b0 * p.npw, F + (size_t)b0 * p.npw, std::min(nbb, nbnd - b0), Zt, Yb, true);
    const int rc = fl.run(c);
    if (rc) return rc;
  }
  return HPSI_OK;
}

// Several problems in one launch per kernel; zt[i], yb[i] hold item i's stick rows (local_row_bytes).
int local_fast_apply_multi(Context& c, int nitem, const int* prob, const int* nbnd, const double2* const* psi,
                           double2* const* hpsi, void* const* zt, void* const* yb) {
  if (cur_prec(c) == HPSI_FP64) return local_fixed_apply_multi(c, nitem, prob, nbnd, psi, hpsi, zt, yb);
  static thread_local FastLaunch fl;
  for (int i0 = 0; i0 < nitem; i0 += kMaxLocalItems) {
    fl.reset();
    for (int i = i0; i < std::min(nitem, i0 + kMaxLocalItems); ++i)
      fl.add(c, c.probs[prob[i]], psi[i], hpsi[i], nbnd[i], zt[i], yb[i]);
    const int rc = fl.run(c);
    if (rc) return rc;
  }
  return HPSI_OK;
}

// The whole hpsi_apply_batch in one persistent launch: every item on the fast path with one box edge, at most
// kMaxLocalItems of them (and kNlBatch with a nonlocal term in float64).  with_nl: the float64 nonlocal term of the
// items joins the launch.  *done = false: nothing was launched and the caller takes the launch-per-kernel path.
int local_batch_persistent(Context& c, int nitem, const int* prob, const int* nbnd, const double2* const* psi,
                           double2* const* hpsi, void* const* zt, void* const* yb, bool with_nl, bool* done) {
  *done = false;
  if (nitem < 1 || nitem > kMaxLocalItems || nitem > kNlBatch || c.force_generic) return HPSI_OK;
  const int pr = cur_prec(c);
  for (int i = 0; i < nitem; ++i) {
    const Problem& p = c.probs[prob[i]];
    if (!local_fast_ok(p, pr) || p.n[0] != c.probs[prob[0]].n[0] || nbnd[i] < 1) return HPSI_OK;
  }
  if (pr == HPSI_FP64) return local_fixed_persistent(c, nitem, prob, nbnd, psi, hpsi, zt, yb, with_nl, done);
  static thread_local FastLaunch fl;
  static thread_local NlBatch nl;
  fl.reset();
  for (int i = 0; i < nitem; ++i) fl.add(c, c.probs[prob[i]], psi[i], hpsi[i], nbnd[i], zt[i], yb[i]);
  nl.nitems = 0;
  if (with_nl) {
    const int rc = persistent_nl_batch(c, nitem, prob, nbnd, psi, hpsi, nl);
    if (rc) return rc;
  }
  const int rc = ensure_buffer(c, &c.ws.pbar, &c.ws.pbarbytes, 256);
  if (rc) return rc;
  return fl.persistent(c, nl, static_cast<unsigned*>(c.ws.pbar), done);
}

}  // namespace hpsi
