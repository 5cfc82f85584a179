// The in-place two-stage line transforms of the local paths (fixed_fft.cuh describes the slots and the two forms), as
// stages over the lines of a tile in shared memory.  A stage's items, one R-point DFT each, are dealt over all threads of the
// CTA, so warps are full whatever the factors are.  The arithmetic C gives the value type V, Dft<R>, the
// twiddle type Tw and twiddle(v, w).  Included inside an anonymous namespace of namespace hpsi.
#pragma once

constexpr int kMaxLocalItems = 32;   // problems per launch

template <int R> struct Rx {
  static constexpr int value = R;
};
template <int MAXR, typename F>
__device__ __forceinline__ void radix_switch(int r, F&& f) {
  switch (r) {
    case 2: f(Rx<2>()); break;
    case 3: f(Rx<3>()); break;
    case 4: f(Rx<4>()); break;
    case 5: f(Rx<5>()); break;
    case 6: f(Rx<6>()); break;
    case 8: f(Rx<8>()); break;
    case 9: f(Rx<9>()); break;
    case 10: f(Rx<10>()); break;
    default:
      if constexpr (MAXR > 10) {
        switch (r) {
          case 12: f(Rx<12>()); break;
          default:
            if constexpr (MAXR > 12) {
              if (r == 15) f(Rx<15>());
              else f(Rx<16>());
            }
        }
      }
  }
}

// it = a cnt + b with b < cnt, for the small non-negative numbers of a tile
__device__ __forceinline__ void split_index(int it, int cnt, float inv, int& a, int& b) {
  a = (int)(((float)it + 0.5f) * inv);
  b = it - a * cnt;
}

// The lines of a tile: element (line, cell) at p[line ls + cell cs]
template <typename V> struct LineView {
  V* p;
  int ls, cs;
};
struct AsIs {
  template <typename V> __device__ __forceinline__ V operator()(V v) const { return v; }
};

// Stage 1 (or, REV, the last stage of the reversed sequence) of `cnt` lines, in place: item (t, line), lines fastest over
// the threads.  f is applied to the values as they are read.
template <typename C, int MAXR, bool REV, typename F = AsIs>
__device__ __forceinline__ void line_stage1(const LineAxis& ax, int cnt, const typename C::Tw* tw,
                                            LineView<typename C::V> w, F f = F()) {
  radix_switch<MAXR>(ax.r1, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    const int items = cnt * ax.r2, step = ax.r2 * w.cs;
    const float inv = 1.0f / (float)cnt;
    for (int it = threadIdx.x; it < items; it += blockDim.x) {
      int t, line;
      split_index(it, cnt, inv, t, line);
      typename C::V* q = w.p + line * w.ls + t * w.cs;
      typename C::V v[R];
#pragma unroll
      for (int a = 0; a < R; ++a) v[a] = f(q[a * step]);
      C::template Dft<R>::run(v);
      if (!REV && ax.twiddled) {
#pragma unroll
        for (int a = 1; a < R; ++a) v[a] = C::twiddle(v[a], tw[t * a]);
      }
#pragma unroll
      for (int a = 0; a < R; ++a) q[a * step] = v[a];
    }
  });
}

// Stage 2 (or, REV, the first stage of the reversed sequence): item (k1, line)
template <typename C, int MAXR, bool REV, typename F = AsIs>
__device__ __forceinline__ void line_stage2(const LineAxis& ax, int cnt, const typename C::Tw* tw,
                                            LineView<typename C::V> w, F f = F()) {
  radix_switch<MAXR>(ax.r2, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    const int items = cnt * ax.r1;
    const float inv = 1.0f / (float)cnt;
    for (int it = threadIdx.x; it < items; it += blockDim.x) {
      int k1, line;
      split_index(it, cnt, inv, k1, line);
      typename C::V* q = w.p + line * w.ls + k1 * R * w.cs;
      typename C::V v[R];
#pragma unroll
      for (int b = 0; b < R; ++b) v[b] = f(q[b * w.cs]);
      C::template Dft<R>::run(v);
      if (REV && ax.twiddled) {
#pragma unroll
        for (int b = 1; b < R; ++b) v[b] = C::twiddle(v[b], tw[k1 * b]);
      }
#pragma unroll
      for (int b = 0; b < R; ++b) q[b * w.cs] = v[b];
    }
  });
}

// The x stages read and write rows of the plane array, one row per m1-plane: for every item t the rows' offsets of its r1
// entries (natural index (r2 a + s2 t) mod n), `none` for an index without a plane.
__device__ __forceinline__ int row_table_width(int r1) { return (r1 + 3) & ~3; }
__device__ __forceinline__ void build_row_table(int* xo, const LineAxis& ax, const int* xmap, int row, int none) {
  const int wd = row_table_width(ax.r1);
  for (int i = threadIdx.x; i < ax.r2 * wd; i += blockDim.x) {
    const int t = i / wd, a = i - t * wd;
    int off = none;
    if (a < ax.r1) {
      const int pp = xmap[(ax.r2 * a + ax.s2 * t) % ax.n];
      if (pp >= 0) off = pp * row;
    }
    xo[i] = off;
  }
}
template <int R>
__device__ __forceinline__ void load_rows(int (&o)[(R + 3) / 4 * 4], const int* xo, int t) {
  const int4* q = reinterpret_cast<const int4*>(xo + t * ((R + 3) & ~3));
#pragma unroll
  for (int i = 0; i < (R + 3) / 4; ++i) {
    const int4 w = q[i];
    o[4 * i] = w.x;
    o[4 * i + 1] = w.y;
    o[4 * i + 2] = w.z;
    o[4 * i + 3] = w.w;
  }
}
// Stage 1 of columns of the plane array into the x tile (absent planes read the row of zeros at `none`), and the last
// reversed stage back from it.
template <typename C, int MAXR, typename F = AsIs>
__device__ __forceinline__ void x_stage1(const LineAxis& ax, int cnt, const typename C::Tw* tw, const int* xo,
                                         const typename C::V* P, LineView<typename C::V> w, F f = F()) {
  radix_switch<MAXR>(ax.r1, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    const int items = cnt * ax.r2, step = ax.r2 * w.cs;
    const float inv = 1.0f / (float)cnt;
    for (int it = threadIdx.x; it < items; it += blockDim.x) {
      int t, line;
      split_index(it, cnt, inv, t, line);
      int o[(R + 3) / 4 * 4];
      load_rows<R>(o, xo, t);
      typename C::V v[R];
#pragma unroll
      for (int a = 0; a < R; ++a) v[a] = f(P[o[a] + line]);
      C::template Dft<R>::run(v);
      if (ax.twiddled) {
#pragma unroll
        for (int a = 1; a < R; ++a) v[a] = C::twiddle(v[a], tw[t * a]);
      }
      typename C::V* q = w.p + line * w.ls + t * w.cs;
#pragma unroll
      for (int a = 0; a < R; ++a) q[a * step] = v[a];
    }
  });
}
template <typename C, int MAXR, typename G>
__device__ __forceinline__ void x_stage1_rev(const LineAxis& ax, int cnt, const int* xo, int none,
                                             LineView<typename C::V> w, typename C::V* P, G&& seen) {
  radix_switch<MAXR>(ax.r1, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    const int items = cnt * ax.r2, step = ax.r2 * w.cs;
    const float inv = 1.0f / (float)cnt;
    for (int it = threadIdx.x; it < items; it += blockDim.x) {
      int t, line;
      split_index(it, cnt, inv, t, line);
      const typename C::V* q = w.p + line * w.ls + t * w.cs;
      typename C::V v[R];
#pragma unroll
      for (int a = 0; a < R; ++a) v[a] = q[a * step];
      C::template Dft<R>::run(v);
      int o[(R + 3) / 4 * 4];
      load_rows<R>(o, xo, t);
#pragma unroll
      for (int a = 0; a < R; ++a)
        if (o[a] != none) {
          seen(v[a]);
          P[o[a] + line] = v[a];
        }
    }
  });
}

template <typename Tw>
__device__ __forceinline__ void load_table(Tw* dst, const Tw* src, const LineAxis& ax) {
  if (!ax.twiddled) return;   // the prime-factor form has none
  for (int i = threadIdx.x; i < ax.n; i += blockDim.x) dst[i] = src[i];
}

// for (i = thread; i < n; i += threads) with four iterations' loads in flight: a tile's tables and rows come from L2, and
// one chained load per iteration was a third of a plane's time
template <typename LD, typename ST>
__device__ __forceinline__ void staged_loop(int n, LD&& ld, ST&& st) {
  const int T = blockDim.x;
  for (int i0 = threadIdx.x; i0 < n; i0 += 4 * T) {
    decltype(ld(0)) v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (i0 + j * T < n) v[j] = ld(i0 + j * T);
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (i0 + j * T < n) st(i0 + j * T, v[j]);
  }
}

// The item of tile t in the running counts off[0 .. n]
__device__ __forceinline__ int tile_item(const int* off, int n, int t) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (off[mid] <= t) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}
