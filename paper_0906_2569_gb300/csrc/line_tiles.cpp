// Shape of the plane kernels' CTAs (local_fast.cu, local_fixed.cu).
#include <algorithm>

#include "hpsi_internal.h"

namespace hpsi {

// A stage with I items of radix R takes ceil(I / block) rounds of ~R steps, and every stage ends in a barrier (counted as 4
// steps): the shape with the most CTAs per SM over the CTA's rounds wins.  (On the 90^3 box the planes' time hardly depends
// on it: 5 CTAs of 192 threads and 18 columns, or 4 of 256 and 30, both take 758 us in float32 for 160 bands.)
void plane_shape(const LineAxis& x, const LineAxis& y, int npl, size_t base, size_t col, size_t smem_optin, int threads,
                 int* cw, int* block) {
  *cw = *block = 0;
  double best = 0.0;
  for (int ctas = 1; ctas <= 8; ++ctas) {
    const size_t room = smem_optin / ctas - 1100;
    if (room < base + col) break;
    for (int chunks = 1, last = 0; chunks <= y.n; ++chunks) {
      const int w = (y.n + chunks - 1) / chunks;
      if (w == last) continue;
      last = w;
      if (w < 4 && w < y.n) break;
      if (base + col * w > room) continue;
      for (int b = std::min(96, threads / ctas / 32 * 32); b * ctas <= threads; b += 32) {
        if (b < 64) continue;
        auto rounds = [&](int items) { return (items + b - 1) / b; };
        int t = 2 * (rounds(npl * y.r2) * (y.r1 + 2) + rounds(npl * y.r1) * (y.r2 + 2)) + 4 * 8;
        for (int c0 = 0; c0 < y.n; c0 += w) {
          const int n = std::min(w, y.n - c0);
          t += 2 * rounds(n * x.r2) * (x.r1 + 3) + rounds(n * x.r1) * (2 * x.r2 + 4) + 3 * 4;
        }
        const double score = (double)ctas / t;
        if (score > best) {
          best = score;
          *cw = w;
          *block = b;
        }
      }
      if (w < 12 && chunks > 8) break;   // narrower chunks only add barriers
    }
  }
}

}  // namespace hpsi
