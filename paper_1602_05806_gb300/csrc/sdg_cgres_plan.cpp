// Tile of the resident CG kernel (sdg_cgres.cuh) for a handle's grid.
#include <algorithm>

#include "sdg_internal.h"

namespace sdg {

// Candidates are the tilings with at most one CTA per SM whose lines, registers
// and shared memory fit a CTA; the cheapest by a count of issue cycles per
// iteration wins.  FP64: a warp instruction holds the SM's FP64 unit for 16
// cycles whichever of its lanes are active, so the count is of full warps and
// small grids spread over as many SMs as have a full warp.  FP32: four
// schedulers share the warps, and below about three warps per scheduler the
// latency of a line's dependent instructions shows instead.
ResPlan res_plan(const sdg_handle* h, bool fp32) {
  ResPlan best{};
  best.state = 2;
  const int dim = h->dim, n1 = h->g.n1;
  if (dim == 3 && n1 > kResMaxN1_3d) return best;
  const int npe = h->g.npe, lines_pe = npe / n1;
  const size_t es = (size_t)lines_pe * (n1 + 1), sz = fp32 ? 4 : 8;
  const int maxthr = fp32 ? 512 : 256, maxlpt = fp32 && n1 <= 8 ? 2 : 1;
  const double line = dim * (1.5 * n1 * n1 + (fp32 ? 14.0 : 6.0) * n1) + (fp32 ? 22.0 : 12.0) * n1;
  double best_cost = 0.0;
  int ts[3], nt[3];
  auto canonical = [&](int d, int t) {  // extents that differ by their tile count only once
    nt[d] = (h->g.n[d] + t - 1) / t;
    ts[d] = t;
    return (h->g.n[d] + nt[d] - 1) / nt[d] == t;
  };
  const long long most = std::min(h->nsm, kResMaxCtas);
  const long long max_te = (long long)maxthr * maxlpt / lines_pe;
  for (int tz = 1; tz <= h->g.n[2]; ++tz) {
    if (tz > max_te || !canonical(2, tz) || nt[2] > most) continue;
    for (int ty = 1; ty <= h->g.n[1]; ++ty) {
      if ((long long)tz * ty > max_te) break;
      if (!canonical(1, ty) || (long long)nt[2] * nt[1] > most) continue;
      for (int tx = 1; tx <= h->g.n[0]; ++tx) {
        const long long te = (long long)tz * ty * tx;
        if (te > max_te) break;
        if (!canonical(0, tx)) continue;
        const long long nblk = (long long)nt[2] * nt[1] * nt[0];
        if (nblk > most) continue;
        long long nh = 0;
        for (int d = 0; d < dim; ++d)
          if (nt[d] > 1) nh += 2 * (te / ts[d]);
        const size_t smem =
            ((te + nh) * es + (size_t)(dim - 1) * te * es + (size_t)2 * nh * npe) * sz + (te * 2 * dim + nh) * sizeof(int);
        // (the replacement kernel of the FP64 plan keeps the kernel patterns instead of the halo's r and Ap)
        const size_t smem2 =
            fp32 ? 0 : ((te + nh) * es + (size_t)(dim - 1) * te * es + (size_t)8 * npe) * sz + (te * 2 * dim + nh) * sizeof(int);
        if (std::max(smem, smem2) > (size_t)kResMaxSmem) continue;
        const long long lines = te * lines_pe, warps = (lines + 31) / 32, hw = (nh * npe + 31) / 32;
        const double exchange = nblk > 1 ? 1500.0 + 4.0 * nblk : 0.0;
        const double cost = exchange + (fp32 ? line * std::max<long long>((warps + 3) / 4, 3) + 25.0 * ((hw + 3) / 4)
                                             : 16.0 * (line * std::max<long long>(warps, 2) + 2.0 * hw));
        if (best.state == 1 && cost >= best_cost) continue;
        best_cost = cost;
        best.state = 1;
        for (int d = 0; d < 3; ++d) {
          best.ts[d] = ts[d];
          best.nt[d] = nt[d];
        }
        best.lpt = lines > maxthr ? 2 : 1;
        const long long thr = (lines + best.lpt - 1) / best.lpt;
        best.threads = (int)std::max<long long>(128, (thr + 31) / 32 * 32);
        best.smem = std::max(smem, smem2);
      }
    }
  }
  if (best.state == 1 || !fp32 || dim != 2) return best;
  // larger 2D FP32 tiles: as few rounds of lines per thread as possible, then
  // the smallest halo
  const int epr = kBigThreads / 32 * (32 / n1);
  for (int ty = 1; ty <= h->g.n[1]; ++ty) {
    if (!canonical(1, ty) || nt[1] > most) continue;
    for (int tx = 1; tx <= h->g.n[0]; ++tx) {
      const long long te = (long long)ty * tx;
      if (te > (long long)big_rounds(n1) * epr) break;
      if (!canonical(0, tx) || (long long)nt[1] * nt[0] > most) continue;
      const long long nh = (nt[0] > 1 ? 2 * ty : 0) + (nt[1] > 1 ? 2 * tx : 0);
      const size_t smem = big_smem(n1, te, nh);
      if (smem > (size_t)kResMaxSmem) continue;
      const double cost = (double)((te + epr - 1) / epr) * epr + 0.25 * nh;
      if (best.state == 1 && cost >= best_cost) continue;
      best_cost = cost;
      best.state = 1;
      best.big = 1;
      best.ts[0] = tx;
      best.ts[1] = ty;
      best.ts[2] = 1;
      best.nt[0] = nt[0];
      best.nt[1] = nt[1];
      best.nt[2] = 1;
      best.lpt = big_rounds(n1);
      best.threads = kBigThreads;
      best.smem = smem;
    }
  }
  return best;
}

}  // namespace sdg
