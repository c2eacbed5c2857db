// Residual replacement of the resident CG (sdg_cgres.cuh) in one cooperative
// launch: x += correction, r = b - A x in FP64 with the accurate operator, its
// norm, its projection onto the range of the operator (singular system), the
// decisions, and the vector the iterations go on with.  The start of a solve
// (first residual, its floor) is the same kernel.
//
// As nine launches and two host round trips a replacement took 140 us on
// 64 x 64 cells, N = 5, against 4.2 us for an iteration of the solve; its
// arithmetic is one operator application.  Here every CTA keeps its tile of x
// in shared memory and its lines of x and r in registers between the
// grid-wide sums, which travel like those of sdg_cgres.cuh (tagged words,
// bounded waits, fixed order).
#pragma once

#include "sdg_cgres.cuh"

namespace sdg {

constexpr int kResidMaxKd = 8;  // kernel patterns: 2^dim at most

template <int DIM, int N1>
struct ResidParams {
  Coef<double, N1> c;
  double w[N1];
  double s[3];
  double cmass;
  int n[3], ts[3], nt[3];
  const double* b;
  double* x;
  double* x0;           // copy of the start vector (singular system)
  float* x32;           // FP32 iterations: their correction (scaled by sigma), else null
  // by parity of the iteration count
  double* r[2];         // FP64 iterations: the residual
  float* r32[2];        // FP32 iterations: the residual, scaled (else null)
  const double* p[2];   // pending step of an iteration stopped at maxit
  const float* p32[2];
  const double* kb;     // kd x npe orthonormal kernel patterns
  int kd;               // 0: nothing to project
  double ncell, inv_ncell;
  SolverState* st;
  unsigned long long* slots;  // [2 parities][nslot][16 sums][2 words]
  int nslot;
  unsigned tag;
  int polls;            // of a wait before it gives up
  int start;            // 1: start of a solve
  double rtol, delta;
  int maxit;
};

// The sums v[0..15] of every thread of the grid, in s_sum of every CTA.
// Exchange number `tag`, in the words at `slot`.  All threads of the block call it;
// false (for all of them) when a wait of the CTA ran out: it leaves then.
__device__ __forceinline__ bool resid_exchange(double (&v)[16], unsigned long long* slot, unsigned tag, int limit,
                                               double (*s_red)[16], double* s_sum, int* s_fail) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
  // lanes halve the values between them: lane pair 2 i, 2 i + 1 ends with value i
#pragma unroll
  for (int h = 8; h >= 1; h >>= 1) {
    const bool up = lane & (2 * h);
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const double keep = up ? v[i + h] : v[i], give = up ? v[i] : v[i + h];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, give, 2 * h);
    }
  }
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
  if (!(lane & 1)) s_red[wid][lane >> 1] = v[0];
  __syncthreads();
  const int c = lane & 15, h2 = lane >> 4;
  if (wid == 0) {
    double t = 0.0;
    for (int w = h2; w < nw; w += 2) t += s_red[w][c];
    t += __shfl_xor_sync(0xffffffffu, t, 16);
    if (lane < 16) {
      if (gridDim.x > 1) {
        unsigned q[2];
        ResAcc<double>::pack(t, q);
        res_store_words(slot + 32 * blockIdx.x + 2 * lane, q[0], q[1], tag);
      } else {
        s_sum[lane] = t;
      }
    }
  }
  __syncthreads();
  if (gridDim.x > 1) {
    // a warp load covers two CTAs; warp w takes the pairs w, w + nw, ...
    constexpr int PB = 8;
    double t = 0.0;
    bool ok = true;
    for (int i0 = 2 * wid + h2; i0 < (int)gridDim.x && ok; i0 += PB * nw * 2) {
      unsigned long long q0[PB], q1[PB];
      int polls = 0;
      do {
        ok = true;
#pragma unroll
        for (int u = 0; u < PB; ++u)
          if (i0 + u * nw * 2 < (int)gridDim.x) res_load_words(slot + 32 * (i0 + u * nw * 2) + 2 * c, q0[u], q1[u]);
#pragma unroll
        for (int u = 0; u < PB; ++u)
          if (i0 + u * nw * 2 < (int)gridDim.x)
            ok = ok && (unsigned)(q0[u] >> 32) == tag && (unsigned)(q1[u] >> 32) == tag;
      } while (!ok && ++polls < limit);
      if (ok) {
#pragma unroll
        for (int u = 0; u < PB; ++u)
          if (i0 + u * nw * 2 < (int)gridDim.x) t += ResAcc<double>::unpack((unsigned)q0[u], (unsigned)q1[u]);
      }
    }
    if (!ok) *s_fail = 1;
    __syncwarp();
    t += __shfl_xor_sync(0xffffffffu, t, 16);
    if (lane < 16) s_red[wid][lane] = t;
    __syncthreads();
    if (tid < 16) {
      double z = 0.0;
      for (int w = 0; w < nw; ++w) z += s_red[w][tid];
      s_sum[tid] = z;
    }
  }
  __syncthreads();
  return *s_fail == 0;
}

// 2^floor(log2 |x|) / (2^52 2 sqrt 3) with the sign of an integer hash of the
// node's index (k_rounding_perturbation)
__device__ __forceinline__ double resid_perturb(double x, unsigned long long i) {
  const double scale = 0.5 / 1.7320508075688772 / 4503599627370496.0;
  const double pw = __longlong_as_double(__double_as_longlong(x) & 0x7FF0000000000000LL);
  unsigned long long z = i + 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  z ^= z >> 31;
  return ((z >> 63) ? -scale : scale) * pw;
}

template <int DIM, int N1>
__global__ void __launch_bounds__(256, 1) k_cg_resid(const __grid_constant__ ResidParams<DIM, N1> a) {
  using E = ResEl<DIM, N1>;
  constexpr int NPE = E::NPE, LINES = E::LINES, ES = E::ES;
  const ResTile<DIM> tile(a.n, a.ts, a.nt);
  const int TE = tile.TE, NH = tile.NH;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* s_p = reinterpret_cast<double*>(smem_raw);       // (TE + NH) ES: x
  double* s_o = s_p + (size_t)(TE + NH) * ES;              // (DIM - 1) TE ES
  double* s_kb = s_o + (size_t)(DIM - 1) * TE * ES;        // kd NPE
  int* s_nb = reinterpret_cast<int*>(s_kb + (size_t)a.kd * NPE);
  int* s_hel = s_nb + TE * 2 * DIM;
  __shared__ double s_w[N1];
  __shared__ double s_red[8][16];
  __shared__ double s_sum[16];
  __shared__ double s_dd[4];
  __shared__ int s_di[4];
  __shared__ int s_fail;

  SolverState* st = a.st;
  const int tid = threadIdx.x, nth = blockDim.x;
  if (tid < N1) s_w[tid] = a.w[tid];
  if (tid == 0) s_fail = 0;
  for (int i = tid; i < a.kd * NPE; i += nth) s_kb[i] = a.kb[i];
  tile.tables(a.n, a.nt, ES, s_nb, s_hel);

  const bool start = a.start != 0, f32 = a.r32[0] != nullptr;
  const int cur = start ? 0 : st->iter & 1;
  const int seg_done = start ? 0 : st->done, seg_status = start ? SDG_OK : st->status;
  const double sigma0 = start ? 1.0 : st->sigma, inv = start ? 1.0 : st->inv_sigma;
  // the iteration stopped at maxit with its last step not yet in x
  const bool pend = seg_done && seg_status == SDG_ERR_NOT_CONVERGED;
  const double al = st->alpha;
  const float alf = st->alpha_f;
  auto xval = [&](size_t i) -> double {
    double v = a.x[i];
    if (start) return v;
    if (f32) {
      float c = a.x32[i];
      if (pend) c = fmaf(alf, a.p32[cur][i], c);
      return v + (double)c * inv;
    }
    return pend ? fma(al, a.p[cur][i], v) : v;
  };

  // one x-line per thread
  const bool act = tid < TE * LINES;
  const int e = act ? tid / LINES : 0, lam = act ? tid - e * LINES : 0;
  size_t gl = 0;
  double x[N1], r[N1], xc[N1], val[N1];
#pragma unroll
  for (int m = 0; m < N1; ++m) x[m] = r[m] = val[m] = 0.0;
  if (act) {
    const int l[3] = {e % tile.V[0], (e / tile.V[0]) % tile.V[1], e / (tile.V[0] * tile.V[1])};
    gl = (((size_t)(tile.o[2] + l[2]) * a.n[1] + (tile.o[1] + l[1])) * a.n[0] + (tile.o[0] + l[0])) * NPE +
         (size_t)lam * N1;
#pragma unroll
    for (int m = 0; m < N1; ++m) s_p[e * ES + E::xline(lam) + m] = x[m] = xval(gl + m);
  }
  __syncthreads();  // s_hel
  for (int v = tid; v < NH * NPE; v += nth) {
    const int s = v / NPE, q = v - s * NPE;
    s_p[(TE + s) * ES + E::node(q)] = xval((size_t)s_hel[s] * NPE + q);
  }
  __syncthreads();

  // r = b - A x; sums r, r^2, b^2, (start: A u, (A u)^2), K_j . r
  double v[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = 0.0;
  res_cross_passes<double, DIM, N1, 1>(a.c, a.s, s_w, s_p, s_o, s_nb, TE);
  __syncthreads();
  if (act) {
    res_x_line<double, DIM, N1>(a.c, a.s[0], a.cmass, s_w, s_p, s_o, s_nb, TE, e, lam, xc, val);
#pragma unroll
    for (int m = 0; m < N1; ++m) {
      const double bi = a.b[gl + m];
      r[m] = bi - val[m];
      v[0] += r[m];
      v[1] = fma(r[m], r[m], v[1]);
      v[2] = fma(bi, bi, v[2]);
    }
#pragma unroll
    for (int j = 0; j < kResidMaxKd; ++j) {
      if (j >= a.kd) break;
#pragma unroll
      for (int m = 0; m < N1; ++m) v[5 + j] = fma(s_kb[j * NPE + lam * N1 + m], r[m], v[5 + j]);
    }
  }
  if (start) {
    // residual floor: the operator on a perturbation of the size of x's rounding
    __syncthreads();
    if (act) {
#pragma unroll
      for (int m = 0; m < N1; ++m) s_p[e * ES + E::xline(lam) + m] = resid_perturb(x[m], gl + m);
    }
    for (int q0 = tid; q0 < NH * NPE; q0 += nth) {
      const int s = q0 / NPE, q = q0 - s * NPE;
      double* t = s_p + (TE + s) * ES + E::node(q);
      *t = resid_perturb(*t, (unsigned long long)s_hel[s] * NPE + q);
    }
    __syncthreads();
    res_cross_passes<double, DIM, N1, 1>(a.c, a.s, s_w, s_p, s_o, s_nb, TE);
    __syncthreads();
    if (act) {
      res_x_line<double, DIM, N1>(a.c, a.s[0], a.cmass, s_w, s_p, s_o, s_nb, TE, e, lam, xc, val);
#pragma unroll
      for (int m = 0; m < N1; ++m) {
        v[3] += val[m];
        v[4] = fma(val[m], val[m], v[4]);
      }
    }
  }
  // a CTA whose wait ran out posts nothing more and writes no vector
  auto give_up = [&] {
    if (tid == 0) st->wait_failed = 1;
  };
  unsigned long long* const slot1 = a.slots + (size_t)a.nslot * 32;  // the other parity's words
  if (!resid_exchange(v, a.slots, a.tag, a.polls, s_red, s_sum, &s_fail)) return give_up();
  const double ndof = a.ncell * (double)NPE;
  const double bb = s_sum[2], uu0 = s_sum[4], us = s_sum[3];
  double ss = s_sum[1];
  if (a.kd > 0) {
    // the part in the kernel of the operator (round-off of b and of A x) goes
    if (act) {
#pragma unroll
      for (int j = 0; j < kResidMaxKd; ++j) {
        if (j >= a.kd) break;
        const double cj = s_sum[5 + j] * a.inv_ncell;
#pragma unroll
        for (int m = 0; m < N1; ++m) r[m] = fma(-cj, s_kb[j * NPE + lam * N1 + m], r[m]);
      }
    }
    __syncthreads();  // s_sum is read
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = 0.0;
#pragma unroll
    for (int m = 0; m < N1; ++m) v[0] = fma(r[m], r[m], v[0]);
    if (!resid_exchange(v, slot1, a.tag + 1, a.polls, s_red, s_sum, &s_fail)) return give_up();
    ss = s_sum[0];
  }

  // ---- decisions, by one warp (FP64 divisions are slow), the same in every CTA ----
  if (tid < 32) {
    const double sg = !start ? sigma0 : (!f32 || !(bb > 0.0)) ? 1.0 : 1.0 / sqrt(bb);
    const double rr = ss * sg * sg;
    double tol2 = start ? a.rtol * a.rtol * bb * sg * sg : st->tol2;
    int done = bb == 0.0 || rr <= tol2, status = seg_status, floored = 0;
    double floor_res = 0.0;
    if (start && !done) {
      const double mean = a.kd > 0 ? us / ndof : 0.0;
      double uu = uu0 - ndof * mean * mean;
      if (uu < 0.0) uu = 0.0;
      floor_res = bb > 0.0 ? sqrt(uu / bb) : 0.0;
      floored = 1;
      if (3.0 * floor_res > a.rtol) {
        tol2 = 9.0 * floor_res * floor_res * bb * sg * sg;
        done = rr <= tol2;
      }
    }
    if (!isfinite(rr)) {
      done = 1;
      status = SDG_ERR_BREAKDOWN;
    }
    if (tid == 0) {
      s_dd[0] = sg;
      s_dd[1] = rr;
      s_dd[2] = tol2;
      s_dd[3] = floor_res;
      s_di[0] = done;
      s_di[1] = status;
      s_di[2] = floored;
      // a converged singular solve gives x the kernel part of the start vector back
      s_di[3] = a.kd > 0 && done && !start && !seg_done && status == SDG_OK;
    }
  }
  __syncthreads();
  const double sigma = s_dd[0];
  const bool restore = s_di[3];
  if (restore) {
    __syncthreads();  // s_sum is read
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = 0.0;
    if (act) {
#pragma unroll
      for (int m = 0; m < N1; ++m) {
        const double d = x[m] - a.x0[gl + m];
#pragma unroll
        for (int j = 0; j < kResidMaxKd; ++j)
          if (j < a.kd) v[5 + j] = fma(s_kb[j * NPE + lam * N1 + m], d, v[5 + j]);
      }
    }
    if (!resid_exchange(v, a.slots, a.tag + 2, a.polls, s_red, s_sum, &s_fail)) return give_up();
    if (act) {
#pragma unroll
      for (int j = 0; j < kResidMaxKd; ++j) {
        if (j >= a.kd) break;
        const double cj = s_sum[5 + j] * a.inv_ncell;
#pragma unroll
        for (int m = 0; m < N1; ++m) x[m] = fma(-cj, s_kb[j * NPE + lam * N1 + m], x[m]);
      }
    }
  }
  if (act) {
#pragma unroll
    for (int m = 0; m < N1; ++m) {
      if (start) {
        if (a.kd > 0) a.x0[gl + m] = x[m];
        if (f32) a.x32[gl + m] = 0.0f;
      } else {
        if (f32 || pend || restore) a.x[gl + m] = x[m];
        if (f32) a.x32[gl + m] = 0.0f;
      }
      if (f32) a.r32[cur][gl + m] = (float)(r[m] * sigma);
      else a.r[cur][gl + m] = r[m];
    }
  }
  if (blockIdx.x == 0 && tid == 0) {
    if (start) {
      st->bnorm2 = bb;
      st->sigma = sigma;
      st->inv_sigma = 1.0 / sigma;
      st->iter = 0;
      st->maxit = a.maxit;
      st->updates = 0;
      st->reliable = 1;
      st->delta2 = a.delta * a.delta;
      st->alpha = 0.0;
      st->pAp = 0.0;
      st->xpend = 0;
      st->rr_old = s_dd[1];
      st->red[0] = s_dd[3];
      st->red[1] = (double)s_di[2];
    } else {
      st->updates += 1;
    }
    st->rr = s_dd[1];
    st->maxrr = s_dd[1];
    st->tol2 = s_dd[2];
    st->pause = 0;
    st->done = s_di[0];
    st->status = s_di[1];
    st->seg_done = seg_done;
    st->seg_status = seg_status;
    st->restored = restore;
  }
}

template <int DIM, int N1>
cudaError_t launch_resid_t(const sdg_handle* h, const ResPlan& pl, const ResidArgs& in, cudaStream_t stream) {
  ResidParams<DIM, N1> p;
  ApplyParams<double, DIM, N1> q;
  ApplyArgs<double> aa{};
  for (int d = 0; d < 3; ++d) aa.s[d] = in.s[d];
  aa.cmass = in.cmass;
  fill_apply_params<double, DIM, N1>(h, aa, &q);
  p.c = q.c;
  for (int i = 0; i < N1; ++i) p.w[i] = q.w[i];
  p.cmass = q.cmass;
  for (int d = 0; d < 3; ++d) {
    p.s[d] = q.s[d];
    p.n[d] = q.n[d];
    p.ts[d] = pl.ts[d];
    p.nt[d] = pl.nt[d];
  }
  p.b = in.b;
  p.x = in.x;
  p.x0 = in.x0;
  p.x32 = in.x32;
  for (int k = 0; k < 2; ++k) {
    p.r[k] = in.r[k];
    p.r32[k] = in.r32[k];
    p.p[k] = in.p[k];
    p.p32[k] = in.p32[k];
  }
  p.kb = h->kbasis;
  p.kd = in.project ? h->kd : 0;
  p.ncell = (double)h->g.ncell;
  p.inv_ncell = 1.0 / (double)h->g.ncell;
  p.st = in.st;
  p.slots = h->res_slots + (size_t)2 * h->res_ctas * 8;
  p.nslot = h->res_ctas;
  p.tag = in.tag;
  p.polls = h->polls;
  p.start = in.start;
  p.rtol = in.rtol;
  p.delta = in.delta;
  p.maxit = in.maxit;
  static PerDevice attr_set;
  return launch_coop(k_cg_resid<DIM, N1>, p, h, pl, &attr_set, stream);
}

}  // namespace sdg
