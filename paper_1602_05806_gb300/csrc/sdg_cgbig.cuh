// Resident conjugate gradients for 2D FP32 grids with many lines per thread:
// the scheme of sdg_cgres.cuh (one cooperative launch, one exchange of tagged
// words per iteration) with the vectors placed so that up to 28672 nodes fit
// an SM (256 x 256 cells at N = 7 on 152 SMs).
//
// What bounds the two-launch iteration at this size is instruction issue and
// the trips of r, p, Ap and x between L2 and the SMs (36 B/DOF; 30 us operator
// + 11 us update at 256 x 256, N = 7).  Here
//   p   stays in shared memory (with the face halo, which its owners publish
//       as they form it and which is fetched behind the first interior lines),
//   r   in registers, by x-lines,
//   Ap  in registers for the first AR rounds of lines and in shared memory for
//       the rest (at 256 x 256, N = 7 both are full: 225 KB, 255 registers),
//   x   in global memory: read and written once per iteration, 8 B/DOF.
// A warp works on whole elements, 32 / N1 at a time with a line per lane, and
// a thread on two rounds of them at once, a line of each in one P2; the two
// passes of an element exchange its values inside the warp, in the element's
// place of the Ap store, with no block barrier.
//
// Measured, us per iteration of the mixed solver, two launches -> here: 39.2
// -> 25.6 (256 x 256, N = 7), 47.3 -> 30.9 (256 x 256, N = 6), 30.2 -> 19.9
// (256 x 256, N = 5), 18.8 -> 9.4 (256 x 256, N = 3), 41.8 -> 25.8 (128 x 128,
// N = 11).  Cycles of the first, its sums still plain along a line (52000):
// update 14400 (of which x 5800), passes 27000, halo 4700, sums, exchange and
// decisions 6500.  512 threads with one line at a time took 1.5 us more, a
// scalar form with 256 threads twice as long.
#pragma once

#include "sdg_cgres.cuh"
#include "sdg_el2.cuh"

namespace sdg {

template <int N1>
struct BigEl : El2<N1> {
  static constexpr int NT = kBigThreads, AR = kBigRegRounds, ROUNDS = big_rounds(N1);
  static constexpr int EPW = 32 / N1;       // elements of a warp
  static constexpr int EPR = NT / 32 * EPW;  // elements of a round
};

// Two words of consecutive nodes.
__device__ __forceinline__ void big_publish2(unsigned long long* w, float a, float b, unsigned tag) {
  res_store_words(w, __float_as_uint(a), __float_as_uint(b), tag);
}

// Fetch the neighbours' p of this exchange into the halo slots: all loads of
// a thread in flight together (by fours they took 9800 of 70000 cycles).
template <int N1>
__device__ __forceinline__ bool big_fetch_halo(float* s_p, const int* s_hel, int TE, int NH,
                                               const unsigned long long* hw, unsigned tag, int limit) {
  using B = BigEl<N1>;
  constexpr int NPE = N1 * N1, NT = B::NT, W = NPE % 2 == 0 ? 2 : 1, HB = 12;
  const int nv = NH * (NPE / W);
  bool fail = false;
  for (int v0 = threadIdx.x; v0 < nv && !fail; v0 += HB * NT) {
    unsigned long long w0[HB], w1[HB];
    bool ok;
    int polls = 0;
    do {
      ok = true;
#pragma unroll
      for (int u = 0; u < HB; ++u) {
        const int v = v0 + u * NT, s = v / (NPE / W);
        w0[u] = w1[u] = (unsigned long long)tag << 32;
        if (v >= nv) continue;
        const unsigned long long* at = hw + ((unsigned)s_hel[s] * (unsigned)NPE + (unsigned)((v - s * (NPE / W)) * W));
        if constexpr (W == 2) res_load_words(at, w0[u], w1[u]);
        else asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(w0[u]) : "l"(at) : "memory");
      }
#pragma unroll
      for (int u = 0; u < HB; ++u) ok = ok && (unsigned)(w0[u] >> 32) == tag && (unsigned)(w1[u] >> 32) == tag;
    } while (!ok && ++polls < limit);
    fail = !ok;
#pragma unroll
    for (int u = 0; u < HB; ++u) {
      const int v = v0 + u * NT, s = v / (NPE / W);
      if (v >= nv) continue;
      const int q = (v - s * (NPE / W)) * W, k = q / N1, l = q - k * N1;
      float* to = s_p + B::node(TE + s, k, l);
      to[0] = __uint_as_float((unsigned)w0[u]);
      if constexpr (W == 2) {
        const int k1 = (q + 1) / N1;
        s_p[B::node(TE + s, k1, q + 1 - k1 * N1)] = __uint_as_float((unsigned)w1[u]);
      }
    }
  }
  return !fail;
}

template <int N1>
struct BigParams : ResParams<float, 2, N1> {
  Coef<C2, N1> c2;
};

template <int N1>
__global__ void __launch_bounds__(kBigThreads, 1) k_cg_big(const __grid_constant__ BigParams<N1> a) {
  using B = BigEl<N1>;
  using TA = ResAcc<float>;
  constexpr int NPE = N1 * N1, NT = B::NT, R = B::ROUNDS, AR = B::AR, EPR = B::EPR;
  SolverState* st = a.st;
  if (st->done || st->pause) return;  // uniform over the grid

  const ResTile<2> tile(a.n, a.ts, a.nt);
  const int TE = tile.TE, NH = tile.NH;
  extern __shared__ __align__(256) unsigned char smem_raw[];
  float* s_p = reinterpret_cast<float*>(smem_raw);   // (TE + NH) ES
  float* s_ap = s_p + (size_t)(TE + NH) * B::ES;     // Ap of the rounds from AR on; at least two rounds
  const int apn = TE > (AR + 2) * EPR ? TE - AR * EPR : 2 * EPR;
  // per element in order of processing (those that read the halo last): its
  // slot, its x and y neighbours' slots (16 bits each), its global element
  // with bit 31 set when a neighbouring CTA reads it
  // (on a 16-byte boundary: an odd number of elements of 360 bytes is not)
  int4* s_tab = reinterpret_cast<int4*>(smem_raw + (((size_t)(TE + NH + apn) * B::ES * 4 + 15) & ~size_t(15)));
  int* s_hel = reinterpret_cast<int*>(s_tab + TE);   // NH
  __shared__ float s_w[N1];
  __shared__ F2 s_red[16][4];
  __shared__ F2 s_tot[8][4];
  __shared__ float s_ab[2];
  __shared__ int s_flow, s_fail;
  __shared__ ResLoop<float> s_lp;

  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int eidx = lane / N1, lam = lane - eidx * N1;
  const bool on = eidx < B::EPW;
  if (tid < N1) s_w[tid] = a.w[tid];
  if (tid == 0) s_fail = 0;
  const int ax = a.nt[0] > 1, ay = a.nt[1] > 1;
  const int VX = tile.V[0], VY = tile.V[1];
  const int IW = max(VX - 2 * ax, 0), IH = max(VY - 2 * ay, 0), NI = IW * IH;
  for (int e = tid; e < TE; e += NT) {
    const int ex = e % VX, ey = e / VX;
    int xl = e - 1, xr = e + 1, yl = e - VX, yr = e + VX;
    if (ex == 0) xl = ax ? TE + ey : e + VX - 1;
    if (ex == VX - 1) xr = ax ? TE + VY + ey : e - (VX - 1);
    if (ey == 0) yl = ay ? TE + tile.hoff[1] + ex : e + (VY - 1) * VX;
    if (ey == VY - 1) yr = ay ? TE + tile.hoff[1] + VX + ex : e - (VY - 1) * VX;
    // interior elements before e in row order
    const int full = min(max(ey - ay, 0), IH);
    const bool row_in = ey >= ay && ey < ay + IH;
    const int before = full * IW + (row_in ? min(max(ex - ax, 0), IW) : 0);
    const bool inner = row_in && ex >= ax && ex < ax + IW;
    const unsigned ge = (unsigned)((tile.o[1] + ey) * a.n[0] + tile.o[0] + ex);
    s_tab[inner ? before : NI + e - before] =
        make_int4(e, xl | (xr << 16), yl | (yr << 16), (int)(ge | (inner ? 0u : 0x80000000u)));
  }
  for (int s = tid; s < NH; s += NT) {
    int gx, gy;
    if (s < tile.hoff[1]) {  // x faces
      gx = s < VY ? tile.o[0] - 1 : tile.o[0] + VX;
      gy = tile.o[1] + (s < VY ? s : s - VY);
    } else {
      const int t = s - tile.hoff[1];
      gx = tile.o[0] + (t < VX ? t : t - VX);
      gy = t < VX ? tile.o[1] - 1 : tile.o[1] + VY;
    }
    gx = gx < 0 ? gx + a.n[0] : (gx >= a.n[0] ? gx - a.n[0] : gx);
    gy = gy < 0 ? gy + a.n[1] : (gy >= a.n[1] ? gy - a.n[1] : gy);
    s_hel[s] = gy * a.n[0] + gx;
  }
  __syncthreads();

  const int it0 = st->iter;
  const bool fresh = it0 == 0;
  const int b0 = it0 & 1;
  float r[R][N1], apr[AR][N1];
  // the table row of a round's element (x < 0: none); its line's first node in global memory
  auto elem = [&](int j) -> int4 {
    int w = wid;
    asm volatile("" : "+r"(w));
    const int pos = (j * (NT / 32) + w) * B::EPW + eidx;
    return on && pos < TE ? s_tab[pos] : make_int4(-1, 0, 0, 0);
  };
  auto gnode = [&](int4 t) -> unsigned { return (unsigned)(t.w & 0x7fffffff) * (unsigned)NPE + (unsigned)(lam * N1); };
  // place of a round's element in the Ap store (rounds in registers pass
  // their y parts through the first round's places)
  const int ap0 = wid * B::EPW + eidx;
  auto aplace = [&](int j) -> int {
    int p = ap0;
    asm volatile("" : "+r"(p));  // not worth a register per round and row
    return (j < AR ? j & 1 : j - AR) * EPR + p;
  };
#pragma unroll
  for (int j = 0; j < R; ++j) {
    const int4 t = elem(j);
#pragma unroll
    for (int m = 0; m < N1; ++m) r[j][m] = 0.0f;
    if (j < AR) {
#pragma unroll
      for (int m = 0; m < N1; ++m) apr[j][m] = 0.0f;
    }
    if (t.x < 0) continue;
    const unsigned g = gnode(t);
    float pv[N1], av[N1];
#pragma unroll
    for (int m = 0; m < N1; ++m) {
      r[j][m] = a.r[b0][g + m];
      pv[m] = fresh ? 0.0f : a.p[b0][g + m];
      av[m] = fresh ? 0.0f : a.ap[b0][g + m];
    }
    B::store_row(s_p, t.x, lam, pv);
    if (j < AR) {
#pragma unroll
      for (int m = 0; m < N1; ++m) apr[j][m] = av[m];
    } else {
      B::store_row(s_ap, aplace(j), lam, av);
    }
  }
  // (a thread updates the rows it loaded itself: no barrier needed here)

  float alpha = fresh ? 0.0f : st->alpha_f;
  float beta = fresh ? 0.0f : st->beta_f;
  // (warp 0's recursion waits in shared memory between the decisions: registers are full)
  if (tid == 0) s_lp.init(st, a.delta2, a.cap);

  for (int k = 0;; ++k) {
    const unsigned tag = a.tag + (unsigned)k;
    unsigned long long* hw = a.halo + (size_t)(k & 1) * a.ndof;
    // sums: compensated term by term along a line, float pairs across lines
    F2 s_pa{0.0f, 0.0f}, s_rr{0.0f, 0.0f}, s_ra{0.0f, 0.0f}, s_aa{0.0f, 0.0f};

    // ---- r -= alpha Ap, x += alpha p, p = r + beta p; r.r; boundary lines
    // first, their p published at once ----
    // (two rounds per turn of a loop, the next turn's x loaded ahead: one round
    // at a time, each load behind the last round's store, their latencies add up)
    const int nr = (TE + EPR - 1) / EPR;
    auto load_x = [&](int j, float (&xv)[2][N1], int (&slot)[2], unsigned (&g)[2]) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int4 t = elem(j + u);
        slot[u] = t.x < 0 ? -1 : t.x | (t.w < 0 ? 0x10000 : 0);
        g[u] = gnode(t);
        if (t.x < 0) continue;
        if constexpr (N1 % 4 == 0) {
#pragma unroll
          for (int m = 0; m < N1; m += 4) {
            const float4 q = *reinterpret_cast<const float4*>(a.x + g[u] + m);
            xv[u][m] = q.x; xv[u][m + 1] = q.y; xv[u][m + 2] = q.z; xv[u][m + 3] = q.w;
          }
        } else {
#pragma unroll
          for (int m = 0; m < N1; ++m) xv[u][m] = __ldcg(a.x + g[u] + m);
        }
      }
    };
    float xn[2][N1];
    int sn[2];
    unsigned gn[2];
    load_x((nr - 1) & ~1, xn, sn, gn);
#pragma unroll 1
    for (int j = (nr - 1) & ~1; j >= 0; j -= 2) {
      float xv[2][N1];
      int slot[2];
      unsigned g[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
#pragma unroll
        for (int m = 0; m < N1; ++m) xv[u][m] = xn[u][m];
        slot[u] = sn[u];
        g[u] = gn[u];
      }
      if (j >= 2) load_x(j - 2, xn, sn, gn);
      float av[2][N1];
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (j >= AR) B::load_row(s_ap, slot[u] >= 0 ? aplace(j + u) : 0, lam, av[u]);
      // r of the two rounds (av: r's new values from here on)
#pragma unroll
      for (int q = 0; q < R; q += 2) {
        if (j != q) continue;
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int m = 0; m < N1; ++m) {
            const float ap = q < AR ? apr[q < AR ? q + u : 0][m] : av[u][m];
            r[q + u][m] = fmaf(-alpha, ap, r[q + u][m]);
            av[u][m] = r[q + u][m];
          }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        if (slot[u] < 0) continue;
        const int e = slot[u] & 0xffff;
        float po[N1];
        B::load_row(s_p, e, lam, po);
        KDot<float> rr;
#pragma unroll
        for (int m = 0; m < N1; ++m) {
          xv[u][m] = fmaf(alpha, po[m], xv[u][m]);
          po[m] = fmaf(beta, po[m], av[u][m]);
          rr.add(av[u][m], av[u][m]);
        }
        s_rr = f2_add(s_rr, pair(rr));
        B::store_row(s_p, e, lam, po);
        if (slot[u] & 0x10000) {
          if constexpr (N1 % 2 == 0) {
#pragma unroll
            for (int m = 0; m < N1; m += 2) big_publish2(hw + g[u] + m, po[m], po[m + 1], tag);
          } else {
#pragma unroll
            for (int m = 0; m < N1; ++m) res_publish(hw, (long long)g[u] + m, po[m], tag);
          }
        }
        if constexpr (N1 % 4 == 0) {
#pragma unroll
          for (int m = 0; m < N1; m += 4)
            __stcg(reinterpret_cast<float4*>(a.x + g[u] + m),
                   make_float4(xv[u][m], xv[u][m + 1], xv[u][m + 2], xv[u][m + 3]));
        } else {
#pragma unroll
          for (int m = 0; m < N1; ++m) __stcg(a.x + g[u] + m, xv[u][m]);
        }
      }
    }
    __syncthreads();
    // the last turn of the loop below before one that reads the halo
    const bool early = NI < 2 * EPR;
    const int jf = early ? -1 : (NI / (2 * EPR) - 1) * 2;
    if (NH > 0 && early) {
      if (!big_fetch_halo<N1>(s_p, s_hel, TE, NH, hw, tag, a.polls)) s_fail = st->wait_failed = 1;
      __syncthreads();
    }

    // ---- Ap, two rounds at a time: a line of each in one P2.  A loop, not
    // unrolled (the registers of a round are reached through a switch) ----
#pragma unroll 1
    for (int j = 0; j < nr; j += 2) {
      const int4 t0 = elem(j);
      int4 t1 = j + 1 < nr ? elem(j + 1) : make_int4(-1, 0, 0, 0);
      const bool two = t1.x >= 0;
      if (!two) t1 = t0;  // computed twice, counted once
      const int pl0 = aplace(j), pl1 = two ? aplace(j + 1) : pl0;
      const float wl = s_w[lam];
      if (t0.x >= 0) {  // y pass: column lam
        P2 xl[N1], xc[N1], xr[N1], val[N1];
        B::load_cols(s_p, B::col(t0.z & 0xffff, lam), B::col(t1.z & 0xffff, lam), xl);
        B::load_cols(s_p, B::col(t0.x, lam), B::col(t1.x, lam), xc);
        B::load_cols(s_p, B::col((unsigned)t0.z >> 16, lam), B::col((unsigned)t1.z >> 16, lam), xr);
        line_apply<P2, N1, true>(a.c2, xl, xc, xr, P2(a.s[1] * wl), val);
        B::store_cols(s_ap, B::col(pl0, lam), B::col(pl1, lam), val);
      }
      __syncwarp();
      if (t0.x >= 0) {  // x pass: row lam
        P2 xl[N1], xc[N1], xr[N1], val[N1], po[N1];
        B::load_rows(s_p, t0.y & 0xffff, t1.y & 0xffff, lam, xl);
        B::load_rows(s_p, t0.x, t1.x, lam, xc);
        B::load_rows(s_p, (unsigned)t0.y >> 16, (unsigned)t1.y >> 16, lam, xr);
        line_apply<P2, N1, true>(a.c2, xl, xc, xr, P2(a.s[0] * wl), val);
        asm volatile("" ::: "memory");  // p again rather than held through the contraction
        B::load_rows(s_p, t0.x, t1.x, lam, xc);
        B::load_rows(s_ap, pl0, pl1, lam, po);
        if (a.cmass != 0.0f) {
#pragma unroll
          for (int m = 0; m < N1; ++m) val[m] = fma(a.cmass * wl * s_w[m], xc[m], val[m]);
        }
        KDot<P2> pa, ra, aa;
#pragma unroll
        for (int m = 0; m < N1; ++m) {
          val[m] = val[m] + po[m];
          pa.add(xc[m], val[m]);
          aa.add(val[m], val[m]);
        }
#pragma unroll
        for (int q = 0; q < R; q += 2) {
          if (j != q) continue;
#pragma unroll
          for (int m = 0; m < N1; ++m) ra.add(P2(r[q][m], r[q + 1][m]), val[m]);
          if (q < AR) {
#pragma unroll
            for (int m = 0; m < N1; ++m) {
              apr[q < AR ? q : 0][m] = val[m].lo();
              apr[q < AR ? q + 1 : 0][m] = val[m].hi();
            }
          }
        }
        s_pa = f2_add(s_pa, pair_lo(pa));
        s_ra = f2_add(s_ra, pair_lo(ra));
        s_aa = f2_add(s_aa, pair_lo(aa));
        if (two) {
          s_pa = f2_add(s_pa, pair_hi(pa));
          s_ra = f2_add(s_ra, pair_hi(ra));
          s_aa = f2_add(s_aa, pair_hi(aa));
        }
        if (j >= AR) B::store_rows(s_ap, pl0, pl1, lam, val);
      }
      __syncwarp();  // the next rounds may use the same places
      if (j == jf && NH > 0) {
        if (!big_fetch_halo<N1>(s_p, s_hel, TE, NH, hw, tag, a.polls)) s_fail = st->wait_failed = 1;
        __syncthreads();
      }
    }

    // ---- sums, alpha, beta, decisions ----
    F2 v4[4] = {s_pa, s_rr, s_ra, s_aa};
    unsigned long long* slot = a.slots + (size_t)(k & 1) * a.nslot * 8;
    // (sums formed with an old halo are not posted; s_fail is the same for all
    // threads here, the fetch being behind a barrier)
    if (!s_fail) {
      res_post_sums<float>(v4, slot, tag, s_red, s_tot);
      if (!res_poll_sums<float>(slot, tag, a.polls, s_tot)) s_fail = st->wait_failed = 1;
    }
    __syncthreads();
    if (wid == 0) {
      ResLoop<float> lp = s_lp;
      ++lp.it;
      lp.decide(s_tot, s_fail, s_ab, &s_flow);
      __syncwarp();
      if (lane == 0) s_lp = lp;
    }
    __syncthreads();
    alpha = s_ab[0];
    beta = s_ab[1];
    if (s_flow) break;
  }

  // ---- leave r, p, Ap of the last iteration (x is without its step) ----
  const int b1 = s_lp.it & 1;
#pragma unroll
  for (int j = 0; j < R; ++j) {
    const int4 t = elem(j);
    if (t.x < 0) continue;
    const unsigned g = gnode(t);
    float pv[N1], av[N1];
    B::load_row(s_p, t.x, lam, pv);
    if (j >= AR) B::load_row(s_ap, aplace(j), lam, av);
#pragma unroll
    for (int m = 0; m < N1; ++m) {
      a.r[b1][g + m] = r[j][m];
      a.p[b1][g + m] = pv[m];
      a.ap[b1][g + m] = j < AR ? apr[j < AR ? j : 0][m] : av[m];
    }
  }
  if (blockIdx.x == 0 && tid == 0) s_lp.store(st, a.delta2);
}

template <int N1>
cudaError_t launch_big(const sdg_handle* h, const ResPlan& pl, const ResArgs<float>& in, cudaStream_t stream) {
  BigParams<N1> p;
  fill_res_params<float, 2, N1>(h, pl, in, &p);
  dup_coef(p.c, &p.c2);
  static PerDevice attr_set;
  return launch_coop(k_cg_big<N1>, p, h, pl, &attr_set, stream);
}

}  // namespace sdg
