// Line-wise kernels of the step's stages (Sec. 2.2, 2.3): one thread per
// (element, line along d), every length a compile-time constant, the 1D
// matrices in the kernel-parameter bank.
//
// All of these are bound by the FP64 pipe (two lanes per SM and clock on
// GB300), so what counts is FP64 instructions per node.  The Gauss-Legendre
// nodes are symmetric, which halves the contractions:
//   * pair transforms y = K a + s (J K J) b  (J: reversal of a line; the L2
//     projections with s = 1: M^L = J M^R J; weak gradient and divergence
//     with s = -1: L~ = J R~ J, L-bar = J R-bar J) become, with c = J b,
//       y + J y = (K + J K)(a + s c) ,   y - J y = (K - J K)(a - s c) :
//     n^2 instead of 2 n^2 multiply-adds per line.  (Not the divergence: its
//     terms cancel to 1e-6 and less, and the sums and differences of a and c
//     are two more roundings of each: 3.6e-11 of a right-hand side on 48^3
//     cells, N = 4, against 1.9e-11 term by term, for 0.2 of 4.9 ms.  And not
//     for n = 2, where those two roundings count: errors against extended
//     precision 1.2 to 1.5 times those of the term by term form in the
//     projections and 1.0 to 1.4 times in the velocity update's gradient,
//     against 0.5 to 1.1 times for n >= 3, where on the mean over degrees,
//     rough and smooth data they are 0.94 and 0.86 times as large);
//   * the volume term of the convection, an anti-centrosymmetric matrix,
//     splits into two blocks of (n/2)^2.
#pragma once

#include <algorithm>
#include <type_traits>

#include "sdg_device.cuh"

namespace sdg {

// Where a thread's line lies: element, its neighbour along the line, offsets.
struct LineGeo {
  int n[3];
  int d;       // direction of the line
  int st;      // node stride along the line
  unsigned nlines;
};

// K + J K (rows m < (n+1)/2; the middle row counts once) and K - J K (rows
// m < n/2), halved, so that y_m = e + o, y_{n-1-m} = e - o
template <int N1>
struct PairMat {
  static constexpr int H = N1 / 2, HE = (N1 + 1) / 2, HO = H > 0 ? H : 1;
  double E[HE * N1], O[HO * N1];
  void fill(const double* K) {
    for (int m = 0; m < HE; ++m)
      for (int q = 0; q < N1; ++q)
        E[m * N1 + q] = 2 * m == N1 - 1 ? K[m * N1 + q] : 0.5 * (K[m * N1 + q] + K[(N1 - 1 - m) * N1 + q]);
    for (int m = 0; m < H; ++m)
      for (int q = 0; q < N1; ++q) O[m * N1 + q] = 0.5 * (K[m * N1 + q] - K[(N1 - 1 - m) * N1 + q]);
  }
};

// y = K a + s (J K J) b
template <int N1, bool PLUS>
__device__ __forceinline__ void pair_apply(const PairMat<N1>& k, const double (&a)[N1], const double (&b)[N1],
                                           double (&y)[N1]) {
  constexpr int H = N1 / 2, HE = (N1 + 1) / 2;
  double e[N1], o[N1];
#pragma unroll
  for (int q = 0; q < N1; ++q) {
    const double c = b[N1 - 1 - q];
    e[q] = PLUS ? a[q] + c : a[q] - c;
    o[q] = PLUS ? a[q] - c : a[q] + c;
  }
  double yE[HE], yO[HE];
#pragma unroll
  for (int m = 0; m < HE; ++m) {
    double t = 0.0;
#pragma unroll
    for (int q = 0; q < N1; ++q) t = fma(k.E[m * N1 + q], e[q], t);
    yE[m] = t;
  }
#pragma unroll
  for (int m = 0; m < H; ++m) {
    double t = 0.0;
#pragma unroll
    for (int q = 0; q < N1; ++q) t = fma(k.O[m * N1 + q], o[q], t);
    yO[m] = t;
  }
#pragma unroll
  for (int m = 0; m < H; ++m) {
    y[m] = yE[m] + yO[m];
    y[N1 - 1 - m] = yE[m] - yO[m];
  }
  if constexpr (N1 % 2) y[H] = yE[H];  // row H of K a + s J K J b is K_H (a + s c)
}

// R and -s L themselves, for the term by term form.
template <int N1>
struct PairFull {
  double A[N1 * N1], B[N1 * N1];
  void fill(const double* R, const double* L, bool plus) {
    for (int i = 0; i < N1 * N1; ++i) {
      A[i] = R[i];
      B[i] = plus ? -L[i] : L[i];
    }
  }
};

// y = A a - B b
template <int N1>
__device__ __forceinline__ void full_apply(const PairFull<N1>& k, const double (&a)[N1], const double (&b)[N1],
                                           double (&y)[N1]) {
#pragma unroll
  for (int m = 0; m < N1; ++m) {
    double t = 0.0;
#pragma unroll
    for (int q = 0; q < N1; ++q) {
      t = fma(k.A[m * N1 + q], a[q], t);
      t = fma(-k.B[m * N1 + q], b[q], t);
    }
    y[m] = t;
  }
}

// the pair transform is formed term by term, for accuracy, for n = 2
constexpr bool pair_full(int n1) { return n1 == 2; }

template <int N1>
struct PairParams {
  typename std::conditional<pair_full(N1), PairFull<N1>, PairMat<N1>>::type k;
  double wi[N1];         // 1 / w (term by term)
  int n[3];
  unsigned nlines;
  int sa, sb;            // elements along d from which the line multiplied by R (K), by L (J K J) is read
  // MIX: both lines are of c1 x + c2 x2; read and mixed per direction rather
  // than once into a buffer, so that the call needs no scratch
  const double *x, *x2;
  double c1, c2;
  struct Dir {
    int d, st;           // direction, node stride along it
    const double* base;  // what the result is added to (null: nothing)
    double scale;
    double* out;
  } dir[3];              // by blockIdx.y
};

// out = base + scale (1 / w) (R a + s L b) along a direction, a and b lines of x
template <int DIM, int N1, bool PLUS, bool MIX>
__global__ void __launch_bounds__(256) k_pair_line(const __grid_constant__ PairParams<N1> p) {
  constexpr int LINES = DIM == 2 ? N1 : N1 * N1, NPE = LINES * N1;
  const auto& q = p.dir[blockIdx.y];
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= p.nlines) return;
  const unsigned el = t / LINES;
  const int lam = (int)(t - el * LINES);
  const int q0 = lam % N1, q1 = lam / N1;
  const int lb = DIM == 2 ? (q.d == 0 ? lam * N1 : lam)
                          : (q.d == 0 ? lam * N1 : q.d == 1 ? q0 + q1 * N1 * N1 : lam);
  // the neighbours along d
  const unsigned nx = p.n[0], ny = p.n[1];
  const unsigned ex = el % nx, ey = (el / nx) % ny;
  const int pos = q.d == 0 ? (int)ex : q.d == 1 ? (int)ey : (int)(el / (nx * ny));
  const long long str = q.d == 0 ? 1 : q.d == 1 ? (long long)nx : (long long)nx * ny;
  const int nd = p.n[q.d];
  auto nb = [&](int s) -> size_t {
    long long e = (long long)el + s * str;
    if (s < 0 && pos == 0) e += nd * str;
    if (s > 0 && pos == nd - 1) e -= nd * str;
    return (size_t)e * NPE + lb;
  };
  const size_t ia = nb(p.sa), ib = nb(p.sb);
  const size_t io = (size_t)el * NPE + lb;
  const int st = q.st;
  double a[N1], b[N1], y[N1];
#pragma unroll
  for (int k = 0; k < N1; ++k) {
    a[k] = p.x[ia + k * st];
    b[k] = p.x[ib + k * st];
    if (MIX) {
      a[k] = fma(p.c1, a[k], p.c2 * p.x2[ia + k * st]);
      b[k] = fma(p.c1, b[k], p.c2 * p.x2[ib + k * st]);
    }
  }
  if constexpr (pair_full(N1)) full_apply<N1>(p.k, a, b, y);
  else pair_apply<N1, PLUS>(p.k, a, b, y);
#pragma unroll
  for (int m = 0; m < N1; ++m) {
    const double f = pair_full(N1) ? q.scale * p.wi[m] : q.scale;
    q.out[io + m * st] = q.base ? fma(f, y[m], q.base[io + m * st]) : f * y[m];
  }
}

// ---- divergence -------------------------------------------------------------
// out = base + sum_d f_d M^{perp d} (R U_d[e] - L U_d[e-1]), and the sum of out
// into st->red[0].  A CTA takes runs of G elements and adds the directions up
// in shared memory (rows of N1 values padded to an odd length), so that base
// and out move once.  A launch per direction, with the sums through out, costs
// a launch latency each: right-hand side on 8 x 8 cells, N = 3, 29.7 instead of
// 24.7 us, on 64 x 64, N = 5, 43.6 instead of 37.0, on 48^3, N = 4, 2 % more.
template <int N1>
struct DivParams {
  PairFull<N1> k;
  double w[N1];
  int n[3];
  unsigned ncell;
  int G;
  const double* U[3];
  double f[3];
  const double* base;  // null: nothing
  double* out;
  SolverState* st;
  double* partials;
};

template <int DIM, int N1>
constexpr int div_group() {  // elements of a run at most
  constexpr int lines = DIM == 2 ? N1 : N1 * N1;
  return lines >= 256 ? 1 : 256 / lines;
}

template <int DIM, int N1>
__global__ void __launch_bounds__(256) k_div_line(const __grid_constant__ DivParams<N1> p) {
  constexpr int LINES = DIM == 2 ? N1 : N1 * N1, NPE = LINES * N1;
  constexpr int RS = N1 | 1, ES = LINES * RS;
  __shared__ double s_acc[div_group<DIM, N1>() * ES];
  __shared__ double s_w[N1];
  const int tid = threadIdx.x, nth = blockDim.x;
  if (tid < N1) s_w[tid] = p.w[tid];
  const int es = tid / LINES, lam = tid - es * LINES;
  const int q0 = lam % N1, q1 = lam / N1;
  auto at = [](int i) { return i / N1 * RS + i % N1; };  // place of value i of the run
  const unsigned nrun = (p.ncell + p.G - 1) / p.G;
  double sum = 0.0;
  for (unsigned run = blockIdx.x; run < nrun; run += gridDim.x) {
    const unsigned e0 = run * p.G;
    const int ne = min((unsigned)p.G, p.ncell - e0);
    const size_t g0 = (size_t)e0 * NPE;
    for (int i = tid; i < ne * NPE; i += nth) s_acc[at(i)] = p.base ? p.base[g0 + i] : 0.0;
    __syncthreads();
    const unsigned el = e0 + es;
    const unsigned nx = p.n[0], ny = p.n[1];
    const unsigned e[3] = {el % nx, (el / nx) % ny, el / (nx * ny)};
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
      if (es < ne) {
        constexpr int PS = LINES;  // node stride along z
        const int st = d == 0 ? 1 : d == 1 ? N1 : PS;
        const int lb = DIM == 2 ? (d == 0 ? lam * N1 : lam) : (d == 0 ? lam * N1 : d == 1 ? q0 + q1 * N1 * N1 : lam);
        const size_t str = d == 0 ? 1 : d == 1 ? (size_t)nx : (size_t)nx * ny;
        const size_t em = e[d] == 0 ? el + (p.n[d] - 1) * str : el - str;
        const double* U = p.U[d];
        const size_t ia = (size_t)el * NPE + lb, ib = em * NPE + lb;
        double a[N1], b[N1], y[N1];
#pragma unroll
        for (int k = 0; k < N1; ++k) {
          a[k] = U[ia + k * st];
          b[k] = U[ib + k * st];
        }
        full_apply<N1>(p.k, a, b, y);
        const double f = p.f[d] * (DIM == 2 ? s_w[lam] : s_w[q0] * s_w[q1]);
        // rows hold x-lines: a step along y is a row, along z N1 rows
        const int sst = d == 0 ? 1 : d == 1 ? RS : N1 * RS;
        double* s = s_acc + es * ES +
                    (d == 0 ? lam * RS : DIM == 2 ? lam : d == 1 ? q0 + q1 * N1 * RS : q0 + q1 * RS);
#pragma unroll
        for (int m = 0; m < N1; ++m) s[m * sst] = fma(f, y[m], s[m * sst]);
      }
      __syncthreads();
    }
    for (int i = tid; i < ne * NPE; i += nth) {
      const double v = s_acc[at(i)];
      p.out[g0 + i] = v;
      sum += v;
    }
    __syncthreads();
  }
  double v1[1] = {sum}, tot[1];
  if (grid_sum<1>(v1, p.partials, &p.st->counter, tot) && tid == 0) p.st->red[0] = tot[0];
}

// ---- convection -------------------------------------------------------------
// out_c = a V0_c + b (V_c + dt L_c), L the collocated Rusanov DG operator
//   L(q) = - sum_d (1/dx_d) M_d^-1 [phi(1) F^_{e+1/2} - phi(0) F^_{e-1/2} - Dn^T W (q v_d)]
// F^ = (q^- v^- + q^+ v^+)/2 - s (q^+ - q^-)/2,  s = 2 max(|v_d^-|, |v_d^+|).
// A launch per direction: the first writes L, the next add to it, the last
// forms the output.  A CTA takes a run of elements along d with one more at
// either end; every thread forms the two traces of its own line once and
// reads its neighbours' from shared memory.
template <int N1>
struct ConvMat {
  static constexpr int H = N1 / 2, HO = H > 0 ? H : 1, HE = (N1 + 1) / 2;
  // volume matrix D = (1/dx) M^-1 Dn^T W: e_m = P_m . f_O (the middle row
  // too), o_m = Q_m . f_E, where vol_m = e_m + o_m, vol_{n-1-m} = e_m - o_m
  double P[HE * HO], Q[HO * HE];
  double phi0[N1], phi1[N1];
  double we[HE], wo[HO];  // lifts (1/dx) M^-1 phi(0, 1): half sum, half difference
};

template <int DIM, int N1>
struct ConvParams {
  ConvMat<N1> c;
  LineGeo g;
  int run;           // elements per run
  int first, last;
  const double* V0[3];
  const double* V[3];
  double* L[3];
  double* out[3];
  double a, b, dt;
};

template <int DIM, int N1>
constexpr int conv_slots() {  // elements a CTA holds (a run and its two ends)
  constexpr int lines = DIM == 2 ? N1 : N1 * N1;
  return lines >= 128 ? 3 : (256 / lines > 34 ? 34 : 256 / lines < 3 ? 3 : 256 / lines);
}

template <int DIM, int N1>
__global__ void __launch_bounds__(conv_slots<DIM, N1>() * (DIM == 2 ? N1 : N1 * N1))
    k_conv_line(const __grid_constant__ ConvParams<DIM, N1> p) {
  constexpr int LINES = DIM == 2 ? N1 : N1 * N1, NPE = LINES * N1, S = conv_slots<DIM, N1>();
  constexpr int H = N1 / 2, HE = (N1 + 1) / 2, HO = H > 0 ? H : 1;
  constexpr bool MID = (N1 % 2) == 1;
  __shared__ double s_t[2][DIM][S * LINES];  // traces at xi = 0, 1
  const int d = p.g.d, st = p.g.st, nd = p.g.n[d];
  const int slot = threadIdx.x / LINES, lam = threadIdx.x - slot * LINES;
  // run of the CTA: first element along d, and the other coordinates
  const unsigned nrun = (nd + p.run - 1) / p.run;
  const unsigned rb = blockIdx.x % nrun;
  unsigned rest = blockIdx.x / nrun;
  int e[3] = {0, 0, 0};
  const int i0 = (int)rb * p.run, len = min(p.run, nd - i0);
  {
    const int da = d == 0 ? 1 : 0, db = DIM == 3 ? (d == 2 ? 1 : 2) : 2;
    e[da] = (int)(rest % (unsigned)p.g.n[da]);
    rest /= (unsigned)p.g.n[da];
    if (DIM == 3) e[db] = (int)rest;
  }
  const bool in = slot < len + 2;
  int pos = i0 + slot - 1;
  pos = pos < 0 ? pos + nd : (pos >= nd ? pos - nd : pos);
  e[d] = pos;
  const int q0 = lam % N1, q1 = lam / N1;
  const int lb = DIM == 2 ? (d == 0 ? lam * N1 : lam) : (d == 0 ? lam * N1 : d == 1 ? q0 + q1 * N1 * N1 : lam);
  const size_t io = (((size_t)e[2] * p.g.n[1] + e[1]) * p.g.n[0] + e[0]) * NPE + lb;

  // own lines and traces
  double q[DIM][N1];
#pragma unroll
  for (int c = 0; c < DIM; ++c) {
    double t0 = 0.0, t1 = 0.0;
#pragma unroll
    for (int m = 0; m < N1; ++m) {
      q[c][m] = in ? p.V[c][io + (size_t)m * st] : 0.0;
      t0 = fma(p.c.phi0[m], q[c][m], t0);
      t1 = fma(p.c.phi1[m], q[c][m], t1);
    }
    s_t[0][c][threadIdx.x] = t0;
    s_t[1][c][threadIdx.x] = t1;
  }
  __syncthreads();
  if (slot < 1 || slot > len) return;
  const int il = threadIdx.x - LINES, ic = threadIdx.x, ir = threadIdx.x + LINES;
  // normal velocity on both faces and its line
  double vd[N1];
  double vlm = 0.0, vlp = 0.0, vrm = 0.0, vrp = 0.0;
#pragma unroll
  for (int c = 0; c < DIM; ++c) {
    if (c != d) continue;
#pragma unroll
    for (int m = 0; m < N1; ++m) vd[m] = q[c][m];
    vlm = s_t[1][c][il];
    vlp = s_t[0][c][ic];
    vrm = s_t[1][c][ic];
    vrp = s_t[0][c][ir];
  }
  const double hl = fmax(fabs(vlm), fabs(vlp)), hr = fmax(fabs(vrm), fabs(vrp));  // s / 2
#pragma unroll
  for (int c = 0; c < DIM; ++c) {
    const double qlm = s_t[1][c][il], qlp = s_t[0][c][ic], qrm = s_t[1][c][ic], qrp = s_t[0][c][ir];
    const double fl = 0.5 * (qlm * vlm + qlp * vlp) - hl * (qlp - qlm);
    const double fr = 0.5 * (qrm * vrm + qrp * vrp) - hr * (qrp - qrm);
    const double fd = fr - fl, fs = fr + fl;
    // f = q v_d, split
    double fE[HE], fO[HO];
#pragma unroll
    for (int k = 0; k < H; ++k) {
      const double x0 = q[c][k] * vd[k], x1 = q[c][N1 - 1 - k] * vd[N1 - 1 - k];
      fE[k] = x0 + x1;
      fO[k] = x0 - x1;
    }
    if constexpr (MID) fE[H] = q[c][H] * vd[H];
    double L[N1];
#pragma unroll
    for (int m = 0; m < HE; ++m) {
      double ev = -p.c.we[m] * fd;
#pragma unroll
      for (int k = 0; k < H; ++k) ev = fma(p.c.P[m * HO + k], fO[k], ev);
      if (m < H) {
        double ov = -p.c.wo[m] * fs;
#pragma unroll
        for (int k = 0; k < HE; ++k) ov = fma(p.c.Q[m * HE + k], fE[k], ov);
        L[m] = ev + ov;
        L[N1 - 1 - m] = ev - ov;
      } else {
        L[m] = ev;
      }
    }
#pragma unroll
    for (int m = 0; m < N1; ++m) {
      const size_t i = io + (size_t)m * st;
      const double Lv = p.first ? L[m] : p.L[c][i] + L[m];
      if (p.last) {
        const double t = p.b * fma(p.dt, Lv, q[c][m]);
        p.out[c][i] = p.a != 0.0 ? fma(p.a, p.V0[c][i], t) : t;
      } else {
        p.L[c][i] = Lv;
      }
    }
  }
}

// ---- launchers --------------------------------------------------------------
inline LineGeo line_geo(const Geo& g, int d) {
  LineGeo q;
  for (int k = 0; k < 3; ++k) q.n[k] = g.n[k];
  q.d = d;
  q.st = d == 0 ? 1 : (d == 1 ? g.n1 : g.n1 * g.n1);
  q.nlines = (unsigned)(g.ndof / g.n1);
  return q;
}

template <int DIM, int N1>
cudaError_t launch_pair(const sdg_handle* h, const PairArgs& in, cudaStream_t s) {
  PairParams<N1> p;
  const double* w = h->basis.w;
  if constexpr (pair_full(N1)) {
    p.k.fill(in.R, in.L, in.plus);
  } else {
    // the mean of the two computed matrices (each carries the rounding of its
    // own quadrature), rows scaled by 1 / w
    double K[N1 * N1];
    for (int i = 0; i < N1 * N1; ++i) K[i] = 0.5 * (in.R[i] + in.L[N1 * N1 - 1 - i]) / w[i / N1];
    p.k.fill(K);
  }
  for (int i = 0; i < N1; ++i) p.wi[i] = 1.0 / w[i];
  for (int k = 0; k < 3; ++k) p.n[k] = h->g.n[k];
  p.nlines = (unsigned)(h->g.ndof / N1);
  p.sa = in.sa;
  p.sb = in.sb;
  p.x = in.x;
  p.x2 = in.x2;
  p.c1 = in.c1;
  p.c2 = in.c2;
  for (int k = 0; k < in.ndir; ++k) {
    const int d = in.dir[k].d;
    p.dir[k] = {d, line_geo(h->g, d).st, in.dir[k].base, in.dir[k].scale, in.dir[k].out};
  }
  // As many threads in a CTA as leave every SM one: on few lines the FP64 pipes
  // of a few SMs held whole CTAs of 256 while the others idled (projection on
  // 31 x 21 cells, N = 8: 12.3 us with 23 CTAs, 7.3 us with 184).
  const unsigned per_sm = (p.nlines * in.ndir + h->nsm - 1) / h->nsm;
  const unsigned threads = per_sm >= 256 ? 256 : (per_sm + 31) / 32 * 32;
  const dim3 grid((p.nlines + threads - 1) / threads, in.ndir);
  if (in.plus) k_pair_line<DIM, N1, true, false><<<grid, threads, 0, s>>>(p);
  else if (in.x2) k_pair_line<DIM, N1, false, true><<<grid, threads, 0, s>>>(p);
  else k_pair_line<DIM, N1, false, false><<<grid, threads, 0, s>>>(p);
  return cudaGetLastError();
}

template <int DIM, int N1>
cudaError_t launch_div(const sdg_handle* h, const DivArgs& in, cudaStream_t s) {
  constexpr int LINES = DIM == 2 ? N1 : N1 * N1, G = div_group<DIM, N1>();
  DivParams<N1> p;
  p.k.fill(h->basis.Rb, h->basis.Lb, false);
  for (int i = 0; i < N1; ++i) p.w[i] = h->basis.w[i];
  for (int k = 0; k < 3; ++k) {
    p.n[k] = h->g.n[k];
    p.U[k] = k < DIM ? in.U[k] : nullptr;
    p.f[k] = k < DIM ? in.scale / h->dx[k] : 0.0;
  }
  p.ncell = (unsigned)h->g.ncell;
  // (as for the pairs: no more elements in a run than leave every SM one)
  p.G = (int)std::min<long long>(G, (h->g.ncell + h->nsm - 1) / h->nsm);
  p.base = in.base;
  p.out = in.out;
  p.st = in.st;
  p.partials = in.partials;
  const long long runs = (h->g.ncell + p.G - 1) / p.G;
  const int threads = (p.G * LINES + 31) / 32 * 32;
  k_div_line<DIM, N1><<<(unsigned)std::min<long long>(runs, kReduceBlocks), threads, 0, s>>>(p);
  return cudaGetLastError();
}

template <int DIM, int N1>
cudaError_t launch_conv(const sdg_handle* h, const ConvArgs& in, cudaStream_t s) {
  constexpr int H = N1 / 2, HE = (N1 + 1) / 2, HO = H > 0 ? H : 1, LINES = DIM == 2 ? N1 : N1 * N1;
  constexpr int S = conv_slots<DIM, N1>();
  const Basis1D& B = h->basis;
  ConvParams<DIM, N1> p;
  p.c = ConvMat<N1>{};
  for (int d = 0; d < DIM; ++d) {
    const double invdx = 1.0 / h->dx[d];
    auto D = [&](int m, int k) { return invdx * B.Dn[k * N1 + m] * B.w[k] / B.w[m]; };
    for (int m = 0; m < HE; ++m) {
      const bool mid = 2 * m == N1 - 1;
      const double l0 = invdx * B.phi0[m] / B.w[m], l1 = invdx * B.phi1[m] / B.w[m];
      p.c.we[m] = mid ? l1 : 0.5 * (l1 + l0);
      for (int k = 0; k < H; ++k) p.c.P[m * HO + k] = mid ? D(m, k) : 0.5 * (D(m, k) - D(m, N1 - 1 - k));
      if (mid) continue;
      p.c.wo[m] = 0.5 * (l1 - l0);
      for (int k = 0; k < H; ++k) p.c.Q[m * HE + k] = 0.5 * (D(m, k) + D(m, N1 - 1 - k));
      if (N1 % 2) p.c.Q[m * HE + H] = D(m, H);
    }
    for (int m = 0; m < N1; ++m) {
      p.c.phi0[m] = B.phi0[m];
      p.c.phi1[m] = B.phi1[m];
    }
    p.g = line_geo(h->g, d);
    p.run = S - 2 < h->g.n[d] ? S - 2 : h->g.n[d];
    p.first = d == 0;
    p.last = d == DIM - 1;
    for (int c = 0; c < 3; ++c) {
      p.V0[c] = c < DIM && in.V0 ? in.V0[c] : nullptr;
      p.V[c] = c < DIM ? in.V[c] : nullptr;
      p.L[c] = c < DIM ? h->Lc[c] : nullptr;
      p.out[c] = c < DIM ? in.out[c] : nullptr;
    }
    p.a = in.a;
    p.b = in.b;
    p.dt = in.dt;
    const long long runs = (h->g.n[d] + p.run - 1) / p.run;
    const long long grid = runs * (h->g.ncell / h->g.n[d]);
    // whole warps, and no more slots than a run needs
    const int threads = ((p.run + 2) * LINES + 31) / 32 * 32;
    k_conv_line<DIM, N1><<<(unsigned)grid, threads < S * LINES ? threads : S * LINES, 0, s>>>(p);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace sdg
