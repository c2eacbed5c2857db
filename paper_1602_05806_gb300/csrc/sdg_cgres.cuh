// Resident conjugate gradients: one cooperative launch runs many iterations
// of the CG of Sec. 2.1 on a grid whose element tiles all fit on the GPU at
// once, one CTA per tile.
//
// What bounds the per-launch iteration on such grids is not the data but the
// launches: two launches per iteration cost 15-17 us of host time (7.4 us
// each) for 2-10 us of device work.  Here r, x, p and Ap of a tile stay in
// registers and shared memory from one iteration to the next, and an
// iteration has one grid-wide exchange: every CTA publishes the Ap of its
// boundary elements and four sums (p.Ap, r.r, r.Ap, Ap.Ap), then forms from
// the totals alpha of this iteration and beta of the next one,
//   ||r_{k+1}||^2 = r.r - 2 alpha r.Ap + alpha^2 Ap.Ap ,
// exactly as the one-launch form does (cg_iteration_finish), and every CTA
// takes the same decisions from the same totals (fixed summation order).
//
// The sums are compensated term by term where the launches of the two-launch
// form compensate theirs (in FP32 all, in FP64 p.Ap).  Plain sums along a line
// have 1.2 (N = 1) to 5 (N = 11) times the error in FP32 and save 2 % of an
// iteration (64 x 64 cells, N = 5: 4.21 against 4.30 us; FP64 24.3 against
// 25.2).  For FP32 data alpha and beta come from float pairs: over beta from
// 1e-4 to 30 the floats the vectors take are off by at most 5.96e-8, as from
// FP64 divisions, which take 0.5 us an iteration.
//
// The exchange has no counter, flag or fence: sums and Ap travel in 64-bit
// words of 32 data bits and a 32-bit tag (the exchange's number), so a reader
// that sees the tag has the data, in one memory round trip.  (With a fence
// between the published Ap and the sums, and one after the waits, an exchange
// took 2100 cycles longer; with one sum of 32 CTAs per warp load instead of
// all sums of eight, 7000 cycles instead of 2300 among 152 CTAs: the readers
// of a line delay its writers, so few whole lines are best.)  Two parities of
// words alternate: a CTA writes exchange k + 2 only after every CTA has
// written k + 1, that is, has read all it needs of k.  Waits are bounded: a
// CTA that gives up sets the state's wait_failed and leaves without posting
// anything more, and so does every CTA that waits for it; the host reports
// SDG_ERR_CUDA.
//
// A CTA keeps its copy of the neighbours' r and p on its face halo and
// advances it with the published Ap (the same arithmetic as the owner's), so
// one vector moves per iteration, on boundary elements only.
//
// Thread t owns the x-lines t, t + blockDim, ... (LPT of them): r, x and Ap of
// their nodes are registers.  p lives in shared memory (padded rows as in
// k_apply); the y (and z) passes leave their part of Ap in accumulators of
// their own, the x pass adds them up in the owner's registers.
#pragma once

#include "sdg_apply.cuh"

namespace sdg {

// threads per CTA the kernel is compiled for: 255 registers in FP64, 128 in FP32
template <typename T>
constexpr int res_max_threads() { return sizeof(T) == 8 ? 256 : 512; }

template <typename T, int DIM, int N1>
struct ResParams {
  Coef<T, N1> c;
  T w[N1];
  T s[3];
  T cmass;
  int n[3];
  int ts[3];   // tile extents
  int nt[3];   // tiles per direction
  // vectors of iteration j at index j & 1 (as in the one-launch form)
  T* r[2];
  T* p[2];
  T* ap[2];
  T* x;
  SolverState* st;
  unsigned long long* slots;  // [2 parities][nslot][4 sums][2 words]
  int nslot;
  unsigned long long* halo;   // [2 parities][ndof] words (FP64: pairs of them)
  long long ndof;
  unsigned tag;               // exchange k of this launch carries tag + k
  int cap;                    // most iterations of this launch
  int polls;                  // of a wait before it gives up
  double delta2;              // pause when r.r < delta2 (its largest value so far)
};

// ---- scalars of the iteration: float pairs (FP32 data) or doubles ----------
template <typename T>
struct ResAcc;
template <>
struct ResAcc<float> {
  using A = F2;
  static __device__ __forceinline__ A zero() { return F2{0.0f, 0.0f}; }
  using Dot = KDot<float>;
  static __device__ __forceinline__ A value(const Dot& d) { return pair(d); }
  static __device__ __forceinline__ A add(A a, A b) { return f2_add(a, b); }
  static __device__ __forceinline__ A shfl(A a, int o) {
    return F2{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
  }
  static __device__ __forceinline__ A from(A a, int l) {  // of lane l
    return F2{__shfl_sync(0xffffffffu, a.hi, l), __shfl_sync(0xffffffffu, a.lo, l)};
  }
  static __device__ __forceinline__ void pack(A a, unsigned w[2]) {
    w[0] = __float_as_uint(a.hi);
    w[1] = __float_as_uint(a.lo);
  }
  static __device__ __forceinline__ A unpack(unsigned w0, unsigned w1) {
    return F2{__uint_as_float(w0), __uint_as_float(w1)};
  }
  static __device__ __forceinline__ float hi(A a) { return a.hi + a.lo; }
  static __device__ __forceinline__ double dbl(A a) { return (double)a.hi + (double)a.lo; }
  // float-pair arithmetic (products through fma, sums through TwoSum)
  static __device__ __forceinline__ A norm(float h, float l) {
    const float s = h + l;
    return F2{s, l - (s - h)};
  }
  static __device__ __forceinline__ A mul(A a, A b) {
    const float p = a.hi * b.hi;
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return norm(p, e);
  }
  static __device__ __forceinline__ A sub(A a, A b) {
    const A s = f2_add(a, F2{-b.hi, -b.lo});
    return norm(s.hi, s.lo);
  }
  static __device__ __forceinline__ A one() { return F2{1.0f, 0.0f}; }
  static __device__ __forceinline__ A inv(A b) {  // one Newton step from the rounded reciprocal
    b = norm(b.hi, b.lo);
    const float q = 1.0f / b.hi;
    const float e = fmaf(-q, b.lo, fmaf(-q, b.hi, 1.0f));
    return norm(q, q * e);
  }
};
template <>
struct ResAcc<double> {
  using A = double;
  static __device__ __forceinline__ A zero() { return 0.0; }
  struct Dot {
    double s = 0.0;
    __device__ __forceinline__ void add(double a, double b) { s = fma(a, b, s); }
  };
  static __device__ __forceinline__ A value(const Dot& d) { return d.s; }
  static __device__ __forceinline__ A value(const KDot<double>& d) { return d.s + d.e; }
  static __device__ __forceinline__ A add(A a, A b) { return a + b; }
  static __device__ __forceinline__ A shfl(A a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
  static __device__ __forceinline__ A from(A a, int l) { return __shfl_sync(0xffffffffu, a, l); }
  static __device__ __forceinline__ void pack(A a, unsigned w[2]) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(a);
    w[0] = (unsigned)u;
    w[1] = (unsigned)(u >> 32);
  }
  static __device__ __forceinline__ A unpack(unsigned w0, unsigned w1) {
    return __longlong_as_double((long long)(((unsigned long long)w1 << 32) | w0));
  }
  static __device__ __forceinline__ double hi(A a) { return a; }
  static __device__ __forceinline__ double dbl(A a) { return a; }
  static __device__ __forceinline__ A norm(double h, double) { return h; }
  static __device__ __forceinline__ A mul(A a, A b) { return a * b; }
  static __device__ __forceinline__ A sub(A a, A b) { return a - b; }
  static __device__ __forceinline__ A one() { return 1.0; }
  static __device__ __forceinline__ A inv(A b) { return 1.0 / b; }
};

__device__ __forceinline__ void res_store_words(unsigned long long* a, unsigned w0, unsigned w1, unsigned tag) {
  const unsigned long long t = (unsigned long long)tag << 32;
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(a), "l"(t | w0), "l"(t | w1) : "memory");
}
__device__ __forceinline__ void res_load_words(const unsigned long long* a, unsigned long long& v0,
                                               unsigned long long& v1) {
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(v0), "=l"(v1) : "l"(a) : "memory");
}

// one published value: a word (FP32) or two (FP64)
__device__ __forceinline__ void res_publish(unsigned long long* base, long long i, float v, unsigned tag) {
  const unsigned long long w = ((unsigned long long)tag << 32) | __float_as_uint(v);
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(base + i), "l"(w) : "memory");
}
__device__ __forceinline__ void res_publish(unsigned long long* base, long long i, double v, unsigned tag) {
  unsigned w[2];
  ResAcc<double>::pack(v, w);
  res_store_words(base + 2 * i, w[0], w[1], tag);
}
// ---- the sums of an iteration ------------------------------------------------
// p.Ap, r.r, r.Ap, Ap.Ap of a CTA (from its threads' v4) posted in exchange
// `tag`: lanes halve the four sums between them first.  64 bytes per CTA, so
// that the store and the readers' loads are whole lines.  All threads call it.
template <typename T>
__device__ __forceinline__ void res_post_sums(typename ResAcc<T>::A (&v4)[4], unsigned long long* slot, unsigned tag,
                                              typename ResAcc<T>::A (*s_red)[4], typename ResAcc<T>::A (*s_tot)[4]) {
  using TA = ResAcc<T>;
  using A = typename TA::A;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const bool h16 = lane & 16, h8 = lane & 8;
  A k0 = h16 ? v4[2] : v4[0], k1 = h16 ? v4[3] : v4[1];
  A g0 = h16 ? v4[0] : v4[2], g1 = h16 ? v4[1] : v4[3];
  k0 = TA::add(k0, TA::shfl(g0, 16));
  k1 = TA::add(k1, TA::shfl(g1, 16));
  A m0 = h8 ? k1 : k0, m1 = h8 ? k0 : k1;
  m0 = TA::add(m0, TA::shfl(m1, 8));
#pragma unroll
  for (int s = 4; s > 0; s >>= 1) m0 = TA::add(m0, TA::shfl(m0, s));
  if ((lane & 7) == 0) s_red[wid][(h16 ? 2 : 0) + (h8 ? 1 : 0)] = m0;
  __syncthreads();
  if (wid == 0) {
    const int c4 = lane & 3, w8 = lane >> 2;
    A t = w8 < nw ? s_red[w8][c4] : TA::zero();
    if (w8 + 8 < nw) t = TA::add(t, s_red[w8 + 8][c4]);
#pragma unroll
    for (int s = 16; s >= 4; s >>= 1) t = TA::add(t, TA::shfl(t, s));
    if (lane < 4) {
      if (gridDim.x > 1) {
        unsigned w[2];
        TA::pack(t, w);
        res_store_words(slot + 8 * blockIdx.x + 2 * lane, w[0], w[1], tag);
      } else {
        s_tot[0][lane] = t;
      }
    }
  }
}

// polling warps of a CTA: each warp load covers eight CTAs
__device__ __forceinline__ int res_poll_warps() { return gridDim.x == 1 ? 1 : (blockDim.x >> 5) >= 8 ? 8 : 4; }

// The sums of every CTA, added by the polling warps into s_tot; a lane's loads
// are in flight together.  False when a wait ran out.
template <typename T>
__device__ __forceinline__ bool res_poll_sums(const unsigned long long* slot, unsigned tag, int limit,
                                              typename ResAcc<T>::A (*s_tot)[4]) {
  using TA = ResAcc<T>;
  using A = typename TA::A;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int c4 = lane & 3, w8 = lane >> 2, PW = res_poll_warps();
  bool fail = false;
  if (wid < PW && gridDim.x > 1) {
    constexpr int PB = 5;
    A t = TA::zero();
    for (int i0 = wid * 8 + w8; i0 < (int)gridDim.x && !fail; i0 += PB * PW * 8) {
      unsigned long long q0[PB], q1[PB];
      bool ok;
      int polls = 0;
      do {
        ok = true;
#pragma unroll
        for (int u = 0; u < PB; ++u)
          if (i0 + u * PW * 8 < (int)gridDim.x) res_load_words(slot + 8 * (i0 + u * PW * 8) + 2 * c4, q0[u], q1[u]);
#pragma unroll
        for (int u = 0; u < PB; ++u)
          if (i0 + u * PW * 8 < (int)gridDim.x)
            ok = ok && (unsigned)(q0[u] >> 32) == tag && (unsigned)(q1[u] >> 32) == tag;
      } while (!ok && ++polls < limit);
      fail = !ok;
      if (ok) {
#pragma unroll
        for (int u = 0; u < PB; ++u)
          if (i0 + u * PW * 8 < (int)gridDim.x) t = TA::add(t, TA::unpack((unsigned)q0[u], (unsigned)q1[u]));
      }
    }
    __syncwarp();
#pragma unroll
    for (int s = 16; s >= 4; s >>= 1) t = TA::add(t, TA::shfl(t, s));
    if (lane < 4) s_tot[wid][lane] = t;
  }
  return !fail;
}

// Warp 0's copy of the recursion, the same in every CTA.
template <typename T>
struct ResLoop {
  using TA = ResAcc<T>;
  using A = typename TA::A;
  A alpha, beta, rr, rr_old, pap;
  T maxrr, tol2, delta2;
  int it0, it, maxit, cap, done, pause, status;
  bool reliable;
  __device__ __forceinline__ void init(const SolverState* st, double d2, int cap_) {
    alpha = beta = rr = rr_old = pap = TA::zero();
    maxrr = (T)st->maxrr;
    tol2 = (T)st->tol2;
    delta2 = (T)d2;
    it = it0 = st->iter;
    maxit = st->maxit;
    cap = cap_;
    done = pause = 0;
    status = st->status;
    reliable = st->reliable != 0;
  }
  // alpha, beta and the decisions (cg_iteration_finish) from the totals, by
  // warp 0; s_ab and s_flow tell the others
  __device__ __forceinline__ void decide(A (*s_tot)[4], int fail, T* s_ab, int* s_flow) {
    const int lane = threadIdx.x & 31, c4 = lane & 3, w8 = lane >> 2;
    A t = w8 < res_poll_warps() ? s_tot[w8][c4] : TA::zero();
#pragma unroll
    for (int s = 16; s >= 4; s >>= 1) t = TA::add(t, TA::shfl(t, s));
    const A pa = TA::from(t, 0), r2 = TA::from(t, 1), ra = TA::from(t, 2), aa = TA::from(t, 3);
    const T pa_h = (T)TA::hi(pa), rr_h = (T)TA::hi(r2);
    pap = pa;
    rr_old = rr;
    rr = r2;
    if (rr_h > maxrr) maxrr = rr_h;
    if (fail) {
      done = 1;
      status = SDG_ERR_CUDA;
    } else if (!(pa_h > T(0)) || !isfinite(pa_h) || !isfinite(rr_h)) {
      done = 1;
      status = SDG_ERR_BREAKDOWN;
      alpha = TA::zero();
      beta = TA::zero();
    } else {
      // beta = ||r_{k+1}||^2 / ||r_k||^2 = 1 - (2 r.Ap - alpha Ap.Ap) / p.Ap
      const A iv = TA::inv(pa);
      alpha = TA::mul(r2, iv);
      beta = TA::sub(TA::one(), TA::mul(TA::sub(TA::add(ra, ra), TA::mul(alpha, aa)), iv));
      if (!((T)TA::hi(beta) > T(0))) beta = TA::zero();
      if (rr_h <= tol2) {
        if (reliable) pause = 1;
        else { done = 1; status = SDG_OK; }
      } else if (reliable && rr_h < delta2 * maxrr) {
        pause = 1;
      } else if (it >= maxit) {
        done = 1;
        status = SDG_ERR_NOT_CONVERGED;
      }
    }
    if (lane == 0) {
      s_ab[0] = (T)TA::hi(alpha);
      s_ab[1] = (T)TA::hi(beta);
      *s_flow = done || pause || it - it0 >= cap;
    }
  }
  __device__ __forceinline__ void store(SolverState* st, double d2) const {
    st->pAp = TA::dbl(pap);
    st->rr_old = it - it0 > 1 ? TA::dbl(rr_old) : st->rr;
    st->rr = TA::dbl(rr);
    st->alpha = TA::dbl(alpha);
    st->beta = TA::dbl(beta);
    st->alpha_f = (float)TA::hi(alpha);
    st->beta_f = (float)TA::hi(beta);
    st->maxrr = (double)maxrr;
    st->delta2 = d2;
    st->iter = it;
    st->done = done;
    st->pause = pause;
    st->status = status;
  }
};

// ---- tile of a CTA ----------------------------------------------------------
// Position and extents of the CTA's tile; face halo x-, x+, y-, y+, z-, z+
// (a direction with a single tile wraps inside it and has none): slots
// [0, TE) are the tile's elements, [TE, TE + NH) the halo's.
template <int DIM>
struct ResTile {
  int o[3], V[3], TE, NH, hoff[DIM + 1];
  __device__ __forceinline__ ResTile(const int (&n)[3], const int (&ts)[3], const int (&nt)[3]) {
    const int b[3] = {(int)blockIdx.x % nt[0], ((int)blockIdx.x / nt[0]) % nt[1], (int)blockIdx.x / (nt[0] * nt[1])};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      o[d] = b[d] * ts[d];
      V[d] = min(ts[d], n[d] - o[d]);
    }
    TE = V[0] * V[1] * V[2];
    hoff[0] = 0;
#pragma unroll
    for (int d = 0; d < DIM; ++d) hoff[d + 1] = hoff[d] + (nt[d] > 1 ? 2 * (TE / V[d]) : 0);
    NH = hoff[DIM];
  }
  // neighbour slots (times ES) of every element, global element of every halo slot
  __device__ __forceinline__ void tables(const int (&n)[3], const int (&nt)[3], int ES, int* s_nb, int* s_hel) const {
    const int tid = threadIdx.x, nth = blockDim.x;
    for (int e = tid; e < TE; e += nth) {
      const int l[3] = {e % V[0], (e / V[0]) % V[1], e / (V[0] * V[1])};
#pragma unroll
      for (int d = 0; d < DIM; ++d) {
        const int str = d == 0 ? 1 : d == 1 ? V[0] : V[0] * V[1];
        // position of this element in the face normal to d
        const int f = d == 0 ? l[2] * V[1] + l[1] : d == 1 ? l[2] * V[0] + l[0] : l[1] * V[0] + l[0];
        const int F = TE / V[d];
        int lo = e - str, hi = e + str;
        if (l[d] == 0) lo = nt[d] > 1 ? TE + hoff[d] + f : e + (V[d] - 1) * str;
        if (l[d] == V[d] - 1) hi = nt[d] > 1 ? TE + hoff[d] + F + f : e - (V[d] - 1) * str;
        s_nb[e * 2 * DIM + 2 * d] = lo * ES;
        s_nb[e * 2 * DIM + 2 * d + 1] = hi * ES;
      }
    }
    for (int s = tid; s < NH; s += nth) {
      int d = 0;
#pragma unroll
      for (int k = 1; k < DIM; ++k)
        if (s >= hoff[k]) d = k;
      const int F = TE / V[d];
      const int side = (s - hoff[d]) / F, f = (s - hoff[d]) % F;
      int g[3] = {0, 0, 0};
      const int d0 = d == 0 ? 1 : 0, d1 = d == 2 ? 1 : 2;  // the face's directions
      g[d0] = o[d0] + f % V[d0];
      g[d1] = DIM == 3 ? o[d1] + f / V[d0] : 0;
      g[d] = side ? o[d] + V[d] : o[d] - 1;
      if (g[d] < 0) g[d] += n[d];
      if (g[d] >= n[d]) g[d] -= n[d];
      s_hel[s] = (g[2] * n[1] + g[1]) * n[0] + g[0];
    }
  }
};

// Shared-memory layout of an element: rows of N1 values padded to RS.
template <int DIM, int N1>
struct ResEl {
  static constexpr int NPE = ipow(N1, DIM), LINES = ipow(N1, DIM - 1);
  static constexpr int RS = N1 + 1, PS = N1 * RS, ES = DIM == 2 ? PS : N1 * PS;
  static __device__ __forceinline__ int xline(int lam) { return DIM == 2 ? lam * RS : (lam % N1) * RS + (lam / N1) * PS; }
  static __device__ __forceinline__ int node(int q) { return (q / N1) * RS + q % N1; }
};

// y (and z) passes over the tile's lines, each into an accumulator of its own
template <typename T, int DIM, int N1, int LPT>
__device__ __forceinline__ void res_cross_passes(const Coef<T, N1>& c, const T (&sd)[3], const T* s_w, const T* s_p,
                                                 T* s_o, const int* s_nb, int TE) {
  using E = ResEl<DIM, N1>;
  const int nl = TE * E::LINES;
#pragma unroll
  for (int d = DIM - 1; d >= 1; --d) {
#pragma unroll
    for (int j = 0; j < LPT; ++j) {
      const int id = threadIdx.x + j * blockDim.x;
      if (id >= nl) continue;
      const int e = id / E::LINES, lam = id - e * E::LINES;
      const int q0 = lam % N1, q1 = lam / N1;
      const int stride = d == 1 ? E::RS : E::PS;
      const int base = DIM == 2 ? lam : (d == 1 ? q0 + q1 * E::PS : q0 + q1 * E::RS);
      const T wp = DIM == 2 ? s_w[lam] : s_w[q0] * s_w[q1];
      const T* pl = s_p + s_nb[e * 2 * DIM + 2 * d] + base;
      const T* pr = s_p + s_nb[e * 2 * DIM + 2 * d + 1] + base;
      const T* pc = s_p + e * E::ES + base;
      T xl[N1], xc[N1], xr[N1], val[N1];
#pragma unroll
      for (int m = 0; m < N1; ++m) {
        xl[m] = pl[m * stride];
        xc[m] = pc[m * stride];
        xr[m] = pr[m * stride];
      }
      line_apply<T, N1, true>(c, xl, xc, xr, sd[d] * wp, val);
      T* out = s_o + (size_t)(d - 1) * TE * E::ES + e * E::ES + base;
#pragma unroll
      for (int m = 0; m < N1; ++m) out[m * stride] = val[m];
    }
  }
}

// x pass of line lam of element e, the other passes' parts and the mass term
// added: the operator's values on the line's nodes (xc: the centre values)
template <typename T, int DIM, int N1>
__device__ __forceinline__ void res_x_line(const Coef<T, N1>& c, T s0, T cmass, const T* s_w, const T* s_p,
                                           const T* s_o, const int* s_nb, int TE, int e, int lam, T (&xc)[N1],
                                           T (&val)[N1]) {
  using E = ResEl<DIM, N1>;
  const int base = E::xline(lam);
  const T wp = DIM == 2 ? s_w[lam] : s_w[lam % N1] * s_w[lam / N1];
  const T* pl = s_p + s_nb[e * 2 * DIM] + base;
  const T* pr = s_p + s_nb[e * 2 * DIM + 1] + base;
  const T* pc = s_p + e * E::ES + base;
  const T* po = s_o + e * E::ES + base;
  T xl[N1], xr[N1];
#pragma unroll
  for (int m = 0; m < N1; ++m) {
    xl[m] = pl[m];
    xc[m] = pc[m];
    xr[m] = pr[m];
  }
  line_apply<T, N1, true>(c, xl, xc, xr, s0 * wp, val);
#pragma unroll
  for (int m = 0; m < N1; ++m) {
    T v = val[m];
    if (cmass != T(0)) v = fma(cmass * wp * s_w[m], xc[m], v);
    v += po[m];
    if (DIM == 3) v += po[(size_t)TE * E::ES + m];
    val[m] = v;
  }
}

// The neighbours' published values of exchange `tag` into s_ah (a halo element
// after the other), all loads of a thread in flight together; in FP32 two
// words per load where elements hold an even number of nodes.  False when a
// wait ran out.
template <typename T, int NPE>
__device__ __forceinline__ bool res_fetch(T* s_ah, const int* s_hel, int NH, const unsigned long long* hw, unsigned tag,
                                          int limit) {
  constexpr int W = sizeof(T) == 4 && NPE % 2 == 0 ? 2 : 1, HB = 8;
  constexpr int NV = NPE / W;
  const int tid = threadIdx.x, nth = blockDim.x, nv = NH * NV;
  bool fail = false;
  for (int v0 = tid; v0 < nv && !fail; v0 += HB * nth) {
    unsigned long long w0[HB], w1[HB];
    bool ok;
    int polls = 0;
    do {
      ok = true;
#pragma unroll
      for (int u = 0; u < HB; ++u) {
        const int v = v0 + u * nth, s = v / NV;
        w0[u] = w1[u] = (unsigned long long)tag << 32;
        if (v >= nv) continue;
        const unsigned long long* at = hw + (sizeof(T) / 4) * ((size_t)s_hel[s] * NPE + (size_t)((v - s * NV) * W));
        if constexpr (sizeof(T) == 8 || W == 2) res_load_words(at, w0[u], w1[u]);
        else asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(w0[u]) : "l"(at) : "memory");
      }
#pragma unroll
      for (int u = 0; u < HB; ++u) ok = ok && (unsigned)(w0[u] >> 32) == tag && (unsigned)(w1[u] >> 32) == tag;
    } while (!ok && ++polls < limit);
    fail = !ok;
#pragma unroll
    for (int u = 0; u < HB; ++u) {
      const int v = v0 + u * nth;
      if (v >= nv) continue;
      if constexpr (sizeof(T) == 8) {
        s_ah[v] = ResAcc<double>::unpack((unsigned)w0[u], (unsigned)w1[u]);
      } else {
        s_ah[v * W] = __uint_as_float((unsigned)w0[u]);
        if constexpr (W == 2) s_ah[v * W + 1] = __uint_as_float((unsigned)w1[u]);
      }
    }
  }
  return !fail;
}

template <typename T, int DIM, int N1, int LPT>
__global__ void __launch_bounds__(res_max_threads<T>(), 1) k_cg_res(const __grid_constant__ ResParams<T, DIM, N1> a) {
  using TA = ResAcc<T>;
  using A = typename TA::A;
  using E = ResEl<DIM, N1>;
  constexpr int NPE = E::NPE, LINES = E::LINES, ES = E::ES;

  SolverState* st = a.st;
  if (st->done || st->pause) return;  // uniform over the grid

  const ResTile<DIM> tile(a.n, a.ts, a.nt);
  const int TE = tile.TE, NH = tile.NH;

  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* s_p = reinterpret_cast<T*>(smem_raw);             // (TE + NH) ES: p
  T* s_o = s_p + (size_t)(TE + NH) * ES;               // (DIM - 1) TE ES: parts of Ap
  T* s_rh = s_o + (size_t)(DIM - 1) * TE * ES;         // NH NPE: r of the halo
  T* s_ah = s_rh + (size_t)NH * NPE;                   // NH NPE: Ap of the halo, last iteration's
  int* s_nb = reinterpret_cast<int*>(s_ah + (size_t)NH * NPE);  // TE 2 DIM: neighbour slots
  int* s_hel = s_nb + TE * 2 * DIM;                    // NH: global element of a halo slot
  __shared__ T s_w[N1];
  __shared__ A s_red[16][4];   // the warps' sums
  __shared__ A s_tot[8][4];    // totals, by polling warp
  __shared__ T s_ab[2];        // alpha, beta
  __shared__ int s_flow;       // the CTA leaves the loop
  __shared__ int s_fail;

  const int tid = threadIdx.x, nth = blockDim.x;
  const int wid = tid >> 5;
  if (tid < N1) s_w[tid] = a.w[tid];
  if (tid == 0) s_fail = 0;
  tile.tables(a.n, a.nt, ES, s_nb, s_hel);
  __syncthreads();

  // ---- this thread's x-lines ----
  const int nl = TE * LINES;
  const int it0 = st->iter;
  const int b0 = it0 & 1;
  const bool fresh = it0 == 0;
  T r[LPT][N1], x[LPT][N1], ap[LPT][N1];
  size_t gl[LPT];    // global index of the line's first node
  bool act[LPT], pub[LPT];
#pragma unroll
  for (int k = 0; k < LPT; ++k) {
    const int id = tid + k * nth;
    act[k] = id < nl;
    pub[k] = false;
    gl[k] = 0;
    if (!act[k]) continue;
    const int e = id / LINES, lam = id - e * LINES;
    const int l[3] = {e % tile.V[0], (e / tile.V[0]) % tile.V[1], e / (tile.V[0] * tile.V[1])};
    const size_t ge = ((size_t)(tile.o[2] + l[2]) * a.n[1] + (tile.o[1] + l[1])) * a.n[0] + (tile.o[0] + l[0]);
    gl[k] = ge * NPE + (size_t)lam * N1;
#pragma unroll
    for (int d = 0; d < DIM; ++d)
      if (a.nt[d] > 1 && (l[d] == 0 || l[d] == tile.V[d] - 1)) pub[k] = true;
    const int base = e * ES + E::xline(lam);
#pragma unroll
    for (int m = 0; m < N1; ++m) {
      r[k][m] = a.r[b0][gl[k] + m];
      x[k][m] = a.x[gl[k] + m];
      ap[k][m] = fresh ? T(0) : a.ap[b0][gl[k] + m];
      s_p[base + m] = fresh ? T(0) : a.p[b0][gl[k] + m];
    }
  }
  for (int v = tid; v < NH * NPE; v += nth) {
    const int s = v / NPE, q = v - s * NPE;
    const size_t gi = (size_t)s_hel[s] * NPE + q;
    s_rh[v] = a.r[b0][gi];
    s_ah[v] = fresh ? T(0) : a.ap[b0][gi];
    s_p[(TE + s) * ES + E::node(q)] = fresh ? T(0) : a.p[b0][gi];
  }

  T alpha = fresh ? T(0) : (sizeof(T) == 4 ? (T)st->alpha_f : (T)st->alpha);
  T beta = fresh ? T(0) : (sizeof(T) == 4 ? (T)st->beta_f : (T)st->beta);
  ResLoop<T> lp;
  lp.init(st, a.delta2, a.cap);

  for (int k = 0;; ++k) {
    const unsigned tag = a.tag + (unsigned)k;  // of this iteration's exchange
    unsigned long long* hout = a.halo + (size_t)(k & 1) * a.ndof * (sizeof(T) / 4);
    // ---- r -= alpha Ap, x += alpha p, p = r + beta p ----
    // (halo: with the neighbours' Ap of the last iteration; iteration 0 takes p = r)
#pragma unroll
    for (int j = 0; j < LPT; ++j) {
      if (!act[j]) continue;
      const int id = tid + j * nth;
      const int e = id / LINES, lam = id - e * LINES;
      const int base = e * ES + E::xline(lam);
#pragma unroll
      for (int m = 0; m < N1; ++m) {
        const T po = s_p[base + m];
        r[j][m] = fma(-alpha, ap[j][m], r[j][m]);
        x[j][m] = fma(alpha, po, x[j][m]);
        s_p[base + m] = fma(beta, po, r[j][m]);
      }
    }
    for (int v = tid; v < NH * NPE; v += nth) {
      const int s = v / NPE, si = (TE + s) * ES + E::node(v - s * NPE);
      const T rh = fma(-alpha, s_ah[v], s_rh[v]);
      s_rh[v] = rh;
      s_p[si] = fma(beta, s_p[si], rh);
    }
    __syncthreads();

    // ---- Ap: z and y passes into accumulators, x pass in registers ----
    res_cross_passes<T, DIM, N1, LPT>(a.c, a.s, s_w, s_p, s_o, s_nb, TE);
    __syncthreads();
    // (compensated term by term: p.Ap, in FP32 all)
    KDot<T> d_pa;
    typename TA::Dot d_rr, d_ra, d_aa;
#pragma unroll
    for (int j = 0; j < LPT; ++j) {
      if (!act[j]) continue;
      const int id = tid + j * nth;
      const int e = id / LINES, lam = id - e * LINES;
      T xc[N1];
      res_x_line<T, DIM, N1>(a.c, a.s[0], a.cmass, s_w, s_p, s_o, s_nb, TE, e, lam, xc, ap[j]);
      if (pub[j]) {
#pragma unroll
        for (int m = 0; m < N1; ++m) res_publish(hout, (long long)gl[j] + m, ap[j][m], tag);
      }
#pragma unroll
      for (int m = 0; m < N1; ++m) {
        d_pa.add(xc[m], ap[j][m]);
        d_rr.add(r[j][m], r[j][m]);
        d_ra.add(r[j][m], ap[j][m]);
        d_aa.add(ap[j][m], ap[j][m]);
      }
    }
    A v4[4] = {TA::value(d_pa), TA::value(d_rr), TA::value(d_ra), TA::value(d_aa)};
    unsigned long long* slot = a.slots + (size_t)(k & 1) * a.nslot * 8;
    res_post_sums<T>(v4, slot, tag, s_red, s_tot);
    // the neighbours' Ap for the next update, published before their sums
    bool fail = NH > 0 && !res_fetch<T, NPE>(s_ah, s_hel, NH, hout, tag, a.polls);
    fail = !res_poll_sums<T>(slot, tag, a.polls, s_tot) || fail;
    if (fail) s_fail = st->wait_failed = 1;
    __syncthreads();

    ++lp.it;
    if (wid == 0) lp.decide(s_tot, s_fail, s_ab, &s_flow);
    __syncthreads();
    alpha = s_ab[0];
    beta = s_ab[1];
    if (s_flow) break;
  }

  // ---- leave r, p, Ap of the last iteration and x (without its step) ----
  const int b1 = lp.it & 1;
#pragma unroll
  for (int j = 0; j < LPT; ++j) {
    if (!act[j]) continue;
    const int id = tid + j * nth;
    const int e = id / LINES, lam = id - e * LINES;
    const int base = e * ES + E::xline(lam);
#pragma unroll
    for (int m = 0; m < N1; ++m) {
      a.r[b1][gl[j] + m] = r[j][m];
      a.x[gl[j] + m] = x[j][m];
      a.ap[b1][gl[j] + m] = ap[j][m];
      a.p[b1][gl[j] + m] = s_p[base + m];
    }
  }
  if (blockIdx.x == 0 && tid == 0) lp.store(st, a.delta2);
}

// launchers, one per translation unit (sdg_cgres_*.cu)
template <typename T, int DIM, int N1>
void fill_res_params(const sdg_handle* h, const ResPlan& pl, const ResArgs<T>& in, ResParams<T, DIM, N1>* pp) {
  ResParams<T, DIM, N1>& p = *pp;
  ApplyParams<T, DIM, N1> q;
  ApplyArgs<T> aa{};
  for (int d = 0; d < 3; ++d) aa.s[d] = in.s[d];
  aa.cmass = in.cmass;
  fill_apply_params<T, DIM, N1>(h, aa, &q);
  p.c = q.c;
  for (int i = 0; i < N1; ++i) p.w[i] = q.w[i];
  p.cmass = q.cmass;
  for (int d = 0; d < 3; ++d) {
    p.s[d] = q.s[d];
    p.n[d] = q.n[d];
    p.ts[d] = pl.ts[d];
    p.nt[d] = pl.nt[d];
  }
  for (int k = 0; k < 2; ++k) {
    p.r[k] = in.r[k];
    p.p[k] = in.p[k];
    p.ap[k] = in.ap[k];
  }
  p.x = in.x;
  p.st = in.st;
  p.slots = h->res_slots;
  p.nslot = h->res_ctas;
  p.halo = h->res_halo;
  p.ndof = h->g.ndof;
  p.tag = in.tag;
  p.cap = in.cap;
  p.polls = h->polls;
  p.delta2 = in.delta2;
}

// Cooperative launch (all CTAs resident: they wait for one another) of a
// kernel on the plan's tiles.  The shared-memory attribute is set once per
// instantiation and device.
template <typename P>
cudaError_t launch_coop(void (*kern)(P), const P& p, const sdg_handle* h, const ResPlan& pl, PerDevice* attr_set,
                        cudaStream_t stream) {
  if (!attr_set->get(h->device)) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kResMaxSmem);
    if (e != cudaSuccess) return e;
    attr_set->set(h->device, 1);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(pl.nt[0] * pl.nt[1] * pl.nt[2]));
  cfg.blockDim = dim3(pl.threads);
  cfg.dynamicSmemBytes = pl.smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, kern, p);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

template <typename T, int DIM, int N1, int LPT>
cudaError_t launch_res(const sdg_handle* h, const ResPlan& pl, const ResArgs<T>& in, cudaStream_t stream) {
  ResParams<T, DIM, N1> p;
  fill_res_params<T, DIM, N1>(h, pl, in, &p);
  static PerDevice attr_set;
  return launch_coop(k_cg_res<T, DIM, N1, LPT>, p, h, pl, &attr_set, stream);
}

// two x-lines per thread in FP32 where their registers fit (n1 <= 8)
template <typename T, int DIM, int N1>
cudaError_t launch_res_t(const sdg_handle* h, const ResPlan& pl, const ResArgs<T>& in, cudaStream_t stream) {
  if constexpr (sizeof(T) == 4 && N1 <= 8) {
    if (pl.lpt == 2) return launch_res<T, DIM, N1, 2>(h, pl, in, stream);
  }
  return launch_res<T, DIM, N1, 1>(h, pl, in, stream);
}

}  // namespace sdg
