// 3D operator kernel that marches through z (block hepta-diagonal system of
// Eq. pSyst, applied dimension by dimension as 1D contractions, Eq. tensorP1).
//
// One CTA owns a column of TX x TY elements in x and y and a run of zc planes
// in z.  It keeps three planes of the column (z-1, z, z+1) in a shared-memory
// ring and, per step, loads one new plane plus the x/y face halo of the plane
// it computes: every element is read about 1 + 2 (TX + TY) / (TX TY) + 2 / zc
// times (about 2.2 for 4 x 4 and zc = 12) instead of once per face
// neighbour.  Each thread owns one 1D line of one element of the plane per
// direction and applies the line operator (line_apply: the same accurate
// contraction as the element-tile kernel).  The store adds the accumulators
// of the directions, and each plane is stored as it is finished.
//
// FP32 waits for its loads unless they are under way early (AHEAD): the z
// lines of a plane come first, after which plane z-1 is done with, and the
// next plane and face halo are copied (cp.async) while the x and y lines are
// computed; p = r + beta p_old is formed where they land.  48^3 cells, N = 4:
// plain apply 82 -> 62 us, the CG operator 116 -> 101 us (cold), now bound by
// instruction issue (61 % of the slots; 40 % of them FP32 arithmetic) and
// barriers.  It takes rows of whole vectors (odd N1, nx a multiple of the
// vector): value by value the copies cost more than the waiting (47 x 45 x 41
// cells: 256 -> 328 us per iteration).  FP64 is bound by its pipe (80 % of
// it), gains nothing by it (48^3: 1283 -> 1320 us) and loads when needed,
// one accumulator per direction and no barrier between the passes.
//
// Modes as in k_apply: plain apply (fuse 0), the operator of the two-launch
// CG iteration (fuse 1: p = r + beta p_old, x += alpha p_old when the state
// asks for it, and the block's p.Ap total for the update launch) and the one-launch CG
// iteration (ONE: r -= alpha Ap_old, x += alpha p_old, p = r + beta p_old,
// Ap, and p.Ap, r.r, r.Ap, Ap.Ap).  Planes z0 - 1 and z0 + zc belong to the
// neighbouring runs: this CTA forms their values but writes nothing there.
#pragma once

#include "sdg_apply.cuh"

namespace sdg {

template <int N1>
struct March3 {
  static constexpr int TX = 4, TY = 4;
  static constexpr int PE = TX * TY;           // elements of one plane of the column
  static constexpr int NPE = N1 * N1 * N1;
  static constexpr int LINES = N1 * N1;        // lines of an element per direction
  static constexpr int THREADS = PE * LINES;
  // rows of N1 values, padded for even N1 only: for odd N1 the strided line
  // reads of a warp already fall on distinct banks, and the unpadded layout
  // makes staging a plain copy
  static constexpr int RS = (N1 % 2) ? N1 : N1 + 1;
  static constexpr int PS = N1 * RS;
  static constexpr int ES = N1 * PS;
  static constexpr int HALO = 2 * TX + 2 * TY;  // x and y face halo of a plane
};

// shared-memory offset of element-local node q (x fastest)
template <int N1>
__device__ __forceinline__ int m3_sidx(int q) {
  using M = March3<N1>;
  if constexpr (M::RS == N1) return q;
  const int row = q / N1;
  return row * M::RS + (q - row * N1);
}

// x-face halo slot of the marching kernel: an element rounded up to whole
// vectors of T
template <typename T, int N1>
__host__ __device__ constexpr int m3_halo_slot() {
  return (March3<N1>::ES + VecOf<T>::W - 1) / VecOf<T>::W * VecOf<T>::W;
}

// Resident CTAs per SM the kernel is compiled for (a register cap: without
// barriers between the passes the compiler keeps more values live): three of
// 400 threads in FP32 for N1 = 5 (48 registers per thread), two in FP64, and
// what the registers of the passes allow below (N1 = 4: 80 in FP64; with the
// 88 it would take of itself two CTAs fit, and a CG iteration on 30 x 24 x 27
// cells took 267 instead of 239 us)
template <typename T, int N1>
constexpr int march3_min_blocks() {
  if (sizeof(T) == 4) return N1 == 5 ? 3 : N1 >= 3 ? 5 : 8;
  return N1 == 5 ? 2 : N1 == 4 ? 3 : N1 == 3 ? 4 : 8;
}

// Shared memory of a mode (0 plain apply, 1 operator of the two-launch CG
// iteration, 2 one-launch iteration), in values: what is copied ahead of its
// use is what still lets the CTAs above share an SM.
template <typename T, int N1, int MODE, bool AHEAD>
struct March3Smem {
  using M = March3<N1>;
  static constexpr int HALO_SZ = 2 * M::TY * m3_halo_slot<T, N1>() + 2 * M::TX * M::ES;
  static constexpr int HB = AHEAD ? 2 : 1;      // face-halo buffers
  static constexpr int ACCS = AHEAD ? 2 : 3;    // accumulators: z + x, y lines / z, y, x lines
  static constexpr int SZ = (3 + ACCS) * M::PE * M::ES + HB * HALO_SZ +
                            (MODE == 2 ? 3 * M::PE * M::ES : AHEAD && MODE == 1 ? M::PE * M::ES + HALO_SZ : 0);
};

// v as a value of unknown origin
template <typename I>
__device__ __forceinline__ void keep(I& v) { asm volatile("" : "+r"(v)); }

// asynchronous copy of 16 bytes, global to shared memory; copy_async_wait
// waits for the calling thread's copies
__device__ __forceinline__ void copy_async(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <typename T, int N1, bool ACC, int MODE, bool AHEAD>
__global__ void __launch_bounds__(March3<N1>::THREADS, (march3_min_blocks<T, N1>()))
    k_apply3m(const __grid_constant__ ApplyParams<T, 3, N1> a) {
  using M = March3<N1>;
  using L = March3Smem<T, N1, MODE, AHEAD>;
  constexpr bool ONE = MODE == 2, fuse = MODE != 0;
  constexpr int TX = M::TX, TY = M::TY, PE = M::PE, NPE = M::NPE, LINES = M::LINES;
  constexpr int RS = M::RS, PS = M::PS, ES = M::ES, HALO = M::HALO, THREADS = M::THREADS;
  using VT = typename VecOf<T>::V;
  constexpr int VW = VecOf<T>::W;
  constexpr int HS = m3_halo_slot<T, N1>();  // x-halo slot: ES rounded up to whole vectors
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* ring = reinterpret_cast<T*>(smem_raw);  // 3 planes: 3 * PE * ES
  T* halo = ring + 3 * PE * ES;              // face halo, 1 or 2 buffers (L::HB)
  T* s_out = halo + L::HB * L::HALO_SZ;      // accumulators (see March3Smem)
  T* extra = s_out + L::ACCS * PE * ES;            // CG: p_old of the incoming plane and halo / one launch: r_k by ring slot
  T* hpo = extra + PE * ES;

  pdl_trigger();
  const int bx = blockIdx.x % a.ntile[0];
  const int by = (blockIdx.x / a.ntile[0]) % a.ntile[1];
  const int bz = blockIdx.x / (a.ntile[0] * a.ntile[1]);
  const int nx = a.n[0], ny = a.n[1], nz = a.n[2];
  const int ox = bx * TX, oy = by * TY, z0 = bz * a.zc;
  const int VX = min(TX, nx - ox), VY = min(TY, ny - oy);
  const int NZ = min(a.zc, nz - z0);  // planes owned by this CTA

  pdl_wait();
  bool first = false, xupd = false;
  T beta = T(0), alpha = T(0);
  if constexpr (fuse) {
    if (a.st->done || a.st->pause) return;  // uniform: written by the previous kernel
    first = (a.st->iter == 0);
    if (!first) {
      beta = sizeof(T) == 4 ? (T)a.st->beta_f : (T)a.st->beta;
      alpha = sizeof(T) == 4 ? (T)a.st->alpha_f : (T)a.st->alpha;
      // two-launch form: x += alpha_{k-1} p_{k-1} on the owned nodes
      xupd = !ONE && a.xsol != nullptr && a.st->xpend != 0;
    }
  }

  // the value of node gi that the passes read: x (plain), p = r + beta p_old
  // (CG); for an owned node also the CG writes (kept r_k in *rk)
  auto stage = [&](size_t gi, bool owned, T* rk) -> T {
    T r = a.x[gi];
    if constexpr (!fuse) return r;
    if constexpr (ONE) {
      if (!first) {
        const T po = a.p_old[gi];
        r = fma(-alpha, a.ap_old[gi], r);
        const T p = fma(beta, po, r);
        if (owned) {
          a.xsol[gi] = fma(alpha, po, a.xsol[gi]);
          a.r_out[gi] = r;
          a.p_out[gi] = p;
          *rk = r;
        }
        return p;
      }
      if (owned) {
        a.r_out[gi] = r;
        a.p_out[gi] = r;
        *rk = r;
      }
      return r;
    } else {
      if (first) {
        if (owned) a.p_out[gi] = r;
        return r;
      }
      const T po = a.p_old[gi];
      const T p = fma(beta, po, r);
      if (owned) {
        a.p_out[gi] = p;
        if (xupd) a.xsol[gi] = fma(alpha, po, a.xsol[gi]);
      }
      return p;
    }
  };
  auto wrapz = [nz](int z) { return z < 0 ? z + nz : (z >= nz ? z - nz : z); };

  // Rows of the column (TX elements along x) are contiguous runs of TX NPE
  // values in global memory and, with unpadded rows, in shared memory; when
  // the column is full in x and nx is a multiple of the vector width they
  // start on 16-byte boundaries, and box planes, y-face halo and stores move
  // as float4 / double2 with one index computation per vector.
  constexpr int RV = TX * NPE / VW;  // vectors per row
  const size_t plane = (size_t)nx * ny * NPE;
  // (byte offsets within a plane are 32-bit in the vector path)
  const bool vec = AHEAD || ((RS == N1) && (TX * NPE) % VW == 0 && VX == TX && nx % VW == 0 &&
                             plane * sizeof(T) < (size_t(1) << 32));
  // x-face halo elements in the vector path: element ox - 1 ends and element
  // ox + VX starts on a vector boundary (both neighbour a full, aligned row
  // of the column, or wrap to a row end / start), so each moves as the HS / VW
  // vectors that end (x = -1) or start (x = VX) there; the x = -1 element then
  // sits LOFF values into its slot, the few values before it are unused
  constexpr int LOFF = (VW - NPE % VW) % VW;
  const int loff = vec ? LOFF : 0;
  // the vector at byte off of the plane that starts at value zb: a pointer
  // common to the block and 32 bits per thread
  auto vat = [](auto* v, size_t zb, unsigned off) {
    using C = std::conditional_t<std::is_const_v<std::remove_pointer_t<decltype(v)>>, const VT, VT>;
    using B = std::conditional_t<std::is_const_v<std::remove_pointer_t<decltype(v)>>, const char, char>;
    return reinterpret_cast<C*>(reinterpret_cast<B*>(v + zb) + off);
  };
  // stage() on the VW values of one vector
  // (rs, ps, xs: where r, p_old and x already are, null: read them here)
  auto stage_vec = [&](size_t zb, unsigned off, bool owned, VT* rk, const VT* rs, const VT* ps, const VT* xs) -> VT {
    VT out;
    T* o = reinterpret_cast<T*>(&out);
    VT r = rs ? *rs : *vat(a.x, zb, off);
    if constexpr (!fuse) return r;
    T* rp = reinterpret_cast<T*>(&r);
    if constexpr (ONE) {
      if (!first) {
        const VT po = *vat(a.p_old, zb, off);
        const VT ao = *vat(a.ap_old, zb, off);
        const T* pp = reinterpret_cast<const T*>(&po);
        const T* ap = reinterpret_cast<const T*>(&ao);
#pragma unroll
        for (int k = 0; k < VW; ++k) {
          rp[k] = fma(-alpha, ap[k], rp[k]);
          o[k] = fma(beta, pp[k], rp[k]);
        }
        if (owned) {
          VT xv = *vat(a.xsol, zb, off);
          T* xp = reinterpret_cast<T*>(&xv);
#pragma unroll
          for (int k = 0; k < VW; ++k) xp[k] = fma(alpha, pp[k], xp[k]);
          *vat(a.xsol, zb, off) = xv;
        }
      } else {
        out = r;
      }
      if (owned) {
        *vat(a.r_out, zb, off) = r;
        *vat(a.p_out, zb, off) = out;
        *rk = r;
      }
      return out;
    } else {
      if (first) {
        out = r;
      } else {
        const VT po = ps ? *ps : *vat(a.p_old, zb, off);
        const T* pp = reinterpret_cast<const T*>(&po);
#pragma unroll
        for (int k = 0; k < VW; ++k) o[k] = fma(beta, pp[k], rp[k]);
        if (owned && xupd) {
          VT xv = xs ? *xs : *vat(a.xsol, zb, off);
          T* xp = reinterpret_cast<T*>(&xv);
#pragma unroll
          for (int k = 0; k < VW; ++k) xp[k] = fma(alpha, pp[k], xp[k]);
          *vat(a.xsol, zb, off) = xv;
        }
      }
      if (owned) *vat(a.p_out, zb, off) = out;
      return out;
    }
  };

  // Per-thread vectors of the vector path, fixed over the march: box rows
  // (boff: offset in a plane of the global arrays, bsi: in a ring slot), the
  // y-face rows (yoff) and the x-face elements (xoff); -1 = none.  Rows and
  // slots follow one another unpadded, so vector v of a buffer lies at v VW.
  constexpr int HV = HS / VW;                                  // vectors per x-face element
  constexpr int NBV = (PE * NPE) / VW;                         // box vectors of a plane
  constexpr int KP = (NBV + THREADS - 1) / THREADS;
  constexpr int KY = (2 * RV + THREADS - 1) / THREADS;
  constexpr int KX = (2 * TY * HV + THREADS - 1) / THREADS;
  constexpr unsigned NONE = ~0u;
  unsigned boff[KP], yoff[KY], xoff[KX];
#pragma unroll
  for (int k = 0; k < KP; ++k) {
    const int v = threadIdx.x + k * THREADS;
    boff[k] = NONE;
    if (vec && v < VY * RV) {
      const int row = v / RV, i = v - row * RV;
      boff[k] = (((oy + row) * nx + ox) * NPE + i * VW) * (unsigned)sizeof(T);
    }
  }
#pragma unroll
  for (int k = 0; k < KY; ++k) {
    const int v = threadIdx.x + k * THREADS;
    yoff[k] = NONE;
    if (vec && v < 2 * RV) {
      const int side = v / RV, i = v - side * RV;
      int gy = side ? oy + VY : oy - 1;
      gy = gy < 0 ? gy + ny : (gy >= ny ? gy - ny : gy);
      yoff[k] = ((gy * nx + ox) * NPE + i * VW) * (unsigned)sizeof(T);
    }
  }
#pragma unroll
  for (int k = 0; k < KX; ++k) {
    const int v = threadIdx.x + k * THREADS;
    xoff[k] = NONE;
    if (vec && v < 2 * TY * HV) {
      const int s = v / HV, j = v - s * HV;
      const int sy = s < TY ? s : s - TY;
      if (sy < VY) {
        int gx = s < TY ? ox - 1 : ox + VX;
        gx = gx < 0 ? gx + nx : (gx >= nx ? gx - nx : gx);
        const int ge = (oy + sy) * nx + gx;
        xoff[k] = ((s < TY ? (ge + 1) * NPE - HS : ge * NPE) + j * VW) * (unsigned)sizeof(T);
      }
    }
  }

  const int v0 = threadIdx.x * VW;
  constexpr int VS = THREADS * VW;
  // box of plane iz (relative to z0) into dst; owned iff 0 <= iz < NZ.  HOW 0
  // loads the values; 1 starts copies of r (x) and, in CG, p_old into dst and
  // extra; 2 completes a started box in CG (p, the writes of owned nodes).
  // The thread that completes a value is the one that started its copy.
  VT xv[KP];
  auto load_x = [&](int iz) {
    if (vec && xupd && iz < NZ) {
#pragma unroll
      for (int k = 0; k < KP; ++k)
        if (boff[k] != NONE) xv[k] = *vat(a.xsol, (size_t)wrapz(z0 + iz) * plane, boff[k]);
    }
  };
  auto load_plane = [&](int iz, T* dst, auto how) {
    constexpr int HOW = decltype(how)::value;
    const int z = wrapz(z0 + iz);
    const bool owned = iz >= 0 && iz < NZ;
    T* ex = ONE ? extra + (dst - ring) : extra;
    if (vec) {
      const size_t zb = (size_t)z * plane;
#pragma unroll
      for (int k = 0; k < KP; ++k) {
        if (boff[k] == NONE) continue;
        const int si = v0 + k * VS;
        if constexpr (HOW == 1) {
          copy_async(dst + si, vat(a.x, zb, boff[k]));
          if (fuse && !first) copy_async(ex + si, vat(a.p_old, zb, boff[k]));
        } else {
          VT rk;
          VT* at = reinterpret_cast<VT*>(dst + si);
          VT* po = reinterpret_cast<VT*>(ex + si);
          *at = stage_vec(zb, boff[k], owned, &rk, HOW == 2 ? at : nullptr, HOW == 2 ? po : nullptr, HOW == 2 ? xv + k : nullptr);
          if constexpr (ONE) {
            if (owned) *po = rk;
          }
        }
      }
      return;
    }
    if constexpr (HOW != 1) {
      for (int v = threadIdx.x; v < PE * NPE; v += THREADS) {
        const int s = v / NPE, q = v - s * NPE;
        const int sx = s % TX, sy = s / TX;
        if (sx >= VX || sy >= VY) continue;
        const long long ge = ((long long)z * ny + (oy + sy)) * nx + (ox + sx);
        const size_t gi = (size_t)ge * NPE + q;
        const int si = s * ES + m3_sidx<N1>(q);
        T rk = T(0);
        dst[si] = stage(gi, owned, &rk);
        if constexpr (ONE) {
          if (owned) ex[si] = rk;
        }
      }
    }
  };
  // x and y face halo of plane iz into dst: x-halo slots [0, TY) x = -1,
  // [TY, 2 TY) x = VX; then y-halo slots [0, TX) y = -1, [TX, 2 TX) y = VY
  auto load_halo = [&](int iz, T* dst, auto how) {
    constexpr int HOW = decltype(how)::value;
    const int z = wrapz(z0 + iz);
    // one vector: plane at zb, byte off in it, place si in a halo buffer
    auto vec1 = [&](size_t zb, unsigned off, int si) {
      if constexpr (HOW == 1) {
        copy_async(dst + si, vat(a.x, zb, off));
        if (fuse && !first) copy_async(hpo + si, vat(a.p_old, zb, off));
      } else {
        VT rk;
        VT* at = reinterpret_cast<VT*>(dst + si);
        *at = stage_vec(zb, off, false, &rk, HOW == 2 ? at : nullptr, HOW == 2 ? reinterpret_cast<VT*>(hpo + si) : nullptr, nullptr);
      }
    };
    if (vec) {
      const size_t zb = (size_t)z * plane;
#pragma unroll
      for (int k = 0; k < KY; ++k)
        if (yoff[k] != NONE) vec1(zb, yoff[k], 2 * TY * HS + v0 + k * VS);
#pragma unroll
      for (int k = 0; k < KX; ++k)
        if (xoff[k] != NONE) vec1(zb, xoff[k], v0 + k * VS);
      return;
    }
    if constexpr (HOW != 1) {
      for (int v = threadIdx.x; v < HALO * NPE; v += THREADS) {
        const int s = v / NPE, q = v - s * NPE;
        int sx, sy, so;
        if (s < 2 * TY) {
          sy = s < TY ? s : s - TY;
          sx = s < TY ? -1 : VX;
          if (sy >= VY) continue;
          so = s * HS;
        } else {
          const int u = s - 2 * TY;
          sx = u < TX ? u : u - TX;
          sy = u < TX ? -1 : VY;
          if (sx >= VX) continue;
          so = 2 * TY * HS + u * ES;
        }
        int gx = ox + sx, gy = oy + sy;
        gx = gx < 0 ? gx + nx : (gx >= nx ? gx - nx : gx);
        gy = gy < 0 ? gy + ny : (gy >= ny ? gy - ny : gy);
        const size_t gi = (size_t)(((long long)z * ny + gy) * nx + gx) * NPE + q;
        const int si = so + m3_sidx<N1>(q);
        T rk;
        dst[si] = stage(gi, false, &rk);
      }
    }
  };
  constexpr std::integral_constant<int, 0> LOAD{};
  constexpr std::integral_constant<int, 1> START{};
  constexpr std::integral_constant<int, 2> FINISH{};

  // reductions: p.Ap (fuse 1, compensated); ONE: p.Ap, r.r (compensated), r.Ap, Ap.Ap
  T s_pa = T(0), c_pa = T(0), s_rr = T(0), c_rr = T(0), s_ra = T(0), s_aa = T(0);
  auto reduce = [&](T y, T pv, T r) {
    const T t1 = fma(pv, y, -c_pa);
    const T u1 = s_pa + t1;
    c_pa = (u1 - s_pa) - t1;
    s_pa = u1;
    if constexpr (ONE) {
      const T t2 = fma(r, r, -c_rr);
      const T u2 = s_rr + t2;
      c_rr = (u2 - s_rr) - t2;
      s_rr = u2;
      s_ra = fma(r, y, s_ra);
      s_aa = fma(y, y, s_aa);
    }
  };
  // y = sum of the accumulators of plane iz, stored; reduced in CG modes
  auto store_plane = [&](int iz, const T* cur) {
    const int z = z0 + iz;
    const T* rk = extra + (cur - ring);  // ONE
    if (vec) {
      const size_t zb = (size_t)z * plane;
#pragma unroll
      for (int k = 0; k < KP; ++k) {
        if (boff[k] == NONE) continue;
        const int si = v0 + k * VS;
        VT yv = *reinterpret_cast<const VT*>(s_out + si);
        const VT y1 = *reinterpret_cast<const VT*>(s_out + PE * ES + si);
        T* yw = reinterpret_cast<T*>(&yv);
        const T* a1 = reinterpret_cast<const T*>(&y1);
        VT y2;
        if constexpr (!AHEAD) y2 = *reinterpret_cast<const VT*>(s_out + 2 * PE * ES + si);
        const T* a2 = reinterpret_cast<const T*>(&y2);
#pragma unroll
        for (int m = 0; m < VW; ++m) yw[m] += AHEAD ? a1[m] : a1[m] + a2[m];
        *vat(a.y, zb, boff[k]) = yv;
        if constexpr (fuse) {
          const VT pv4 = *reinterpret_cast<const VT*>(cur + si);
          const T* pp = reinterpret_cast<const T*>(&pv4);
          VT rv4;
          if constexpr (ONE) rv4 = *reinterpret_cast<const VT*>(rk + si);
          const T* rp = reinterpret_cast<const T*>(&rv4);
#pragma unroll
          for (int m = 0; m < VW; ++m) reduce(yw[m], pp[m], ONE ? rp[m] : T(0));
        }
      }
      return;
    }
    if constexpr (!AHEAD) {
      for (int v = threadIdx.x; v < PE * NPE; v += THREADS) {
        const int s = v / NPE, q = v - s * NPE;
        const int sx = s % TX, sy = s / TX;
        if (sx >= VX || sy >= VY) continue;
        const long long ge = ((long long)z * ny + (oy + sy)) * nx + (ox + sx);
        const int si = s * ES + m3_sidx<N1>(q);
        const T y = (s_out[PE * ES + si] + s_out[2 * PE * ES + si]) + s_out[si];
        a.y[(size_t)ge * NPE + q] = y;
        if constexpr (fuse) reduce(y, cur[si], ONE ? rk[si] : T(0));
      }
    }
  };

  // this thread's line in each direction: offset of its first node in a plane
  // of the ring (o) and of the neighbour elements' lines (l, r: in the same
  // plane, or, complemented, in the face halo)
  const int t = threadIdx.x;
  const int te = t / LINES, lam = t - te * LINES;
  const int lx = te % TX, ly = te / TX;
  const int q0 = lam % N1, q1 = lam / N1;
  int o0 = te * ES + q0 * RS + q1 * PS, o1 = te * ES + q0 + q1 * PS, o2 = te * ES + q0 + q1 * RS;
  int l0 = lx > 0 ? o0 - ES : ~(o0 - te * ES + ly * HS + loff);
  int r0 = lx + 1 < VX ? o0 + ES : ~(o0 - te * ES + (TY + ly) * HS);
  int l1 = ly > 0 ? o1 - TX * ES : ~(o1 - te * ES + 2 * TY * HS + lx * ES);
  int r1 = ly + 1 < VY ? o1 + TX * ES : ~(o1 - te * ES + 2 * TY * HS + (TX + lx) * ES);
  if (lx >= VX || ly >= VY) o0 = -1;  // no line
  const T wp = a.w[q0] * a.w[q1];
  // opaque to the compiler, which would otherwise form them anew for every
  // line from threadIdx (a quarter of all instructions) to save registers
  // (FP32; the FP64 kernels wait for the FP64 pipe and would spill)
  if constexpr (sizeof(T) == 4) {
    keep(o0), keep(o1), keep(o2), keep(l0), keep(r0), keep(l1), keep(r1);
#pragma unroll
    for (int k = 0; k < KP; ++k) keep(boff[k]);
#pragma unroll
    for (int k = 0; k < KY; ++k) keep(yoff[k]);
#pragma unroll
    for (int k = 0; k < KX; ++k) keep(xoff[k]);
  }

  // one pass: this thread's line along d of plane cur (pm, pp: the planes
  // below and above, hx: the plane's face halo)
  auto pass = [&](auto dir, const T* pm, const T* cur, const T* pp, const T* hx) {
    constexpr int d = decltype(dir)::value;
    if (o0 < 0) return;
    constexpr int stride = d == 0 ? 1 : d == 1 ? RS : PS;
    const int o = d == 0 ? o0 : d == 1 ? o1 : o2;
    const T* pc = cur + o;
    const T *pl, *pr;
    if constexpr (d == 2) {
      pl = pm + o;
      pr = pp + o;
    } else {
      const int l = d == 0 ? l0 : l1, r = d == 0 ? r0 : r1;
      pl = l >= 0 ? cur + l : hx + ~l;
      pr = r >= 0 ? cur + r : hx + ~r;
    }
    T xl[N1], xc[N1], xr[N1];
#pragma unroll
    for (int k = 0; k < N1; ++k) {
      xl[k] = pl[k * stride];
      xc[k] = pc[k * stride];
      xr[k] = pr[k * stride];
    }
    T val[N1];
    line_apply<T, N1, ACC>(a.c, xl, xc, xr, a.s[d] * wp, val);
    T* out = s_out + (d == 1 ? PE * ES : d == 0 && !AHEAD ? 2 * PE * ES : 0) + o;
#pragma unroll
    for (int m = 0; m < N1; ++m) {
      T v = val[m];
      if (d == 0) {
        if (a.cmass != T(0)) v = fma(a.cmass * wp * a.w[m], xc[m], v);
        if constexpr (AHEAD) v += out[m];
      }
      out[m * stride] = v;
    }
  };

  // March: planes iz - 1, iz, iz + 1 are in the ring when plane iz is
  // computed.  The z lines come first: then the plane iz - 1 is done with,
  // and the copies of plane iz + 2 into its place run while the x and y lines
  // are computed, those of the next face halo from the start of the plane.
  constexpr int SL = PE * ES;
  load_plane(-1, ring, LOAD);
  load_plane(0, ring + SL, LOAD);
  load_plane(1, ring + 2 * SL, LOAD);
  load_halo(0, halo, LOAD);
  __syncthreads();
  T *pm = ring, *cur = ring + SL, *pp = ring + 2 * SL;
  T* hx = halo;
  T* hn = L::HB == 2 ? halo + L::HALO_SZ : halo;  // halo of the next plane
  for (int iz = 0; iz < NZ; ++iz) {
    const bool more = iz + 1 < NZ;  // uniform over the CTA
    if constexpr (AHEAD) {
      if (more) load_halo(iz + 1, hn, START);
    }
    pass(std::integral_constant<int, 2>{}, pm, cur, pp, hx);
    if constexpr (AHEAD) {
      __syncthreads();
      if (more) load_plane(iz + 2, pm, START);
    }
    pass(std::integral_constant<int, 0>{}, pm, cur, pp, hx);
    pass(std::integral_constant<int, 1>{}, pm, cur, pp, hx);
    if constexpr (AHEAD && MODE == 1) {
      if (more) load_x(iz + 2);
    }
    __syncthreads();
    store_plane(iz, cur);
    if (more) {
      copy_async_wait();
      if constexpr (!AHEAD) load_plane(iz + 2, pm, LOAD);
      else if constexpr (fuse) load_plane(iz + 2, pm, FINISH);
      if constexpr (!AHEAD) load_halo(iz + 1, hn, LOAD);
      else if constexpr (fuse) load_halo(iz + 1, hn, FINISH);
      __syncthreads();
    }
    T* t0 = pm;
    pm = cur;
    cur = pp;
    pp = t0;
    t0 = hx;
    hx = hn;
    hn = t0;
  }

  if constexpr (!fuse) {
  } else if constexpr (ONE) {
    double tot[4];
    bool last;
    if constexpr (sizeof(T) == 4) {
      F2 v4[4] = {F2{(float)s_pa, -(float)c_pa}, F2{(float)s_rr, -(float)c_rr}, F2{(float)s_ra, 0.0f},
                  F2{(float)s_aa, 0.0f}};
      last = grid_sum_f2<4>(v4, a.partials, &a.st->counter, tot);
    } else {
      double v4[4] = {(double)s_pa - (double)c_pa, (double)s_rr - (double)c_rr, (double)s_ra, (double)s_aa};
      last = grid_sum<4>(v4, a.partials, &a.st->counter, tot);
    }
    if (last && threadIdx.x == 0) cg_iteration_finish(a.st, tot[0], tot[1], tot[2], tot[3]);
  } else {
    // the block's p.Ap total for the update launch, which forms alpha
    __shared__ double s_opr[32];
    if constexpr (sizeof(T) == 4) op_partial_f2(F2{(float)s_pa, -(float)c_pa}, a.partials, s_opr);
    else op_partial_f64((double)s_pa - (double)c_pa, a.partials, s_opr);
    if (blockIdx.x == 0 && threadIdx.x == 0) a.st->nop = (int)gridDim.x;
  }
}

// z-run length: the shortest runs whose CTAs all fit on the GPU at once
// (slots = SMs x resident CTAs per SM), so that the launch is one wave; at
// least 2 planes per run (fewer only on grids with fewer planes)
inline int march3_zc(int ntx, int nty, int nz, long long slots) {
  const long long cols = (long long)ntx * nty;
  if (slots < 1) slots = 1;
  long long zc = (nz * cols + slots - 1) / slots;
  if (zc < 2) zc = 2;
  if (zc > nz) zc = nz;
  return (int)zc;
}

template <typename T, int N1, bool ACC, int MODE, bool AHEAD>
cudaError_t launch_apply3m(const sdg_handle* h, const ApplyArgs<T>& in, cudaStream_t stream) {
  using M = March3<N1>;
  ApplyParams<T, 3, N1> p;
  fill_apply_params<T, 3, N1>(h, in, &p);
  const size_t smem = (size_t)March3Smem<T, N1, MODE, AHEAD>::SZ * sizeof(T);
  // resident CTAs per SM of this instantiation (fixed: threads and shared
  // memory do not depend on the grid), asked once per device
  static PerDevice occ_of;
  int occ = occ_of.get(h->device);
  if (occ == 0) {
    cudaError_t e = cudaFuncSetAttribute(k_apply3m<T, N1, ACC, MODE, AHEAD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_apply3m<T, N1, ACC, MODE, AHEAD>, M::THREADS, smem);
    if (e != cudaSuccess) return e;
    if (occ < 1) occ = 1;
    occ_of.set(h->device, occ);
  }
  p.ntile[0] = (p.n[0] + M::TX - 1) / M::TX;
  p.ntile[1] = (p.n[1] + M::TY - 1) / M::TY;
  p.zc = march3_zc(p.ntile[0], p.ntile[1], p.n[2], (long long)h->nsm * occ);
  p.ntile[2] = (p.n[2] + p.zc - 1) / p.zc;
  const long long nblk = (long long)p.ntile[0] * p.ntile[1] * p.ntile[2];
  if (nblk > h->max_blocks) return cudaErrorInvalidConfiguration;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)nblk);
  cfg.blockDim = dim3(M::THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = in.pdl ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, k_apply3m<T, N1, ACC, MODE, AHEAD>, p);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

// 3D dispatch for small degrees: the marching kernel for every mode
template <typename T, int N1>
cudaError_t launch_apply3m_t(const sdg_handle* h, const ApplyArgs<T>& in, cudaStream_t stream) {
  if (in.fuse == 2) return launch_apply3m<T, N1, true, 2, false>(h, in, stream);
  if constexpr (sizeof(T) == 4 && N1 % 2 == 1) {
    // planes copied ahead: whole vectors everywhere (see March3Smem)
    const long long plane = (long long)h->g.n[0] * h->g.n[1] * March3<N1>::NPE;
    if (h->g.n[0] % VecOf<T>::W == 0 && plane * (long long)sizeof(T) < (1LL << 32)) {
      if (in.fuse == 1) return launch_apply3m<T, N1, true, 1, true>(h, in, stream);
      return launch_apply3m<T, N1, true, 0, true>(h, in, stream);
    }
  }
  if (in.fuse == 1) return launch_apply3m<T, N1, true, 1, false>(h, in, stream);
  if (sizeof(T) == 8 && !in.accurate) return launch_apply3m<T, N1, false, 0, false>(h, in, stream);
  return launch_apply3m<T, N1, true, 0, false>(h, in, stream);
}

}  // namespace sdg
