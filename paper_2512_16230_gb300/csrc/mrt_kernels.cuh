// The per-cell MRT collision in the Hermite basis and the fused pull collide-stream kernel.
//
// One thread owns one cell (k_step) or, from 80,000 cells in FP32 and 16-bit storage, two neighbouring ones
// (k_step_pair). It gathers the Q populations of its cells from the neighbours
// x - e_i of the previous step (pull form of the propagation, Eq. (2-2b)), collides them
// (Eq. (2-3) with the Hermite-moment collision Eq. (H-MRT-LB-1)) and writes the post-collision
// populations back at its own cells (aligned, coalesced stores). The stored array is therefore
// the post-collision state of the last step; the pre-collision f-bar(x, t_n) of the paper is
// its pull-gather.
//
// The collision is evaluated in the reduced form that Eq. (H-MRT-LB-1) gives when every row
// of order >= 4 relaxes with one rate s_h:
//   f*_i = (1 - s_h) f_i + w_i sum_{r<R} H_ri / N_r [ s_h m^eq_r - (s_r - s_h)(m_r - m^eq_r)
//                                                     + sigma_r ],
// because the W-orthogonal complement of span(H0..H3) carries the same rate in every row.
// The two contractions with the Hermite matrix are factored through the monomials of the integer
// velocities (raw_moments and back_project: small integers known at compile time, so zero products
// vanish, the +-e pairs share one pass and the directions that differ by reflections share their
// sums), and through the rows' few entries below the diagonal (collide_moments). Everything is in
// lattice units: the axis speeds sit in the constants (LatTables, Rates).
//
// What bounds it: HBM on large FP32 grids, the arithmetic and its latency elsewhere (k_step_pair has the counters),
// and the FP64 pipe (2 FMAs per clock and SM) in FP64. The shared sums, the scaled rows and s_h = 1 without the old
// populations take rD3Q53 from about 830 to 600 FP32 operations per cell; whole solves on GB300:
// rD2Q25 64x48 FP64 x 100 steps 1424 -> 996 us, rD3Q33 64^3 FP32 x 64 816 -> 693 us, rD2Q13
// 1024x768 FP32 x 100 1361 -> 1190 us, rD3Q53 256x256x192 x 24 FP32 21.8 -> 20.4 ms and FP16
// 16.4 -> 13.9 ms.
#pragma once

#include <algorithm>

#include "lbm_internal.cuh"

// Tuning knobs of k_step, one cell per thread, which runs FP64, grids below 80,000 cells and the steps without a
// collision, and of the batched kernel's blocks (k_step_pair has its own block counts, pair_blocks). 4 blocks
// of 128 threads per SM leave 128 registers. Measured best while it ran every grid, rD3Q53 256x256x192, FP32 / FP16 ms
// a step with 4 blocks 0.833 / 0.686, with 5 (96 registers) 0.883 / 0.732, with 6 0.989 / 0.756; evict-first loads or
// stores were slower. (k_step_pair takes 0.759 / 0.44 there.)
//   LBM_K1_MIN_BLOCKS  minimum resident blocks per SM requested through __launch_bounds__
//   LBM_K1_LOAD        1: evict-first (__ldcs), 2: plain load. The read-only path (ld.global.nc) is
//                      not offered: a chained launch starts while the kernel that writes its input
//                      still runs, so the input is not constant over the launch's lifetime and a
//                      read-only load could be moved above the wait for that kernel.
//   LBM_K1_STORE       0: plain store, 1: evict-first streaming store (__stcs)
#ifndef LBM_K1_MIN_BLOCKS
#define LBM_K1_MIN_BLOCKS 4
#endif
#ifndef LBM_K1_LOAD
#define LBM_K1_LOAD 2
#endif
#ifndef LBM_K1_STORE
#define LBM_K1_STORE 0
#endif

namespace lbm {

template <class T>
__device__ __forceinline__ T k1_load(const T* p) {
#if LBM_K1_LOAD == 1
  return __ldcs(p);
#else
  return *p;
#endif
}

template <class T>
__device__ __forceinline__ void k1_store(T* p, T v) {
#if LBM_K1_STORE == 1
  __stcs(p, v);
#else
  *p = v;
#endif
}

template <class CT>
__device__ __forceinline__ CT fmaf_t(CT a, CT b, CT c) {
  if constexpr (std::is_same<CT, F2>::value) return fma2(a, b, c);
  else return fma(a, b, c);
}

// a b where the product's only use is in a sum. The assembler fuses a packed product into the packed
// addition that takes it, whatever the rounding modifiers say, and would round once where the scalar
// kernels round twice; a multiply-add with zero is not fused. (For every product it costs registers:
// rD3Q53 FP16 256x256x192 448 -> 472 us a step.)
template <class V>
__device__ __forceinline__ V product(V a, V b) {
  if constexpr (std::is_same<V, F2>::value) return fma2(a, b, F2(0.f));
  else return a * b;
}

// acc + c * x for a compile-time integer c
template <int C, class CT>
__device__ __forceinline__ CT axpy_c(CT x, CT acc) {
  if constexpr (C == 1) return acc + x;
  else if constexpr (C == -1) return acc - x;
  else return fmaf_t(CT(C), x, acc);
}

// Sums of one primitive direction d: s_deg = sum_m m^deg (f_md +- f_-md), + for even degree, - for
// odd (m = 1 is on every lattice).
template <class V>
struct DirSums {
  V s0, s1, s2, s3;
};
template <class L, int DX, int DY, int DZ, class V>
__device__ __forceinline__ DirSums<V> dir_sums(const V (&f)[L::Q]) {
  constexpr Vel d{DX, DY, DZ};
  const V p1 = f[velocity_index<L>(d, 1)] + f[velocity_index<L>(d, -1)];
  const V m1 = f[velocity_index<L>(d, 1)] - f[velocity_index<L>(d, -1)];
  DirSums<V> r{p1, m1, p1, m1};
  static_for<2>([&](auto mm) {
    constexpr int M = decltype(mm)::value + 2;
    constexpr int ip = velocity_index<L>(d, M), im = velocity_index<L>(d, -M);
    if constexpr (ip >= 0) {
      const V sp = f[ip] + f[im];
      const V sm = f[ip] - f[im];
      r.s0 = r.s0 + sp;
      r.s1 = axpy_c<M>(sm, r.s1);
      r.s2 = axpy_c<M * M>(sp, r.s2);
      r.s3 = axpy_c<M * M * M>(sm, r.s3);
    }
  });
  return r;
}

// Signed sums of four values over (sign along b, sign along g) = ++, +-, -+, --: the plain sum, the
// sums signed by b, by g and by both (8 additions for the four).
template <class V>
struct Signed4 {
  V s, b, g, bg;
};
template <class V>
__device__ __forceinline__ Signed4<V> signed4(V pp, V pm, V mp, V mm) {
  const V a0 = pp + pm, a1 = pp - pm, c0 = mp + mm, c1 = mp - mm;
  return Signed4<V>{a0 + c0, a0 - c0, a1 + c1, a1 - c1};
}

// Raw moments mu_k = sum_i mono_k(e_i) f_i, k < R. The directions of one plane (1, 1), (1, -1) and the
// four space diagonals enter the monomials with the same magnitude and a sign, so their signed sums
// are formed once: for rD3Q53 104 operations in dir_sums and 88 here, against 152 with one
// multiply-add per direction and monomial.
template <class L, class V>
__device__ __forceinline__ void raw_moments_2d(V f0, const DirSums<V>& X, const DirSums<V>& Y, const DirSums<V>& P,
                                               const DirSums<V>& M, V (&mu)[L::R]) {
  mu[0] = (f0 + (X.s0 + Y.s0)) + (P.s0 + M.s0);
  mu[1] = X.s1 + (P.s1 + M.s1);
  mu[2] = Y.s1 + (P.s1 - M.s1);
  const V d2 = P.s2 + M.s2, o3 = P.s3 + M.s3, q3 = P.s3 - M.s3;
  mu[row2<2>(0, 0)] = X.s2 + d2;
  mu[row2<2>(1, 1)] = Y.s2 + d2;
  mu[row2<2>(0, 1)] = P.s2 - M.s2;
  mu[row3<2>(0, 1, 1)] = o3;
  mu[row3<2>(0, 0, 1)] = q3;
  if constexpr (!L::SINGLE) {
    mu[row3<2>(0, 0, 0)] = X.s3 + o3;
    mu[row3<2>(1, 1, 1)] = Y.s3 + q3;
  }
}

template <class L, class V>
__device__ __forceinline__ void raw_moments(const V (&f)[L::Q], V (&mu)[L::R]) {
  constexpr int D = L::D;
  if constexpr (D == 2) {
    raw_moments_2d<L>(f[0], dir_sums<L, 1, 0, 0>(f), dir_sums<L, 0, 1, 0>(f), dir_sums<L, 1, 1, 0>(f),
                      dir_sums<L, 1, -1, 0>(f), mu);
  } else {
    const DirSums<V> ax[3] = {dir_sums<L, 1, 0, 0>(f), dir_sums<L, 0, 1, 0>(f), dir_sums<L, 0, 0, 1>(f)};
    // space diagonals (1, +-1, +-1)
    const DirSums<V> pp = dir_sums<L, 1, 1, 1>(f), pm = dir_sums<L, 1, 1, -1>(f);
    const DirSums<V> mp = dir_sums<L, 1, -1, 1>(f), mm = dir_sums<L, 1, -1, -1>(f);
    const V c0 = (pp.s0 + pm.s0) + (mp.s0 + mm.s0);
    const Signed4<V> c2 = signed4(pp.s2, pm.s2, mp.s2, mm.s2), c3 = signed4(pp.s3, pm.s3, mp.s3, mm.s3);
    const V c1[3] = {(pp.s1 + pm.s1) + (mp.s1 + mm.s1), (pp.s1 + pm.s1) - (mp.s1 + mm.s1),
                     (pp.s1 - pm.s1) + (mp.s1 - mm.s1)};
    const V c3a[3] = {c3.s, c3.b, c3.g};
    const V c2ab[3] = {c2.b, c2.g, c2.bg};  // planes xy, xz, yz
    V m0 = f[0] + c0, m1[3], m2[3], m3[3];
    static_for<3>([&](auto aa) {
      constexpr int A = decltype(aa)::value;
      m0 = m0 + ax[A].s0;
      m1[A] = ax[A].s1 + c1[A];
      m2[A] = ax[A].s2 + c2.s;
      m3[A] = ax[A].s3;
    });
    // planes (a, b): e_a + e_b and e_a - e_b
    static_for<3>([&](auto pl) {
      constexpr int PL = decltype(pl)::value;
      constexpr int A = PL == 2 ? 1 : 0, B = PL == 0 ? 1 : 2;
      const DirSums<V> P = dir_sums<L, A == 0, (A == 1) + (B == 1), B == 2>(f);
      const DirSums<V> M = dir_sums<L, A == 0, (A == 1) - (B == 1), -(B == 2)>(f);
      const V d2 = P.s2 + M.s2, o3 = P.s3 + M.s3, q3 = P.s3 - M.s3;
      m0 = m0 + (P.s0 + M.s0);
      m1[A] = m1[A] + (P.s1 + M.s1);
      m1[B] = m1[B] + (P.s1 - M.s1);
      m2[A] = m2[A] + d2;
      m2[B] = m2[B] + d2;
      mu[row2<3>(A, B)] = (P.s2 - M.s2) + c2ab[PL];
      const V abb = o3 + c3a[A], baa = q3 + c3a[B];
      mu[row3<3>(A, B, B)] = abb;
      mu[row3<3>(B, A, A)] = baa;
      // a cube takes both planes of its axis and the space diagonals once (in its first plane)
      constexpr bool firstA = PL == 0, firstB = PL <= 1;
      m3[A] = m3[A] + (firstA ? abb : o3);
      m3[B] = m3[B] + (firstB ? baa : q3);
    });
    mu[0] = m0;
    static_for<3>([&](auto aa) {
      constexpr int A = decltype(aa)::value;
      mu[1 + A] = m1[A];
      mu[row2<3>(A, A)] = m2[A];
      if constexpr (!L::SINGLE) mu[row3<3>(A, A, A)] = m3[A];
    });
    mu[row3<3>(0, 1, 2)] = c3.bg;
  }
}

// The two populations of a direction at every speed m present:
// f_{+-md} = (1 - s_h) f_{+-md} + w (E_0 + m^2 E_2 +- m (E_1 + m^2 E_3)), E_deg = sum_{deg(k) = deg}
// mono_k(d) h_k. KEEP = false: s_h = 1, the old populations drop out.
template <class L, int DX, int DY, int DZ, bool KEEP, class V>
__device__ __forceinline__ void dir_out(V (&f)[L::Q], const LatTables<V>& lt, V oms, V E0, V E1, V E2, V E3) {
  constexpr Vel d{DX, DY, DZ};
  static_for<3>([&](auto mi) {
    constexpr int M = decltype(mi)::value + 1;
    constexpr int ip = velocity_index<L>(d, M), im = velocity_index<L>(d, -M);
    if constexpr (ip >= 0) {
      const V we = lt.w[ip] * axpy_c<M * M>(E2, E0);
      V odd = E1;
      if constexpr (!(L::SINGLE && iabs(DX) + iabs(DY) + iabs(DZ) == 1)) odd = axpy_c<M * M>(E3, E1);
      if constexpr (KEEP) {
        f[ip] = fmaf_t(oms, f[ip], fmaf_t(lt.wm[ip], odd, we));
        f[im] = fmaf_t(oms, f[im], fmaf_t(lt.wm[im], odd, we));
      } else {
        f[ip] = fmaf_t(lt.wm[ip], odd, we);
        f[im] = fmaf_t(lt.wm[im], odd, we);
      }
    }
  });
}

// The populations of one direction of a 2D lattice: W = 0 (1, 0) and the rest, 1 (0, 1), 2 (1, 1), 3 (1, -1).
template <class L, bool KEEP, int W, class V>
__device__ __forceinline__ void back_direction_2d(V (&f)[L::Q], const LatTables<V>& lt, const V (&h)[L::R], V oms) {
  const V h0 = h[0];
  if constexpr (W == 0) {
    if constexpr (KEEP) f[0] = fmaf_t(oms, f[0], lt.w[0] * h0);
    else f[0] = lt.w[0] * h0;
  }
  if constexpr (W < 2) {
    V cube = V(0.f);
    if constexpr (!L::SINGLE) cube = h[row3<2>(W, W, W)];
    dir_out<L, W == 0, W == 1, 0, KEEP>(f, lt, oms, h0, h[1 + W], h[row2<2>(W, W)], cube);
  } else {
    V ox = h[row3<2>(0, 1, 1)], oy = h[row3<2>(0, 0, 1)];
    if constexpr (!L::SINGLE) {
      ox = h[row3<2>(0, 0, 0)] + ox;
      oy = h[row3<2>(1, 1, 1)] + oy;
    }
    const V s2 = h[row2<2>(0, 0)] + h[row2<2>(1, 1)], m = h[row2<2>(0, 1)];
    if constexpr (W == 2) dir_out<L, 1, 1, 0, KEEP>(f, lt, oms, h0, h[1] + h[2], s2 + m, ox + oy);
    else dir_out<L, 1, -1, 0, KEEP>(f, lt, oms, h0, h[1] - h[2], s2 - m, ox - oy);
  }
}

// f_i = (1 - s_h) f_i + w_i sum_k mono_k(e_i) h_k, with the sums of raw_moments transposed.
template <class L, bool KEEP, class V>
__device__ __forceinline__ void back_project(V (&f)[L::Q], const LatTables<V>& lt, const V (&h)[L::R], V oms) {
  constexpr int D = L::D;
  if constexpr (D == 2) {
    static_for<4>([&](auto w) { back_direction_2d<L, KEEP, decltype(w)::value>(f, lt, h, oms); });
  } else {
    const V h0 = h[0];
    if constexpr (KEEP) f[0] = fmaf_t(oms, f[0], lt.w[0] * h0);
    else f[0] = lt.w[0] * h0;
    V cube[3];
    static_for<3>([&](auto aa) {
      constexpr int A = decltype(aa)::value;
      if constexpr (L::SINGLE) cube[A] = V(0.f);
      else cube[A] = h[row3<3>(A, A, A)];
      dir_out<L, A == 0, A == 1, A == 2, KEEP>(f, lt, oms, h0, h[1 + A], h[row2<3>(A, A)], cube[A]);
    });
    V t3[3];  // per axis: cube + both mixed rows
    static_for<3>([&](auto pl) {
      constexpr int PL = decltype(pl)::value;
      constexpr int A = PL == 2 ? 1 : 0, B = PL == 0 ? 1 : 2;
      const V abb = h[row3<3>(A, B, B)], baa = h[row3<3>(B, A, A)];
      V oa = abb, ob = baa;
      if constexpr (!L::SINGLE) {
        oa = cube[A] + abb;
        ob = cube[B] + baa;
      }
      const V s2 = h[row2<3>(A, A)] + h[row2<3>(B, B)], m = h[row2<3>(A, B)];
      dir_out<L, A == 0, (A == 1) + (B == 1), B == 2, KEEP>(f, lt, oms, h0, h[1 + A] + h[1 + B], s2 + m, oa + ob);
      dir_out<L, A == 0, (A == 1) - (B == 1), -(B == 2), KEEP>(f, lt, oms, h0, h[1 + A] - h[1 + B], s2 - m, oa - ob);
      if constexpr (PL == 0) {
        t3[0] = oa;
        t3[1] = ob;
      } else if constexpr (PL == 1) {
        t3[0] = t3[0] + abb;
        t3[2] = ob;
      } else {
        t3[1] = t3[1] + abb;
        t3[2] = t3[2] + baa;
      }
    });
    const V S = (h[row2<3>(0, 0)] + h[row2<3>(1, 1)]) + h[row2<3>(2, 2)];
    // over the signs (along y, along z): ++, +-, -+, --
    const Signed4<V> e2 = signed4(S, h[row2<3>(0, 1)], h[row2<3>(0, 2)], h[row2<3>(1, 2)]);
    const Signed4<V> e3 = signed4(t3[0], t3[1], t3[2], h[row3<3>(0, 1, 2)]);
    const V xy = h[1] + h[2], xmy = h[1] - h[2];
    dir_out<L, 1, 1, 1, KEEP>(f, lt, oms, h0, xy + h[3], e2.s, e3.s);
    dir_out<L, 1, 1, -1, KEEP>(f, lt, oms, h0, xy - h[3], e2.b, e3.b);
    dir_out<L, 1, -1, 1, KEEP>(f, lt, oms, h0, xmy + h[3], e2.g, e3.g);
    dir_out<L, 1, -1, -1, KEEP>(f, lt, oms, h0, xmy - h[3], e2.bg, e3.bg);
  }
}

// h_k = sum_{r >= k} T'_rk gN_r: the coefficients of the monomials from those of the rows.
template <class L, class V>
__device__ __forceinline__ void rows_to_monomials(const LatTables<V>& lt, const V (&gN)[L::R], V (&h)[L::R]) {
  constexpr int D = L::D;
  h[0] = gN[0];
  static_for<D>([&](auto aa) {
    constexpr int A = decltype(aa)::value;
    h[0] = fmaf_t(lt.nd0[A], gN[row2<D>(A, A)], h[0]);
    h[row2<D>(A, A)] = gN[row2<D>(A, A)];
    h[1 + A] = gN[1 + A];
    if constexpr (!L::SINGLE) {
      const V g3 = gN[row3<D>(A, A, A)];
      h[row3<D>(A, A, A)] = g3;
      h[1 + A] = fmaf_t(lt.l3[A], g3, h[1 + A]);
    }
    static_for<D - 1>([&](auto ii) {
      constexpr int I = decltype(ii)::value, B = other_axis(A, I);
      V g = gN[row3<D>(A, B, B)];
      if constexpr (!L::SINGLE) g = fmaf_t(lt.be[A][I], gN[row3<D>(A, A, A)], g);
      h[row3<D>(A, B, B)] = g;
      h[1 + A] = fmaf_t(lt.nd0[B], g, h[1 + A]);
      if constexpr (B > A) h[row2<D>(A, B)] = gN[row2<D>(A, B)];
    });
  });
  if constexpr (D == 3) h[row3<3>(0, 1, 2)] = gN[row3<3>(0, 1, 2)];
}

// Hermite moments of the NSE equilibrium in the scaled rows, from rho, j'_a = rho u'_a and u'_a. The
// continuous moments (Eq. (M-NSEs-6a), Eq. (M-NSEs-6-1) with k = 0, M30 = rho u u u, p = rho cs2_eq)
// are M2 = j u + p I and M3 = j u u + p (u delta)_sym, which gives in the rows
//   aa: rho (u'_a^2 + q_a)   ab: j'_a u'_b   abb: u'_a m_bb   abg: j'_a u'_b u'_g
//   aaa: u'_a rho (u'_a^2 + k3_a) + be_a0 m_abb + be_a1 m_agg.
// Single-speed lattices (k = 1) take M30 = 0: abb: j'_a q_b, abg: 0, no cubes. cub[a] is the part of
// the cube row before the be terms.
template <class L, class V>
__device__ __forceinline__ void eq_rows_nse(const LatTables<V>& lt, const Rates<V>& rt, V rho, const V (&j)[3],
                                            const V (&u)[3], V (&me)[L::R], V (&cub)[3]) {
  constexpr int D = L::D;
  me[0] = rho;
  static_for<D>([&](auto aa) {
    constexpr int A = decltype(aa)::value;
    me[1 + A] = j[A];
    me[row2<D>(A, A)] = fmaf_t(j[A], u[A], rho * rt.q[A]);
  });
  static_for<D>([&](auto aa) {
    constexpr int A = decltype(aa)::value;
    static_for<D - 1>([&](auto ii) {
      constexpr int I = decltype(ii)::value, B = other_axis(A, I);
      if constexpr (B > A) me[row2<D>(A, B)] = j[A] * u[B];
      if constexpr (L::SINGLE) me[row3<D>(A, B, B)] = j[A] * rt.q[B];
      else me[row3<D>(A, B, B)] = u[A] * me[row2<D>(B, B)];
    });
    if constexpr (!L::SINGLE) {
      cub[A] = u[A] * fmaf_t(j[A], u[A], rho * rt.k3[A]);
      V v = cub[A];
      static_for<D - 1>([&](auto ii) {
        constexpr int I = decltype(ii)::value, B = other_axis(A, I);
        v = fmaf_t(lt.be[A][I], me[row3<D>(A, B, B)], v);
      });
      me[row3<D>(A, A, A)] = v;
    }
  });
  if constexpr (D == 3) {
    if constexpr (L::SINGLE) me[row3<3>(0, 1, 2)] = V(0.f);
    else me[row3<3>(0, 1, 2)] = me[row2<3>(0, 1)] * u[2];
  }
}

// D(phi) = phi + nonlin phi^3 / 3 and the second-order normal row of the NCDE equilibrium (Eq.
// (M-NCDE-6), M20 = 0): M0 = phi, M1 = u phi, M2 = cs2_eq D(phi) I; third-order moments zero.
template <class V>
__device__ __forceinline__ V ncde_flux(const Rates<V>& rt, V phi) {
  return fmaf_t(rt.nonlin_third, phi * phi * phi, phi);
}

// One collision (Eq. (2-3)) of the populations f of one cell, in place.
// F: body force at the cell (NSE); phi_prev / phi_now: the NCDE field at t_{n-1} and t_n.
// DEV: f holds deviations f - w rho_ref (16-bit storage). The moments of the reference state are
// added back (only 1 and the squares c_a^2 have non-zero lattice moments), and the update
// f* - w rho_ref = (1 - s_h)(f - w rho_ref) + w H(h) - s_h w rho_ref folds the last term into h_0.

// The collision in moment space: from the raw moments mu_k = sum_i mono_k(e_i) f_i (k < R) to
// the monomial-basis coefficients h of the update f*_i = (1 - s_h) f_i + w_i sum_k mono_k(e_i) h_k.
// Per row gN_r = [s_h m^eq_r - (s_r - s_h)(m_r - m^eq_r) + sigma_r] / N'_r, where on the normal
// second-order rows the d x d block S_n takes the place of s_r (it carries the bulk coupling of
// Eq. (4-27)). sigma: NSE (1 - s/2) F on order 1 and M2G = (I - S2/2)(uF + Fu) on order 2, plus, given
// gr (single-speed lattices), the diagonal (delta4 . u) . grad rho of Eq. (M2Ga); NCDE M1G =
// (I - S1/2) u d_t phi - S1 A1 d_t(u phi) on order 1, minus S1 A2 grad psi given gr (Eq. (M-NCDE-6),
// D-bar = psi I), and, for the CDE variant, M0G = (1 - s0/2) S_G on order 0. The conserved rows of the
// NSE are exact: with j = mu_a + F/2 the first-order row is s_h mu_a + F whatever its own rate.
// F: the body force over c_a (read only when forced); phi_now receives phi (NCDE) or rho (NSE).
template <class L, class V, int EQ, bool DEV>
__device__ __forceinline__ void collide_moments(V (&mu)[L::R], const LatTables<V>& lt, const Rates<V>& rt, bool forced,
                                                const V (&F)[3], V phi_prev, V& phi_now, V (&h)[L::R],
                                                const V* gr = nullptr) {
  constexpr int R = L::R, D = L::D;
  if constexpr (DEV) {
    mu[0] = mu[0] + lt.wmr[0];
    static_for<D>([&](auto a) {
      constexpr int A = decltype(a)::value;
      mu[row2<D>(A, A)] = mu[row2<D>(A, A)] + lt.wmr[1 + A];
    });
  }
  V gN[R], me[R], neq[R];
  // FP32: A mu, the momentum's own part of the first-order rows, is added last. The force and what the third-order
  // rows add are a few units in its last place. Added to it one after the other, each would be rounded the same
  // way at every step, a drift of the momentum (u = 0.04: rD3Q45 and the cubic rD3Q53 -4.2e-8 a step, so -0.4e-8 ..
  // 0.2e-8).
  constexpr bool LAST = EQ == LBM_NSE && !std::is_same<V, double>::value;
  if constexpr (EQ == LBM_NSE) {
    // Eq. (2-4-2) with S = 0, F_F = F: rho = sum f, rho u = sum c f + F / 2
    const V rho = mu[0];
    const V inv = V(1.f) / rho;
    phi_now = rho;
    V j[3], u[3], cub[3];
    static_for<D>([&](auto a) {
      constexpr int A = decltype(a)::value;
      j[A] = mu[1 + A];
      if (forced) j[A] = fmaf_t(V(0.5f), F[A], j[A]);
      u[A] = j[A] * inv;
    });
    eq_rows_nse<L>(lt, rt, rho, j, u, me, cub);
    gN[0] = rt.A[0] * rho;
    static_for<D>([&](auto a) {
      constexpr int A = decltype(a)::value;
      if constexpr (LAST) {
        gN[1 + A] = V(0.f);
      } else {
        gN[1 + A] = rt.A[1 + A] * mu[1 + A];
        if (forced) gN[1 + A] = fmaf_t(lt.iN[1 + A], F[A], gN[1 + A]);
      }
      constexpr int AA = row2<D>(A, A);
      neq[AA] = fmaf_t(lt.nd0[A], rho, mu[AA]) - me[AA];
    });
    static_for<D>([&](auto a) {
      constexpr int A = decltype(a)::value;
      static_for<D - 1>([&](auto ii) {
        constexpr int I = decltype(ii)::value, B = other_axis(A, I), ABB = row3<D>(A, B, B);
        if constexpr (B > A) neq[row2<D>(A, B)] = mu[row2<D>(A, B)] - me[row2<D>(A, B)];
        neq[ABB] = fmaf_t(lt.nd0[B], mu[1 + A], mu[ABB]) - me[ABB];
      });
      if constexpr (!L::SINGLE) {
        constexpr int AAA = row3<D>(A, A, A);
        V v = fmaf_t(lt.l3[A], mu[1 + A], mu[AAA]) - cub[A];
        static_for<D - 1>([&](auto ii) {
          constexpr int I = decltype(ii)::value, B = other_axis(A, I);
          v = fmaf_t(lt.be[A][I], neq[row3<D>(A, B, B)], v);
        });
        neq[AAA] = v;
      }
    });
    if constexpr (D == 3) neq[row3<3>(0, 1, 2)] = mu[row3<3>(0, 1, 2)] - me[row3<3>(0, 1, 2)];
    static_for<R>([&](auto r) {
      constexpr int Rr = decltype(r)::value;
      if constexpr (degree(mono<D>(Rr)) >= 2) {
        constexpr int na = normal_index<D>(Rr);
        V g = rt.A[Rr] * me[Rr];
        if constexpr (na >= 0) {
          static_for<D>([&](auto b) {
            constexpr int B = decltype(b)::value;
            g = fmaf_t(rt.NBn[na][B], neq[row2<D>(B, B)], g);
          });
        } else {
          g = fmaf_t(rt.NB[Rr], neq[Rr], g);
        }
        gN[Rr] = g;
      }
    });
    if (forced || gr != nullptr) {
      if (LAST && forced) {
        static_for<D>([&](auto a) {
          constexpr int A = decltype(a)::value;
          gN[1 + A] = product(lt.iN[1 + A], F[A]);
        });
      }
      V t[3];
      static_for<D>([&](auto b) {
        constexpr int B = decltype(b)::value;
        V v = V(0.f);
        if (forced) v = F[B] + F[B];
        if (gr != nullptr) v = v + gr[B];
        t[B] = u[B] * v;
      });
      static_for<D>([&](auto a) {
        constexpr int A = decltype(a)::value;
        static_for<D>([&](auto b) {
          constexpr int B = decltype(b)::value;
          gN[row2<D>(A, A)] = fmaf_t(rt.Cn[A][B], t[B], gN[row2<D>(A, A)]);
          if constexpr (B > A) {
            constexpr int AB = row2<D>(A, B);
            if (forced) gN[AB] = fmaf_t(rt.C[AB], fmaf_t(u[A], F[B], u[B] * F[A]), gN[AB]);
          }
        });
      });
    }
  } else {
    // Eq. (2-4-1) with S = 0: phi = sum f (+ S_G / 2, lambda = 1, for the CDE variant)
    V phi = mu[0], sg = V(0.f);
    if (rt.ncde_variant == LBM_NCDE_CDE) {
      // S_G = -u . grad phi with grad_a phi = -s_a M1_a^ne / cs2 (M1 = 0)
      static_for<D>([&](auto a) {
        constexpr int A = decltype(a)::value;
        sg = fmaf_t(rt.cde_coef[A], mu[1 + A], sg);
      });
      phi = fmaf_t(V(0.5f), sg, phi);
    }
    phi_now = phi;
    const V dphi = phi - phi_prev;
    const V Dphi = ncde_flux(rt, phi);
    gN[0] = rt.A[0] * phi;
    if (rt.ncde_variant == LBM_NCDE_CDE) gN[0] = gN[0] + fmaf_t(rt.NB[0], mu[0] - phi, rt.half0 * sg);
    static_for<D>([&](auto a) {
      constexpr int A = decltype(a)::value;
      const V m1 = rt.u_const[A] * phi;
      const V n1 = mu[1 + A] - m1;
      V s1 = rt.s1[A];
      if (rt.ncde_variant == LBM_NCDE_RATE) {
        // s_a(phi) = 1 / ((1/s_a - 1/2)(1 + nonlin phi^2) + 1/2)
        const V g = fmaf_t(rt.nonlin_rate, phi * phi, V(1.f));
        s1 = V(1.f) / fmaf_t(rt.kfac[A], g, V(0.5f));
        const V half1 = V(1.f) - product(s1, V(0.5f) + rt.a1);
        const V relax = product(s1 - rt.s_high, n1);
        gN[1 + A] = lt.iN[1 + A] * (fmaf_t(rt.s_high, m1, half1 * (rt.u_const[A] * dphi)) - relax);
      } else {
        gN[1 + A] = fmaf_t(rt.A[1 + A], m1, fmaf_t(rt.NB[1 + A], n1, rt.h1[A] * dphi));
      }
      if (gr != nullptr) gN[1 + A] = gN[1 + A] - product(lt.iN[1 + A], s1 * gr[A]);
      constexpr int AA = row2<D>(A, A);
      me[AA] = fmaf_t(rt.pc[A], Dphi, lt.nd0[A] * phi);
      neq[AA] = fmaf_t(lt.nd0[A], mu[0], mu[AA]) - me[AA];
    });
    static_for<D>([&](auto a) {
      constexpr int A = decltype(a)::value, AA = row2<D>(A, A);
      V g = rt.A[AA] * me[AA];
      static_for<D>([&](auto b) {
        constexpr int B = decltype(b)::value;
        if constexpr (B == A) g = fmaf_t(rt.NBn[A][A], neq[AA], g);  // no bulk block in the NCDE
      });
      gN[AA] = g;
      static_for<D - 1>([&](auto ii) {
        constexpr int I = decltype(ii)::value, B = other_axis(A, I), ABB = row3<D>(A, B, B);
        if constexpr (B > A) gN[row2<D>(A, B)] = product(rt.NB[row2<D>(A, B)], mu[row2<D>(A, B)]);
        neq[ABB] = fmaf_t(lt.nd0[B], mu[1 + A], mu[ABB]);
        gN[ABB] = product(rt.NB[ABB], neq[ABB]);
      });
      if constexpr (!L::SINGLE) {
        constexpr int AAA = row3<D>(A, A, A);
        V v = fmaf_t(lt.l3[A], mu[1 + A], mu[AAA]);
        static_for<D - 1>([&](auto ii) {
          constexpr int I = decltype(ii)::value, B = other_axis(A, I);
          v = fmaf_t(lt.be[A][I], neq[row3<D>(A, B, B)], v);
        });
        gN[AAA] = product(rt.NB[AAA], v);
      }
    });
    if constexpr (D == 3) gN[row3<3>(0, 1, 2)] = product(rt.NB[row3<3>(0, 1, 2)], mu[row3<3>(0, 1, 2)]);
  }
  rows_to_monomials<L>(lt, gN, h);
  if constexpr (LAST) {  // (A to twice the precision: a rounded factor would be a bias of every step)
    static_for<D>([&](auto a) {
      constexpr int A = decltype(a)::value;
      h[1 + A] = fmaf_t(rt.A[1 + A], mu[1 + A], fmaf_t(rt.Alo[A], mu[1 + A], h[1 + A]));
    });
  }
  if constexpr (DEV) h[0] = h[0] - rt.sh_rho_ref;
}

// KEEP = false: every row of order >= 4 relaxes with s_h = 1 (the default), so that f* depends on the
// moments alone and the populations need not stay in registers through the collision.
template <class L, class V, int EQ, bool DEV, bool KEEP>
__device__ __forceinline__ void collide(V (&f)[L::Q], const LatTables<V>& lt, const Rates<V>& rt, bool forced,
                                        const V (&F)[3], V phi_prev, V& phi_now, const V* gr = nullptr) {
  V mu[L::R];
  raw_moments<L>(f, mu);
  V h[L::R];
  collide_moments<L, V, EQ, DEV>(mu, lt, rt, forced, F, phi_prev, phi_now, h, gr);
  back_project<L, KEEP>(f, lt, h, rt.one_minus_sh);
}

// Equilibrium populations of given fields, Eq. (feq-1): f^eq_i = w_i sum_r H_ri m^eq_r / N_r
// (u: the velocity over c_a).
template <class L, class V, int EQ>
__device__ __forceinline__ void equilibrium(V (&f)[L::Q], const LatTables<V>& lt, const Rates<V>& rt, V rho_or_phi,
                                            const V (&u)[3]) {
  constexpr int R = L::R, D = L::D;
  V me[R];
  static_for<R>([&](auto r) { me[decltype(r)::value] = V(0.f); });
  if constexpr (EQ == LBM_NSE) {
    V j[3], cub[3];
    static_for<D>([&](auto a) { j[decltype(a)::value] = rho_or_phi * u[decltype(a)::value]; });
    eq_rows_nse<L>(lt, rt, rho_or_phi, j, u, me, cub);
  } else {
    const V phi = rho_or_phi;
    const V Dphi = ncde_flux(rt, phi);
    me[0] = phi;
    static_for<D>([&](auto a) {
      constexpr int A = decltype(a)::value;
      me[1 + A] = rt.u_const[A] * phi;
      me[row2<D>(A, A)] = fmaf_t(rt.pc[A], Dphi, lt.nd0[A] * phi);
    });
  }
  V gN[R];
  static_for<R>([&](auto r) {
    constexpr int Rr = decltype(r)::value;
    gN[Rr] = me[Rr] * lt.iN[Rr];
  });
  V h[R];
  rows_to_monomials<L>(lt, gN, h);
  back_project<L, false>(f, lt, h, V(0.f));
}

}  // namespace lbm

#include "high.cuh"

namespace lbm {

// Cell coordinates and periodic neighbour offsets.
template <class L>
struct Neigh {
  static constexpr int RM = L::RMAX;
  int xo[2 * RM + 1], yo[2 * RM + 1], zo[2 * RM + 1];
  int x, y, z;
  template <class CT>
  __device__ __forceinline__ Neigh(int cell, const StepParams<CT>& p) : Neigh(cell, p.n, p.div_m, p.div_s) {}
  __device__ __forceinline__ Neigh(int cell, const int (&n)[3], const unsigned (&div_m)[2], const int (&div_s)[2]) {
    const int nx = n[0], ny = n[1];
    // the velocity components are at most RM <= every extent, so one wrap suffices and only on
    // the side a displacement can cross
    const int t = int(__umulhi(unsigned(cell), div_m[0]) >> div_s[0]);
    x = cell - t * nx;
    if constexpr (L::D == 2) {
      y = t;
      z = 0;
    } else {
      z = int(__umulhi(unsigned(t), div_m[1]) >> div_s[1]);
      y = t - z * ny;
    }
#pragma unroll
    for (int s = -RM; s <= RM; ++s) {
      xo[s + RM] = wrap1(x - s, s, nx);
      yo[s + RM] = wrap1(y - s, s, ny) * nx;
      if constexpr (L::D == 3) zo[s + RM] = wrap1(z - s, s, n[2]) * nx * ny;
      else zo[s + RM] = 0;
    }
  }
  __device__ __forceinline__ static int wrap1(int v, int s, int n) {
    if (s > 0) return v < 0 ? v + n : v;
    if (s < 0) return v >= n ? v - n : v;
    return v;
  }
  // cell index of x - e (pull source) for a compile-time velocity
  template <int I>
  __device__ __forceinline__ int src() const {
    constexpr Vel v = L::e(I);
    return xo[RM + v.x] + yo[RM + v.y] + (L::D == 3 ? zo[RM + v.z] : 0);
  }
};

// Body force over c_a at a cell; false (and F unset) without one.
template <class CT>
__device__ __forceinline__ bool body_force(int force_a, int force_b, const CT* force_tab, const CT (&invc)[3], int x,
                                           int y, int z, CT (&F)[3]) {
  if (force_b < 0) return false;
  const int ib = force_b == 0 ? x : (force_b == 1 ? y : z);
  const CT v = force_tab[ib];
  F[0] = force_a == 0 ? v * invc[0] : CT(0);
  F[1] = force_a == 1 ? v * invc[1] : CT(0);
  F[2] = force_a == 2 ? v * invc[2] : CT(0);
  return true;
}

// The same for two cells.
__device__ __forceinline__ bool body_force(int force_a, int force_b, const float* force_tab, const F2 (&invc)[3],
                                           const int (&c0)[3], const int (&c1)[3], F2 (&F)[3]) {
  if (force_b < 0) return false;
  const F2 v(force_tab[force_b == 0 ? c0[0] : (force_b == 1 ? c0[1] : c0[2])],
             force_tab[force_b == 0 ? c1[0] : (force_b == 1 ? c1[1] : c1[2])]);
  F[0] = force_a == 0 ? v * invc[0] : F2(0.f);
  F[1] = force_a == 1 ? v * invc[1] : F2(0.f);
  F[2] = force_a == 2 ? v * invc[2] : F2(0.f);
  return true;
}

// Gradient terms of the source moments: the delta4 term of M2G (Eq. (M2Ga)) on the single-speed
// lattices needs grad rho, the cross-diffusion term of M1G (Eq. (M-NCDE-6)) grad psi. Both take
// gr_a = gscale_a (g(x + e_a) - g(x - e_a)), the central difference of the cell field p.grad_in at
// the periodic neighbours of cell (x, y, z); nullptr when the term is off.
template <class L, int EQ>
struct GradTerm {
  static constexpr bool kOn = (L::SINGLE && EQ == LBM_NSE) || EQ == LBM_NCDE;
};
template <class L, class CT>
__device__ __forceinline__ void field_differences(const int (&n)[3], const CT* g, int cell, int x, int y, int z,
                                                  CT (&d)[3]) {
  const int nx = n[0], ny = n[1];
  const int xp = x + 1 == nx ? -x : 1, xm = x == 0 ? nx - 1 : -1;
  d[0] = g[cell + xp] - g[cell + xm];
  const int yp = (y + 1 == ny ? -y : 1) * nx, ym = (y == 0 ? ny - 1 : -1) * nx;
  d[1] = g[cell + yp] - g[cell + ym];
  if constexpr (L::D == 3) {
    const int nz = n[2], nxy = nx * ny;
    const int zp = (z + 1 == nz ? -z : 1) * nxy, zm = (z == 0 ? nz - 1 : -1) * nxy;
    d[2] = g[cell + zp] - g[cell + zm];
  }
}
template <class L, class CT>
__device__ __forceinline__ const CT* cell_field_gradient(const Rates<CT>& p, const int (&n)[3], const CT* g, int cell,
                                                         int x, int y, int z, CT (&gr)[3]) {
  if (!p.grad_on) return nullptr;
  field_differences<L>(n, g, cell, x, y, z, gr);
  static_for<L::D>([&](auto a) { gr[decltype(a)::value] = p.gscale[decltype(a)::value] * gr[decltype(a)::value]; });
  return gr;
}
// The same for two cells, the second one following the first in memory.
template <class L>
__device__ __forceinline__ const F2* cell_field_gradient(const Rates<F2>& p, const int (&n)[3], const float* g,
                                                         int cell, const int (&c0)[3], const int (&c1)[3],
                                                         F2 (&gr)[3]) {
  if (!p.grad_on) return nullptr;
  float d0[3], d1[3];
  field_differences<L>(n, g, cell, c0[0], c0[1], c0[2], d0);
  field_differences<L>(n, g, cell + 1, c1[0], c1[1], c1[2], d1);
  static_for<L::D>([&](auto a) {
    constexpr int A = decltype(a)::value;
    gr[A] = p.gscale[A] * F2(d0[A], d1[A]);
  });
  return gr;
}

// K1 (COLLIDE) / K2 (stream only): pull gather, collide, aligned store.
template <class L, class CT, class ST, int EQ, bool COLLIDE, bool KEEP>
__global__ void __launch_bounds__(kBlock, LBM_K1_MIN_BLOCKS) k_step(const StepParams<CT> p, const ST* fin, ST* fout,
                                                                        CT* phi) {
  chain_release_if(p.release, kReleaseFirst);
  const int cell = blockIdx.x * kBlock + threadIdx.x;
  if (cell >= p.ncells) return;
  const Neigh<L> nb(cell, p);
  chain_wait();
  chain_release_if(p.release, kReleaseAfterWait);
  const size_t N = size_t(p.ncells);
  CT f[L::Q];
  constexpr bool DEV = is_deviation_storage<ST>();
  static_for<L::Q>([&](auto i) {
    constexpr int I = decltype(i)::value;
    if constexpr (DEV) f[I] = RawCodec<ST>::dec(k1_load(fin + size_t(I) * N + nb.template src<I>()));
    else f[I] = Codec<ST>::dec(k1_load(fin + size_t(I) * N + nb.template src<I>()), p.wref[I]);
  });
  if constexpr (COLLIDE) {
    CT F[3];
    const bool forced = body_force(p.force_a, p.force_b, p.force_tab, p.invc, nb.x, nb.y, nb.z, F);
    CT phi_prev = CT(0), phi_now = CT(0);
    if constexpr (EQ == LBM_NCDE) phi_prev = phi[cell];
    constexpr bool AG = GradTerm<L, EQ>::kOn;
    CT gr[3];
    const CT* grad = nullptr;
    if constexpr (AG) grad = cell_field_gradient<L>(p, p.n, p.grad_in, cell, nb.x, nb.y, nb.z, gr);
    collide<L, CT, EQ, DEV, KEEP>(f, p, p, forced, F, phi_prev, phi_now, grad);
    if constexpr (EQ == LBM_NCDE) phi[cell] = phi_now;
    if constexpr (AG && EQ == LBM_NSE) {
      if (p.grad_on) p.rho_out[cell] = phi_now;
    }
  }
  chain_release_if(p.release, kReleaseLast);
  static_for<L::Q>([&](auto i) {
    constexpr int I = decltype(i)::value;
    if constexpr (DEV) k1_store(fout + size_t(I) * N + cell, RawCodec<ST>::enc(f[I]));
    else k1_store(fout + size_t(I) * N + cell, Codec<ST>::enc(f[I], p.wref[I]));
  });
}

// Two 16-bit values in one word, decoded.
template <class ST>
__device__ __forceinline__ F2 dec_word(uint32_t b) {
  if constexpr (std::is_same<ST, __half>::value) {
    const float2 v = __half22float2(*reinterpret_cast<const __half2*>(&b));
    return F2(v.x, v.y);
  } else {
    return F2(__uint_as_float(b << 16), __uint_as_float(b & 0xFFFF0000u));
  }
}
template <class ST>
__device__ __forceinline__ uint32_t enc_word(float a, float b) {
  uint32_t r;
  if constexpr (std::is_same<ST, __half>::value) {
    const __half2 h = __floats2half2_rn(a, b);
    r = *reinterpret_cast<const uint32_t*>(&h);
  } else {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    r = *reinterpret_cast<const uint32_t*>(&h);
  }
  return r;
}

// K1 on two neighbouring cells per thread in packed FP32 arithmetic (f32x2.cuh), for FP32 and 16-bit
// storage: bitwise the populations of k_step. EVEN: n_x is even, the cells are (x, x + 1) of one row
// with x even; an even e_x is one load of both sources, the stores are pairs. Otherwise the cells are
// 2 t and 2 t + 1 of the array and every access is by cell (the last cell of an odd grid is done alone).
//
// What bounds it: HBM on large FP32 grids; elsewhere memory, the FMA pipe and latency at 11 to 15 warps per SM
// together (busy on rD3Q53, DRAM / heavy FMA pipe / issue: FP16 256x256x96 74 / 69 / 50%, BF16 on odd rows 56 / 48 /
// 50%, FP32 with per-order rates 63 / 41 / 42%). Packing halves the FP32 instructions. us a step on GB300, one cell / two cells per thread: rD2Q13 1024x768 FP32 11.5 / 8.8, rD3Q33 64^3 FP32
// 10.2 / 8.4, rD3Q53 256x256x192 FP32 776 / 759, rD3Q53 150x131x147 BF16 153 / 111, rD3Q45 101x103x97
// FP32 62.8 / 57.5. 4 blocks per SM leave 128 registers; on rD3Q53 the single accesses spill at that, with 3
// blocks 81^3 FP32 takes 39.0 us (one cell per thread 40.0) and 149x131x147 BF16 139 us (156). s_h != 1
// (KEEP) holds the old populations as well: 3 blocks, spilling a little, against 2 without: rD3Q53 256x128x96
// FP32 218 -> 198, FP16 168 -> 136, rD3Q45 FP32 187 -> 165, FP16 148 -> 114.
//
// HI: with the operator of the higher rows (hc). FP32 storage waits for memory and takes one block per SM
// more than 16-bit storage, at about 290 bytes of spills a thread on rD3Q53 (they stay in L1); 16-bit storage is bound
// by issue (96 bytes of spills on even rows of rD3Q53), and its blocks stay resident, so that each stages the operator once. us a
// step, with 2, 3, 4 blocks per SM (Q > 33, >= 27, below) / with one more: rD3Q53 160x144x120 FP32 245 / 232, FP16 202 /
// 225; rD3Q45 205 / 175, 159 / 169; rD2Q25 1024x768 26.5 / 25.5, 21.5 / 22.7. Blocks that stay resident: FP32 265 (245 with a block per 256 cells), FP16 202 (220). Also measured: the
// sources of the next two cells copied to shared memory meanwhile (cp.async, 64 threads, 4 blocks per SM): 311.
struct NoCoefs {};
template <class L, class ST>
constexpr int pair_high_blocks() {
  return (L::Q > 33 ? 2 : (L::Q >= 27 ? 3 : 4)) + (is_deviation_storage<ST>() ? 0 : 1);
}
template <class L, class ST, bool KEEP, bool EVEN, bool HI>
constexpr int pair_blocks() {
  if (HI) return pair_high_blocks<L, ST>();
  if (KEEP && L::Q > 33) return 3;
  return L::Q > 45 && (!EVEN || is_deviation_storage<ST>()) ? 3 : 4;
}
template <class L, class ST, int EQ, bool KEEP, bool EVEN, bool HI = false, bool LATE = false>
__global__ void __launch_bounds__(kBlock, pair_blocks<L, ST, KEEP, EVEN, HI>())
    k_step_pair(const StepParams<F2, float> p, const std::conditional_t<HI, HighCoefs<float>, NoCoefs> hc, const ST* fin,
                ST* fout, float* phi) {
  constexpr int Q = L::Q, RM = L::RMAX;
  constexpr bool DEV = is_deviation_storage<ST>();
  __shared__ std::conditional_t<HI, HighCoefs<float>, NoCoefs> coefs;
  if constexpr (HI) {
    stage_coefs<L>(coefs, hc);
    __syncthreads();
  }
  if constexpr (!LATE && EVEN) chain_release();
  const size_t N = size_t(p.ncells);
  auto step = [&](int cell) {
    const bool two = EVEN || cell + 1 < p.ncells;
    const Neigh<L> n0(cell, p.n, p.div_m, p.div_s);
    F2 f[Q];
    auto one = [&](const ST* a) -> float {
      if constexpr (DEV) return RawCodec<ST>::dec(k1_load(a));
      else return k1_load(a);
    };
    int c0[3] = {n0.x, n0.y, n0.z}, c1[3] = {n0.x + 1, n0.y, n0.z};
    if constexpr (EVEN) {
      // x positions of the second cell's sources; the first cell's for e_x = -RM .. RM are n0.xo
      int x1[2 * RM + 1];
#pragma unroll
      for (int sh = -RM; sh <= RM; ++sh) x1[sh + RM] = Neigh<L>::wrap1(n0.x + 1 - sh, sh == 0 ? 1 : sh, p.n[0]);
      chain_wait();
      static_for<Q>([&](auto i) {
        constexpr int I = decltype(i)::value;
        constexpr Vel v = L::e(I);
        const int yz = n0.yo[RM + v.y] + (L::D == 3 ? n0.zo[RM + v.z] : 0);
        const ST* a = fin + size_t(I) * N + (n0.xo[RM + v.x] + yz);
        if constexpr (v.x % 2 == 0) {
          if constexpr (DEV) f[I] = dec_word<ST>(*reinterpret_cast<const uint32_t*>(a));
          else f[I] = *reinterpret_cast<const F2*>(a);
        } else {
          f[I] = F2(one(a), one(fin + size_t(I) * N + (x1[RM + v.x] + yz)));
        }
      });
    } else {
      const Neigh<L> n1(two ? cell + 1 : cell, p.n, p.div_m, p.div_s);
      c1[0] = n1.x;
      c1[1] = n1.y;
      c1[2] = n1.z;
      chain_wait();
      if constexpr (!LATE) chain_release();
      static_for<Q>([&](auto i) {
        constexpr int I = decltype(i)::value;
        f[I] = F2(one(fin + size_t(I) * N + n0.template src<I>()), one(fin + size_t(I) * N + n1.template src<I>()));
      });
    }
    F2 F[3];
    const bool forced = body_force(p.force_a, p.force_b, p.force_tab, p.invc, c0, c1, F);
    F2 phi_prev(0.f), phi_now(0.f);
    if constexpr (EQ == LBM_NCDE) {
      if constexpr (EVEN) phi_prev = *reinterpret_cast<const F2*>(phi + cell);
      else phi_prev = F2(phi[cell], phi[two ? cell + 1 : cell]);
    }
    constexpr bool AG = GradTerm<L, EQ>::kOn;
    F2 gr[3];
    const F2* grad = nullptr;
    if constexpr (AG) {
      if (two) {
        grad = cell_field_gradient<L>(p, p.n, p.grad_in, cell, c0, c1, gr);
      } else if (p.grad_on) {
        float d[3];
        field_differences<L>(p.n, p.grad_in, cell, c0[0], c0[1], c0[2], d);
        static_for<L::D>([&](auto a) { gr[decltype(a)::value] = p.gscale[decltype(a)::value] * F2(d[decltype(a)::value]); });
        grad = gr;
      }
    }
    if constexpr (HI) collide_high<L, F2, EQ, DEV>(f, coefs.c, p, p, forced, F, phi_prev, phi_now, grad);
    else collide<L, F2, EQ, DEV, KEEP>(f, p, p, forced, F, phi_prev, phi_now, grad);
    float a, b;
    auto field_out = [&](float* g) {
      if constexpr (EVEN) {
        *reinterpret_cast<F2*>(g + cell) = phi_now;
      } else {
        phi_now.get(a, b);
        g[cell] = a;
        if (two) g[cell + 1] = b;
      }
    };
    if constexpr (EQ == LBM_NCDE) field_out(phi);
    if constexpr (AG && EQ == LBM_NSE) {
      if (p.grad_on) field_out(p.rho_out);
    }
    if constexpr (LATE) chain_release();
    static_for<Q>([&](auto i) {
      constexpr int I = decltype(i)::value;
      ST* o = fout + size_t(I) * N + cell;
      if constexpr (EVEN && !DEV) {
        *reinterpret_cast<F2*>(o) = f[I];
      } else {
        f[I].get(a, b);
        if constexpr (EVEN) {
          *reinterpret_cast<uint32_t*>(o) = enc_word<ST>(a, b);
        } else if constexpr (DEV) {
          k1_store(o, RawCodec<ST>::enc(a));
          if (two) k1_store(o + 1, RawCodec<ST>::enc(b));
        } else {
          k1_store(o, a);
          if (two) k1_store(o + 1, b);
        }
      }
    });
  };
  const int first = 2 * (blockIdx.x * kBlock + threadIdx.x);
  if constexpr (HI && DEV) {
    // (as many blocks as are resident: the operator is staged once by each)
    const int64_t stride = int64_t(2) * kBlock * gridDim.x;
    for (int64_t cell = first; cell < p.ncells; cell += stride) step(int(cell));
  } else {
    if (first < p.ncells) step(first);
  }
}

// K1 on a small 2D grid in FP64, four threads per cell. GB300 runs one FP64 warp instruction per 64
// clocks and SM sub-partition, whatever the number of active lanes, so a grid with fewer warps of cells
// than there are sub-partitions (608) takes the time of one cell's instructions on a few of them. Here warp
// W of a block owns direction W of 32 cells: it loads, sums and writes that direction's populations, the
// sums go through shared memory, warps 0 and 1 do the even and the odd rows of the moment-space part, and its
// result goes through shared memory too. Same operations in the same order as k_step, bitwise the same
// results. rD2Q25 64x48: 9.5 us per step with one thread per cell, 4.9 here, of which 1.9 is a launch in a
// chain; the longest chain is now the even or odd rows' (a quarter of the cell's operations each).
template <class L, int EQ, bool KEEP, int W>
__device__ __forceinline__ void split_direction(const StepParams<double>& p, const double* fin, double* fout,
                                                double* phi, const Neigh<L>& nb, int cell, bool live,
                                                double (&sums)[17][32], double (&coef)[10][32]) {
  constexpr int Q = L::Q;
  constexpr int DX = W != 1, DY = W == 0 ? 0 : (W == 3 ? -1 : 1);
  const int lane = threadIdx.x & 31;
  const size_t N = size_t(p.ncells);
  double f[Q];
  double phi_prev = 0.0, phi_now = 0.0;
  auto mine = [](int i) constexpr {
    return i == 0 ? W == 0 : same_vel(primitive(L::e(i)), Vel{DX, DY, 0});
  };
  if (live) {
    static_for<Q>([&](auto i) {
      constexpr int I = decltype(i)::value;
      if constexpr (mine(I)) f[I] = k1_load(fin + size_t(I) * N + nb.template src<I>());
    });
    if constexpr (EQ == LBM_NCDE) phi_prev = phi[cell];
    const DirSums<double> r = dir_sums<L, DX, DY, 0>(f);
    sums[4 * W][lane] = r.s0;
    sums[4 * W + 1][lane] = r.s1;
    sums[4 * W + 2][lane] = r.s2;
    sums[4 * W + 3][lane] = r.s3;
    if constexpr (W == 0) sums[16][lane] = f[0];
  }
  asm volatile("bar.sync 1, 128;" ::: "memory");  // one barrier for the block's four warps, each from its own code
  // W = 0: the coefficients of 1, aa, ab; W = 1: of a and the third order (what the other needs is dropped by
  // the compiler)
  auto mine_row = [](int r) constexpr { return (degree(mono<2>(r)) % 2 == 0) == (W == 0); };
  double h[L::R];
  if (W < 2 && live) {
    auto dir = [&](int d) {
      return DirSums<double>{sums[4 * d][lane], sums[4 * d + 1][lane], sums[4 * d + 2][lane], sums[4 * d + 3][lane]};
    };
    double mu[L::R], F[3], gr[3];
    raw_moments_2d<L>(sums[16][lane], dir(0), dir(1), dir(2), dir(3), mu);
    const bool forced = body_force(p.force_a, p.force_b, p.force_tab, p.invc, nb.x, nb.y, 0, F);
    constexpr bool AG = GradTerm<L, EQ>::kOn;
    const double* grad = nullptr;
    if constexpr (AG) grad = cell_field_gradient<L>(p, p.n, p.grad_in, cell, nb.x, nb.y, 0, gr);
    collide_moments<L, double, EQ, false>(mu, p, p, forced, F, phi_prev, phi_now, h, grad);
    if constexpr (W == 0 && EQ == LBM_NCDE) phi[cell] = phi_now;
    if constexpr (W == 0 && AG && EQ == LBM_NSE) {
      if (p.grad_on) p.rho_out[cell] = phi_now;
    }
    static_for<L::R>([&](auto r) {
      constexpr int Rr = decltype(r)::value;
      if constexpr (mine_row(Rr)) coef[Rr][lane] = h[Rr];
    });
  }
  asm volatile("bar.sync 1, 128;" ::: "memory");
  if (!live) return;
  static_for<L::R>([&](auto r) { h[decltype(r)::value] = coef[decltype(r)::value][lane]; });
  back_direction_2d<L, KEEP, W>(f, p, h, p.one_minus_sh);
  static_for<Q>([&](auto i) {
    constexpr int I = decltype(i)::value;
    if constexpr (mine(I)) k1_store(fout + size_t(I) * N + cell, f[I]);
  });
}

template <class L, int EQ, bool KEEP>
__global__ void __launch_bounds__(128) k_step_split(const StepParams<double> p, const double* fin, double* fout,
                                                    double* phi) {
  __shared__ double sums[17][32];  // per direction and degree, and the rest population
  __shared__ double coef[10][32];  // the coefficients of the monomials
  const int raw_cell = blockIdx.x * 32 + (threadIdx.x & 31);
  const bool live = raw_cell < p.ncells;
  const int cell = live ? raw_cell : p.ncells - 1;
  const Neigh<L> nb(cell, p);
  chain_wait();
  chain_release();
  switch (threadIdx.x >> 5) {
    case 0: split_direction<L, EQ, KEEP, 0>(p, fin, fout, phi, nb, cell, live, sums, coef); break;
    case 1: split_direction<L, EQ, KEEP, 1>(p, fin, fout, phi, nb, cell, live, sums, coef); break;
    case 2: split_direction<L, EQ, KEEP, 2>(p, fin, fout, phi, nb, cell, live, sums, coef); break;
    default: split_direction<L, EQ, KEEP, 3>(p, fin, fout, phi, nb, cell, live, sums, coef); break;
  }
}

// K1 with distinct rates for the orders >= 4: the same gather / collide / store with the operator of the
// higher rows (high.cuh), one cell per thread. Bound by issue and by too few warps to hide the loads: us a
// step of rD3Q53 160x144x120 FP32 with 3 / 4 / 5 blocks per SM 270 / 241 / 246 (4: 128 registers, 20 bytes
// spilled); the rows' two contractions instead of the operator took 555 (2.45 ms on 256x256x192).
template <class L, class CT, class ST, int EQ>
__global__ void __launch_bounds__(kBlock, std::is_same<CT, double>::value ? 2 : 4)
    k_step_high(const StepParams<CT> p, const HighCoefs<CT> hc, const ST* fin, ST* fout, CT* phi) {
  __shared__ HighCoefs<CT> coefs;
  stage_coefs<L>(coefs, hc);
  __syncthreads();
  const int cell = blockIdx.x * kBlock + threadIdx.x;
  if (cell >= p.ncells) return;
  const Neigh<L> nb(cell, p);
  chain_wait();
  chain_release();
  const size_t N = size_t(p.ncells);
  CT f[L::Q];
  constexpr bool DEV = is_deviation_storage<ST>();
  static_for<L::Q>([&](auto i) {
    constexpr int I = decltype(i)::value;
    if constexpr (DEV) f[I] = RawCodec<ST>::dec(k1_load(fin + size_t(I) * N + nb.template src<I>()));
    else f[I] = Codec<ST>::dec(k1_load(fin + size_t(I) * N + nb.template src<I>()), p.wref[I]);
  });
  CT F[3];
  const bool forced = body_force(p.force_a, p.force_b, p.force_tab, p.invc, nb.x, nb.y, nb.z, F);
  CT phi_prev = CT(0), phi_now = CT(0);
  if constexpr (EQ == LBM_NCDE) phi_prev = phi[cell];
  constexpr bool AG = GradTerm<L, EQ>::kOn;
  CT gr[3];
  const CT* grad = nullptr;
  if constexpr (AG) grad = cell_field_gradient<L>(p, p.n, p.grad_in, cell, nb.x, nb.y, nb.z, gr);
  collide_high<L, CT, EQ, DEV>(f, coefs.c, p, p, forced, F, phi_prev, phi_now, grad);
  if constexpr (EQ == LBM_NCDE) phi[cell] = phi_now;
  if constexpr (AG && EQ == LBM_NSE) {
    if (p.grad_on) p.rho_out[cell] = phi_now;
  }
  static_for<L::Q>([&](auto i) {
    constexpr int I = decltype(i)::value;
    if constexpr (DEV) k1_store(fout + size_t(I) * N + cell, RawCodec<ST>::enc(f[I]));
    else k1_store(fout + size_t(I) * N + cell, Codec<ST>::enc(f[I], p.wref[I]));
  });
}

// Initialisation: f-bar(t=0) = f^eq(fields), written to the stored array at x - e_i so that the
// next pull gather yields it; the NCDE previous-step field starts at phi^0, the previous-step
// density of the single-speed NSE (phi non-null) at rho^0.
template <class L, class CT, class ST, int EQ>
__global__ void __launch_bounds__(kBlock) k_init(const StepParams<CT> p, const double* rho_or_phi,
                                                 const double* u, ST* __restrict__ fout,
                                                 CT* __restrict__ phi) {
  const int cell = blockIdx.x * kBlock + threadIdx.x;
  if (cell >= p.ncells) return;
  const Neigh<L> nb(cell, p);
  const size_t N = size_t(p.ncells);
  const CT r = CT(rho_or_phi[cell]);
  CT uu[3] = {CT(0), CT(0), CT(0)};
  if constexpr (EQ == LBM_NSE) {
    for (int a = 0; a < L::D; ++a) uu[a] = CT(u[size_t(a) * N + cell]) * p.invc[a];
    if (phi != nullptr) phi[cell] = r;
  } else {
    phi[cell] = r;
  }
  CT f[L::Q];
  equilibrium<L, CT, EQ>(f, p, p, r, uu);
  static_for<L::Q>([&](auto i) {
    constexpr int I = decltype(i)::value;
    fout[size_t(I) * N + nb.template src<I>()] = Codec<ST>::enc(f[I], p.wref[I]);
  });
}

// K6: persistent batched collide-stream. The grid is the resident capacity of the GPU; each
// block walks the tile work-list of the group (tiles of BLOCK cells from every solve), stages
// the descriptor of the tile's solve in shared memory when it changes, and runs the same per-cell
// gather / collide / store as k_step.
template <int BLOCK>
constexpr int batch_min_blocks() {
  return BLOCK >= 256 ? 2 : (BLOCK >= 128 ? LBM_K1_MIN_BLOCKS : 10);
}

// One cell of a batched step: the same gather / collide / store as k_step, with the solve's
// parameters from its staged descriptor (HI: hc, the staged operator of a per-order-rate group).
template <class L, class CT, class ST, int EQ, bool KEEP, bool HI>
__device__ __forceinline__ void batch_cell(const LatTables<CT>& t, const SolveDesc<CT>& sd, int cell, int parity,
                                           const CT* hc) {
  const Neigh<L> nb(cell, sd.n, sd.div_m, sd.div_s);
  const size_t N = size_t(sd.ncells);
  const ST* fin = static_cast<const ST*>(sd.f[parity]);
  ST* fout = static_cast<ST*>(sd.f[parity ^ 1]);
  constexpr bool DEV = is_deviation_storage<ST>();
  CT f[L::Q];
  static_for<L::Q>([&](auto i) {
    constexpr int I = decltype(i)::value;
    if constexpr (DEV) f[I] = RawCodec<ST>::dec(k1_load(fin + size_t(I) * N + nb.template src<I>()));
    else f[I] = Codec<ST>::dec(k1_load(fin + size_t(I) * N + nb.template src<I>()), t.wref[I]);
  });
  CT F[3];
  const bool forced = body_force(sd.force_a, sd.force_b, sd.force_tab, t.invc, nb.x, nb.y, nb.z, F);
  CT phi_prev = CT(0), phi_now = CT(0);
  if constexpr (EQ == LBM_NCDE) phi_prev = sd.phi[cell];
  constexpr bool AG = GradTerm<L, EQ>::kOn;
  CT gr[3];
  const CT* grad = nullptr;
  if constexpr (AG) grad = cell_field_gradient<L>(sd, sd.n, sd.grad_in[parity], cell, nb.x, nb.y, nb.z, gr);
  if constexpr (HI) collide_high<L, CT, EQ, DEV>(f, hc, t, sd, forced, F, phi_prev, phi_now, grad);
  else collide<L, CT, EQ, DEV, KEEP>(f, t, sd, forced, F, phi_prev, phi_now, grad);
  if constexpr (EQ == LBM_NCDE) sd.phi[cell] = phi_now;
  if constexpr (AG && EQ == LBM_NSE) {
    if (sd.grad_on) sd.rho_out[parity][cell] = phi_now;
  }
  chain_release();  // of the block's first tile: before the stores, as a step of one wave
  static_for<L::Q>([&](auto i) {
    constexpr int I = decltype(i)::value;
    if constexpr (DEV) k1_store(fout + size_t(I) * N + cell, RawCodec<ST>::enc(f[I]));
    else k1_store(fout + size_t(I) * N + cell, Codec<ST>::enc(f[I], t.wref[I]));
  });
}

// Stage the descriptor of solve `solve` in shared memory (block-wide; call with the whole block).
template <class CT, int BLOCK>
__device__ __forceinline__ void stage_desc(SolveDesc<CT>& sd, const SolveDesc<CT>* descs, int solve) {
  constexpr int kWords = int(sizeof(SolveDesc<CT>) / sizeof(int4));
  static_assert(sizeof(SolveDesc<CT>) % sizeof(int4) == 0, "descriptor must be a whole number of int4");
  const int4* src = reinterpret_cast<const int4*>(descs + solve);
  int4* dst = reinterpret_cast<int4*>(&sd);
  for (int w = threadIdx.x; w < kWords; w += BLOCK) dst[w] = src[w];
}

template <class L, class CT, class ST, int EQ, int BLOCK, bool KEEP>
__global__ void __launch_bounds__(BLOCK, batch_min_blocks<BLOCK>())
    k_step_batch(const LatTables<CT> t, const SolveDesc<CT>* descs, const Tile* tiles, int ntiles, int parity) {
  __shared__ SolveDesc<CT> sd;
  chain_wait();
  int staged = -1;
  for (int ti = blockIdx.x; ti < ntiles; ti += gridDim.x) {
    const Tile tile = tiles[ti];
    if (tile.solve != staged) {
      __syncthreads();
      stage_desc<CT, BLOCK>(sd, descs, tile.solve);
      __syncthreads();
      staged = tile.solve;
    }
    const int cell = tile.cell0 + int(threadIdx.x);
    if (cell >= sd.ncells) continue;
    batch_cell<L, CT, ST, EQ, KEEP, false>(t, sd, cell, parity, nullptr);
  }
}

// The batched step of a group whose solves have one rate per order >= 4: tiles of kBlock cells,
// and the solve's operator of the higher rows staged in shared memory with its descriptor.
template <class L, class CT, class ST, int EQ>
__global__ void __launch_bounds__(kBlock, 3)
    k_step_batch_high(const LatTables<CT> t, const SolveDesc<CT>* descs, const HighCoefs<CT>* highs,
                      const Tile* tiles, int ntiles, int parity) {
  __shared__ SolveDesc<CT> sd;
  __shared__ HighCoefs<CT> coefs;
  chain_wait();
  int staged = -1;
  for (int ti = blockIdx.x; ti < ntiles; ti += gridDim.x) {
    const Tile tile = tiles[ti];
    if (tile.solve != staged) {
      __syncthreads();
      stage_desc<CT, kBlock>(sd, descs, tile.solve);
      stage_coefs<L>(coefs, highs[tile.solve]);
      __syncthreads();
      staged = tile.solve;
    }
    const int cell = tile.cell0 + int(threadIdx.x);
    if (cell >= sd.ncells) continue;
    batch_cell<L, CT, ST, EQ, true, true>(t, sd, cell, parity, coefs.c);
  }
}

}  // namespace lbm

#include "io_kernels.cuh"
#include "resident.cuh"
#include "tc_kernels.cuh"

namespace lbm {

template <class L, class CT, class ST, int EQ, class F>
lbm_status batch_by_block(int block, bool keep, F&& fn) {
  auto go = [&](auto k) -> lbm_status {
    constexpr bool K = decltype(k)::value;
    switch (block) {
      case 64: return fn(k_step_batch<L, CT, ST, EQ, 64, K>);
      case 128: return fn(k_step_batch<L, CT, ST, EQ, 128, K>);
      case 256: return fn(k_step_batch<L, CT, ST, EQ, 256, K>);
    }
    return set_error(LBM_ERR_ARG, "batched tile size must be 64, 128 or 256 cells");
  };
  return keep ? go(std::true_type{}) : go(std::false_type{});
}

template <class L, class F>
lbm_status batch_kernel_high(int store, int eq, F&& fn) {
  if (store == LBM_F32) {
    if (eq == LBM_NSE) return fn(k_step_batch_high<L, float, float, LBM_NSE>);
    return fn(k_step_batch_high<L, float, float, LBM_NCDE>);
  }
  if (store == LBM_F16_DEV) {
    if (eq == LBM_NSE) return fn(k_step_batch_high<L, float, __half, LBM_NSE>);
    return fn(k_step_batch_high<L, float, __half, LBM_NCDE>);
  }
  if (store == LBM_BF16_DEV) {
    if (eq == LBM_NSE) return fn(k_step_batch_high<L, float, __nv_bfloat16, LBM_NSE>);
    return fn(k_step_batch_high<L, float, __nv_bfloat16, LBM_NCDE>);
  }
  return set_error(LBM_ERR_NOT_IMPLEMENTED, "batched execution supports F32, F16_DEV and BF16_DEV storage");
}

template <class L, class F>
lbm_status batch_kernel(int store, int eq, int block, bool keep, F&& fn) {
  if (store == LBM_F32) {
    if (eq == LBM_NSE) return batch_by_block<L, float, float, LBM_NSE>(block, keep, fn);
    return batch_by_block<L, float, float, LBM_NCDE>(block, keep, fn);
  }
  if (store == LBM_F16_DEV) {
    if (eq == LBM_NSE) return batch_by_block<L, float, __half, LBM_NSE>(block, keep, fn);
    return batch_by_block<L, float, __half, LBM_NCDE>(block, keep, fn);
  }
  if (store == LBM_BF16_DEV) {
    if (eq == LBM_NSE) return batch_by_block<L, float, __nv_bfloat16, LBM_NSE>(block, keep, fn);
    return batch_by_block<L, float, __nv_bfloat16, LBM_NCDE>(block, keep, fn);
  }
  return set_error(LBM_ERR_NOT_IMPLEMENTED, "batched execution supports F32, F16_DEV and BF16_DEV storage");
}

template <int KIND>
lbm_status BatchLaunch<KIND>::launch(const BatchGroup& g, int parity, cudaStream_t stream) {
  using L = Lat<KIND>;
  if (g.high) {
    return batch_kernel_high<L>(g.store, g.eq, [&](auto kernel) -> lbm_status {
      const LatTables<float>& t = *static_cast<const LatTables<float>*>(g.tables);
      cudaError_t err = launch_chained(kernel, g.grid, kBlock, 0, stream, t,
                                       static_cast<const SolveDesc<float>*>(g.d_desc),
                                       static_cast<const HighCoefs<float>*>(g.d_high), g.d_tiles, g.ntiles, parity);
      return err == cudaSuccess ? LBM_OK : cuda_error(err, "batched step launch");
    });
  }
  return batch_kernel<L>(g.store, g.eq, g.block, g.keep != 0, [&](auto kernel) -> lbm_status {
    const LatTables<float>& t = *static_cast<const LatTables<float>*>(g.tables);
    cudaError_t err = launch_chained(kernel, g.grid, g.block, 0, stream, t,
                                     static_cast<const SolveDesc<float>*>(g.d_desc), g.d_tiles, g.ntiles, parity);
    return err == cudaSuccess ? LBM_OK : cuda_error(err, "batched step launch");
  });
}

template <int KIND>
lbm_status BatchLaunch<KIND>::occupancy(const BatchGroup& g, int* blocks_per_sm) {
  using L = Lat<KIND>;
  if (g.high) {
    return batch_kernel_high<L>(g.store, g.eq, [&](auto kernel) -> lbm_status {
      cudaError_t err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, kernel, kBlock, 0);
      return err == cudaSuccess ? LBM_OK : cuda_error(err, "occupancy query");
    });
  }
  return batch_kernel<L>(g.store, g.eq, g.block, g.keep != 0, [&](auto kernel) -> lbm_status {
    cudaError_t err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, kernel, g.block, 0);
    return err == cudaSuccess ? LBM_OK : cuda_error(err, "occupancy query");
  });
}

// Cells from which a step takes two of them per thread. Below, the halved number of threads leaves SMs
// short of warps (us a step, one cell / two cells per thread: rD2Q21 256x200 2.44 / 2.61, 333x301 4.16 /
// 3.77; rD3Q45 36^3 5.6 / 6.3, 45^3 6.6 / 5.9, 64^3 14.0 / 11.4).
constexpr int kPairCells = 80000;
// Cells below which the two-cell kernel releases the next launch before its stores (few waves: a block of the
// next step takes a free place while others of this one end), and above which at its start (ragged grids: once
// the wait is over, where the second cell's indices are ready). us a step,
// rD3Q33 64^3 8.4 at the start of every block (8.9 with the point picked at run time), rD3Q53 150x131x147 BF16
// 110.8 (114.8), rD2Q25 512x384 before the stores 5.3 (5.4). (The kernels with s_high != 1 and with per-order rates
// release at the start on every size; where else they might was not measured.)
constexpr int kPairLateCells = 200000;

// Host launchers for one lattice kind (instantiated in k_<lattice>.cu).
template <class L, class CT, class ST>
lbm_status launch_step_typed(lbm_model* m, int64_t nsteps, bool collide_on) {
  StepParams<CT> p;
  make_step_params(m, &p);
  const int grid = (m->ncells + kBlock - 1) / kBlock;
  CT* phi = static_cast<CT*>(m->phi_prev);
  const bool high = collide_on && has_high_rates(m);
  // tcgen05 when asked for (on FP32 storage only the higher rows go to the tensor cores), and for per-order
  // rates with a forced row-staged gather, which has no other form, or where the row-staged tcgen05 kernel
  // is the faster one: its blocks of 256 threads need nearly full rows, many of them per block, and a
  // lattice of many rows. us a step in FP16, CUDA cores / tcgen05: rD3Q53 256x128x96 227 / 214, 256x64x64
  // 80 / 86, 192x96x96 130 / 158, 160x144x120 201 / 267; rD3Q45 256x128x96 180 / 185.
  [[maybe_unused]] bool tensor =
      collide_on && (m->tensor_cores || (m->tc_auto && high && m->gather == LBM_GATHER_ROWS));
  if constexpr (is_deviation_storage<ST>() && L::Q > 45) {
    RowPlan wide;
    if (high && !tensor && m->tc_auto && m->gather == LBM_GATHER_AUTO && m->n[0] >= 240 &&
        m->ncells / m->n[0] >= 64 * sm_count(m->device))
      tensor = RowLaunch<L::KIND>::plan(m, &wide, true, true);
  }
  [[maybe_unused]] const bool tensor32 = std::is_same<ST, float>::value && tensor && high;
  TcParams tp;
  [[maybe_unused]] Tc32Params tp32;
  int tgrid = 0;
  size_t tsmem = 0;
  [[maybe_unused]] auto tc_kernel = [&](auto hi_tag, auto eq_tag) {
    return k_step_tc<L, ST, decltype(eq_tag)::value, decltype(hi_tag)::value>;
  };
  if constexpr (is_deviation_storage<ST>()) {
    if (tensor) {
      make_tc_params(m, &tp);
      using NSE_ = std::integral_constant<int, LBM_NSE>;
      using NCDE_ = std::integral_constant<int, LBM_NCDE>;
      const void* k = nullptr;
      if (high) {
        tsmem = sizeof(TcSmem<L, true>);
        k = m->eq == LBM_NSE ? reinterpret_cast<const void*>(tc_kernel(std::true_type{}, NSE_{}))
                             : reinterpret_cast<const void*>(tc_kernel(std::true_type{}, NCDE_{}));
        tgrid = tc_grid(m, tp.ntiles, k, TcShape<L, true>::CTAS, tsmem);
      } else {
        tsmem = sizeof(TcSmem<L, false>);
        k = m->eq == LBM_NSE ? reinterpret_cast<const void*>(tc_kernel(std::false_type{}, NSE_{}))
                             : reinterpret_cast<const void*>(tc_kernel(std::false_type{}, NCDE_{}));
        tgrid = tc_grid(m, tp.ntiles, k, TcShape<L, false>::CTAS, tsmem);
      }
    }
  }
  if constexpr (std::is_same<ST, float>::value) {
    if (tensor32) {
      make_tc32_params(m, &tp32);
      // With many tiles a CTA, as much shared memory as lets no further CTA beside CTAS of them: the next launch, released
      // early, would else place its CTAs on the SMs that have room and leave others short of work. us a step with
      // room / without: rD2Q13 1024x768 27.8 / 20.5, rD3Q33 96^3 70.5 / 59.9 (15 tiles a CTA); 512x384 7.2 / 7.4, rD2Q25
      // 10.8 / 11.7 (3.4 tiles: the next launch's tables are made meanwhile). rD3Q45 and larger fill the SM anyway.
      tsmem = sizeof(Tc32Smem<L>);
      int sm_smem = 0;
      if (tp32.ntiles >= 4 * Tc32Shape<L>::CTAS * sm_count(m->device)) {
        if (cudaDeviceGetAttribute(&sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, m->device) != cudaSuccess)
          cudaGetLastError();
        tsmem = std::max(tsmem, size_t(sm_smem) / (Tc32Shape<L>::CTAS + 1));
      }
      const void* k = m->eq == LBM_NSE ? reinterpret_cast<const void*>(k_step_tc32_high<L, LBM_NSE>)
                                       : reinterpret_cast<const void*>(k_step_tc32_high<L, LBM_NCDE>);
      tgrid = tc_grid(m, tp32.ntiles, k, Tc32Shape<L>::CTAS, tsmem);
    }
  }
  // 16-bit storage: the row-staged gather on tcgen05, for a step without a collision, or when forced. On the
  // CUDA cores the per-thread kernels are the faster ones since they take two cells per thread: us a step of
  // FP16, row-staged / per thread: rD3Q53 256x256x192 460 / 441, 96^3 43 / 35, 32^3 5.6 / 3.3, with s_h != 1
  // 256x128x96 150 / 136; rD3Q33 64^3 10.6 / 7.4; rD2Q17 256x4096 14.7 / 11.5. (A step without a collision on
  // 256x256x192: 439 row-staged, 550 per thread.)
  [[maybe_unused]] RowPlan rplan;
  [[maybe_unused]] StepParams<F2, float> p2;  // the row-staged CUDA-core kernel works on two cells at a time
  bool rows = false;
  if constexpr (is_deviation_storage<ST>()) {
    if (m->gather == LBM_GATHER_ROWS && high && !tensor)
      return set_error(LBM_ERR_NOT_IMPLEMENTED,
                       "the row-staged gather runs per-order rates on the tensor cores only");
    if (m->gather == LBM_GATHER_ROWS || (m->gather == LBM_GATHER_AUTO && (tensor || !collide_on))) {
      rows = RowLaunch<L::KIND>::plan(m, &rplan, tensor, high);
      if (!rows && m->gather == LBM_GATHER_ROWS) return set_error(LBM_ERR_ARG, "the row-staged gather does not apply");
      if (rows && nsteps > 0) {
        const lbm_status st = RowLaunch<L::KIND>::configure(m, rplan, collide_on);
        if (st != LBM_OK) return st;
        make_step_params(m, &p2);
      }
    }
  }
  // small 2D grids: the whole call in one launch, the populations in a cluster's shared memory
  if constexpr (!std::is_same<CT, double>::value && L::D == 2) {
    int ctas = 0;
    if (collide_on && !high && !tensor && resident_plan<L, ST>(m, nsteps, &ctas)) {
      constexpr int64_t kMost = 1 << 16;  // steps of one launch
      while (nsteps > 0) {
        const int n = int(std::min<int64_t>(kMost, nsteps));
        cudaError_t err;
        if (m->eq == LBM_NSE)
          err = m->s_high == 1.0 ? launch_resident<L, ST, LBM_NSE, false>(m, p, n, ctas, phi)
                                 : launch_resident<L, ST, LBM_NSE, true>(m, p, n, ctas, phi);
        else
          err = m->s_high == 1.0 ? launch_resident<L, ST, LBM_NCDE, false>(m, p, n, ctas, phi)
                                 : launch_resident<L, ST, LBM_NCDE, true>(m, p, n, ctas, phi);
        if (err != cudaSuccess) {  // no room for the cluster (a partitioned GPU): step by step
          cudaGetLastError();
          break;
        }
        m->cur ^= n & 1;  // as n launches would have left it
        m->launches += 1;
        m->steps += n;
        nsteps -= n;
      }
      if (nsteps == 0) return LBM_OK;
    }
  }
  // two cells per thread where the halved thread count still fills the GPU (with the higher rows' operator
  // not on ragged FP32 grids of the largest lattice: rD3Q53 101x103x97 99 us a step against 94 with one)
  [[maybe_unused]] const bool pairs = !std::is_same<CT, double>::value && collide_on && !tensor && !rows &&
                                      m->ncells >= kPairCells &&
                                      !(high && L::Q > 45 && std::is_same<ST, float>::value && m->n[0] % 2 != 0);
  if (pairs) make_step_params(m, &p2);
  HighCoefs<CT> hc;
  if (high && !tensor) make_high_coefs(m, &hc);
  const int grid2 = (m->ncells / 2 + m->ncells % 2 + kBlock - 1) / kBlock;
  // FP64 on a small 2D grid: four threads per cell while every block of 32 cells has an SM of its own. Us per
  // step, one thread per cell against four (a first version): 80x60 cells, 150 blocks, rD2Q13 6.4 / 5.2, rD2Q25
  // 9.6 / 6.1; 100x76, 238 blocks, 6.4 / 7.7 and 9.6 / 9.2; 128x96 6.5 / 10.5 and 9.6 / 13.
  [[maybe_unused]] const int grid_split = (m->ncells + 31) / 32;
  [[maybe_unused]] bool split = false;
  if constexpr (std::is_same<CT, double>::value && L::D == 2)
    split = collide_on && !high && grid_split <= sm_count(m->device);
  const bool hist = collide_on && m->m2g_aniso;
  int release = -1;
  p.grad_on = collide_on && p.grad_on;
  if (rows || pairs) p2.grad_on = p.grad_on;
  for (int64_t s = 0; s < nsteps; ++s) {
    const ST* fin = static_cast<const ST*>(m->f[m->cur]);
    ST* fout = static_cast<ST*>(m->f[m->cur ^ 1]);
    if (hist) {
      p.grad_in = static_cast<const CT*>(m->rho_hist[m->hist_cur]);
      p.rho_out = static_cast<CT*>(m->rho_hist[m->hist_cur ^ 1]);
      if constexpr (std::is_same<CT, float>::value) {
        p2.grad_in = p.grad_in;
        p2.rho_out = p.rho_out;
      }
    }
    cudaError_t err = cudaSuccess;
    auto go = [&](auto kernel, int blocks, int threads, size_t smem, const auto&... args) {
      if (release < 0) release = release_point(kernel, blocks, threads, smem, m->device);
      p.release = p2.release = release;
      err = launch_chained(kernel, blocks, threads, smem, m->stream, args..., fin, fout, phi);
    };
    bool done = false;
    if constexpr (is_deviation_storage<ST>()) {
      if (rows) {
        const lbm_status st = RowLaunch<L::KIND>::launch(m, rplan, p, p2, fin, fout, phi, collide_on);
        if (st != LBM_OK) return st;
        done = true;
      } else if (tensor) {
        if (high) {
          if (m->eq == LBM_NSE) go(k_step_tc<L, ST, LBM_NSE, true>, tgrid, 128, tsmem, p, tp);
          else go(k_step_tc<L, ST, LBM_NCDE, true>, tgrid, 128, tsmem, p, tp);
        } else {
          if (m->eq == LBM_NSE) go(k_step_tc<L, ST, LBM_NSE, false>, tgrid, 128, tsmem, p, tp);
          else go(k_step_tc<L, ST, LBM_NCDE, false>, tgrid, 128, tsmem, p, tp);
        }
        done = true;
      }
    }
    if constexpr (std::is_same<ST, float>::value) {
      if (tensor32) {
        if (m->eq == LBM_NSE) go(k_step_tc32_high<L, LBM_NSE>, tgrid, 128, tsmem, p, tp32);
        else go(k_step_tc32_high<L, LBM_NCDE>, tgrid, 128, tsmem, p, tp32);
        done = true;
      }
    }
    if constexpr (!std::is_same<CT, double>::value) {
      if (pairs) {
        auto pick = [&](auto eq, auto even) {
          constexpr int E = decltype(eq)::value;
          constexpr bool EV = decltype(even)::value;
          if (high) {
            go(k_step_pair<L, ST, E, true, EV, true>,
               is_deviation_storage<ST>() ? std::min(grid2, sm_count(m->device) * pair_high_blocks<L, ST>()) : grid2, kBlock, 0,
               p2, hc);
          } else if (m->s_high == 1.0 && m->ncells < kPairLateCells) {
            go(k_step_pair<L, ST, E, false, EV, false, true>, grid2, kBlock, 0, p2, NoCoefs{});
          } else if (m->s_high == 1.0) {
            go(k_step_pair<L, ST, E, false, EV>, grid2, kBlock, 0, p2, NoCoefs{});
          } else {
            go(k_step_pair<L, ST, E, true, EV>, grid2, kBlock, 0, p2, NoCoefs{});
          }
        };
        auto by_even = [&](auto eq) {
          if (m->n[0] % 2 == 0) pick(eq, std::true_type{});
          else pick(eq, std::false_type{});
        };
        if (m->eq == LBM_NSE) by_even(std::integral_constant<int, LBM_NSE>{});
        else by_even(std::integral_constant<int, LBM_NCDE>{});
        done = true;
      }
    }
    if constexpr (std::is_same<CT, double>::value && L::D == 2) {
      if (split) {
        if (m->eq == LBM_NSE) {
          if (m->s_high == 1.0) go(k_step_split<L, LBM_NSE, false>, grid_split, 128, 0, p);
          else go(k_step_split<L, LBM_NSE, true>, grid_split, 128, 0, p);
        } else {
          if (m->s_high == 1.0) go(k_step_split<L, LBM_NCDE, false>, grid_split, 128, 0, p);
          else go(k_step_split<L, LBM_NCDE, true>, grid_split, 128, 0, p);
        }
        done = true;
      }
    }
    if (done) {
    } else if (high) {
      if (m->eq == LBM_NSE) go(k_step_high<L, CT, ST, LBM_NSE>, grid, kBlock, 0, p, hc);
      else go(k_step_high<L, CT, ST, LBM_NCDE>, grid, kBlock, 0, p, hc);
    } else if (!collide_on) {
      go(k_step<L, CT, ST, LBM_NSE, false, true>, grid, kBlock, 0, p);
    } else if (m->eq == LBM_NSE) {
      if (m->s_high == 1.0) go(k_step<L, CT, ST, LBM_NSE, true, false>, grid, kBlock, 0, p);
      else go(k_step<L, CT, ST, LBM_NSE, true, true>, grid, kBlock, 0, p);
    } else {
      if (m->s_high == 1.0) go(k_step<L, CT, ST, LBM_NCDE, true, false>, grid, kBlock, 0, p);
      else go(k_step<L, CT, ST, LBM_NCDE, true, true>, grid, kBlock, 0, p);
    }
    if (err != cudaSuccess) return cuda_error(err, "collide-stream launch");
    m->cur ^= 1;
    if (hist) m->hist_cur ^= 1;
    m->launches += 1;
    if (collide_on) m->steps += 1;
  }
  return LBM_OK;
}

template <class L, class CT, class ST>
lbm_status launch_init_typed(lbm_model* m, const double* rho_or_phi, const double* u) {
  StepParams<CT> p;
  make_step_params(m, &p);
  const int grid = (m->ncells + kBlock - 1) / kBlock;
  ST* fout = static_cast<ST*>(m->f[m->cur]);
  CT* phi = static_cast<CT*>(m->eq == LBM_NSE ? m->rho_hist[m->hist_cur] : m->phi_prev);
  if (m->eq == LBM_NSE)
    k_init<L, CT, ST, LBM_NSE><<<grid, kBlock, 0, m->stream>>>(p, rho_or_phi, u, fout, phi);
  else
    k_init<L, CT, ST, LBM_NCDE><<<grid, kBlock, 0, m->stream>>>(p, rho_or_phi, u, fout, phi);
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return cuda_error(err, "init launch");
  m->launches += 1;
  return LBM_OK;
}

template <int KIND>
lbm_status Launch<KIND>::step(lbm_model* m, int64_t nsteps, bool collide_on) {
  using L = Lat<KIND>;
  switch (m->store) {
    case LBM_F64: return launch_step_typed<L, double, double>(m, nsteps, collide_on);
    case LBM_F32: return launch_step_typed<L, float, float>(m, nsteps, collide_on);
    case LBM_BF16_DEV: return launch_step_typed<L, float, __nv_bfloat16>(m, nsteps, collide_on);
    case LBM_F16_DEV: return launch_step_typed<L, float, __half>(m, nsteps, collide_on);
  }
  return set_error(LBM_ERR_ARG, "unknown storage dtype");
}

template <int KIND>
lbm_status Launch<KIND>::init(lbm_model* m, const double* rho_or_phi, const double* u) {
  using L = Lat<KIND>;
  switch (m->store) {
    case LBM_F64: return launch_init_typed<L, double, double>(m, rho_or_phi, u);
    case LBM_F32: return launch_init_typed<L, float, float>(m, rho_or_phi, u);
    case LBM_BF16_DEV: return launch_init_typed<L, float, __nv_bfloat16>(m, rho_or_phi, u);
    case LBM_F16_DEV: return launch_init_typed<L, float, __half>(m, rho_or_phi, u);
  }
  return set_error(LBM_ERR_ARG, "unknown storage dtype");
}

}  // namespace lbm

#define LBM_INSTANTIATE_LATTICE(KIND) \
  template struct lbm::Launch<KIND>;     \
  template struct lbm::BatchLaunch<KIND>;
