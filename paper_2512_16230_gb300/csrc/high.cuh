// The full Q x Q collision with one rate per order >= 4 (Eq. (H-MRT-LB)), beside the reduced form.
//
// The rows of order >= 4 add w_i sum_r alpha_r H_r(c_i) sum_j H_r(c_j) f_j, alpha_r = -(s_r - s_high) / N_r, to
// the update: a symmetric Q x Q operator. The velocity sets, the weights and the orders are invariant
// under the reflections of the axes, so the operator is block diagonal over functions of one parity
// class. Those functions are the signed sums over the velocities m (+-a), m (+-a +- b), m (+-a +- b +- c) that
// the raw moments are made of: with a_k = sum_i phi_k(c_i) f_i (phi_k = +-1 on the velocities of one speed
// and reflection class, 0 elsewhere) the update is w_i sum_k phi_k(c_i) b_k, b = M a in blocks. For
// rD3Q53 the blocks are 15, 3 x 4, 3 x 8 and 2 functions wide: 469 multiply-adds per cell, where the rows
// themselves take 2 x 33 x 27 and the dense operator 53 x 53. (1 - s_high) f_i is the diagonal entry
// (1 - s_high) / (w_i times the number of velocities of phi_k), so the old populations are not kept.
#pragma once

namespace lbm {

// Speeds m = 1 .. n of the axis, plane-diagonal and space-diagonal directions.
template <class L>
struct Speeds {
  static constexpr int count(Vel d) {
    int n = 0;
    while (velocity_index<L>(d, n + 1) >= 0) ++n;
    return n;
  }
  static constexpr int A = count(Vel{1, 0, 0}), P = count(Vel{1, 1, 0}), C = L::D == 3 ? count(Vel{1, 1, 1}) : 0;
};

// Indices of the functions, class by class: even (rest, axes, planes, space diagonals), (odd, odd) of each
// plane, odd of each axis, odd in all three.
template <class L>
struct Adapted {
  using S = Speeds<L>;
  static constexpr int D = L::D, NP = D == 3 ? 3 : 1;  // planes xy, xz, yz
  static constexpr int N0 = 1 + D * S::A + NP * S::P + S::C, N2 = S::P + S::C, N1 = S::A + (D - 1) * S::P + S::C,
                       N3 = S::C;
  static_assert(N0 + NP * N2 + D * N1 + N3 == L::Q, "the functions are a basis");
  static constexpr int plane(int a, int b) { return D == 2 ? 0 : a + b - 1; }
  static constexpr int off2(int pl) { return N0 + pl * N2; }
  static constexpr int off1(int a) { return N0 + NP * N2 + a * N1; }
  static constexpr int off3() { return N0 + NP * N2 + D * N1; }
  // m counts from 1
  static constexpr int axis_even(int a, int m) { return 1 + a * S::A + m - 1; }
  static constexpr int plane_even(int pl, int m) { return 1 + D * S::A + pl * S::P + m - 1; }
  static constexpr int corner_even(int m) { return 1 + D * S::A + NP * S::P + m - 1; }
  static constexpr int plane_odd2(int pl, int m) { return off2(pl) + m - 1; }
  static constexpr int corner_odd2(int pl, int m) { return off2(pl) + S::P + m - 1; }
  static constexpr int axis_odd(int a, int m) { return off1(a) + m - 1; }
  // the i-th other axis of a (other_axis)
  static constexpr int plane_odd(int a, int b, int m) {
    return off1(a) + S::A + (D == 2 ? 0 : (other_axis(a, 0) == b ? 0 : 1)) * S::P + m - 1;
  }
  static constexpr int corner_odd(int a, int m) { return off1(a) + S::A + (D - 1) * S::P + m - 1; }
  static constexpr int corner_odd3(int m) { return off3() + m - 1; }
  // blocks: 0 even, 1 .. NP planes, then axes, then all three
  static constexpr int blocks() { return 1 + NP + D + (D == 3 ? 1 : 0); }
  static constexpr int block_off(int b) {
    return b == 0 ? 0 : (b <= NP ? off2(b - 1) : (b <= NP + D ? off1(b - NP - 1) : off3()));
  }
  static constexpr int block_size(int b) { return b == 0 ? N0 : (b <= NP ? N2 : (b <= NP + D ? N1 : N3)); }
  static constexpr int coef_off(int b) {
    int o = 0;
    for (int i = 0; i < b; ++i) o += block_size(i) * block_size(i);
    return o;
  }
};

template <class L, int DX, int DY, int DZ, int M, class V>
__device__ __forceinline__ void pair_sums(const V (&f)[L::Q], V& s, V& d) {
  constexpr int ip = velocity_index<L>(Vel{DX, DY, DZ}, M), im = velocity_index<L>(Vel{DX, DY, DZ}, -M);
  s = f[ip] + f[im];
  d = f[ip] - f[im];
}

// a_k = sum_i phi_k(c_i) f_i
template <class L, class V>
__device__ __forceinline__ void adapt(const V (&f)[L::Q], V (&a)[L::Q]) {
  using B = Adapted<L>;
  using S = Speeds<L>;
  constexpr int D = L::D;
  a[0] = f[0];
  static_for<D>([&](auto aa) {
    constexpr int A = decltype(aa)::value;
    static_for<S::A>([&](auto mm) {
      constexpr int M = decltype(mm)::value + 1;
      pair_sums<L, A == 0, A == 1, A == 2, M>(f, a[B::axis_even(A, M)], a[B::axis_odd(A, M)]);
    });
  });
  static_for<B::NP>([&](auto pp) {
    constexpr int PL = decltype(pp)::value, X = PL == 2 ? 1 : 0, Y = PL == 0 ? 1 : 2;
    static_for<S::P>([&](auto mm) {
      constexpr int M = decltype(mm)::value + 1;
      V sp, dp, sm, dm;
      pair_sums<L, X == 0, (X == 1) + (Y == 1), Y == 2, M>(f, sp, dp);
      pair_sums<L, X == 0, (X == 1) - (Y == 1), -(Y == 2), M>(f, sm, dm);
      a[B::plane_even(PL, M)] = sp + sm;
      a[B::plane_odd2(PL, M)] = sp - sm;
      a[B::plane_odd(X, Y, M)] = dp + dm;
      a[B::plane_odd(Y, X, M)] = dp - dm;
    });
  });
  if constexpr (D == 3) {
    static_for<S::C>([&](auto mm) {
      constexpr int M = decltype(mm)::value + 1;
      V s[4], d[4];
      pair_sums<L, 1, 1, 1, M>(f, s[0], d[0]);
      pair_sums<L, 1, 1, -1, M>(f, s[1], d[1]);
      pair_sums<L, 1, -1, 1, M>(f, s[2], d[2]);
      pair_sums<L, 1, -1, -1, M>(f, s[3], d[3]);
      const Signed4<V> e = signed4(s[0], s[1], s[2], s[3]), o = signed4(d[0], d[1], d[2], d[3]);
      a[B::corner_even(M)] = e.s;
      a[B::corner_odd2(0, M)] = e.b;
      a[B::corner_odd2(1, M)] = e.g;
      a[B::corner_odd2(2, M)] = e.bg;
      a[B::corner_odd(0, M)] = o.s;
      a[B::corner_odd(1, M)] = o.b;
      a[B::corner_odd(2, M)] = o.g;
      a[B::corner_odd3(M)] = o.bg;
    });
  }
}

// Raw moments mu_k = sum_i mono_k(e_i) f_i from the adapted sums: m^deg times the sums of one kind, over the speeds.
template <class L, class V>
__device__ __forceinline__ void adapted_moments(const V (&a)[L::Q], V (&mu)[L::R]) {
  using B = Adapted<L>;
  using S = Speeds<L>;
  constexpr int D = L::D;
  V m0 = a[0], m1[3], m2[3], m3[3], x3[6];
  static_for<D>([&](auto aa) {
    constexpr int A = decltype(aa)::value;
    m0 = m0 + a[B::axis_even(A, 1)];
    m1[A] = a[B::axis_odd(A, 1)];
    m2[A] = a[B::axis_even(A, 1)];
    m3[A] = m1[A];
    static_for<S::A - 1>([&](auto mm) {
      constexpr int M = decltype(mm)::value + 2;
      m0 = m0 + a[B::axis_even(A, M)];
      m1[A] = axpy_c<M>(a[B::axis_odd(A, M)], m1[A]);
      m2[A] = axpy_c<M * M>(a[B::axis_even(A, M)], m2[A]);
      m3[A] = axpy_c<M * M * M>(a[B::axis_odd(A, M)], m3[A]);
    });
  });
  V c2 = V(0.f), c3[3];
  if constexpr (D == 3) {
    c2 = a[B::corner_even(1)];
    m0 = m0 + c2;
    V xyz = a[B::corner_odd3(1)];
    static_for<3>([&](auto aa) {
      constexpr int A = decltype(aa)::value;
      c3[A] = a[B::corner_odd(A, 1)];
      m1[A] = m1[A] + c3[A];
    });
    static_for<S::C - 1>([&](auto mm) {
      constexpr int M = decltype(mm)::value + 2;
      m0 = m0 + a[B::corner_even(M)];
      c2 = axpy_c<M * M>(a[B::corner_even(M)], c2);
      xyz = axpy_c<M * M * M>(a[B::corner_odd3(M)], xyz);
      static_for<3>([&](auto aa) {
        constexpr int A = decltype(aa)::value;
        m1[A] = axpy_c<M>(a[B::corner_odd(A, M)], m1[A]);
        c3[A] = axpy_c<M * M * M>(a[B::corner_odd(A, M)], c3[A]);
      });
    });
    mu[row3<3>(0, 1, 2)] = xyz;
    static_for<3>([&](auto aa) { m2[decltype(aa)::value] = m2[decltype(aa)::value] + c2; });
  }
  static_for<B::NP>([&](auto pp) {
    constexpr int PL = decltype(pp)::value, X = PL == 2 ? 1 : 0, Y = PL == 0 ? 1 : 2;
    V s2 = a[B::plane_even(PL, 1)], q2 = a[B::plane_odd2(PL, 1)];
    V xo = a[B::plane_odd(X, Y, 1)], yo = a[B::plane_odd(Y, X, 1)];
    m0 = m0 + s2;
    m1[X] = m1[X] + xo;
    m1[Y] = m1[Y] + yo;
    static_for<S::P - 1>([&](auto mm) {
      constexpr int M = decltype(mm)::value + 2;
      m0 = m0 + a[B::plane_even(PL, M)];
      s2 = axpy_c<M * M>(a[B::plane_even(PL, M)], s2);
      q2 = axpy_c<M * M>(a[B::plane_odd2(PL, M)], q2);
      m1[X] = axpy_c<M>(a[B::plane_odd(X, Y, M)], m1[X]);
      m1[Y] = axpy_c<M>(a[B::plane_odd(Y, X, M)], m1[Y]);
      xo = axpy_c<M * M * M>(a[B::plane_odd(X, Y, M)], xo);
      yo = axpy_c<M * M * M>(a[B::plane_odd(Y, X, M)], yo);
    });
    m2[X] = m2[X] + s2;
    m2[Y] = m2[Y] + s2;
    m3[X] = m3[X] + xo;
    m3[Y] = m3[Y] + yo;
    if constexpr (D == 3) {
      static_for<S::C>([&](auto mm) {
        constexpr int M = decltype(mm)::value + 1;
        q2 = axpy_c<M * M>(a[B::corner_odd2(PL, M)], q2);
      });
      xo = xo + c3[X];
      yo = yo + c3[Y];
    }
    mu[row2<D>(X, Y)] = q2;
    mu[row3<D>(X, Y, Y)] = xo;
    mu[row3<D>(Y, X, X)] = yo;
  });
  mu[0] = m0;
  static_for<D>([&](auto aa) {
    constexpr int A = decltype(aa)::value;
    mu[1 + A] = m1[A];
    mu[row2<D>(A, A)] = m2[A];
    if constexpr (!L::SINGLE) {
      if constexpr (D == 3) mu[row3<D>(A, A, A)] = m3[A] + c3[A];
      else mu[row3<D>(A, A, A)] = m3[A];
    }
  });
}

// 16 bytes of coefficients from shared memory.
template <class C>
__device__ __forceinline__ void load_coefs(const C* c, C (&v)[16 / sizeof(C)]) {
  if constexpr (std::is_same<C, float>::value) {
    const float4 q = *reinterpret_cast<const float4*>(c);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  } else {
    const double2 q = *reinterpret_cast<const double2*>(c);
    v[0] = q.x; v[1] = q.y;
  }
}

// c * x + acc with an unpacked coefficient. On two cells these are two scalar multiply-adds: the packed one takes
// the FMA pipe for as long, and would need the coefficient twice (8 bytes of shared memory reads for each).
template <class V>
__device__ __forceinline__ V coef_fma(typename Coef<V>::type c, V x, V acc) {
  if constexpr (std::is_same<V, F2>::value) {
    float x0, x1, a0, a1;
    x.get(x0, x1);
    acc.get(a0, a1);
    return F2(fmaf(c, x0, a0), fmaf(c, x1, a1));
  } else {
    return fma(c, x, acc);
  }
}
template <class V>
__device__ __forceinline__ V coef_mul(typename Coef<V>::type c, V x) {
  if constexpr (std::is_same<V, F2>::value) {
    float x0, x1;
    x.get(x0, x1);
    return F2(c * x0, c * x1);
  } else {
    return c * x;
  }
}

// b = M a, in place, block by block. The coefficients are used in the order in which they lie in shared
// memory, one vector load for 16 bytes of them (as kernel parameters each would have to be brought
// into registers, and the allocator keeps many of them there: 490 bytes of spills at 168 registers).
template <class L, class V>
__device__ __forceinline__ void high_operator(V (&a)[L::Q], const typename Coef<V>::type* c) {
  using B = Adapted<L>;
  using C = typename Coef<V>::type;
  constexpr int VEC = 16 / sizeof(C);
  C v[VEC];
  static_for<B::blocks()>([&](auto bb) {
    constexpr int BL = decltype(bb)::value, O = B::block_off(BL), N = B::block_size(BL), CO = B::coef_off(BL);
    V t[N > 0 ? N : 1];
    static_for<N * N>([&](auto ii) {
      constexpr int I = decltype(ii)::value, K = I / N, J = I % N;
      if constexpr ((CO + I) % VEC == 0) load_coefs(c + CO + I, v);
      if constexpr (J == 0) t[K] = coef_mul<V>(v[(CO + I) % VEC], a[O]);
      else t[K] = coef_fma<V>(v[(CO + I) % VEC], a[O + J], t[K]);
    });
    static_for<N>([&](auto kk) { a[O + decltype(kk)::value] = t[decltype(kk)::value]; });
  });
}

// Block-wide copy of the operator into shared memory (a barrier has to follow).
template <class L, class C>
__device__ __forceinline__ void stage_coefs(HighCoefs<C>& dst, const HighCoefs<C>& src) {
  constexpr int n = Adapted<L>::coef_off(Adapted<L>::blocks());
  for (int k = threadIdx.x; k < n; k += blockDim.x) dst.c[k] = src.c[k];
}

// The two populations at speed M of a direction, f_{+-md} = w (E_0 + m^2 E_2 + B_e +- (m (E_1 + m^2 E_3) + B_o)); the
// odd functions' rows of M are over m, so that B_o / m comes in (E_1, E_2, E_3 as in dir_out).
template <class L, int DX, int DY, int DZ, int M, class V>
__device__ __forceinline__ void pair_out(V (&f)[L::Q], const LatTables<V>& lt, V E0, V E1, V E2, V E3, V Be, V Bo) {
  constexpr int ip = velocity_index<L>(Vel{DX, DY, DZ}, M), im = velocity_index<L>(Vel{DX, DY, DZ}, -M);
  const V we = lt.w[ip] * (axpy_c<M * M>(E2, E0) + Be);
  V odd = E1;
  if constexpr (!(L::SINGLE && iabs(DX) + iabs(DY) + iabs(DZ) == 1)) odd = axpy_c<M * M>(E3, E1);
  odd = odd + Bo;
  f[ip] = fmaf_t(lt.wm[ip], odd, we);
  f[im] = fmaf_t(lt.wm[im], odd, we);
}

// f_i = w_i (sum_k mono_k(e_i) h_k + sum_k phi_k(c_i) b_k)
template <class L, class V>
__device__ __forceinline__ void back_project_high(V (&f)[L::Q], const LatTables<V>& lt, const V (&h)[L::R],
                                                  const V (&b)[L::Q]) {
  using B = Adapted<L>;
  using S = Speeds<L>;
  constexpr int D = L::D;
  const V h0 = h[0];
  f[0] = lt.w[0] * (h0 + b[0]);
  V cube[3], t3[3];
  static_for<D>([&](auto aa) {
    constexpr int A = decltype(aa)::value;
    if constexpr (L::SINGLE) cube[A] = V(0.f);
    else cube[A] = h[row3<D>(A, A, A)];
    t3[A] = cube[A];
    static_for<S::A>([&](auto mm) {
      constexpr int M = decltype(mm)::value + 1;
      pair_out<L, A == 0, A == 1, A == 2, M>(f, lt, h0, h[1 + A], h[row2<D>(A, A)], cube[A], b[B::axis_even(A, M)],
                                             b[B::axis_odd(A, M)]);
    });
  });
  static_for<B::NP>([&](auto pp) {
    constexpr int PL = decltype(pp)::value, X = PL == 2 ? 1 : 0, Y = PL == 0 ? 1 : 2;
    const V abb = h[row3<D>(X, Y, Y)], baa = h[row3<D>(Y, X, X)];
    V ox = abb, oy = baa;
    if constexpr (!L::SINGLE) {
      ox = cube[X] + abb;
      oy = cube[Y] + baa;
    }
    t3[X] = t3[X] + abb;
    t3[Y] = t3[Y] + baa;
    const V s2 = h[row2<D>(X, X)] + h[row2<D>(Y, Y)], q = h[row2<D>(X, Y)];
    const V e1p = h[1 + X] + h[1 + Y], e1m = h[1 + X] - h[1 + Y];
    const V e2p = s2 + q, e2m = s2 - q, e3p = ox + oy, e3m = ox - oy;
    static_for<S::P>([&](auto mm) {
      constexpr int M = decltype(mm)::value + 1;
      const V be = b[B::plane_even(PL, M)], bd = b[B::plane_odd2(PL, M)];
      const V bx = b[B::plane_odd(X, Y, M)], by = b[B::plane_odd(Y, X, M)];
      pair_out<L, X == 0, (X == 1) + (Y == 1), Y == 2, M>(f, lt, h0, e1p, e2p, e3p, be + bd, bx + by);
      pair_out<L, X == 0, (X == 1) - (Y == 1), -(Y == 2), M>(f, lt, h0, e1m, e2m, e3m, be - bd, bx - by);
    });
  });
  if constexpr (D == 3) {
    const V ss = (h[row2<3>(0, 0)] + h[row2<3>(1, 1)]) + h[row2<3>(2, 2)];
    const Signed4<V> e2 = signed4(ss, h[row2<3>(0, 1)], h[row2<3>(0, 2)], h[row2<3>(1, 2)]);
    const Signed4<V> e3 = signed4(t3[0], t3[1], t3[2], h[row3<3>(0, 1, 2)]);
    const V xy = h[1] + h[2], xmy = h[1] - h[2];
    static_for<S::C>([&](auto mm) {
      constexpr int M = decltype(mm)::value + 1;
      const Signed4<V> be = signed4(b[B::corner_even(M)], b[B::corner_odd2(0, M)], b[B::corner_odd2(1, M)],
                                    b[B::corner_odd2(2, M)]);
      const Signed4<V> bo = signed4(b[B::corner_odd(0, M)], b[B::corner_odd(1, M)], b[B::corner_odd(2, M)],
                                    b[B::corner_odd3(M)]);
      pair_out<L, 1, 1, 1, M>(f, lt, h0, xy + h[3], e2.s, e3.s, be.s, bo.s);
      pair_out<L, 1, 1, -1, M>(f, lt, h0, xy - h[3], e2.b, e3.b, be.b, bo.b);
      pair_out<L, 1, -1, 1, M>(f, lt, h0, xmy + h[3], e2.g, e3.g, be.g, bo.g);
      pair_out<L, 1, -1, -1, M>(f, lt, h0, xmy - h[3], e2.bg, e3.bg, be.bg, bo.bg);
    });
  }
}

// The collision of collide() with the operator of the higher rows (c: its blocks, constant or shared memory).
template <class L, class V, int EQ, bool DEV>
__device__ __forceinline__ void collide_high(V (&f)[L::Q], const typename Coef<V>::type* c, const LatTables<V>& lt,
                                             const Rates<V>& rt, bool forced, const V (&F)[3], V phi_prev, V& phi_now, const V* gr) {
  V a[L::Q], mu[L::R], h[L::R];
  adapt<L>(f, a);
  adapted_moments<L>(a, mu);
  collide_moments<L, V, EQ, DEV>(mu, lt, rt, forced, F, phi_prev, phi_now, h, gr);
  high_operator<L>(a, c);
  back_project_high<L>(f, lt, h, a);
}

// Velocity i reflected in axis a.
template <class L>
struct Reflected {
  int v[3][L::Q];
  constexpr Reflected() : v{} {
    for (int a = 0; a < L::D; ++a)
      for (int i = 0; i < L::Q; ++i) {
        const Vel e = L::e(i);
        while (!same_vel(L::e(v[a][i]), Vel{a == 0 ? -e.x : e.x, a == 1 ? -e.y : e.y, a == 2 ? -e.z : e.z})) ++v[a][i];
      }
  }
};

// Host: the blocks of M for the rates of the model. rep_k: a velocity with phi_k = +1, so that H_r = sum_k
// H_r(rep_k) phi_k over the functions of the row's class (the row's behaviour under the reflections).
template <int KIND>
void Launch<KIND>::high_operator_blocks(const lbm_model* m, double* c) {
  const bool fp64 = m->store == LBM_F64;
  using L = Lat<KIND>;
  using B = Adapted<L>;
  using S = Speeds<L>;
  const lbm_lattice* lat = m->lat;
  constexpr int Q = L::Q, D = L::D;
  int rep[Q] = {}, cls[Q] = {}, mult[Q], members[Q];
  for (int k = 0; k < Q; ++k) mult[k] = members[k] = 1;
  auto set = [&](int k, int cl, Vel d, int mm, int n) {
    rep[k] = velocity_index<L>(d, mm);
    cls[k] = cl;
    mult[k] = mm;
    members[k] = n;
  };
  for (int a = 0; a < D; ++a)
    for (int mm = 1; mm <= S::A; ++mm) {
      const Vel d{a == 0, a == 1, a == 2};
      set(B::axis_even(a, mm), 0, d, mm, 2);
      set(B::axis_odd(a, mm), 1 << a, d, mm, 2);
    }
  for (int pl = 0; pl < B::NP; ++pl) {
    const int x = pl == 2 ? 1 : 0, y = pl == 0 ? 1 : 2;
    const Vel d{x == 0, (x == 1) + (y == 1), y == 2};
    for (int mm = 1; mm <= S::P; ++mm) {
      set(B::plane_even(pl, mm), 0, d, mm, 4);
      set(B::plane_odd2(pl, mm), (1 << x) | (1 << y), d, mm, 4);
      set(B::plane_odd(x, y, mm), 1 << x, d, mm, 4);
      set(B::plane_odd(y, x, mm), 1 << y, d, mm, 4);
    }
  }
  if (D == 3)
    for (int mm = 1; mm <= S::C; ++mm) {
      const Vel d{1, 1, 1};
      set(B::corner_even(mm), 0, d, mm, 8);
      for (int pl = 0; pl < 3; ++pl) {
        const int x = pl == 2 ? 1 : 0, y = pl == 0 ? 1 : 2;
        set(B::corner_odd2(pl, mm), (1 << x) | (1 << y), d, mm, 8);
        set(B::corner_odd(pl, mm), 1 << pl, d, mm, 8);
      }
      set(B::corner_odd3(mm), 7, d, mm, 8);
    }
  // the rows with a rate of their own, by class
  static constexpr Reflected<L> mirror{};
  int rows[8][Q], count[8] = {};
  for (int r = 0; r < lat->nhigh; ++r) {
    if (high_rate(m, lat->h_order[r]) == m->s_high) continue;
    const double* h = lat->Hh + size_t(r) * Q;
    int cl = 0;
    for (int a = 0; a < D; ++a) {
      double s = 0.0;  // <H_r, H_r reflected in axis a>
      for (int i = 0; i < Q; ++i) s += h[i] * h[mirror.v[a][i]];
      if (s < 0.0) cl |= 1 << a;
    }
    rows[cl][count[cl]++] = r;
  }
  // s_high as the kernel has it (make_step_params): A and 1 - s_high come from one value, or the rows that carry
  // mass and momentum would grow by its rounding at every step (s_high = 1.05 in FP32: 4.8e-8)
  const double sh = fp64 ? m->s_high : double(float(m->s_high)), oms = 1.0 - sh;
  for (int b = 0; b < B::blocks(); ++b) {
    const int o = B::block_off(b), n = B::block_size(b);
    double* M = c + B::coef_off(b);
    for (int k = 0; k < n; ++k)
      for (int l = 0; l < n; ++l) {
        double v = k == l ? oms / ((fp64 ? lat->w[rep[o + k]] : double(lat->wf[rep[o + k]])) * members[o + k]) : 0.0;
        for (int q = 0; q < count[cls[o + k]]; ++q) {
          const int r = rows[cls[o + k]][q];
          const double* h = lat->Hh + size_t(r) * Q;
          v -= (high_rate(m, lat->h_order[r]) - sh) / lat->Nh[r] * h[rep[o + k]] * h[rep[o + l]];
        }
        const bool odd = (((cls[o + k] & 1) + ((cls[o + k] >> 1) & 1) + ((cls[o + k] >> 2) & 1)) & 1) != 0;
        M[k * n + l] = odd ? v / mult[o + k] : v;
      }
  }
}

}  // namespace lbm
