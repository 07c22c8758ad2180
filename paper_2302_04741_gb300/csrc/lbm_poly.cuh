// lbm_poly.cuh -- the collision of the FP64 step kernels (IEEE double and
// float-float), evaluated by parity classes instead of direction by direction.
//
// What bounds these kernels: the FP64 step is bound by the SM's FP64 unit (on
// GB300 a warp's FP64 instruction occupies it for 19 cycles, 64 when only one
// of the four sub-partitions uses it, whatever its number of active lanes), the
// float-float step by instruction issue.  In both the time is the number of
// arithmetic operations per site, so this form is chosen to need few.
//
// Equilibrium and force together are, at one site, a polynomial in the lattice
// vector e (total degree 4 on D2Q37, 3 on D3Q39):
//   f*_i - w_i = (1 - om) d_i + w_i G(e_i),
//   G(e) = om drho + rho om p(e) + rho (1 - om/2) F'(e).
// Directions that differ only in signs share the parts of G that are even or
// odd in each component, so G's monomial coefficients are formed once per site
// (PolyCoef) and each mirror group (+-a, +-b) evaluates its four parity parts
// once for its four members; the update of a pair (e, -e) stays
// (even part) +- (odd part), so the rounding of the even part cancels in the
// momentum.  The relaxed d enters as the pair's sum s and difference a, which
// the moments use too.
//
// Measured on GB300 (ten steps of 1024 x 512 D2Q37 sites and their read-out,
// against the same body evaluated pair by pair in t = xi.u): IEEE double 6.46 ->
// 4.50 ms; float-float 2.51 -> 1.70 ms (with df_split free of conversions), 1.33 ms
// in packed FP32 (lbm_df2.cuh); D3Q39, 61 x 47 x 53 in double, 20 steps: 3.60 -> 2.75 ms.
//
// The errors of rho, u, T and q against an 80-bit evaluation of the method are those of
// the pair-by-pair body, each within 4 % or smaller, over channels at speed (3 x 150 up to
// 1,000 steps, 4 x 40 to 70 x 150), convection, Kolmogorov flow, boxes and cylinders (T of a
// 33 x 300 channel after 20 steps 5.8e-16 -> 6.5e-16).  That hangs on the places marked
// "error" below and in site_coefficients: a site whose state hardly changes repeats its
// rounding in every step.
#pragma once

#include "lbm_device.cuh"

namespace lbm {

// Pair index k of the pair (e, -e) whose first member 2k + 1 is (ex, ey, ez);
// -1 when the lattice has none.
template <class L>
__host__ __device__ constexpr int pair_of(int ex, int ey, int ez) {
  for (int k = 0; k < (L::Q - 1) / 2; ++k)
    if (L::E(2 * k + 1, 0) == ex && L::E(2 * k + 1, 1) == ey && L::E(2 * k + 1, 2) == ez) return k;
  return -1;
}

// the entry of pair (X, Y, Z) in an array over pairs
template <class L, int X, int Y, int Z, class R, int N>
__device__ __forceinline__ R at(const R (&v)[N]) {
  constexpr int k = pair_of<L>(X, Y, Z);
  static_assert(k >= 0, "no such pair");
  return v[k];
}

// v times a compile-time integer, and acc + K v
template <int K>
__device__ __forceinline__ double kscale(double v) {
  if constexpr (K == 1) return v;
  else return double(K) * v;
}
template <int K>
__device__ __forceinline__ DF kscale(DF v) {
  if constexpr (K == 1) return v;
  else if constexpr ((K & (K - 1)) == 0) return DF(float(K) * v.hi, float(K) * v.lo);  // exact
  else return df_mulf(float(K), v);
}
template <int K, class R>
__device__ __forceinline__ R kmac(R v, R acc) {
  if constexpr (K == 1) return acc + v;
  else if constexpr (K == -1) return acc - v;
  else if constexpr (std::is_same<R, DF>::value) return K > 0 ? acc + kscale<K>(v) : acc - kscale<-K>(v);
  else return fma(R(K), v, acc);
}
// acc + k v for a quadrature constant k known at compile time
__device__ __forceinline__ double cmac(double k, double v, double acc) { return fma(k, v, acc); }
__device__ __forceinline__ DF cmac(double k, DF v, DF acc) { return fma(DF(k), v, acc); }
__device__ __forceinline__ double cmul(double k, double v) { return k * v; }
__device__ __forceinline__ DF cmul(double k, DF v) { return DF(k) * v; }
// acc + v / 2 and half of v
__device__ __forceinline__ double hmac(double v, double acc) { return fma(0.5, v, acc); }
__device__ __forceinline__ DF hmac(DF v, DF acc) { return acc + DF(0.5f * v.hi, 0.5f * v.lo); }
__device__ __forceinline__ double half_of(double v) { return 0.5 * v; }
__device__ __forceinline__ DF half_of(DF v) { return DF(0.5f * v.hi, 0.5f * v.lo); }
// 3/2 of v
__device__ __forceinline__ double sesqui(double v) { return 1.5 * v; }
__device__ __forceinline__ DF sesqui(DF v) { return df_mulf(1.5f, v); }

// Raw moments of the deviations from the pair sums s and differences a
// (drho, j, k2 as RawMoments): mirror groups first, then the shells.
template <class L, class R>
__device__ __forceinline__ RawMoments<L, R> pair_moments(R d0, const R (&s)[(L::Q - 1) / 2], const R (&a)[(L::Q - 1) / 2]) {
  RawMoments<L, R> r;
  if constexpr (L::D == 2) {
    // sums of the mirror groups (x, +-y): even, odd in x, odd in y
    auto S = [&](auto X, auto Y) { return at<L, X, Y, 0>(s) + at<L, X, -Y, 0>(s); };
    auto Ax = [&](auto X, auto Y) { return at<L, X, Y, 0>(a) + at<L, X, -Y, 0>(a); };
    auto Ay = [&](auto X, auto Y) { return at<L, X, Y, 0>(a) - at<L, X, -Y, 0>(a); };
    constexpr ic<1> _1{};
    constexpr ic<2> _2{};
    constexpr ic<3> _3{};
    const R s1 = at<L, 1, 0, 0>(s) + at<L, 0, 1, 0>(s), s2 = S(_1, _1), s4 = at<L, 2, 0, 0>(s) + at<L, 0, 2, 0>(s), s5 = S(_2, _1) + S(_1, _2),
            s8 = S(_2, _2), s9 = at<L, 3, 0, 0>(s) + at<L, 0, 3, 0>(s), s10 = S(_3, _1) + S(_1, _3);
    r.drho = d0 + (((s1 + s2) + (s4 + s5)) + ((s8 + s9) + s10));
    R k2 = kmac<2>(s2, s1);
    k2 = kmac<4>(s4, k2);
    k2 = kmac<5>(s5, k2);
    k2 = kmac<8>(s8, k2);
    k2 = kmac<9>(s9, k2);
    r.k2 = kmac<10>(s10, k2);
    const R x1 = (at<L, 1, 0, 0>(a) + Ax(_1, _1)) + (Ax(_1, _2) + Ax(_1, _3)), x2 = at<L, 2, 0, 0>(a) + (Ax(_2, _1) + Ax(_2, _2)),
            x3 = at<L, 3, 0, 0>(a) + Ax(_3, _1);
    const R y1 = (at<L, 0, 1, 0>(a) + Ay(_1, _1)) + (Ay(_2, _1) + Ay(_3, _1)), y2 = at<L, 0, 2, 0>(a) + (Ay(_1, _2) + Ay(_2, _2)),
            y3 = at<L, 0, 3, 0>(a) + Ay(_1, _3);
    r.j[0] = kmac<3>(x3, kmac<2>(x2, x1));
    r.j[1] = kmac<3>(y3, kmac<2>(y2, y1));
    r.j[2] = R(0);
  } else {
    const R s1 = at<L, 1, 0, 0>(s) + at<L, 0, 1, 0>(s) + at<L, 0, 0, 1>(s);
    const R s3 = (at<L, 1, 1, 1>(s) + at<L, 1, 1, -1>(s)) + (at<L, 1, -1, 1>(s) + at<L, 1, -1, -1>(s));
    const R s4 = at<L, 2, 0, 0>(s) + at<L, 0, 2, 0>(s) + at<L, 0, 0, 2>(s);
    const R s8 = (at<L, 2, 2, 0>(s) + at<L, 2, -2, 0>(s)) + (at<L, 2, 0, 2>(s) + at<L, 2, 0, -2>(s)) + (at<L, 0, 2, 2>(s) + at<L, 0, 2, -2>(s));
    const R s9 = at<L, 3, 0, 0>(s) + at<L, 0, 3, 0>(s) + at<L, 0, 0, 3>(s);
    r.drho = d0 + ((s1 + s3) + (s4 + (s8 + s9)));
    R k2 = kmac<3>(s3, s1);
    k2 = kmac<4>(s4, k2);
    k2 = kmac<8>(s8, k2);
    r.k2 = kmac<9>(s9, k2);
    const R u = at<L, 1, 1, 1>(a) + at<L, 1, 1, -1>(a), v = at<L, 1, -1, 1>(a) + at<L, 1, -1, -1>(a);
    const R x = at<L, 1, 1, 1>(a) - at<L, 1, 1, -1>(a), y = at<L, 1, -1, 1>(a) - at<L, 1, -1, -1>(a);
    const R x1 = at<L, 1, 0, 0>(a) + (u + v), y1 = at<L, 0, 1, 0>(a) + (u - v), z1 = at<L, 0, 0, 1>(a) + (x + y);
    const R x2 = at<L, 2, 0, 0>(a) + (at<L, 2, 2, 0>(a) + at<L, 2, -2, 0>(a)) + (at<L, 2, 0, 2>(a) + at<L, 2, 0, -2>(a));
    const R y2 = at<L, 0, 2, 0>(a) + (at<L, 2, 2, 0>(a) - at<L, 2, -2, 0>(a)) + (at<L, 0, 2, 2>(a) + at<L, 0, 2, -2>(a));
    const R z2 = at<L, 0, 0, 2>(a) + (at<L, 2, 0, 2>(a) - at<L, 2, 0, -2>(a)) + (at<L, 0, 2, 2>(a) - at<L, 0, 2, -2>(a));
    r.j[0] = kmac<3>(at<L, 3, 0, 0>(a), kmac<2>(x2, x1));
    r.j[1] = kmac<3>(at<L, 0, 3, 0>(a), kmac<2>(y2, y1));
    r.j[2] = kmac<3>(at<L, 0, 0, 3>(a), kmac<2>(z2, z1));
  }
  return r;
}

// Monomial coefficients of G in e.  D = 2: even E00, E20 (x^2), E11, E02, E40,
// E31, E22, E13, E04; odd O10, O01, O30, O21 (x^2 y), O12, O03.  D = 3: even
// e0, e2[a] (a^2), e11 = (xy, xz, yz); odd o1[a], o3[a] (a^3), o21[a][b] (a^2 b),
// o111.
template <class R>
struct PolyCoef2 {
  R E00, E20, E11, E02, E40, E31, E22, E13, E04, O10, O01, O30, O21, O12, O03;
};
template <class R>
struct PolyCoef3 {
  R e0, e2[3], e11[3], o1[3], o3[3], o21[3][3], o111;
};

template <class R>
__device__ __forceinline__ R const_term(const PolyCoef2<R>& k) { return k.E00; }
template <class R>
__device__ __forceinline__ R const_term(const PolyCoef3<R>& k) { return k.e0; }

// What the coefficients are made of: rom = rho om, rk = rho (1 - om/2),
// U = c u, S = rk c g (the force), T = c^2 (theta - 1).
template <class R>
struct SiteState {
  R drho, rho, om, u2, Th, T, rom, rkgu, U[3], S[3];
};

// D2Q37 in double (float-float: poly_coef2).  With b0 = 1 - u2/2 - 2 Th and
// H = (T + U^2) / 2, written so that no product is formed twice and no halving costs
// an operation: E20 = rho om (b0 H - Th U^2 / 2), E31 = U_y times the equilibrium
// part of O30.  Error: 1/24 and 1/6, which are not doubles, multiply U^4 and U^3 only,
// not the terms in T.
template <int FO>
__device__ __forceinline__ void poly_coef(const SiteState<double>& m, PolyCoef2<double>& k) {
  const double X = m.U[0], Y = m.U[1];
  const double xx = X * X, yy = Y * Y, xy = X * Y;
  const double b0 = fma(-0.5, m.u2, fma(-2.0, m.Th, 1.0));
  const double hT = 0.5 * m.T, hx = fma(0.5, xx, hT), hy = fma(0.5, yy, hT);
  const double th2 = 0.5 * m.Th;
  // a00 = -u2/2 - Th + (u2/8 + Th) u2 + Th^2
  const double a00 = fma(fma(0.125, m.u2, m.Th), m.u2, fma(m.Th, m.Th, fma(-0.5, m.u2, -m.Th)));
  k.E00 = fma(m.rom, a00, FO >= 1 ? fma(m.om, m.drho, -m.rkgu) : m.om * m.drho);
  k.E20 = m.rom * fma(b0, hx, -(th2 * xx));
  k.E02 = m.rom * fma(b0, hy, -(th2 * yy));
  k.E11 = m.rom * (b0 - m.Th) * xy;
  const double qT = 0.25 * m.T, e8 = 0.5 * hT * hT;
  k.E40 = m.rom * fma(xx, fma(1.0 / 24.0, xx, qT), e8);
  k.E04 = m.rom * fma(yy, fma(1.0 / 24.0, yy, qT), e8);
  k.E22 = m.rom * hx * hy;
  const double rx = m.rom * X, ry = m.rom * Y;
  k.O30 = rx * fma(1.0 / 6.0, xx, hT);
  k.O03 = ry * fma(1.0 / 6.0, yy, hT);
  k.E31 = k.O30 * Y;
  k.E13 = k.O03 * X;
  if constexpr (FO >= 1) {
    k.E20 = fma(m.S[0], X, k.E20);
    k.E02 = fma(m.S[1], Y, k.E02);
    k.E11 = fma(m.S[0], Y, fma(m.S[1], X, k.E11));
  }
  if constexpr (FO >= 2) {
    const double px = rx + m.S[0], py = ry + m.S[1];
    k.O10 = fma(b0, px, -(m.rkgu * X));
    k.O01 = fma(b0, py, -(m.rkgu * Y));
    k.O30 = fma(hx, m.S[0], k.O30);
    k.O03 = fma(hy, m.S[1], k.O03);
    k.O21 = fma(hx, py, m.S[0] * xy);
    k.O12 = fma(hy, px, m.S[1] * xy);
  } else {
    k.O10 = fma(b0, rx, m.S[0]);
    k.O01 = fma(b0, ry, m.S[1]);
    k.O21 = hx * ry;
    k.O12 = hy * rx;
  }
}

template <int FO, class R>
__device__ __forceinline__ void poly_coef(const SiteState<R>& m, PolyCoef3<R>& k) {
  const R A = hmac(m.u2, sesqui(m.Th));  // u2/2 + 3/2 Th
  k.e0 = fma(m.rom, -A, FO >= 1 ? fma(m.om, m.drho, -m.rkgu) : m.om * m.drho);
  const R b0 = R(1) - (A + m.Th);
  const R hT = half_of(m.T);
  R uu[3], h[3], r[3], p[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    uu[a] = m.U[a] * m.U[a];
    h[a] = hmac(uu[a], hT);
    r[a] = m.rom * m.U[a];
    k.e2[a] = m.rom * h[a];
    k.o3[a] = r[a] * cmac(1.0 / 6.0, uu[a], hT);
    if constexpr (FO >= 1) k.e2[a] = fma(m.S[a], m.U[a], k.e2[a]);
    if constexpr (FO >= 2) {
      p[a] = r[a] + m.S[a];
      k.o1[a] = fma(b0, p[a], -(m.rkgu * m.U[a]));
      k.o3[a] = fma(h[a], m.S[a], k.o3[a]);
    } else {
      p[a] = r[a];
      k.o1[a] = fma(b0, r[a], m.S[a]);
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {  // (x, y), (x, z), (y, z)
    const int a = c == 2 ? 1 : 0, b = c == 0 ? 1 : 2;
    const R ab = m.U[a] * m.U[b];
    k.e11[c] = m.rom * ab;
    k.o21[a][b] = h[a] * p[b];
    k.o21[b][a] = h[b] * p[a];
    if constexpr (FO >= 1) k.e11[c] = fma(m.S[a], m.U[b], fma(m.S[b], m.U[a], k.e11[c]));
    if constexpr (FO >= 2) {
      k.o21[a][b] = fma(m.S[a], ab, k.o21[a][b]);
      k.o21[b][a] = fma(m.S[b], ab, k.o21[b][a]);
    }
    if (c == 0) {
      k.o111 = r[2] * ab;
      if constexpr (FO >= 2) k.o111 = fma(m.S[2], ab, k.o111);
    } else if constexpr (FO >= 2) {
      k.o111 = fma(m.S[c == 1 ? 1 : 0], ab, k.o111);
    }
  }
}

// The sigma-bar terms of the force (FO 3): the odd part gains the cubic
// (gs.e)(e.S.e) - hs.e (see stress_terms).
template <class R>
__device__ __forceinline__ void poly_add_stress(const StressTerms<R>& st, PolyCoef2<R>& k) {
  k.O10 = k.O10 - st.hs[0];
  k.O01 = k.O01 - st.hs[1];
  k.O30 = fma(st.gs[0], st.S[0], k.O30);
  k.O03 = fma(st.gs[1], st.S[1], k.O03);
  k.O21 = fma(st.gs[1], st.S[0], fma(kscale<2>(st.gs[0]), st.S[3], k.O21));
  k.O12 = fma(st.gs[0], st.S[1], fma(kscale<2>(st.gs[1]), st.S[3], k.O12));
}
template <class R>
__device__ __forceinline__ void poly_add_stress(const StressTerms<R>& st, PolyCoef3<R>& k) {
  constexpr int off[3][3] = {{0, 3, 4}, {3, 1, 5}, {4, 5, 2}};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    k.o1[a] = k.o1[a] - st.hs[a];
    k.o3[a] = fma(st.gs[a], st.S[off[a][a]], k.o3[a]);
#pragma unroll
    for (int b = 0; b < 3; ++b)
      if (a != b) k.o21[a][b] = fma(st.gs[b], st.S[off[a][a]], fma(kscale<2>(st.gs[a]), st.S[off[a][b]], k.o21[a][b]));
  }
  const R c = fma(st.gs[0], st.S[5], fma(st.gs[1], st.S[4], st.gs[2] * st.S[3]));
  k.o111 = kmac<2>(c, k.o111);
}

// The weight of direction i in the double collision.  Rounding the weights to double leaves a
// collision that creates a little mass and energy, the same ones in every step of a steady
// site; on D2Q37 two weights are rounded to their other neighbour, which lowers both by an
// eighth at rest (energy 3.0e-17 -> 2.7e-17 a step at theta = 1.1).
template <class L>
__host__ __device__ constexpr double collision_w(int i) {
  if (L::D == 2 && L::E2(L::SH(i)) == 8) return L::W(i) - 0x1p-62;
  if (L::D == 2 && L::E2(L::SH(i)) == 9) return L::W(i) + 0x1p-64;
  return L::W(i);
}

// Even and odd part of w G at every pair, handed to out(pair, w G_even, w G_odd).
template <class L, class R, class OUT>
__device__ __forceinline__ void poly_pairs(const PolyCoef2<R>& k, OUT&& out) {
  auto pair = [&](auto X, auto Y, R wev, R wod) {
    out(ic<pair_of<L>(X, Y, 0)>{}, wev, wod);
  };
  static_for<0, 4>([&](auto A) {
    constexpr int aa = A * A;
    // parts that depend on |e_x| = A only
    R xa = k.E00, xb = k.E02, ya, za, wa = k.O01;
    if constexpr (A > 0) {
      xa = kmac<aa>(kmac<aa>(k.E40, k.E20), k.E00);
      xb = kmac<aa>(k.E22, k.E02);
      ya = kmac<aa>(k.E31, k.E11);
      za = kmac<aa>(k.O30, k.O10);
      wa = kmac<aa>(k.O21, k.O01);
      constexpr double w = collision_w<L>(2 * pair_of<L>(A, 0, 0) + 1);
      pair(A, ic<0>{}, cmul(w, xa), cmul(w * A, za));
    }
    static_for<1, 4>([&](auto B) {
      constexpr int bb = B * B;
      if constexpr (A == 0) {
        constexpr double w = collision_w<L>(2 * pair_of<L>(0, B, 0) + 1);
        pair(A, B, cmul(w, kmac<bb>(kmac<bb>(k.E04, xb), xa)), cmul(w * B, kmac<bb>(k.O03, wa)));
      } else if constexpr (pair_of<L>(A, B, 0) >= 0) {
        constexpr double w = collision_w<L>(2 * pair_of<L>(A, B, 0) + 1);
        const R ee = cmul(w, kmac<bb>(kmac<bb>(k.E04, xb), xa));
        const R oo = kmac<bb>(k.E13, ya);
        const R oe = cmul(w * A, kmac<bb>(k.O12, za));
        const R eo = kmac<bb>(k.O03, wa);
        pair(A, B, cmac(w * A * B, oo, ee), cmac(w * B, eo, oe));
        pair(A, ic<-int(B)>{}, cmac(-w * A * B, oo, ee), cmac(-w * B, eo, oe));
      }
    });
  });
}

template <class L, class R, class OUT>
__device__ __forceinline__ void poly_pairs(const PolyCoef3<R>& k, OUT&& out) {
  auto pair = [&](auto X, auto Y, auto Z, R wev, R wod) {
    out(ic<pair_of<L>(X, Y, Z)>{}, wev, wod);
  };
  constexpr ic<0> _0{};
  constexpr ic<1> _1{};
  constexpr ic<2> _2{};
  constexpr ic<-1> m1{};
  constexpr ic<-2> m2{};
  // axes: (a, 0, 0) and permutations
  static_for<1, 4>([&](auto A) {
    constexpr int aa = A * A;
    constexpr double w = L::W(2 * pair_of<L>(A, 0, 0) + 1);
    pair(A, _0, _0, cmul(w, kmac<aa>(k.e2[0], k.e0)), cmul(w * A, kmac<aa>(k.o3[0], k.o1[0])));
    pair(_0, A, _0, cmul(w, kmac<aa>(k.e2[1], k.e0)), cmul(w * A, kmac<aa>(k.o3[1], k.o1[1])));
    pair(_0, _0, A, cmul(w, kmac<aa>(k.e2[2], k.e0)), cmul(w * A, kmac<aa>(k.o3[2], k.o1[2])));
  });
  {  // (1, 1, 1) and its mirrors
    constexpr double w = L::W(2 * pair_of<L>(1, 1, 1) + 1);
    const R e = cmul(w, k.e0 + k.e2[0] + (k.e2[1] + k.e2[2]));
    const R xy = cmul(w, k.e11[0]), xz = cmul(w, k.e11[1]), yz = cmul(w, k.e11[2]);
    const R X = cmul(w, k.o1[0] + k.o3[0] + (k.o21[1][0] + k.o21[2][0]));
    const R Y = cmul(w, k.o1[1] + k.o3[1] + (k.o21[0][1] + k.o21[2][1]));
    const R Z = cmul(w, k.o1[2] + k.o3[2] + (k.o21[0][2] + k.o21[1][2]));
    const R C = cmul(w, k.o111);
    const R ep = e + xy, em = e - xy, qp = xz + yz, qm = xz - yz;
    const R op = X + Y, om = X - Y, zp = Z + C, zm = Z - C;
    pair(_1, _1, _1, ep + qp, op + zp);
    pair(_1, _1, m1, ep - qp, op - zp);
    pair(_1, m1, _1, em + qm, om + zm);
    pair(_1, m1, m1, em - qm, om - zm);
  }
  {  // (2, 2, 0) and permutations: coefficients of the plane (p, r)
    constexpr double w = L::W(2 * pair_of<L>(2, 2, 0) + 1);
    auto plane = [&](int p, int r, R c11, R& ee, R& oo, R& oe, R& eo) {
      ee = cmul(w, kmac<4>(k.e2[p] + k.e2[r], k.e0));
      oo = c11;
      oe = cmul(2 * w, kmac<4>(k.o3[p] + k.o21[r][p], k.o1[p]));
      eo = kmac<4>(k.o3[r] + k.o21[p][r], k.o1[r]);
    };
    R ee, oo, oe, eo;
    plane(0, 1, k.e11[0], ee, oo, oe, eo);
    pair(_2, _2, _0, cmac(4 * w, oo, ee), cmac(2 * w, eo, oe));
    pair(_2, m2, _0, cmac(-4 * w, oo, ee), cmac(-2 * w, eo, oe));
    plane(0, 2, k.e11[1], ee, oo, oe, eo);
    pair(_2, _0, _2, cmac(4 * w, oo, ee), cmac(2 * w, eo, oe));
    pair(_2, _0, m2, cmac(-4 * w, oo, ee), cmac(-2 * w, eo, oe));
    plane(1, 2, k.e11[2], ee, oo, oe, eo);
    pair(_0, _2, _2, cmac(4 * w, oo, ee), cmac(2 * w, eo, oe));
    pair(_0, _2, m2, cmac(-4 * w, oo, ee), cmac(-2 * w, eo, oe));
  }
}

}  // namespace lbm
