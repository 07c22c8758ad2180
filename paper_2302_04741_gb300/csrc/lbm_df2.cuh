// lbm_df2.cuh -- the float-float FP64 step in packed FP32.
//
// What bounds the float-float step: instruction issue, and the fetch of its
// long code (6,700 instructions a site in scalar form, 107 KB straight-line, with
// no_instruction its top stall at 3.2 per issue).  A packed instruction (add / mul / fma.rn.f32x2) does two float
// operations, rounded as the scalar ones.  The two values of a pack here are the
// two members of an opposite pair, or its even and odd part (sum s and
// difference a, w G_even and w G_odd), or the x and y component: nearly all of
// the step acts on both alike.  A pack's operand may be negated, broadcast or
// swapped at no cost, so (s, a) from (d+, d-) and (f+, f-) from (even, odd) are
// one addition with the signs (1, -1).
// GB300, 1024 x 512 D2Q37, under ncu: 165 us a step in scalar form, 149 packed
// and inline (5,280 instructions), 132 with a pair's ends out of line (5,600
// instructions, no_instruction 0.8); ten steps and the read-out 1.62 -> 1.34 ms.
// The error against 64 bits is that of the scalar form (q after ten steps
// 3.4e-12).
#pragma once

#include "lbm_poly.cuh"

namespace lbm {

struct DF2 {
  float2 hi, lo;
};
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 bx(float2 a) { return make_float2(a.x, a.x); }
__device__ __forceinline__ float2 by(float2 a) { return make_float2(a.y, a.y); }
__device__ __forceinline__ float2 neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ DF2 pack(DF x, DF y) { return DF2{f2(x.hi, y.hi), f2(x.lo, y.lo)}; }
__device__ __forceinline__ DF2 both(DF x) { return DF2{f2(x.hi, x.hi), f2(x.lo, x.lo)}; }
__device__ __forceinline__ DF px(DF2 v) { return DF(v.hi.x, v.lo.x); }
__device__ __forceinline__ DF py(DF2 v) { return DF(v.hi.y, v.lo.y); }
__device__ __forceinline__ DF2 bx(DF2 v) { return DF2{bx(v.hi), bx(v.lo)}; }
__device__ __forceinline__ DF2 by(DF2 v) { return DF2{by(v.hi), by(v.lo)}; }
__device__ __forceinline__ DF2 operator-(DF2 a) { return DF2{neg(a.hi), neg(a.lo)}; }

// s + e: the renormalised pair of a sum s and its error e
__device__ __forceinline__ DF2 renorm(float2 s, float2 e) {
  DF2 r;
  r.hi = __fadd2_rn(s, e);
  r.lo = __fadd2_rn(e, neg(__fadd2_rn(r.hi, neg(s))));
  return r;
}
// sum s of a and b and everything else e (two_sum and the lo parts)
__device__ __forceinline__ void add_parts(DF2 a, DF2 b, float2& s, float2& e) {
  s = __fadd2_rn(a.hi, b.hi);
  const float2 bb = __fadd2_rn(s, neg(a.hi));
  e = __fadd2_rn(__fadd2_rn(a.hi, neg(__fadd2_rn(s, neg(bb)))), __fadd2_rn(b.hi, neg(bb)));
  e = __fadd2_rn(e, __fadd2_rn(a.lo, b.lo));
}
__device__ __forceinline__ DF2 operator+(DF2 a, DF2 b) {
  float2 s, e;
  add_parts(a, b, s, e);
  return renorm(s, e);
}
__device__ __forceinline__ DF2 operator-(DF2 a, DF2 b) { return a + (-b); }
// (a.x + b.x, a.y - b.y), without renormalisation
__device__ __forceinline__ DF2 add_pm(DF2 a, DF2 b) {
  const float2 pm = f2(1.f, -1.f);
  DF2 r;
  r.hi = __ffma2_rn(b.hi, pm, a.hi);
  const float2 bb = __fadd2_rn(r.hi, neg(a.hi));
  const float2 e = __fadd2_rn(__fadd2_rn(a.hi, neg(__fadd2_rn(r.hi, neg(bb)))), __ffma2_rn(b.hi, pm, neg(bb)));
  r.lo = __fadd2_rn(e, __ffma2_rn(b.lo, pm, a.lo));
  return r;
}
__device__ __forceinline__ DF2 operator*(DF2 a, DF2 b) {
  DF2 r;
  r.hi = __fmul2_rn(a.hi, b.hi);
  r.lo = __ffma2_rn(a.lo, b.hi, __ffma2_rn(a.hi, b.lo, __ffma2_rn(a.hi, b.hi, neg(r.hi))));
  return r;
}
// a * b + c
__device__ __forceinline__ DF2 fma(DF2 a, DF2 b, DF2 c) {
  float2 s, e;
  add_parts(a * b, c, s, e);
  return renorm(s, e);
}
// v times exact floats (kx, ky), and acc + that
__device__ __forceinline__ DF2 mulf(float kx, float ky, DF2 v) {
  const float2 k = f2(kx, ky);
  DF2 r;
  r.hi = __fmul2_rn(k, v.hi);
  r.lo = __ffma2_rn(k, v.lo, __ffma2_rn(k, v.hi, neg(r.hi)));
  return r;
}
template <int K>
__device__ __forceinline__ DF2 kmac(DF2 v, DF2 acc) {
  if constexpr (K == 1) return acc + v;
  else if constexpr ((K & (K - 1)) == 0)
    return acc + DF2{__fmul2_rn(f2(K, K), v.hi), __fmul2_rn(f2(K, K), v.lo)};
  else return acc + mulf(K, K, v);
}
// v times the constants (kx, ky), each carried as hi + lo
__device__ __forceinline__ DF2 cmul2(double kx, double ky, DF2 v) {
  const DF x = DF(kx), y = DF(ky);
  return pack(x, y) * v;
}

// Pair sums and differences (s, a) of the deviations from the stored values of
// a pair, and from its deviations.
__device__ __forceinline__ DF2 sum_diff(DF2 d) {
  const DF2 r = add_pm(bx(d), by(d));
  return renorm(r.hi, r.lo);
}

// The ends of a pair's path, out of line: one copy of each for all pairs, so
// that the kernel's code stays near the size of the instruction caches (inline:
// 84 KB, with no_instruction 3.5 stalls per issue).
// (s, a) of the deviations from w of a pair's stored values
static __device__ __noinline__ DF2 pair_in(double fp, double fm, float w_hi, float w_lo) {
  const DF2 f = pack(df_split_raw(fp), df_split_raw(fm));
  return sum_diff(renorm(f.hi, f.lo) - both(DF(w_hi, w_lo)));
}
// The stored values w + (even +- odd) of a relaxed pair, (even, odd) = hom1 (s, a)
// + w G, each rounded to double by the sum of its two parts.
static __device__ __noinline__ double2 pair_out(DF hom1, DF2 v, DF2 wg, float w_hi, float w_lo) {
  const DF2 eo = fma(both(hom1), v, wg);
  float2 hi, lo;
  add_parts(both(DF(w_hi, w_lo)), add_pm(bx(eo), by(eo)), hi, lo);
  return make_double2(df_round(hi.x, lo.x), df_round(hi.y, lo.y));
}

template <class L, int X, int Y, int Z>
__device__ __forceinline__ DF2 at2(const DF2 (&v)[(L::Q - 1) / 2]) {
  constexpr int k = pair_of<L>(X, Y, Z);
  static_assert(k >= 0, "no such pair");
  return v[k];
}

// drho, j and k2 from the (s, a) of the pairs (pair_moments): rows of one |e_a|
// carry the sums for k2 in x and for j_a in y.
template <class L>
__device__ __forceinline__ RawMoments<L, DF> pair_moments2(DF d0, const DF2 (&v)[(L::Q - 1) / 2]) {
  RawMoments<L, DF> r;
  // (k2, j) of one axis from its rows of |e_a| = 1, 2, 3
  auto axis = [](DF2 r1, DF2 r2, DF2 r3, DF& k2, DF& j) {
    const DF2 t = r1 + DF2{__fmul2_rn(f2(4.f, 2.f), r2.hi), __fmul2_rn(f2(4.f, 2.f), r2.lo)};
    const DF2 m = t + mulf(9.f, 3.f, r3);
    k2 = px(m);
    j = py(m);
  };
  DF kx, ky;
  if constexpr (L::D == 2) {
    const DF2 t11 = at2<L, 1, 1, 0>(v) + at2<L, 1, -1, 0>(v), u11 = at2<L, 1, 1, 0>(v) - at2<L, 1, -1, 0>(v);
    const DF2 t22 = at2<L, 2, 2, 0>(v) + at2<L, 2, -2, 0>(v), u22 = at2<L, 2, 2, 0>(v) - at2<L, 2, -2, 0>(v);
    const DF2 t21 = at2<L, 2, 1, 0>(v) + at2<L, 2, -1, 0>(v), u21 = at2<L, 2, 1, 0>(v) - at2<L, 2, -1, 0>(v);
    const DF2 t12 = at2<L, 1, 2, 0>(v) + at2<L, 1, -2, 0>(v), u12 = at2<L, 1, 2, 0>(v) - at2<L, 1, -2, 0>(v);
    const DF2 t31 = at2<L, 3, 1, 0>(v) + at2<L, 3, -1, 0>(v), u31 = at2<L, 3, 1, 0>(v) - at2<L, 3, -1, 0>(v);
    const DF2 t13 = at2<L, 1, 3, 0>(v) + at2<L, 1, -3, 0>(v), u13 = at2<L, 1, 3, 0>(v) - at2<L, 1, -3, 0>(v);
    const DF2 x1 = (at2<L, 1, 0, 0>(v) + t11) + (t12 + t13), x2 = at2<L, 2, 0, 0>(v) + (t21 + t22),
              x3 = at2<L, 3, 0, 0>(v) + t31;
    axis(x1, x2, x3, kx, r.j[0]);
    // the same with the part odd in y
    auto mix = [](DF2 t, DF2 u) { return pack(px(t), py(u)); };
    const DF2 y1 = (at2<L, 0, 1, 0>(v) + mix(t11, u11)) + (mix(t21, u21) + mix(t31, u31)),
              y2 = at2<L, 0, 2, 0>(v) + (mix(t12, u12) + mix(t22, u22)), y3 = at2<L, 0, 3, 0>(v) + mix(t13, u13);
    axis(y1, y2, y3, ky, r.j[1]);
    r.j[2] = DF();
    const DF x0 = (d0 + px(at2<L, 0, 1, 0>(v))) + (px(at2<L, 0, 2, 0>(v)) + px(at2<L, 0, 3, 0>(v)));
    r.drho = (x0 + px(x1)) + (px(x2) + px(x3));
    r.k2 = kx + ky;
  } else {
    auto mix = [](DF2 t, DF2 u) { return pack(px(t), py(u)); };
    const DF2 t1 = at2<L, 1, 1, 1>(v) + at2<L, 1, 1, -1>(v), t2 = at2<L, 1, -1, 1>(v) + at2<L, 1, -1, -1>(v);
    const DF2 u1 = at2<L, 1, 1, 1>(v) - at2<L, 1, 1, -1>(v), u2 = at2<L, 1, -1, 1>(v) - at2<L, 1, -1, -1>(v);
    const DF2 ox = t1 + t2, oy = mix(ox, t1 - t2), oz = mix(ox, u1 + u2);
    const DF2 xy = at2<L, 2, 2, 0>(v) + at2<L, 2, -2, 0>(v), yx = mix(xy, at2<L, 2, 2, 0>(v) - at2<L, 2, -2, 0>(v));
    const DF2 xz = at2<L, 2, 0, 2>(v) + at2<L, 2, 0, -2>(v), zx = mix(xz, at2<L, 2, 0, 2>(v) - at2<L, 2, 0, -2>(v));
    const DF2 yz = at2<L, 0, 2, 2>(v) + at2<L, 0, 2, -2>(v), zy = mix(yz, at2<L, 0, 2, 2>(v) - at2<L, 0, 2, -2>(v));
    DF kz;
    axis(at2<L, 1, 0, 0>(v) + ox, at2<L, 2, 0, 0>(v) + (xy + xz), at2<L, 3, 0, 0>(v), kx, r.j[0]);
    axis(at2<L, 0, 1, 0>(v) + oy, at2<L, 0, 2, 0>(v) + (yx + yz), at2<L, 0, 3, 0>(v), ky, r.j[1]);
    axis(at2<L, 0, 0, 1>(v) + oz, at2<L, 0, 0, 2>(v) + (zx + zy), at2<L, 0, 0, 3>(v), kz, r.j[2]);
    r.k2 = (kx + ky) + kz;
    // the axes' sums of all three |e|, x and y in one pack
    const DF2 sxy = (pack(px(at2<L, 1, 0, 0>(v)), px(at2<L, 0, 1, 0>(v))) + pack(px(at2<L, 2, 0, 0>(v)), px(at2<L, 0, 2, 0>(v)))) +
                    pack(px(at2<L, 3, 0, 0>(v)), px(at2<L, 0, 3, 0>(v)));
    const DF sz = (px(at2<L, 0, 0, 1>(v)) + px(at2<L, 0, 0, 2>(v))) + px(at2<L, 0, 0, 3>(v));
    r.drho = (d0 + (px(sxy) + py(sxy))) + ((sz + px(ox)) + ((px(xy) + px(xz)) + px(yz)));
  }
  return r;
}

// The coefficients of the polynomial (poly_coef, lbm_poly.cuh), those of x and y
// in one pack.
template <int FO>
__device__ __forceinline__ void poly_coef2(const SiteState<DF>& m, PolyCoef2<DF>& k) {
  const DF2 U = pack(m.U[0], m.U[1]), S = pack(m.S[0], m.S[1]);
  const DF2 XX = U * U;
  const DF xy = m.U[0] * m.U[1];
  const DF hu2 = half_of(m.u2);
  const DF b0 = DF(1) - kmac<2>(m.Th, hu2);
  const DF2 AX = both(m.T) + XX, HAX = DF2{__fmul2_rn(f2(0.5f, 0.5f), AX.hi), __fmul2_rn(f2(0.5f, 0.5f), AX.lo)};
  const DF T3 = kscale<3>(m.T), th2 = half_of(m.Th);
  const DF2 T3X = both(T3) + XX;
  const DF a00 = fma(hmac(half_of(hu2), m.Th), m.u2, fma(m.Th, m.Th, -(hu2 + m.Th)));
  k.E00 = fma(m.rom, a00, FO >= 1 ? fma(m.om, m.drho, -m.rkgu) : m.om * m.drho);
  DF2 E2 = both(m.rom) * fma(both(b0), HAX, -(both(th2) * XX));
  k.E11 = m.rom * (b0 - m.Th) * xy;
  const DF q = m.rom * DF(1.0 / 24.0);
  const DF2 E4 = both(q) * fma(XX, kmac<2>(both(T3), XX), both(T3 * m.T));
  k.E22 = m.rom * px(HAX) * py(HAX);
  const DF2 R = both(m.rom) * U;
  DF2 O3 = cmul2(1.0 / 6.0, 1.0 / 6.0, R) * T3X;
  const DF2 E3 = O3 * DF2{f2(U.hi.y, U.hi.x), f2(U.lo.y, U.lo.x)};
  if constexpr (FO >= 1) {
    E2 = fma(S, U, E2);
    k.E11 = fma(m.S[0], m.U[1], fma(m.S[1], m.U[0], k.E11));
  }
  DF2 O1, O2;
  if constexpr (FO >= 2) {
    const DF2 P = R + S;
    O1 = fma(both(b0), P, -(both(m.rkgu) * U));
    O3 = fma(HAX, S, O3);
    O2 = fma(HAX, DF2{f2(P.hi.y, P.hi.x), f2(P.lo.y, P.lo.x)}, S * both(xy));
  } else {
    O1 = fma(both(b0), R, S);
    O2 = HAX * DF2{f2(R.hi.y, R.hi.x), f2(R.lo.y, R.lo.x)};
  }
  k.E20 = px(E2); k.E02 = py(E2);
  k.E40 = px(E4); k.E04 = py(E4);
  k.E31 = px(E3); k.E13 = py(E3);
  k.O10 = px(O1); k.O01 = py(O1);
  k.O30 = px(O3); k.O03 = py(O3);
  k.O21 = px(O2); k.O12 = py(O2);
}

// (w G_even, w G_odd) of every pair, handed to out(pair, value): poly_pairs.
template <class L, class OUT>
__device__ __forceinline__ void poly_pairs2(const PolyCoef2<DF>& k, OUT&& out) {
  static_for<0, 4>([&](auto A) {
    constexpr int a = A, aa = a * a;
    DF2 xz = pack(k.E00, k.O10), yw = pack(k.E11, k.O01);  // (even, odd in x) and (odd in both, odd in y)
    DF xb = k.E02;
    if constexpr (a > 0) {
      xz = kmac<aa>(pack(kmac<aa>(k.E40, k.E20), k.O30), xz);
      yw = kmac<aa>(pack(k.E31, k.O21), yw);
      xb = kmac<aa>(k.E22, k.E02);
      constexpr double w = L::W(2 * pair_of<L>(a, 0, 0) + 1);
      out(ic<pair_of<L>(a, 0, 0)>{}, cmul2(w, w * a, xz));
    }
    static_for<1, 4>([&](auto B) {
      constexpr int b = B, bb = b * b;
      if constexpr (a == 0) {
        constexpr double w = L::W(2 * pair_of<L>(0, b, 0) + 1);
        const DF2 e = kmac<bb>(pack(kmac<bb>(k.E04, xb), k.O03), pack(k.E00, k.O01));
        out(ic<pair_of<L>(0, b, 0)>{}, cmul2(w, w * b, e));
      } else if constexpr (pair_of<L>(a, b, 0) >= 0) {
        constexpr double w = L::W(2 * pair_of<L>(a, b, 0) + 1);
        const DF2 p = cmul2(w, w * a, kmac<bb>(pack(kmac<bb>(k.E04, xb), k.O12), xz));
        const DF2 q = cmul2(w * a * b, w * b, kmac<bb>(pack(k.E13, k.O03), yw));
        out(ic<pair_of<L>(a, b, 0)>{}, p + q);
        out(ic<pair_of<L>(a, -b, 0)>{}, p - q);
      }
    });
  });
}
template <class L, class OUT>
__device__ __forceinline__ void poly_pairs2(const PolyCoef3<DF>& k, OUT&& out) {
  static_for<0, 3>([&](auto C) {
    constexpr int c = C;
    const DF2 o = pack(k.e0, k.o1[c]), s = pack(k.e2[c], k.o3[c]);
    static_for<1, 4>([&](auto A) {
      constexpr int a = A, kp = pair_of<L>(c == 0 ? a : 0, c == 1 ? a : 0, c == 2 ? a : 0);
      constexpr double w = L::W(2 * kp + 1);
      out(ic<kp>{}, cmul2(w, w * a, kmac<a * a>(s, o)));
    });
  });
  {
    constexpr double w = L::W(2 * pair_of<L>(1, 1, 1) + 1);
    const DF2 a = cmul2(w, w, pack(k.e0 + k.e2[0] + (k.e2[1] + k.e2[2]), k.o1[0] + k.o3[0] + (k.o21[1][0] + k.o21[2][0])));
    const DF2 b = cmul2(w, w, pack(k.e11[0], k.o1[1] + k.o3[1] + (k.o21[0][1] + k.o21[2][1])));
    const DF2 f = cmul2(w, w, pack(k.e11[1], k.o1[2] + k.o3[2] + (k.o21[0][2] + k.o21[1][2])));
    const DF2 g = cmul2(w, w, pack(k.e11[2], k.o111));
    const DF2 ep = a + b, em = a - b, qp = f + g, qm = f - g;
    out(ic<pair_of<L>(1, 1, 1)>{}, ep + qp);
    out(ic<pair_of<L>(1, 1, -1)>{}, ep - qp);
    out(ic<pair_of<L>(1, -1, 1)>{}, em + qm);
    out(ic<pair_of<L>(1, -1, -1)>{}, em - qm);
  }
  static_for<0, 3>([&](auto C) {  // planes (x, y), (x, z), (y, z)
    constexpr int c = C, p = c == 2 ? 1 : 0, r = c == 0 ? 1 : 2;
    constexpr int kp = c == 0 ? pair_of<L>(2, 2, 0) : (c == 1 ? pair_of<L>(2, 0, 2) : pair_of<L>(0, 2, 2));
    constexpr int km = c == 0 ? pair_of<L>(2, -2, 0) : (c == 1 ? pair_of<L>(2, 0, -2) : pair_of<L>(0, 2, -2));
    constexpr double w = L::W(2 * kp + 1);
    const DF2 a = cmul2(w, 2 * w, kmac<4>(pack(k.e2[p] + k.e2[r], k.o3[p] + k.o21[r][p]), pack(k.e0, k.o1[p])));
    const DF2 b = cmul2(4 * w, 2 * w, pack(k.e11[c], kmac<4>(k.o3[r] + k.o21[p][r], k.o1[r])));
    out(ic<kp>{}, a + b);
    out(ic<km>{}, a - b);
  });
}

}  // namespace lbm
