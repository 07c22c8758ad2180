// lbm_kernels.cuh -- the kernels of one lattice, included by one .cu per lattice.
//
// Storage: structure of arrays, population i of site s at f[i*N + s], sites
// row-major [nz][ny][nx] with x fastest; two buffers (ping-pong).  The stored
// buffer holds the post-collision distribution f*; a step pulls
// f~_i(x) = f*_i(x - e_i), collides (Eq. lbm) and stores f*_i(x) coalesced.
//
// Launch shape of the per-site kernels: blockDim = (bx, 1, 1) along x,
// grid = (ceil(nx / bx), ny, nz): every block works on one row, so the
// near-wall branch is uniform across a block.
#pragma once

#include "lbm_device.cuh"
#include "lbm_poly.cuh"
#include "lbm_df2.cuh"

namespace lbm {

template <int I>
__host__ __device__ constexpr int opposite() {
  return I == 0 ? 0 : ((I & 1) ? I + 1 : I - 1);
}

__device__ __forceinline__ int wrap3(int v, int n) {
  v += v < 0 ? n : 0;
  v -= v >= n ? n : 0;
  return v;
}

template <int D>
__device__ __forceinline__ void site_force(const StepParams& p, int x, int y, int z, int site,
                                           double (&g)[3]) {
  if (p.gkind == G_UNIFORM) {
    g[0] = p.g0[0]; g[1] = p.g0[1]; g[2] = p.g0[2];
  } else if (p.gkind == G_SINE) {
    const int k = p.gaxis == 0 ? x : (p.gaxis == 1 ? y : z);
    const double s = __ldg(p.gtab + k);
    g[0] = p.g0[0] * s; g[1] = p.g0[1] * s; g[2] = p.g0[2] * s;
  } else {
    g[0] = __ldg(p.gtab + site);
    g[1] = __ldg(p.gtab + (size_t)p.N + site);
    g[2] = D == 3 ? __ldg(p.gtab + 2 * (size_t)p.N + site) : 0.0;
  }
  if (D == 2) g[2] = 0.0;
}

// g(x) in the arithmetic type of the kernel (float kernels read float copies).
template <int D, class R>
__device__ __forceinline__ void site_force_r(const StepParams& p, int x, int y, int z, int site,
                                             R (&g)[3]) {
  using PP = ParamsOf<R>;
  if (p.gkind == G_UNIFORM) {
    g[0] = PP::g0(p, 0); g[1] = PP::g0(p, 1); g[2] = PP::g0(p, 2);
  } else if (p.gkind == G_SINE) {
    const int k = p.gaxis == 0 ? x : (p.gaxis == 1 ? y : z);
    const R s = PP::gtab(p, k);
    g[0] = PP::g0(p, 0) * s; g[1] = PP::g0(p, 1) * s; g[2] = PP::g0(p, 2) * s;
  } else {
    g[0] = PP::gtab(p, site);
    g[1] = PP::gtab(p, (size_t)p.N + site);
    g[2] = D == 3 ? PP::gtab(p, 2 * (size_t)p.N + site) : R(0);
  }
  if (D == 2) g[2] = R(0);
}

// What a pull returns per population: the deviation, the scaled value of an
// FP16-scaled step (see scaled_step), or the stored value itself (FP64 storage:
// the FP64 steps form pair sums and differences from it, see pair_split).
enum { IN_DEV = 0, IN_SCALED = 1, IN_STORED = 2 };
template <class L, int P, int I, int IN>
__device__ __forceinline__ typename Codec<P>::R pulled_value(typename Codec<P>::T v, const StepParams& p) {
  if constexpr (IN == IN_STORED) return v;
  else return step_in<L, P, I, IN == IN_SCALED>(v, p);
}

// Pull of site (x, y, z) of a row that no wall rule touches, with the periodic
// wrap of every axis (IN: what is returned, by default the stored values).
template <class L, int P, class RR, int LD = LD_HINT, int IN = IN_STORED>
__device__ __forceinline__ void pull_stored(const typename Codec<P>::T* __restrict__ fin,
                                          const StepParams& p, int x, int y, int z, RR (&d)[L::Q]) {
  using C = Codec<P>;
  constexpr int D = L::D, Q = L::Q;
  const int nx = p.nx, ny = p.ny, nz = p.nz;
  const size_t N = (size_t)p.N;
  int xs[7], ys[7], zs[7];
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    xs[k] = wrap3(x - (k - 3), nx);
    ys[k] = wrap3(y - (k - 3), ny) * nx;
    zs[k] = D == 3 ? wrap3(z - (k - 3), nz) * nx * ny : 0;
  }
  static_for<0, Q>([&](auto I) {
    constexpr int i = I;
    constexpr int ex = L::E(i, 0), ey = L::E(i, 1), ez = L::E(i, 2);
    const int off = zs[ez + 3] + ys[ey + 3] + xs[ex + 3];
    d[i] = RR(pulled_value<L, P, i, IN>(ldpop<C, LD>(fin + i * N + off, p), p));
  });
}

// Whether layer a of the wall axis pulls through a wall rule.
__device__ __forceinline__ bool near_wall(const StepParams& p, int a, int nA) {
  return p.wall != W_NONE && (a < 3 || a >= nA - 3);
}

// sum + the deviation of a stored value of wall row ROW, in the sum of a thermal
// wall.  FP16 storage: the decode's product is fused into the sum, but for the
// row-2 population along the wall's normal, (0, +-3) or (0, 0, +-3), which is rounded
// first (written out, so that every kernel forms the same wall density).
template <class L, int P, int J, int ROW, class RR>
__device__ __forceinline__ RR add_deviation(RR sum, typename Codec<P>::T v, const StepParams& p) {
  if constexpr (P == P_FP16S && std::is_same<RR, float>::value) {
    if constexpr (ROW == 2 && L::E(J, 0) == 0 && (L::D == 2 || L::E(J, 1) == 0)) return __fadd_rn(sum, __fmul_rn(__half2float(v), p.h_dec[J]));
    else return fmaf(__half2float(v), p.h_dec[J], sum);
  } else {
    return sum + RR(Codec<P>::template decode<L, J>(v, p));
  }
}

// Pull of a site in one of the three rows next to the wall on side SIDE: slots
// whose source lies beyond it follow the wall rule.  The side is a template
// parameter: the populations that leave the column through the wall (26 on
// D2Q37) are then a fixed list, loaded without a predicate each.  SIDE -1: either
// side, known at run time, for a kernel that has no registers for both.
template <class L, int P, class RR, int LD, bool SC, int SIDE>
__device__ __forceinline__ void pull_near(const typename Codec<P>::T* __restrict__ fin, const StepParams& p, int x, int y,
                                          int z, int a, int nA, const int (&xs)[7], const int (&ys)[7],
                                          const int (&zs)[7], RR (&d)[L::Q]) {
  using C = Codec<P>;
  constexpr int D = L::D, Q = L::Q;
  const int nx = p.nx, ny = p.ny;
  const size_t N = (size_t)p.N;
  const int side = SIDE < 0 ? (a < 3 ? 0 : 1) : SIDE;
  const int colbase = D == 2 ? x : (y * nx + x);     // site of the column at wall coord 0
  const int lineA = D == 2 ? nx : nx * ny;           // stride along the wall axis
  RR rm1 = RR(0);                                    // rho_w - 1 of the thermal wall
  if (p.wall == W_THERMAL) {
    RR sum = RR(0);
    static_for<0, 3>([&](auto ROW) {
      constexpr int r = ROW;
      const int row = side == 0 ? r : nA - 1 - r;
      static_for<0, Q>([&](auto J) {
        constexpr int j = J;
        constexpr int eA = L::E(j, D - 1);
        if constexpr ((SIDE != 1 && r + eA < 0) || (SIDE != 0 && r - eA < 0)) {
          if (SIDE >= 0 || (side == 0 ? eA < 0 : eA > 0))
            sum = add_deviation<L, P, j, r>(sum, ldpop<C, LD>(fin + j * N + colbase + row * lineA, p), p);
        }
      });
    });
    rm1 = (ParamsOf<RR>::wallA(p, side) + sum) * ParamsOf<RR>::wall_inv_den(p, side);
  }
  static_for<0, Q>([&](auto I) {
    constexpr int i = I;
    constexpr int ex = L::E(i, 0), ey = L::E(i, 1), ez = L::E(i, 2);
    constexpr int eA = L::E(i, D - 1);
    const int sA = a - eA;
    if ((SIDE == 0 && eA <= 0) || (SIDE == 1 && eA >= 0) || (side == 0 ? sA >= 0 : sA < nA)) {
      const int off = zs[ez + 3] + ys[ey + 3] + xs[ex + 3];
      d[i] = RR(step_in<L, P, i, SC>(ldpop<C, LD>(fin + i * N + off, p), p));
    } else if (p.wall == W_BOUNCE) {
      // d_i = d_io and w_i = w_io: the scaled values agree as well
      constexpr int io = opposite<i>();
      const int mA = side == 0 ? eA - 1 - a : 2 * nA - 1 - sA;
      d[i] = RR(step_in<L, P, io, SC>(ldpop<C, LD>(fin + io * N + colbase + mA * lineA, p), p));
    } else {
      d[i] = step_from_dev<i, SC>(fma(rm1, ParamsOf<RR>::fw(p, side, i), ParamsOf<RR>::fwd(p, side, i)), p);
    }
  });
}

// Pull of all Q populations of site (x, y, z) with the boundary rules, decoded
// to deviations in type RR (SC: the scaled values of an FP16-scaled step, see
// scaled_step).  The wall axis is the last axis (y in 2-D, z in 3-D).
// BOTH: one copy of the wall rows' code for both sides.
template <class L, int P, class RR, int LD = LD_HINT, bool SC = false, bool BOTH = false>
__device__ __forceinline__ void pull(const typename Codec<P>::T* __restrict__ fin,
                                     const StepParams& p, int x, int y, int z, RR (&d)[L::Q]) {
  using C = Codec<P>;
  constexpr int D = L::D, Q = L::Q;
  const int nx = p.nx, ny = p.ny, nz = p.nz;
  const size_t N = (size_t)p.N;
  const int a = D == 2 ? y : z;          // coordinate along the wall axis
  const int nA = D == 2 ? ny : nz;
  int xs[7], ys[7], zs[7];
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    xs[k] = wrap3(x - (k - 3), nx);
    ys[k] = wrap3(y - (k - 3), ny) * nx;
    zs[k] = D == 3 ? wrap3(z - (k - 3), nz) * nx * ny : 0;
  }
  if (!near_wall(p, a, nA)) {
    static_for<0, Q>([&](auto I) {
      constexpr int i = I;
      constexpr int ex = L::E(i, 0), ey = L::E(i, 1), ez = L::E(i, 2);
      const int off = zs[ez + 3] + ys[ey + 3] + xs[ex + 3];
      d[i] = RR(step_in<L, P, i, SC>(ldpop<C, LD>(fin + i * N + off, p), p));
    });
    return;
  }
  // a row next to a wall (block-uniform side)
  if constexpr (BOTH) pull_near<L, P, RR, LD, SC, -1>(fin, p, x, y, z, a, nA, xs, ys, zs, d);
  else if (a < 3) pull_near<L, P, RR, LD, SC, 0>(fin, p, x, y, z, a, nA, xs, ys, zs, d);
  else pull_near<L, P, RR, LD, SC, 1>(fin, p, x, y, z, a, nA, xs, ys, zs, d);
}

// The same into memory, as a call: for a kernel whose registers the wall rows'
// code would overflow.
template <class L, int P, int LD, bool SC>
__device__ __noinline__ void pull_call(const typename Codec<P>::T* __restrict__ fin, const StepParams& p, int x, int y,
                                       int z, typename Codec<P>::R* out) {
  typename Codec<P>::R d[L::Q];
  pull<L, P, typename Codec<P>::R, LD, SC>(fin, p, x, y, z, d);
  static_for<0, L::Q>([&](auto I) { out[I] = d[I]; });
}

// ------------------------------------------------------- solid sites
// A solid site y emits into a fluid neighbour x = y + e_i the wall
// Maxwellian rho_w(x) f0_i(1, 0, T_y) (diffuse thermal wall on a staircase):
// f0_i(1, 0, T) / w_i = 1 + A0 with, for |xi_i|^2 = X2 and Th = T - 1,
//   A0 = Th (X2 - D) / 2 + [NEQ 4] Th^2 (X2^2 - 2 (D + 2) X2 + D (D + 2)) / 8.
// rho_w(x) equals the mass x sends into solid sites (its post-collision slots
// -e_i of the solid-sourced directions) over sum_i f0_i(1, 0, T_y), so every
// fluid site keeps its mass.  In deviations:
//   rho_w - 1 = sum (d*_-i - w_i A0_i) / sum w_i (1 + A0_i),
//   d_i = w_i ((rho_w - 1)(1 + A0_i) + A0_i).
template <class L, int I, class R>
__device__ __forceinline__ R wall_a0(R th) {
  constexpr int D = L::D;
  constexpr double X2 = L::c2 * double(L::E2(L::SH(I)));
  R a0 = R(0.5 * (X2 - D)) * th;
  if constexpr (L::NEQ >= 4) {
    constexpr double q2 = (X2 * X2 - 2.0 * (D + 2) * X2 + double(D * (D + 2))) / 8.0;
    a0 = fma(R(q2) * th, th, a0);
  }
  return a0;
}

// Pull of a fluid site of a grid with solid sites (all axes periodic).
template <class L, int P, class RR>
__device__ __forceinline__ void pull_solid(const typename Codec<P>::T* __restrict__ fin,
                                           const StepParams& p, int x, int y, int z, int site,
                                           RR (&d)[L::Q]) {
  using C = Codec<P>;
  constexpr int D = L::D, Q = L::Q;
  const int nx = p.nx, ny = p.ny, nz = p.nz;
  const size_t N = (size_t)p.N;
  int xs[7], ys[7], zs[7];
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    xs[k] = wrap3(x - (k - 3), nx);
    ys[k] = wrap3(y - (k - 3), ny) * nx;
    zs[k] = D == 3 ? wrap3(z - (k - 3), nz) * nx * ny : 0;
  }
  RR num = RR(0), den = RR(0);
  unsigned long long walls = 0;
  static_for<0, Q>([&](auto I) {
    constexpr int i = I;
    constexpr int ex = L::E(i, 0), ey = L::E(i, 1), ez = L::E(i, 2);
    const int src = zs[ez + 3] + ys[ey + 3] + xs[ex + 3];
    if (__ldg(p.solid + src)) {
      constexpr int io = opposite<i>();
      constexpr RR w = RR(L::W(i));
      const RR a0 = wall_a0<L, i, RR>(ParamsOf<RR>::wall_th(p, src));
      num += RR(C::template decode<L, io>(C::load(fin + io * N + site, p), p)) - w * a0;
      den = fma(w, RR(1) + a0, den);
      walls |= 1ull << i;
      d[i] = a0;  // kept for the second pass
    } else {
      d[i] = RR(C::template decode<L, i>(C::load(fin + i * N + src, p), p));
    }
  });
  if (!walls) return;
  const RR rm1 = num / den;
  static_for<0, Q>([&](auto I) {
    constexpr int i = I;
    if (walls >> i & 1ull) d[i] = RR(L::W(i)) * fma(rm1, RR(1) + d[i], d[i]);
  });
}

// Pull for a warp whose 32 sites neither wrap around x nor touch a wall: every
// source offset relative to the thread's own site, i*N + (row / plane shift)
// - e_ix, is the same for the whole block (rows wrap only through the block's
// y, z), so addresses are a per-thread base plus block-uniform offsets.
template <class L, int P, class RR, int LD = LD_HINT, int IN = IN_DEV>
__device__ __forceinline__ void pull_interior(const typename Codec<P>::T* __restrict__ fsite,
                                              const StepParams& p, int y, int z,
                                              RR (&d)[L::Q]) {
  using C = Codec<P>;
  constexpr int D = L::D, Q = L::Q;
  const long long N = p.N;
  long long dy[7], dz[7];
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    dy[k] = (long long)(wrap3(y - (k - 3), p.ny) - y) * p.nx;
    dz[k] = D == 3 ? (long long)(wrap3(z - (k - 3), p.nz) - z) * p.nx * p.ny : 0;
  }
  static_for<0, Q>([&](auto I) {
    constexpr int i = I;
    constexpr int ex = L::E(i, 0), ey = L::E(i, 1), ez = L::E(i, 2);
    const long long off = i * N + dz[ez + 3] + dy[ey + 3] - ex;
    d[i] = RR(pulled_value<L, P, i, IN>(ldpop<C, LD>(fsite + off, p), p));
  });
}

// ------------------------------------------------------------ the step
// Collision of one site from its pulled deviations d (Eq. lbm) in float and
// store of f*(x) at `site`; shared by all step kernels of the float codecs (FP64
// storage: poly_store below).
//
// f*_i - w_i = d_i (1 - om) + w_i [om drho + rho (om p_i + (1 - om/2) F'_i)],
// with p_i = E +- O the equilibrium polynomial and F'_i = Fe +- Fo the force
// polynomial of the pair (e, -e) (see MidState).  rho om and rho (1 - om/2)
// are folded into per-shell coefficients:
//   even: P0 + t^2 (P2 + t^2 rho om / 24) + s' t,   P0 = rho om A0 + om drho - rho k g.u,
//   odd:  t (Q1 + t^2 rho om / 6) + s' (A1 + t^2 / 2),  Q1 = rho om A1 - rho k g.u
//   (order 1: odd force part is s' alone and Q1 = rho om A1; order 0 also drops
//   the even force part s' t - g.u),
// with t = xi.u, s' = rho k xi.g, k = 1 - om/2 (force order 2; lower orders
// drop terms).  Each pair is stored as even +- odd: the even part (density,
// temperature) is shared by e and -e, so its rounding cancels in the odd part
// that carries the momentum; only the final rounding of each member remains.
// SC (scaled_step): d holds h_i = s d_i / w_i, and every coefficient that
// multiplies w_i above is carried times s instead (exact: s is a power of two).
template <class L, int P, int FO, bool SC = false>
__device__ __forceinline__ void collide_store(typename Codec<P>::R (&d)[L::Q],
                                              const typename Codec<P>::R (&g)[3], int site,
                                              typename Codec<P>::T* __restrict__ fout,
                                              const StepParams& p) {
  using C = Codec<P>;
  using R = typename C::R;
  constexpr int NP = (L::Q - 1) / 2, NS = L::NSHELL, D = L::D;
  constexpr bool EX = P != P_FP16S;  // quadrature constants as hi + lo pairs
  static_assert(!SC || scaled_step<P, FO>(), "scaled values: FP16-scaled storage, FO 0..2");
  static_assert(std::is_same<R, float>::value, "FP64 storage: poly_store");
  const size_t N = (size_t)p.N;
  const RawMoments<L, R> r = SC ? raw_moments_scaled<L, R>(d, R(p.h_inv_scale)) : raw_moments<L, R>(d);
  // times s: the coefficients of w_i in the scaled representation
  auto scl = [&](R v) {
    if constexpr (SC) return v * R(p.h_scale);
    else return v;
  };
  // mid-point state (R1): rho, u = u~ + g/2, theta
  const R rho = R(1) + r.drho;
  const R irho = R(1) / rho;
  R u[3];
  for (int a = 0; a < 3; ++a) u[a] = mul_c<L, R, EX>(r.j[a] * irho) + R(0.5) * g[a];
  const R ut0 = u[0] - R(0.5) * g[0], ut1 = u[1] - R(0.5) * g[1], ut2 = u[2] - R(0.5) * g[2];
  const R g2 = g[0] * g[0] + g[1] * g[1] + g[2] * g[2];
  const R Th = ((mul_c2<L, R, EX>(r.k2) - R(D) * r.drho) * irho - (ut0 * ut0 + ut1 * ut1 + ut2 * ut2)) *
                   R(1.0 / D) + g2 * R(0.25 / D);
  const R u2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  const R gu = g[0] * u[0] + g[1] * u[1] + g[2] * u[2];
  const R om = site_omega<R>(p, rho, R(1) + Th);
  const R om1 = R(1) - om;
  const R hom1 = R(0.5) * om1;
  const R kf = R(1) - R(0.5) * om;
  const R rom0 = rho * om;
  const R rom = scl(rom0);
  const R rkgu = scl(FO >= 1 ? rho * kf * gu : R(0));
  const R rkf = scl(rho * kf);
  R cu[3], cs[3];
  for (int a = 0; a < 3; ++a) {
    cu[a] = mul_c<L, R, EX>(u[a]);
    cs[a] = mul_c<L, R, EX>(rkf * g[a]);
  }
  // per-shell coefficients as polynomials in tx = Th |xi|^2 (constant hi + lo)
  //   A0 = a00 + tx (c1 + tx / 8 [NEQ 4]),  A1 = b0 + tx / 2,  A2 = g0 + tx / 4 [NEQ 4]
  R a00 = R(-0.5) * u2 - R(0.5 * D) * Th;
  R c1 = R(0.5);
  R g0c = R(0.5);
  if constexpr (L::NEQ >= 4) {
    a00 += R(0.125) * u2 * u2 + R(0.25 * (D + 2)) * Th * u2 + R(0.125 * D * (D + 2)) * Th * Th;
    c1 += R(-0.25) * u2 - R(0.25 * (D + 2)) * Th;
    g0c += R(-0.25) * u2 - R(0.25 * (D + 4)) * Th;
  }
  c1 *= Th;  // A0 = a00 + c1 X2 + Th^2 X2^2 / 8 = a00 + (c1 / Th) tx + tx^2 / 8
  const R b0 = R(1) - R(0.5) * u2 - R(0.5 * (D + 2)) * Th;
  R P0[NS], P2[NS], Q1[NS], A1[NS];
  const R base = scl(om * r.drho) - rkgu;
  // rho om multiplies every direction's equilibrium part at this site, so its
  // rounding would act as a common factor (a coherent momentum / energy error
  // per step): carry it as rom + rom_lo, with the exact FMA residual.
  const R rom_lo = scl(fma(rho, om, -rom0));
  static_for<0, NS>([&](auto S) {
    constexpr int sh = S;
    constexpr double X2d = L::c2 * double(L::E2(sh));
    constexpr F2 X2f = f2_of(X2d);
    const R tx = kmul<R, EX>(X2d, X2f, Th);
    R A0, A2;
    if constexpr (L::NEQ >= 4) {
      A0 = fma(R(0.125) * tx, tx, kmul<R, EX>(X2d, X2f, c1) + a00);
      A2 = fma(R(0.25), tx, g0c);
    } else {
      A0 = fma(R(0.5), tx, a00);
      A2 = g0c;
    }
    A1[sh] = fma(R(0.5), tx, b0);
    P0[sh] = fma(rom, A0, fma(rom_lo, A0, base));
    P2[sh] = fma(rom, A2, rom_lo * A2);
    Q1[sh] = fma(rom, A1[sh], fma(rom_lo, A1[sh], FO >= 2 ? -rkgu : R(0)));
  });
  const R P4 = L::NEQ >= 4 ? rom * R(1.0 / 24.0) : R(0);
  const R Q3 = rom * R(1.0 / 6.0);
  // sigma-bar terms (FO 3 = force order 2 with sigma-bar): the odd part gains
  // rho k dF'_i = (k^2 / 2) [(g.xi)(xi.S.xi) - 2 (S g).xi]
  StressTerms<R> st;
  if constexpr (FO == 3) {
    R S[6];
    stress_tensor<L, R>(d, r.drho, rho, Th, u, g, S);
    st = stress_terms<L, R>(S, g, R(0.5) * kf * kf);
  }
  // rest particle: t = s' = 0
  typename C::T* __restrict__ fo = fout + site;
  fo[0] = step_out<L, P, 0, SC>(fma(d[0], om1, SC ? P0[0] : mul_w<L, 0, R, EX>(P0[0])), p);
  static_for<0, NP>([&](auto K) {
    constexpr int ip = 2 * K + 1, im = ip + 1;
    constexpr int sh = L::SH(ip);
    const R t = edot<L, ip>(cu);
    const R t2 = t * t;
    R ev_in = fma(t2, L::NEQ >= 4 ? fma(t2, P4, P2[sh]) : P2[sh], P0[sh]);
    R od_in = t * fma(t2, Q3, Q1[sh]);
    if constexpr (FO >= 1) {
      const R sp = edot<L, ip>(cs);
      ev_in = fma(sp, t, ev_in);
      od_in = FO >= 2 ? fma(sp, fma(R(0.5), t2, A1[sh]), od_in) : od_in + sp;
    } else {
      od_in = od_in + edot<L, ip>(cs);
    }
    if constexpr (FO == 3) od_in += stress_pair<L, ip, R>(st);
    const R ev = fma(d[ip] + d[im], hom1, SC ? ev_in : mul_w<L, ip, R, EX>(ev_in));
    const R od = fma(d[ip] - d[im], hom1, SC ? od_in : mul_w<L, ip, R, EX>(od_in));
    fo[ip * N] = step_out<L, P, ip, SC>(ev + od, p);
    fo[im * N] = step_out<L, P, im, SC>(ev - od, p);
  });
}

// Pair sums s and differences a of the deviations, from the stored values f of
// an FP64 pull: a = f+ - f- and s = a + 2 (f- - w), three operations a pair
// where decoding both members takes four.  f+ - f- and f- - w are exact while
// the members are within a factor of two of each other and of w, so s and a are
// what the decoded deviations give.
template <class L, class R>
__device__ __forceinline__ void pair_split(const R (&f)[L::Q], R& d0, R (&s)[(L::Q - 1) / 2], R (&a)[(L::Q - 1) / 2]) {
  d0 = f[0] - R(L::W(0));
  static_for<0, (L::Q - 1) / 2>([&](auto K) {
    constexpr int k = K, ip = 2 * k + 1;
    a[k] = f[ip] - f[ip + 1];
    s[k] = kmac<2>(f[ip + 1] - R(L::W(ip)), a[k]);
  });
}
// The same from deviations (rows at a wall, sites next to solids).
template <class L, class R>
__device__ __forceinline__ void pair_split_dev(const R (&d)[L::Q], R& d0, R (&s)[(L::Q - 1) / 2], R (&a)[(L::Q - 1) / 2]) {
  d0 = d[0];
  static_for<0, (L::Q - 1) / 2>([&](auto K) {
    constexpr int k = K, ip = 2 * k + 1;
    a[k] = d[ip] - d[ip + 1];
    s[k] = d[ip] + d[ip + 1];
  });
}

// The mid-point state of an FP64 site (R1: rho, u = u~ + g/2, theta) from its raw
// moments, and the polynomial's coefficients.  stress(m, u, S): the tensor S of
// the sigma-bar terms (FO 3).
// Error, in double: u is rounded once (c j / rho and g/2 in one operation; the product
// rounded first, the velocity of a 150-row shear at 1.2 was off by 4.2e-14 after 200 steps,
// now 1.5e-14), and the temperature takes u~ as that u less g/2 (from g.u - u^2, three
// operations fewer, T of a 70 x 150 channel was 7.5e-15 off after 200 steps, now 2.8e-15).
// 0.7 to 1.7 % of a step's time.  Float-float keeps the shorter forms: there they lower the
// errors (13 channels: rho 0.65, u 0.93, T 0.72, q 0.85 of the pair-by-pair body's).
template <class L, class R, int FO, class COEF, class STRESS>
__device__ __forceinline__ void site_coefficients(const RawMoments<L, R>& r, const R (&g)[3], const StepParams& p,
                                                  SiteState<R>& m, COEF& k, STRESS&& stress) {
  constexpr int D = L::D;
  m.drho = r.drho;
  m.rho = R(1) + r.drho;
  const R irho = R(1) / m.rho, cirho = mul_c<L, R>(irho);
  R u[3] = {R(0), R(0), R(0)};
  R gu = R(0);
  m.u2 = R(0);
  R ut2 = R(0), g2 = R(0);
  for (int c = 0; c < D; ++c) {
    if constexpr (std::is_same<R, double>::value) {
      const R h = half_of(g[c]);
      u[c] = fma(r.j[c], cirho, h);
      const R ut = u[c] - h;
      ut2 = c == 0 ? ut * ut : fma(ut, ut, ut2);
      g2 = c == 0 ? g[c] * g[c] : fma(g[c], g[c], g2);
    } else {
      u[c] = hmac(g[c], r.j[c] * cirho);
    }
    m.u2 = c == 0 ? u[c] * u[c] : fma(u[c], u[c], m.u2);
    gu = c == 0 ? g[c] * u[c] : fma(g[c], u[c], gu);
  }
  // D Th = k2 / rho - |u - g/2|^2 + g^2/4
  const R K = cmac(L::c2, r.k2, -kscale<D>(r.drho));
  if constexpr (std::is_same<R, double>::value) {
    m.Th = fma(fma(K, irho, -ut2), R(1.0 / D), R(0.25 / D) * g2);
  } else {
    const R DTh = fma(K, irho, gu - m.u2);
    if constexpr (D == 2) m.Th = half_of(DTh);
    else m.Th = DTh * R(1.0 / D);
  }
  m.om = site_omega<R>(p, m.rho, R(1) + m.Th);
  m.rom = m.rho * m.om;
  const R rk = hmac(-m.rom, m.rho);
  m.rkgu = FO >= 1 ? rk * gu : R(0);
  m.T = mul_c2<L, R>(m.Th);
  const R crk = mul_c<L, R>(rk);
  for (int c = 0; c < 3; ++c) {
    m.U[c] = c < D ? mul_c<L, R>(u[c]) : R(0);
    m.S[c] = c < D ? crk * g[c] : R(0);
  }
  if constexpr (D == 2 && std::is_same<R, DF>::value) poly_coef2<(FO == 3 ? 2 : FO)>(m, k);
  else poly_coef<(FO == 3 ? 2 : FO)>(m, k);
  if constexpr (FO == 3) {
    R S[6];
    stress(m, u, S);
    const R kf = R(1) - half_of(m.om);
    poly_add_stress(stress_terms<L, R>(S, g, half_of(kf * kf)), k);
  }
}
template <class L, class R>
using PolyCoefOf = typename std::conditional<L::D == 2, PolyCoef2<R>, PolyCoef3<R>>::type;

// Collision of one site of an FP64 grid in IEEE double from its pair sums and
// differences, and store of f*(x): see lbm_poly.cuh.
template <class L, int FO>
__device__ __forceinline__ void poly_store(double d0, const double (&s)[(L::Q - 1) / 2],
                                           const double (&a)[(L::Q - 1) / 2], const double (&g)[3], int site,
                                           double* __restrict__ fout, const StepParams& p) {
  const size_t N = (size_t)p.N;
  SiteState<double> m;
  PolyCoefOf<L, double> k;
  site_coefficients<L, double, FO>(pair_moments<L, double>(d0, s, a), g, p, m, k,
                                   [&](const SiteState<double>& st, const double (&u)[3], double (&S)[6]) {
                                     stress_tensor_pairs<L, double>(s, st.drho, st.rho, st.Th, u, g, S);
                                   });
  const double om1 = 1.0 - m.om, hom1 = 0.5 * om1;
  double* __restrict__ fo = fout + site;
  // FP64 storage probe: the stored deviation rounded as a float codec stores it
  const bool probe = p.storage_probe != 0;
  auto put = [&](auto I, double d) {
    constexpr int i = I;
    if (probe) d = probe_round<i>(d, p);
    fo[i * N] = Codec<P_FP64>::template encode<L, i>(d, p);
  };
  put(ic<0>{}, fma(d0, om1, L::W(0) * const_term(k)));
  poly_pairs<L, double>(k, [&](auto K, double wev, double wod) {
    constexpr int kp = K;
    const double ev = fma(hom1, s[kp], wev), od = fma(hom1, a[kp], wod);
    put(ic<2 * kp + 1>{}, ev + od);
    put(ic<2 * kp + 2>{}, ev - od);
  });
}

// The same in float-float, the (s, a) of a pair in one pack (lbm_df2.cuh).
template <class L, int FO>
__device__ __forceinline__ void df2_store(DF d0, const DF2 (&v)[(L::Q - 1) / 2], const DF (&g)[3], int site,
                                          double* __restrict__ fout, const StepParams& p) {
  const size_t N = (size_t)p.N;
  SiteState<DF> m;
  PolyCoefOf<L, DF> k;
  site_coefficients<L, DF, FO>(pair_moments2<L>(d0, v), g, p, m, k,
                               [&](const SiteState<DF>& st, const DF (&u)[3], DF (&S)[6]) {
                                 DF s[(L::Q - 1) / 2];
                                 static_for<0, (L::Q - 1) / 2>([&](auto K) { s[K] = px(v[K]); });
                                 stress_tensor_pairs<L, DF>(s, st.drho, st.rho, st.Th, u, g, S);
                               });
  const DF om1 = DF(1) - m.om;
  const DF hom1 = half_of(om1);
  double* __restrict__ fo = fout + site;
  fo[0] = Codec<P_FP64DF>::template encode<L, 0>(fma(d0, om1, cmul(L::W(0), const_term(k))), p);
  poly_pairs2<L>(k, [&](auto K, DF2 wg) {
    constexpr int kp = K;
    constexpr F2 w = f2_of(L::W(2 * kp + 1));
    const double2 o = pair_out(hom1, v[kp], wg, w.hi, w.lo);
    fo[(2 * kp + 1) * N] = o.x;
    fo[(2 * kp + 2) * N] = o.y;
  });
}

// Resident 256-thread blocks per SM the register cap is sized for: float
// kernels fit 85 registers (3 blocks) -- D2Q37 without spilling, D3Q39 with
// at most 24 B of spill per thread, which measured 7-10 % faster than its
// 128-register, 2-block variant (the batch kernel's two-sites-per-thread
// variants spill more; its tuner measures both); FP64 kernels keep their
// registers.
// LBM_FLOAT_D2Q37_BLOCKS and LBM_FLOAT_D3Q39_BLOCKS override the float values
// at build time (tuning hooks).
#ifndef LBM_FLOAT_D2Q37_BLOCKS
#define LBM_FLOAT_D2Q37_BLOCKS 3
#endif
#ifndef LBM_FLOAT_D3Q39_BLOCKS
#define LBM_FLOAT_D3Q39_BLOCKS 3
#endif
// LBM_DF_BLOCKS: the same for the float-float FP64 step (2: 128 registers,
// about 160 B of spill on D2Q37 and 190 B on D3Q39, mostly around its two calls).
#ifndef LBM_DF_BLOCKS
#define LBM_DF_BLOCKS 2
#endif
// LBM_HALF_D2Q37_BLOCKS, LBM_HALF_D3Q39_BLOCKS: the same for FP16-scaled
// storage (whose 2-byte loads bring half the bytes per load instruction).
#ifndef LBM_HALF_D2Q37_BLOCKS
#define LBM_HALF_D2Q37_BLOCKS LBM_FLOAT_D2Q37_BLOCKS
#endif
#ifndef LBM_HALF_D3Q39_BLOCKS
#define LBM_HALF_D3Q39_BLOCKS LBM_FLOAT_D3Q39_BLOCKS
#endif
template <class L, int P>
constexpr int min_blocks() {
  return P == P_FP64     ? 1
         : P == P_FP64DF ? LBM_DF_BLOCKS
         : P == P_FP16S  ? (L::Q > 37 ? LBM_HALF_D3Q39_BLOCKS : LBM_HALF_D2Q37_BLOCKS)
                         : (L::Q > 37 ? LBM_FLOAT_D3Q39_BLOCKS : LBM_FLOAT_D2Q37_BLOCKS);
}

// Line of the wall axis a block works on.  With walls, the six wall rows
// (whose pull gathers the wall sums and is slower) take the first six block
// indices along that axis, so they start with the first wave instead of
// forming the last blocks of the launch; the bulk rows follow in order.
__device__ __forceinline__ int wall_rows_first(int b, int n, bool walls) {
  if (!walls || n < 6) return b;
  return b < 3 ? b : (b < 6 ? n - 6 + b : b - 3);
}
// The same with the bulk lines in the launch's direction (StepParams::reverse).
__device__ __forceinline__ int launch_line(int b, int n, bool walls, int reverse) {
  if (!walls || n < 6) return reverse ? n - 1 - b : b;
  return b < 3 ? b : (b < 6 ? n - 6 + b : (reverse ? n + 2 - b : b - 3));
}

// Blocks of a launch along y and along z.
constexpr int MAX_GRID_YZ = 65535;

// Class of every site of a grid with solid sites, and the list of the fluid sites next
// to one, a warp for 32 sites of a row as the step has them.  Pass 0: count[0] those
// sites, count[1] the warps that have one, count[2] the warps that have one and a fluid
// site away from all solid ones too.  Pass 1: the list, count[0] its length so far.
template <class L>
__global__ void __launch_bounds__(256) k_classify(const unsigned char* __restrict__ solid, unsigned char* __restrict__ cls,
                                                  int* __restrict__ list, unsigned* __restrict__ count, int pass,
                                                  const StepParams p) {
  const int per_row = (p.nx + 31) / 32, lane = threadIdx.x & 31;
  const long long warp = ((long long)blockIdx.x * 256 + threadIdx.x) / 32;
  if (warp >= (long long)per_row * (p.N / p.nx)) return;
  const int row = (int)(warp / per_row), x = (int)(warp % per_row) * 32 + lane, site = row * p.nx + x;
  unsigned char c = x >= p.nx || solid[site] ? 1 : 0;
  if (!c) {
    const int y = row % p.ny, z = row / p.ny;
    static_for<1, L::Q>([&](auto I) {
      constexpr int i = I;
      const int sx = wrap3(x - L::E(i, 0), p.nx), sy = wrap3(y - L::E(i, 1), p.ny);
      const int sz = L::D == 3 ? wrap3(z - L::E(i, 2), p.nz) : 0;
      if (solid[(sz * p.ny + sy) * p.nx + sx]) c = 2;
    });
  }
  const unsigned wall = __ballot_sync(0xffffffffu, c == 2), plain = __ballot_sync(0xffffffffu, c == 0);
  if (pass == 0) {
    if (x < p.nx) cls[site] = c;
    if (wall && lane < 3 && (lane < 2 || plain)) atomicAdd(count + lane, lane == 0 ? __popc(wall) : 1u);
  } else if (wall) {
    unsigned at = 0u;
    if (lane == 0) at = atomicAdd(count, (unsigned)__popc(wall));
    at = __shfl_sync(0xffffffffu, at, 0) + __popc(wall & ((1u << lane) - 1u));
    if (c == 2) list[at] = site;
  }
}

// Whether a grid keeps the list of its wall sites (SOLID_LIST), from k_classify's counts: the
// FP64 step once it fills the chip, where the list saves work.  In place a warp with a wall
// site takes about twice the time of one without; with the list it takes that for every 32
// wall sites, and a plain pass for each warp that is left with another site.  So the list
// pays for a thin wall, and where nearly every fluid site is at one, not for solids scattered
// so that most warps keep a few sites of both kinds.  GB300, us a step in place -> with the
// list: 512 x 512 annulus 227 -> 192, 0.4 % of the sites solid 326 -> 271, 5 % 430 -> 531, 30 %
// 448 -> 341; 80^3 with 0.4 % 964 -> 673, 5 % 1024 -> 1149, 30 % 1031 -> 579, a ball 626 -> 572.
// (A channel's flat walls, where both sides are equal: 79 -> 64 at 256 x 256 alone, 51 with
// three grids at once either way.)
// Below LBM_WALL_LIST_MIN_SITES a step lasts as long as one warp's pull, and a warp of
// listed sites, whose missing slots differ, runs every slot's wall branch.  GB300,
// cylinders in FP64, us for 40 steps alone / per grid with three at once, list then in
// place: 160 x 160 2809 / 1220, 2303 / 1145; 176 x 176 2830 / 1278, 2766 / 1335;
// 224 x 224 2882 / 1562, 2579 / 1912.  In FP32 the branches are cheap and the list
// never paid (192 x 192: 18.9 us a step, 11.6 in place).
#ifndef LBM_WALL_LIST_MIN_SITES
#define LBM_WALL_LIST_MIN_SITES 28672
#endif
inline bool wall_list(int precision, long long sites, const unsigned (&count)[3]) {
  return precision == P_FP64 && sites >= LBM_WALL_LIST_MIN_SITES && count[2] + count[0] / 16.0 <= 2.0 * count[1];
}

// Lines (y rows in 2-D, z layers in 3-D) that the list of wall sites adds in front
// of a step's grid of blocks of bx threads.
template <int D>
inline int wall_site_lines(const StepParams& p, int bx) {
  const long long line = (long long)((p.nx + bx - 1) / bx) * (D == 2 ? 1 : p.ny) * bx;
  return (int)((p.n_wall_sites + line - 1) / line);
}
// Whether a launch has room for them and the grid.
inline bool wall_list_fits(int D, const StepParams& p, int bx) {
  return p.na + (D == 2 ? wall_site_lines<2>(p, bx) : wall_site_lines<3>(p, bx)) <= MAX_GRID_YZ;
}

// SOLID: the grid has solid sites.  They are skipped; fluid sites next to one take
// the diffuse-wall pull.
//   SOLID_LIST (wall_list): those sites in blocks of their own, the first of the
//   launch.  Left among the others, a warp with one such site ran the wall's FP64
//   operations for all 37 directions, 470 beside the 420 of a plain site, and every
//   site read 37 flags.  256 x 256 cylinders FP64, 20 steps and read-out 1.37 -> 1.03 ms.
//   SOLID_PLACE: among the others, in FP64 only in the warps that have such a site
//   (146 x 146 cylinders, 40 steps and read-out 2.32 -> 1.87 ms, every site before).
enum { SOLID_NONE = 0, SOLID_PLACE = 1, SOLID_LIST = 2 };
template <class L, int P, int FO, int SOLID = SOLID_NONE>
__global__ void __launch_bounds__(256, min_blocks<L, P>())
    k_step(const typename Codec<P>::T* __restrict__ fin, typename Codec<P>::T* __restrict__ fout,
           const StepParams p) {
  using R = typename Codec<P>::R;
  const int lines = SOLID == SOLID_LIST ? (int)(L::D == 2 ? gridDim.y : gridDim.z) - p.na : 0;  // of wall sites (wall_site_lines)
  if constexpr (SOLID == SOLID_LIST) {
    const int line = L::D == 2 ? blockIdx.y : blockIdx.z;
    if (line < lines) {
      const int blk = (L::D == 2 ? line : line * p.ny + (int)blockIdx.y) * gridDim.x + blockIdx.x;
      const int k = blk * blockDim.x + threadIdx.x;
      asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
      if (k >= p.n_wall_sites) return;
      const int site = __ldg(p.wall_sites + k), x = site % p.nx, row = site / p.nx, y = row % p.ny, z = row / p.ny;
      R g[3];
      site_force_r<L::D, R>(p, x, y, z, site, g);
      fin = wait_previous(fin);
      R d[L::Q];
      pull_solid<L, P, R>(fin, p, x, y, z, site, d);
      if constexpr (P == P_FP64) {
        R d0, s[(L::Q - 1) / 2], a[(L::Q - 1) / 2];
        pair_split_dev<L, R>(d, d0, s, a);
        poly_store<L, FO>(d0, s, a, g, site, fout, p);
      } else {
        collide_store<L, P, FO>(d, g, site, fout, p);
      }
      return;
    }
  }
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= p.nx) return;
  // (a grid with solid sites has no walls, and visits its lines in ascending order: the
  // other direction cost FP32 grids of 100 x 100 to 512 x 512 up to a fifth of a step, a
  // channel of 192 x 192 between solid rows 8.9 -> 11.0 us)
  const int reverse = SOLID == SOLID_NONE ? p.reverse : 0;
  const bool walls = SOLID == SOLID_NONE && p.wall != W_NONE;
  const int y = L::D == 2 ? p.a0 + launch_line(blockIdx.y - lines, p.na, walls, reverse)
                          : (reverse ? p.ny - 1 - (int)blockIdx.y : (int)blockIdx.y);
  const int z = L::D == 3 ? p.a0 + launch_line(blockIdx.z - lines, p.na, walls, reverse) : 0;
  const int site = (z * p.ny + y) * p.nx + x;
  if constexpr (SOLID == SOLID_LIST) {
    if (__ldg(p.site_class + site)) return;
  }
  bool at_solid = false;  // a lane of this warp is next to a solid site
  if constexpr (SOLID == SOLID_PLACE) {
    const int cls = __ldg(p.site_class + site);
    at_solid = P != P_FP64 || __any_sync(__activemask(), cls == 2);
    if (cls == 1) return;
  }
  const int a = L::D == 2 ? y : z;
  const int nA = L::D == 2 ? p.ny : p.nz;
  const bool near = near_wall(p, a, nA);
  const int wx0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31);
  const bool interior = !near && wx0 >= 3 && wx0 + 31 <= p.nx - 4;
  // Programmatic dependent launch: let the next step's blocks be scheduled
  // now, and wait for the previous kernel (and its memory) before pulling.
  // Both are no-ops when the launch has no programmatic dependency.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  R g[3];
  site_force_r<L::D, R>(p, x, y, z, site, g);
  fin = wait_previous(fin);
  if constexpr (std::is_same<R, float>::value) {
    constexpr bool SC = scaled_step<P, FO>();
    R d[L::Q];
    if (SOLID == SOLID_PLACE && at_solid) pull_solid<L, P, R>(fin, p, x, y, z, site, d);
    else if (interior) pull_interior<L, P, R, LD_HINT, SC ? IN_SCALED : IN_DEV>(fin + site, p, y, z, d);
    else pull<L, P, R, LD_HINT, SC>(fin, p, x, y, z, d);
    collide_store<L, P, FO, SC>(d, g, site, fout, p);
  } else if constexpr (P == P_FP64) {
    R d0, s[(L::Q - 1) / 2], am[(L::Q - 1) / 2];
    if (SOLID == SOLID_PLACE && at_solid) {
      R d[L::Q];
      pull_solid<L, P, R>(fin, p, x, y, z, site, d);
      pair_split_dev<L, R>(d, d0, s, am);
    } else if (!near) {
      R f[L::Q];
      if (interior) pull_interior<L, P, R, LD_HINT, IN_STORED>(fin + site, p, y, z, f);
      else pull_stored<L, P, R>(fin, p, x, y, z, f);
      pair_split<L, R>(f, d0, s, am);
    } else {
      R d[L::Q];
      pull<L, P, R>(fin, p, x, y, z, d);
      pair_split_dev<L, R>(d, d0, s, am);
    }
    poly_store<L, FO>(d0, s, am, g, site, fout, p);
  } else {
    DF d0;
    DF2 v[(L::Q - 1) / 2];
    if (!near) {
      double f[L::Q];
      if (interior) pull_interior<L, P_FP64, double, LD_HINT, IN_STORED>(fin + site, p, y, z, f);
      else pull_stored<L, P_FP64, double>(fin, p, x, y, z, f);
      d0 = df_split(f[0]) - DF(L::W(0));
      static_for<0, (L::Q - 1) / 2>([&](auto K) {
        constexpr int ip = 2 * K + 1;
        constexpr F2 w = f2_of(L::W(ip));
        v[K] = pair_in(f[ip], f[ip + 1], w.hi, w.lo);
      });
    } else {
      DF d[L::Q];
      pull<L, P, DF>(fin, p, x, y, z, d);
      d0 = d[0];
      static_for<0, (L::Q - 1) / 2>([&](auto K) { v[K] = sum_diff(pack(d[2 * K + 1], d[2 * K + 2])); });
    }
    df2_store<L, FO>(d0, v, g, site, fout, p);
  }
}

// ------------------------------------------------------------ init
// f~_i = f0_i(rho, u, T) - F_i(rho, u, T)/2 as deviations
// d_i = w_i [drho + rho (p_i - F'_i/2)], placed at the slot the next pull of
// (x, i) reads: x - e_i (periodic), or the mirrored slot of the opposite
// direction beyond a wall.
template <class L, int FO, class R>
__device__ __forceinline__ void init_site(const MidState<L, R>& m, R (&d)[L::Q]) {
  constexpr int NP = (L::Q - 1) / 2;
  {
    R E, Fe;
    rest_terms<L, FO, R>(m, E, Fe);
    d[0] = mul_w<L, 0>(fma(m.rho, E - R(0.5) * Fe, m.drho));
  }
  static_for<0, NP>([&](auto K) {
    constexpr int ip = 2 * K + 1, im = ip + 1;
    R E, O, Fe, Fo;
    pair_terms<L, FO, ip, R>(m, E, O, Fe, Fo);
    const R ev = mul_w<L, ip>(fma(m.rho, E - R(0.5) * Fe, m.drho));
    const R od = mul_w<L, ip>(m.rho * (O - R(0.5) * Fo));
    d[ip] = ev + od;
    d[im] = ev - od;
  });
}

// The same in double, by parity classes (lbm_poly.cuh): the polynomial of the
// step with om = 1 and the force's factor 1 - om/2 replaced by -1/2.
template <class L, int FO>
__device__ __forceinline__ void init_site_poly(double drho, const double (&u)[3], double Th, const double (&g)[3],
                                               double (&d)[L::Q]) {
  constexpr int D = L::D;
  SiteState<double> m;
  m.drho = drho;
  m.rho = 1.0 + drho;
  m.om = 1.0;
  m.Th = Th;
  m.T = L::c2 * Th;
  m.rom = m.rho;
  m.u2 = 0.0;
  const double rk = -0.5 * m.rho;
  double gu = 0.0;
  for (int c = 0; c < 3; ++c) {
    m.U[c] = c < D ? L::c * u[c] : 0.0;
    m.S[c] = c < D ? L::c * rk * g[c] : 0.0;
    if (c < D) {
      m.u2 = fma(u[c], u[c], m.u2);
      gu = fma(g[c], u[c], gu);
    }
  }
  m.rkgu = rk * gu;
  typename std::conditional<D == 2, PolyCoef2<double>, PolyCoef3<double>>::type k;
  poly_coef<FO>(m, k);
  d[0] = L::W(0) * const_term(k);
  poly_pairs<L, double>(k, [&](auto K, double ev, double od) {
    d[2 * int(K) + 1] = ev + od;
    d[2 * int(K) + 2] = ev - od;
  });
}

// Deviations of site (x, y, z) from the given fields.
template <class L, class R>
__device__ __forceinline__ void init_deviations(const double* __restrict__ rho, const double* __restrict__ u,
                                                const double* __restrict__ T, int force_order, const StepParams& p,
                                                int x, int y, int z, int site, R (&d)[L::Q]) {
  constexpr int D = L::D;
  const size_t N = (size_t)p.N;
  double gd[3];
  site_force<D>(p, x, y, z, site, gd);
  if constexpr (std::is_same<R, double>::value) {
    const double uu[3] = {u[site], u[N + site], D == 3 ? u[2 * N + site] : 0.0};
    const double drho = rho[site] - 1.0, Th = T[site] - 1.0;
    if (force_order == 0) init_site_poly<L, 0>(drho, uu, Th, gd, d);
    else if (force_order == 1) init_site_poly<L, 1>(drho, uu, Th, gd, d);
    else init_site_poly<L, 2>(drho, uu, Th, gd, d);
  } else {
    const R g[3] = {R(gd[0]), R(gd[1]), R(gd[2])};
    const R uu[3] = {R(u[site]), R(u[N + site]), D == 3 ? R(u[2 * N + site]) : R(0)};
    MidState<L, R> m;
    given_state<L, R>(R(rho[site] - 1.0), uu, R(T[site] - 1.0), g, m);
    if (force_order == 0) init_site<L, 0, R>(m, d);
    else if (force_order == 1) init_site<L, 1, R>(m, d);
    else init_site<L, 2, R>(m, d);
  }
}

// Largest |d_i| of each shell of directions over the sites an FP16 grid
// initialises (as bits; maxbits: L::NSHELL zeroed words): the host divides it
// by the shell's weight for the scale.  (Rounding is monotonic, so this is the
// largest rounded |d_i / w_i|, without a double division per population; and
// one atomic per block and shell instead of one per site.  512 x 512 x 256
// sites: 47.8 ms before.)
template <class L>
__global__ void __launch_bounds__(256) k_init_scale(const double* __restrict__ rho, const double* __restrict__ u,
                                                    const double* __restrict__ T, unsigned int* __restrict__ maxbits,
                                                    int force_order, const StepParams p) {
  constexpr int D = L::D;
  const int layer = D == 2 ? p.nx : p.nx * p.ny;
  const int end = (p.a0 + p.na) * layer;
  unsigned mx[L::NSHELL] = {};  // as bits, in which a NaN is above infinity (fmaxf drops it)
  // (long long: site + stride may pass 2^31)
  for (long long s = (long long)p.a0 * layer + blockIdx.x * 256 + threadIdx.x; s < end; s += (long long)gridDim.x * 256) {
    const int site = (int)s;
    if (p.solid && p.solid[site]) continue;
    const int x = site % p.nx, row = site / p.nx;
    float d[L::Q];
    init_deviations<L, float>(rho, u, T, force_order, p, x, row % p.ny, row / p.ny, site, d);
    static_for<0, L::Q>([&](auto I) {
      constexpr int i = I;
      mx[L::SH(i)] = max(mx[L::SH(i)], __float_as_uint(fabsf(d[i])));
    });
  }
  __shared__ unsigned sh[L::NSHELL];
  if (threadIdx.x < L::NSHELL) sh[threadIdx.x] = 0u;
  __syncthreads();
  for (int k = 0; k < L::NSHELL; ++k) {
    const unsigned m = __reduce_max_sync(0xffffffffu, mx[k]);
    if ((threadIdx.x & 31) == 0) atomicMax(sh + k, m);
  }
  __syncthreads();
  if (threadIdx.x < L::NSHELL) atomicMax(maxbits + threadIdx.x, sh[threadIdx.x]);
}

template <class L, int P>
__global__ void __launch_bounds__(128) k_init(const double* __restrict__ rho, const double* __restrict__ u,
                                              const double* __restrict__ T, typename Codec<P>::T* __restrict__ fout,
                                              int force_order, const StepParams p) {
  using C = Codec<P>;
  using R = typename C::R;
  constexpr int Q = L::Q, D = L::D;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= p.nx) return;
  const int y = D == 2 ? p.a0 + (int)blockIdx.y : (int)blockIdx.y;
  const int z = D == 3 ? p.a0 + (int)blockIdx.z : 0;
  const int nx = p.nx, ny = p.ny, nz = p.nz;
  const int site = (z * ny + y) * nx + x;
  const size_t N = (size_t)p.N;
  if (p.solid && p.solid[site]) return;
  R d[Q];
  init_deviations<L, R>(rho, u, T, force_order, p, x, y, z, site, d);
  const int a = D == 2 ? y : z;
  const int nA = D == 2 ? ny : nz;
  if constexpr (P == P_FP64) {  // storage probe: the initial state as a float codec stores it
    if (p.storage_probe)
      static_for<0, Q>([&](auto I) {
        constexpr int i = I;
        d[i] = probe_round<i>(d[i], p);
      });
  }
  if (!near_wall(p, a, nA) && !p.solid) {  // block-uniform: the slots a plain pull reads
    int xs[7], ys[7], zs[7];
#pragma unroll
    for (int k = 0; k < 7; ++k) {
      xs[k] = wrap3(x - (k - 3), nx);
      ys[k] = wrap3(y - (k - 3), ny) * nx;
      zs[k] = D == 3 ? wrap3(z - (k - 3), nz) * nx * ny : 0;
    }
    static_for<0, Q>([&](auto I) {
      constexpr int i = I;
      fout[i * N + (zs[L::E(i, 2) + 3] + ys[L::E(i, 1) + 3] + xs[L::E(i, 0) + 3])] = C::template encode<L, i>(d[i], p);
    });
    return;
  }
  const int lineA = D == 2 ? nx : nx * ny;
  const int colbase = D == 2 ? x : (y * nx + x);
  static_for<0, Q>([&](auto I) {
    constexpr int i = I;
    constexpr int ex = L::E(i, 0), ey = L::E(i, 1), ez = L::E(i, 2);
    constexpr int eA = L::E(i, D - 1);
    const int sA = a - eA;
    if (p.wall != W_NONE && (sA < 0 || sA >= nA)) {
      constexpr int io = opposite<i>();
      const int mA = sA < 0 ? eA - 1 - a : 2 * nA - 1 - sA;
      fout[io * N + colbase + mA * lineA] = C::template encode<L, io>(d[i], p);
    } else {
      const int sx = wrap3(x - ex, nx);
      const int sy = wrap3(y - ey, ny);
      const int sz = D == 3 ? wrap3(z - ez, nz) : 0;
      const int src = (sz * ny + sy) * nx + sx;
      if (p.solid && p.solid[src]) {
        // pulled from a solid site: the wall emits it; the slot the wall
        // absorbs (-e_i, at this site) holds the local value
        constexpr int io = opposite<i>();
        fout[io * N + site] = C::template encode<L, io>(d[io], p);
      } else {
        fout[i * N + src] = C::template encode<L, i>(d[i], p);
      }
    }
  });
}

// ------------------------------------------------------------ moments
// Physical rho, u, T and heat flux q in double (the FP64 diagnostic), with
// q = 1/2 (1 - 1/(2 tau)) sum_i (f~_i - f0_i + F_i/2) |xi_i - u|^2 (xi_i - u).
// Each of the three sums is a combination of moments of order <= 3, which
// the quadrature integrates exactly for f0 and F (degree 9 >= 4 + 3 on
// D2Q37, 7 >= 3 + 3 on D3Q39), so only the pulled f~ is summed per site:
//   sum f0 |c|^2 c = 0 (the Maxwellian carries no heat flux), and with
//   S = the second moment the force's n = 3 term contracts (rho (u u + theta
//   delta), minus sigma-bar for FO 3; rho delta for orders 0 and 1) and
//   M2 = sum F xi xi (rho (g u + u g) for orders >= 1, else 0),
//   sum F |c|^2 c_a = 2 (S g)_a + g_a tr S - u_a tr M2 - 2 (M2 u)_a
//                     + 2 rho u_a (u.g) + rho u^2 g_a,
// which is (D + 2) rho theta g_a at order 2.  sum f~ |c|^2 c comes from the
// raw moments of the deviations d = f~ - w: m0 = sum d, m1 = sum d e,
// m2 = sum d e e, m3 = sum d |e|^2 e (c = xi - u, xi = c_lat e).
//
// The sums run over mirror groups first (as pair_moments, lbm_poly.cuh): a
// group's even and odd parts feed all moments, so a group of four directions
// takes 4 additions and some 9 more instead of 4 + 8 per pair.
template <class R>
struct HeatMoments {
  R m0, m1[3], m2[6], m3[3];  // m2 as (xx, yy, zz, xy, xz, yz)
};

// An unevaluated sum s + c of two floats as an accumulator: the rounding
// error of every addition goes into c (Knuth's two-sum), which is not
// renormalised, so an addition takes 8 instructions; the result equals the
// FP64 sum to a few units in 2^-48 of the terms' magnitude.  (Explicit
// round-to-nearest operations: a product fused into a following sum would
// break the error-free transformations.)
struct FF {
  float s = 0.f, c = 0.f;
};
__device__ __forceinline__ FF operator+(FF a, FF b) {
  FF r;
  float e;
  df_two_sum(a.s, b.s, r.s, e);
  r.c = __fadd_rn(__fadd_rn(a.c, b.c), e);
  return r;
}
__device__ __forceinline__ FF operator-(FF a, FF b) { return a + FF{-b.s, -b.c}; }
// acc + K v for a compile-time integer K
template <int K>
__device__ __forceinline__ FF kmac(FF v, FF acc) {
  if constexpr (K == 1) {
    return acc + v;
  } else {
    const float p = __fmul_rn(float(K), v.s);
    const float pe = (K & (K - 1)) == 0 ? 0.f : fmaf(float(K), v.s, -p);
    return acc + FF{p, (K & (K - 1)) == 0 ? __fmul_rn(float(K), v.c) : fmaf(float(K), v.c, pe)};
  }
}

// The raw moments from the rest deviation and the pair sums s and differences
// a, in double or as FF pairs.
template <class L, class R>
__device__ __forceinline__ HeatMoments<R> heat_moments(R d0, const R (&s)[(L::Q - 1) / 2], const R (&a)[(L::Q - 1) / 2]) {
  HeatMoments<R> h{};
  if constexpr (L::D == 2) {
    // even part, and the parts odd in x and y, odd in x, odd in y, of the group (+-X, +-Y)
    auto S = [&](auto X, auto Y) { return at<L, X, Y, 0>(s) + at<L, X, -Y, 0>(s); };
    auto O = [&](auto X, auto Y) { return at<L, X, Y, 0>(s) - at<L, X, -Y, 0>(s); };
    auto Ax = [&](auto X, auto Y) { return at<L, X, Y, 0>(a) + at<L, X, -Y, 0>(a); };
    auto Ay = [&](auto X, auto Y) { return at<L, X, Y, 0>(a) - at<L, X, -Y, 0>(a); };
    constexpr ic<1> _1{};
    constexpr ic<2> _2{};
    constexpr ic<3> _3{};
    {
      const R s11 = S(_1, _1), s12 = S(_1, _2), s21 = S(_2, _1), s22 = S(_2, _2), s13 = S(_1, _3), s31 = S(_3, _1);
      // sums over |e_x| = 1, 2, 3, and over |e_y|
      const R x1 = (at<L, 1, 0, 0>(s) + s11) + (s12 + s13), x2 = at<L, 2, 0, 0>(s) + (s21 + s22), x3 = at<L, 3, 0, 0>(s) + s31;
      const R y1 = (at<L, 0, 1, 0>(s) + s11) + (s21 + s31), y2 = at<L, 0, 2, 0>(s) + (s12 + s22), y3 = at<L, 0, 3, 0>(s) + s13;
      const R x0 = (d0 + at<L, 0, 1, 0>(s)) + (at<L, 0, 2, 0>(s) + at<L, 0, 3, 0>(s));
      h.m0 = (x0 + x1) + (x2 + x3);
      h.m2[0] = kmac<9>(x3, kmac<4>(x2, x1));
      h.m2[1] = kmac<9>(y3, kmac<4>(y2, y1));
    }
    h.m2[3] = kmac<4>(O(_2, _2), kmac<3>(O(_1, _3) + O(_3, _1), kmac<2>(O(_1, _2) + O(_2, _1), O(_1, _1))));
    // sum d e_x and sum d |e|^2 e_x, |e|^2 e_x = e_x^3 + e_x e_y^2
    auto odd = [&](R p1, R p2, R p3, R p11, R p12, R p13, R p21, R p22, R p31, R& m1, R& m3) {
      const R x1 = (p1 + p11) + (p12 + p13), x2 = p2 + (p21 + p22), x3 = p3 + p31;
      m1 = kmac<3>(x3, kmac<2>(x2, x1));
      const R c1 = kmac<9>(p13, kmac<4>(p12, p11)), c2 = kmac<4>(p22, p21);  // sums of e_y^2
      m3 = kmac<27>(x3, kmac<8>(x2, x1)) + kmac<3>(p31, kmac<2>(c2, c1));
    };
    odd(at<L, 1, 0, 0>(a), at<L, 2, 0, 0>(a), at<L, 3, 0, 0>(a), Ax(_1, _1), Ax(_1, _2), Ax(_1, _3), Ax(_2, _1), Ax(_2, _2),
        Ax(_3, _1), h.m1[0], h.m3[0]);
    odd(at<L, 0, 1, 0>(a), at<L, 0, 2, 0>(a), at<L, 0, 3, 0>(a), Ay(_1, _1), Ay(_2, _1), Ay(_3, _1), Ay(_1, _2), Ay(_2, _2),
        Ay(_1, _3), h.m1[1], h.m3[1]);
  } else {
    // (1, 1, 1) and its mirrors: even part and the parts odd in two components
    const R ep = at<L, 1, 1, 1>(s) + at<L, 1, 1, -1>(s), eq = at<L, 1, -1, 1>(s) + at<L, 1, -1, -1>(s);
    const R em = at<L, 1, 1, 1>(s) - at<L, 1, 1, -1>(s), en = at<L, 1, -1, 1>(s) - at<L, 1, -1, -1>(s);
    const R s3 = ep + eq;
    const R pxy = at<L, 2, 2, 0>(s) + at<L, 2, -2, 0>(s), pxz = at<L, 2, 0, 2>(s) + at<L, 2, 0, -2>(s),
            pyz = at<L, 0, 2, 2>(s) + at<L, 0, 2, -2>(s);
    h.m2[3] = kmac<4>(at<L, 2, 2, 0>(s) - at<L, 2, -2, 0>(s), ep - eq);
    h.m2[4] = kmac<4>(at<L, 2, 0, 2>(s) - at<L, 2, 0, -2>(s), em + en);
    h.m2[5] = kmac<4>(at<L, 0, 2, 2>(s) - at<L, 0, 2, -2>(s), em - en);
    const R q2x = at<L, 2, 0, 0>(s), q2y = at<L, 0, 2, 0>(s), q2z = at<L, 0, 0, 2>(s);
    h.m2[0] = kmac<9>(at<L, 3, 0, 0>(s), kmac<4>(q2x + (pxy + pxz), at<L, 1, 0, 0>(s) + s3));
    h.m2[1] = kmac<9>(at<L, 0, 3, 0>(s), kmac<4>(q2y + (pxy + pyz), at<L, 0, 1, 0>(s) + s3));
    h.m2[2] = kmac<9>(at<L, 0, 0, 3>(s), kmac<4>(q2z + (pxz + pyz), at<L, 0, 0, 1>(s) + s3));
    const R s1 = (at<L, 1, 0, 0>(s) + at<L, 0, 1, 0>(s)) + at<L, 0, 0, 1>(s);
    const R s9 = (at<L, 3, 0, 0>(s) + at<L, 0, 3, 0>(s)) + at<L, 0, 0, 3>(s);
    h.m0 = ((d0 + s1) + (s3 + s9)) + (((q2x + q2y) + q2z) + ((pxy + pxz) + pyz));
    const R u = at<L, 1, 1, 1>(a) + at<L, 1, 1, -1>(a), v = at<L, 1, -1, 1>(a) + at<L, 1, -1, -1>(a);
    const R x = at<L, 1, 1, 1>(a) - at<L, 1, 1, -1>(a), y = at<L, 1, -1, 1>(a) - at<L, 1, -1, -1>(a);
    // axes a1, a2, a3; o the octet (|e|^2 = 3), p the planes (|e|^2 = 8, component 2)
    auto odd = [&](R a1, R a2, R a3, R o, R p, R& m1, R& m3) {
      m1 = kmac<3>(a3, kmac<2>(a2 + p, a1 + o));
      m3 = kmac<27>(a3, kmac<16>(p, kmac<8>(a2, kmac<3>(o, a1))));
    };
    odd(at<L, 1, 0, 0>(a), at<L, 2, 0, 0>(a), at<L, 3, 0, 0>(a), u + v,
        (at<L, 2, 2, 0>(a) + at<L, 2, -2, 0>(a)) + (at<L, 2, 0, 2>(a) + at<L, 2, 0, -2>(a)), h.m1[0], h.m3[0]);
    odd(at<L, 0, 1, 0>(a), at<L, 0, 2, 0>(a), at<L, 0, 3, 0>(a), u - v,
        (at<L, 2, 2, 0>(a) - at<L, 2, -2, 0>(a)) + (at<L, 0, 2, 2>(a) + at<L, 0, 2, -2>(a)), h.m1[1], h.m3[1]);
    odd(at<L, 0, 0, 1>(a), at<L, 0, 0, 2>(a), at<L, 0, 0, 3>(a), x + y,
        (at<L, 2, 0, 2>(a) - at<L, 2, 0, -2>(a)) + (at<L, 0, 2, 2>(a) - at<L, 0, 2, -2>(a)), h.m1[2], h.m3[2]);
  }
  return h;
}

// The float deviations' moments as float-float values: FF sums, each
// renormalised (an exact two-sum, since c may exceed ulp(s) after a
// cancellation).
template <class L>
__device__ __forceinline__ HeatMoments<DF> heat_moments_df(const float (&d)[L::Q]) {
  constexpr int NP = (L::Q - 1) / 2;
  FF s[NP], a[NP];
  static_for<0, NP>([&](auto K) {
    constexpr int k = K, ip = 2 * k + 1;
    df_two_sum(d[ip], d[ip + 1], s[k].s, s[k].c);
    df_two_sum(d[ip], -d[ip + 1], a[k].s, a[k].c);
  });
  const HeatMoments<FF> f = heat_moments<L, FF>(FF{d[0], 0.f}, s, a);
  HeatMoments<DF> h;
  auto v = [](const FF& x) {
    DF r;
    df_two_sum(x.s, x.c, r.hi, r.lo);
    return r;
  };
  h.m0 = v(f.m0);
  for (int k = 0; k < L::D; ++k) {
    h.m1[k] = v(f.m1[k]);
    h.m3[k] = v(f.m3[k]);
  }
  for (int k = 0; k < 6; ++k)
    if (L::D == 3 || k == 0 || k == 1 || k == 3) h.m2[k] = v(f.m2[k]);
  return h;
}

__device__ __forceinline__ double out_double(double x) { return x; }
__device__ __forceinline__ double out_double(DF x) { return df_to_double(x); }

// rho, u, T and q of one site from the raw moments of its pulled deviations
// (see the comment above HeatMoments), in the arithmetic type R: double for
// FP64 storage, float-float (~48 bits, lbm_df.cuh) for the float codecs,
// whose FP64 combination ran at the FP64 units' rate; each output is one
// rounding to double.
template <class L, class R>
__device__ __forceinline__ void write_moments(const HeatMoments<R>& h, const R (&g)[3], int site, size_t N,
                                              int force_order, const StepParams& p, double* __restrict__ rho,
                                              double* __restrict__ u, double* __restrict__ T,
                                              double* __restrict__ q) {
  constexpr int D = L::D;
  // the D = 2 sums have no z terms: float-float arithmetic does not fold zeros
  auto dot = [](const R* x, const R* y) {
    R r = x[0] * y[0];
    for (int a = 1; a < D; ++a) r = fma(x[a], y[a], r);
    return r;
  };
  const R r = R(1) + h.m0, ir = R(1) / r;
  R J[3], ut[3], uu[3];
  for (int a = 0; a < D; ++a) {
    J[a] = cmul(L::c, h.m1[a]);  // sum f~ xi = rho u~
    ut[a] = J[a] * ir;
    uu[a] = hmac(g[a], ut[a]);
  }
  R k2 = h.m2[0] + h.m2[1];
  if (D == 3) k2 = k2 + h.m2[2];
  const R K = cmul(L::c2, k2);
  const R g2 = dot(g, g);
  const R Th = fma(fma(K - kscale<D>(h.m0), ir, -dot(ut, ut)), R(1.0 / D), cmul(0.25 / D, g2));
  const R th = R(1) + Th;
  if (rho) rho[site] = out_double(r);
  if (T) T[site] = out_double(th);
  if (u)
    for (int a = 0; a < D; ++a) u[a * N + site] = out_double(uu[a]);
  if (!q) return;
  const R om = site_omega<R>(p, r, th);
  const R u2 = dot(uu, uu), uJ = dot(uu, J);
  // with P = c^2 m2 (so sum f~ xi xi = delta + P), sum f~ |c|^2 c_a =
  //   c^3 m3_a - u_a [D + 2 + tr P - 2 u.J + u^2 rho] - 2 (P u)_a + u^2 J_a
  constexpr int off[3][3] = {{0, 3, 4}, {3, 1, 5}, {4, 5, 2}};
  const R B = fma(u2, r, K - kscale<2>(uJ)) + R(D + 2);
  R C3[3];
  for (int a = 0; a < D; ++a) {
    R mu = h.m2[off[a][0]] * uu[0];
    for (int b = 1; b < D; ++b) mu = fma(h.m2[off[a][b]], uu[b], mu);
    C3[a] = fma(u2, J[a], cmac(-2.0 * L::c2, mu, cmul(L::c * L::c2, h.m3[a]) - uu[a] * B));
  }
  // sum F |c|^2 c
  R FC3[3];
  if (force_order >= 2) {
    const R rth = kscale<D + 2>(r * th);
    for (int a = 0; a < D; ++a) FC3[a] = rth * g[a];
    if (force_order == 3) {
      // S = rho (u u + theta delta) - sigma-bar, sigma-bar = -(1 - om/2) S_st
      const R iso = fma(r, Th, h.m0), hr = half_of(r), kf2 = R(2) - om;
      for (int a = 0; a < D; ++a) {
        R Sg = R(0);
        for (int b = 0; b < D; ++b) {
          const R conv = hr * fma(uu[a], g[b] - uu[b], uu[b] * (g[a] - uu[a]));
          R S = cmac(L::c2, h.m2[off[a][b]], conv);
          if (a == b) S = S - iso;
          Sg = fma(S, g[b], Sg);
        }
        FC3[a] = fma(kf2, Sg, FC3[a]);
      }
    }
  } else {
    // S = rho delta; M2 = rho (g u + u g) at order 1, 0 at order 0
    const R ug = dot(uu, g);
    for (int a = 0; a < D; ++a) {
      const R rg = r * g[a], ru = kscale<2>(r * uu[a]);
      FC3[a] = force_order == 1 ? fma(rg, R(D + 2) - u2, -(ru * ug)) : fma(rg, R(D + 2) + u2, ru * ug);
    }
  }
  const R kq = half_of(R(1) - half_of(om));
  for (int a = 0; a < D; ++a) q[a * N + site] = out_double(kq * hmac(FC3[a], C3[a]));
}

// Bound by instruction issue (float storage: compensated sums and a
// float-float combination) or by the FP64 unit (FP64 storage), not by its
// bytes (Q populations in, 2 + 2 D doubles out).  GB300, against the sums pair
// by pair with one instantiation for grids with and without solid sites (146
// registers; now 80 to 96 for the float codecs): 1024 x 512 FP32 85 -> 53 us,
// FP64 289 -> 212 us, 96^3 FP32 160 -> 97 us, 512 x 512 x 256 FP16 9.2 -> 5.8 ms.
// SOLID: the grid has solid sites (an own instantiation: the solid pull runs in
// double and would set the register count of the float codecs' kernel).
template <class L, int P, bool SOLID>
__global__ void __launch_bounds__(128) k_moments(const typename Codec<P>::T* __restrict__ fin,
                                                 double* __restrict__ rho, double* __restrict__ u,
                                                 double* __restrict__ T, double* __restrict__ q,
                                                 int force_order, const StepParams p) {
  constexpr int Q = L::Q, D = L::D;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= p.nx) return;
  const int y = D == 2 ? p.a0 + (int)blockIdx.y : (int)blockIdx.y;
  const int z = D == 3 ? p.a0 + (int)blockIdx.z : 0;
  const int site = (z * p.ny + y) * p.nx + x;
  const size_t N = (size_t)p.N;
  const int cls = SOLID ? p.site_class[site] : 0;
  if constexpr (SOLID) {
    if (cls == 1) {  // solid sites report zeros
      if (rho) rho[site] = 0.0;
      if (T) T[site] = 0.0;
      for (int a = 0; a < D; ++a) {
        if (u) u[a * N + site] = 0.0;
        if (q) q[a * N + site] = 0.0;
      }
      return;
    }
  }
  const bool near = near_wall(p, D == 2 ? y : z, D == 2 ? p.ny : p.nz);
  const int wx0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31);
  const bool interior = !near && wx0 >= 3 && wx0 + 31 <= p.nx - 4;
  if constexpr (P != P_FP64 && !SOLID) {
    // float storage: the deviations are exact floats; compensated float-pair
    // sums and a float-float combination, no FP64 arithmetic but the final
    // rounding of each output
    float d[Q];
    if (interior) pull_interior<L, P, float>(fin + site, p, y, z, d);
    else pull<L, P, float>(fin, p, x, y, z, d);
    const HeatMoments<DF> h = heat_moments_df<L>(d);
    DF g[3];
    site_force_r<D, DF>(p, x, y, z, site, g);
    write_moments<L, DF>(h, g, site, N, force_order, p, rho, u, T, q);
  } else {
    double d0, s[(Q - 1) / 2], a[(Q - 1) / 2];
    if (SOLID && __any_sync(__activemask(), cls)) {  // the warp as one: its lanes would take both pulls in turn
      double d[Q];
      pull_solid<L, P, double>(fin, p, x, y, z, site, d);
      pair_split_dev<L, double>(d, d0, s, a);
    } else if (P == P_FP64 && !near) {
      double f[Q];
      if (interior) pull_interior<L, P, double, LD_HINT, IN_STORED>(fin + site, p, y, z, f);
      else pull_stored<L, P, double>(fin, p, x, y, z, f);
      pair_split<L, double>(f, d0, s, a);
    } else {
      double d[Q];
      pull<L, P, double>(fin, p, x, y, z, d);
      pair_split_dev<L, double>(d, d0, s, a);
    }
    const HeatMoments<double> h = heat_moments<L, double>(d0, s, a);
    double g[3];
    site_force<D>(p, x, y, z, site, g);
    write_moments<L, double>(h, g, site, N, force_order, p, rho, u, T, q);
  }
}

// ------------------------------------------------------ conservation sums
// Compensated (Neumaier) running sum in the arithmetic type R of a kernel:
// the exact sum is s + c up to the rounding of c.
template <class R>
struct RSum {
  R s, c;
  __device__ __forceinline__ void add(R v) {
    const R t = s + v;
    c += fabs(s) >= fabs(v) ? (s - t) + v : (v - t) + s;
    s = t;
  }
  __device__ __forceinline__ void merge(const RSum& o) {
    add(o.s);
    c += o.c;
  }
  __device__ __forceinline__ double value() const { return double(s) + double(c); }
};

// Quantities reduced: 0 mass, 1..3 momentum, 4 energy; plus a count of bad sites.
constexpr int NCONS = 5;
// Doubles per block in the partials array: the NCONS compensated pairs of the
// block's per-site sums, stored in the kernel's type R from the start of the
// slot, then the block's number of fluid sites (a double at index 2 NCONS).
constexpr int CONS_SLOT = 2 * NCONS + 1;

// Block-wide merge of per-thread compensated pairs in a fixed order: the pairs
// go to shared memory, one warp merges a quantity (each lane BS / 32 threads'
// pairs, then five shuffle steps), so a block's merge is BS / 32 + 4 dependent
// merges long.  All in R: with float storage no FP64 instruction runs here, with
// FP64 storage a merge is six of them at 64 cycles each, and this chain (of the
// blocks, and again of the last one) was most of a small grid's pass.  `tot`
// (shared memory) and the counts are valid in every thread afterwards; z is
// left out on two-dimensional grids.
template <class R, int BS, int D>
__device__ __forceinline__ void reduce_block(const RSum<R> (&v)[NCONS], unsigned n, unsigned bad,
                                             RSum<R> (&tot)[NCONS], unsigned& ntot,
                                             unsigned& btot) {
  static_assert(BS % 32 == 0 && BS >= 64, "block size");
  __shared__ R sh_s[NCONS][BS], sh_c[NCONS][BS];
  __shared__ unsigned sh_n[BS / 32], sh_b[BS / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int k = 0; k < NCONS; ++k) {
    if (D == 2 && k == 3) continue;
    sh_s[k][tid] = v[k].s;
    sh_c[k][tid] = v[k].c;
  }
  n = __reduce_add_sync(0xffffffffu, n);
  bad = __reduce_add_sync(0xffffffffu, bad);
  if (lane == 0) {
    sh_n[warp] = n;
    sh_b[warp] = bad;
  }
  __syncthreads();
  constexpr int NK = D == 2 ? NCONS - 1 : NCONS;
  for (int q = warp; q < NK; q += BS / 32) {
    const int k = D == 2 && q == 3 ? 4 : q;
    RSum<R> a{sh_s[k][lane], sh_c[k][lane]};
#pragma unroll
    for (int j = 1; j < BS / 32; ++j) a.merge(RSum<R>{sh_s[k][lane + 32 * j], sh_c[k][lane + 32 * j]});
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
      a.merge(RSum<R>{__shfl_down_sync(0xffffffffu, a.s, off), __shfl_down_sync(0xffffffffu, a.c, off)});
    if (lane == 0) tot[k] = a;
  }
  if (D == 2 && tid == 0) tot[3] = RSum<R>{};
  __syncthreads();
  ntot = 0u;
  btot = 0u;
  for (int w = 0; w < BS / 32; ++w) {
    ntot += sh_n[w];
    btot += sh_b[w];
  }
}

// Mass, momentum and energy (as s, c pairs of doubles: out[2k], out[2k + 1])
// from the grid's sums.  Uniform g: S = (sum drho, sum j, sum k2) and, with
// n fluid sites, mass M = n + S0, momentum c J + M g / 2, energy
// (D n + c^2 K2 + c J.g + M |g|^2 / 2) / 2 (mid-point values of R1).  Other
// forces: S = (sum drho, sum of per-site momentum, sum of per-site energy
// less D / 2), so the momentum is S1..3 and the energy D n / 2 + S4.
template <class L, class R>
__device__ __forceinline__ void conserved_from_sums(const RSum<R> (&S)[NCONS], double n,
                                                    const StepParams& p, double* out) {
  constexpr int D = L::D;
  double v[NCONS];
  for (int k = 0; k < NCONS; ++k) v[k] = S[k].value();
  const double mass = n + v[0];
  double res[NCONS];
  res[0] = mass;
  res[1] = res[2] = res[3] = 0.0;
  if (p.gkind == G_UNIFORM) {
    const double g[3] = {p.g0[0], p.g0[1], D == 3 ? p.g0[2] : 0.0};
    double jg = 0.0;
    for (int a = 0; a < D; ++a) {
      res[1 + a] = L::c * v[1 + a] + 0.5 * g[a] * mass;
      jg += L::c * v[1 + a] * g[a];
    }
    const double g2 = g[0] * g[0] + g[1] * g[1] + g[2] * g[2];
    res[4] = 0.5 * (double(D) * n + L::c2 * v[4] + jg + 0.5 * g2 * mass);
  } else {
    for (int a = 0; a < D; ++a) res[1 + a] = v[1 + a];
    res[4] = 0.5 * double(D) * n + v[4];
  }
  for (int k = 0; k < NCONS; ++k) {
    out[2 * k] = res[k];
    out[2 * k + 1] = 0.0;
  }
}

// Merge of the partials of nblocks blocks (slot layout CONS_SLOT) by one
// block of BS threads, in a fixed order: thread t takes blocks t, t + BS, ...
// then the block merge above.  Thread 0 writes out[0 .. 2 NCONS - 1] (s, c
// pairs) and out[2 NCONS] = the bad-site count.
template <class L, class R, int BS>
__device__ __forceinline__ void reduce_partials(const double* __restrict__ part,
                                                const unsigned* __restrict__ badcount, int nblocks,
                                                const StepParams& p, double* out) {
  RSum<R> f[NCONS] = {};
  unsigned n = 0u, b = 0u;
  for (int blk = threadIdx.x; blk < nblocks; blk += BS) {
    const double* slot = part + (size_t)blk * CONS_SLOT;
    const R* rs = reinterpret_cast<const R*>(slot);
    for (int k = 0; k < NCONS; ++k) f[k].merge(RSum<R>{__ldcg(rs + 2 * k), __ldcg(rs + 2 * k + 1)});
    n += (unsigned)__ldcg(slot + 2 * NCONS);
    b += __ldcg(badcount + blk);
  }
  __shared__ RSum<R> tot[NCONS];
  unsigned ntot, btot;
  reduce_block<R, BS, L::D>(f, n, b, tot, ntot, btot);
  if (threadIdx.x == 0) {
    conserved_from_sums<L, R>(tot, double(ntot), p, out);
    out[2 * NCONS] = double(btot);
  }
}

// Grid-stride pass: block b handles row tiles b, b + gridDim.x, ... (one
// site per thread and tile; threads past the row end contribute nothing).
// Per site only the raw moments are needed, in the codec's arithmetic
// precision: mass rho = 1 + drho, momentum rho u = c j + rho g / 2, energy
// rho (|u|^2 + D theta) / 2 = (K + c j.g + rho |g|^2 / 2) / 2 with
// K = D + c^2 k2 (mid-point values of R1, no division).  With a uniform g
// these are linear in the sums of drho, j and k2, so a thread sums only
// those; otherwise it sums the per-site momentum and energy.  Each thread
// keeps compensated pairs in R; the block merges them (reduce_block) and
// writes its slot of `part` (CONS_SLOT doubles per block) and its bad-site
// count.  The number of blocks is fixed by the caller, so the summation
// order, and the result, are deterministic for a grid.
//
// ticket != nullptr: the last block to finish (by an atomic ticket) also
// reduces all partials in block order into out (the k_conserved_final
// layout, plus out[2 NCONS + 1] = *err, the bounded-wait error flag) and
// resets the ticket; out may be mapped host memory.
// Resident 128-thread blocks per SM the conservation pass is compiled for
// (its grid is LBM_CONSERVED_BLOCKS blocks per SM, a tuning hook).
#ifndef LBM_CONSERVED_BLOCKS
#define LBM_CONSERVED_BLOCKS 4
#endif
template <class L, int P>
__global__ void __launch_bounds__(128, LBM_CONSERVED_BLOCKS) k_conserved(const typename Codec<P>::T* __restrict__ fin,
                                                   double* __restrict__ part,
                                                   unsigned* __restrict__ badcount,
                                                   unsigned* __restrict__ ticket,
                                                   double* __restrict__ out,
                                                   const int* __restrict__ err,
                                                   const StepParams p) {
  using R = typename Codec<P>::R;
  constexpr int Q = L::Q, D = L::D;
  const int ntx = (p.nx + 127) / 128;
  const int ntiles = ntx * (D == 2 ? p.na : p.ny * p.na);
  const bool uniform = p.gkind == G_UNIFORM;
  RSum<R> sums[NCONS] = {};
  unsigned count = 0u, bad = 0u;
  const bool walls = p.wall != W_NONE;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    // the wall rows, whose pull also gathers the wall sums, come first so
    // that they do not form the tail of the pass
    const int xt = t % ntx, row = t / ntx;
    const int y = D == 2 ? p.a0 + wall_rows_first(row, p.na, walls) : row % p.ny;
    const int z = D == 3 ? p.a0 + wall_rows_first(row / p.ny, p.na, walls) : 0;
    const int x = xt * 128 + threadIdx.x;
    if (x >= p.nx) continue;
    const int site = (z * p.ny + y) * p.nx + x;
    const int cls = p.solid ? p.site_class[site] : 0;
    if (cls == 1) continue;
    const int a = D == 2 ? y : z;
    const int nA = D == 2 ? p.ny : p.nz;
    const int wx0 = xt * 128 + (threadIdx.x & ~31);
    const bool near = near_wall(p, a, nA);
    const bool interior = !near && wx0 >= 3 && wx0 + 31 <= p.nx - 4;
    RawMoments<L, R> r;
    if constexpr (P == P_FP64) {  // pair sums and mirror groups: fewer FP64 operations
      R d0, s[(Q - 1) / 2], am[(Q - 1) / 2];
      if (!cls && !near) {
        R f[Q];
        if (interior) pull_interior<L, P, R, LD_HINT, IN_STORED>(fin + site, p, y, z, f);
        else pull_stored<L, P, R>(fin, p, x, y, z, f);
        pair_split<L, R>(f, d0, s, am);
      } else {
        R d[Q];
        if (cls) pull_solid<L, P, R>(fin, p, x, y, z, site, d);
        else pull<L, P, R>(fin, p, x, y, z, d);
        pair_split_dev<L, R>(d, d0, s, am);
      }
      r = pair_moments<L, R>(d0, s, am);
    } else {
      R d[Q];
      if (cls) pull_solid<L, P, R>(fin, p, x, y, z, site, d);
      else if (interior) pull_interior<L, P, R>(fin + site, p, y, z, d);
      else pull<L, P, R>(fin, p, x, y, z, d);
      r = raw_moments<L, R>(d);
    }
    R g[3];
    if (sizeof(R) == sizeof(float) && p.gkind == G_FIELD && p.gtab_f == nullptr) {
      // a caller's double field without a float copy (lbm_conserved_static),
      // rounded to float as a context rounds its copy
      g[0] = R(__ldg(p.gtab + site));
      g[1] = R(__ldg(p.gtab + (size_t)p.N + site));
      g[2] = D == 3 ? R(__ldg(p.gtab + 2 * (size_t)p.N + site)) : R(0);
    } else {
      site_force_r<D, R>(p, x, y, z, site, g);
    }
    ++count;
    sums[0].add(r.drho);
    const R j0 = mul_c<L, R>(r.j[0]), j1 = mul_c<L, R>(r.j[1]), j2 = mul_c<L, R>(r.j[2]);
    const R rr = R(1) + r.drho;
    const R g2 = g[0] * g[0] + g[1] * g[1] + g[2] * g[2];
    if (uniform) {
      for (int a2 = 0; a2 < D; ++a2) sums[1 + a2].add(r.j[a2]);
      sums[4].add(r.k2);
    } else {
      const R hr = R(0.5) * rr;
      sums[1].add(fma(hr, g[0], j0));
      sums[2].add(fma(hr, g[1], j1));
      if (D == 3) sums[3].add(fma(hr, g[2], j2));
      const R jg = j0 * g[0] + j1 * g[1] + j2 * g[2];
      sums[4].add(R(0.5) * (mul_c2<L, R>(r.k2) + jg + R(0.5) * rr * g2));
    }
    // positivity check in the codec's precision, without divisions:
    // D theta = (K - |c j|^2 / rho) / rho + g^2 / 4 with K = D + c^2 k2, so
    // for rho > 0, theta > 0 exactly when e = K rho - |c j|^2 + rho^2 g^2 / 4
    // > 0; a NaN or infinite moment makes e NaN or infinite
    const R K = R(D) + mul_c2<L, R>(r.k2);
    const R e = fma(rr * rr, R(0.25) * g2, fma(K, rr, -(j0 * j0 + j1 * j1 + j2 * j2)));
    bad += (rr > R(0) && e > R(0) && isfinite(e)) ? 0u : 1u;
  }
  {
    __shared__ RSum<R> tot[NCONS];
    unsigned ntot, btot;
    reduce_block<R, 128, D>(sums, count, bad, tot, ntot, btot);
    if (threadIdx.x == 0) {
      double* slot = part + (size_t)blockIdx.x * CONS_SLOT;
      R* rs = reinterpret_cast<R*>(slot);
      for (int k = 0; k < NCONS; ++k) {
        rs[2 * k] = tot[k].s;
        rs[2 * k + 1] = tot[k].c;
      }
      slot[2 * NCONS] = double(ntot);
      badcount[blockIdx.x] = btot;
    }
  }
  if (!ticket) return;
  // the last block to finish reduces every block's partials, in block order
  __shared__ bool last;
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  reduce_partials<L, R, 128>(part, badcount, gridDim.x, p, out);
  if (threadIdx.x == 0) {
    out[2 * NCONS + 1] = err ? double(*(volatile const int*)err) : 0.0;
    *ticket = 0u;
  }
}

// Final pass of the two-kernel form: one block of 128 threads merges the
// partials of k_conserved (launched without a ticket) into out: 2 NCONS
// doubles (s, c pairs) followed by the bad-site count (as double).
template <class L, int P>
__global__ void __launch_bounds__(128) k_conserved_final(const double* __restrict__ part,
                                                         const unsigned* __restrict__ badcount,
                                                         int nblocks, double* __restrict__ out,
                                                         const StepParams p) {
  reduce_partials<L, typename Codec<P>::R, 128>(part, badcount, nblocks, p, out);
}

// ------------------------------------------------------ state access
template <class L, int P>
__global__ void __launch_bounds__(128) k_get_pulled(const typename Codec<P>::T* __restrict__ fin,
                                                    double* __restrict__ out, const StepParams p) {
  constexpr int Q = L::Q, D = L::D;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= p.nx) return;
  const int y = D == 2 ? p.a0 + (int)blockIdx.y : (int)blockIdx.y;
  const int z = D == 3 ? p.a0 + (int)blockIdx.z : 0;
  const int site = (z * p.ny + y) * p.nx + x;
  const size_t N = (size_t)p.N;
  if (p.solid && p.solid[site]) {
    static_for<0, Q>([&](auto I) { out[int(I) * N + site] = 0.0; });
    return;
  }
  double d[Q];
  if (p.solid) pull_solid<L, P, double>(fin, p, x, y, z, site, d);
  else pull<L, P, double>(fin, p, x, y, z, d);
  static_for<0, Q>([&](auto I) {
    constexpr int i = I;
    out[i * N + site] = L::W(i) + d[i];
  });
}

// DIR = 0: out = decode(f) + w ; DIR = 1: f = encode(in - w)
template <class L, int P, int DIR>
__global__ void __launch_bounds__(128) k_state(typename Codec<P>::T* __restrict__ f,
                                               double* __restrict__ io, const StepParams p) {
  using C = Codec<P>;
  constexpr int Q = L::Q, D = L::D;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= p.nx) return;
  const int y = D == 2 ? p.a0 + (int)blockIdx.y : (int)blockIdx.y;
  const int z = D == 3 ? p.a0 + (int)blockIdx.z : 0;
  const int site = (z * p.ny + y) * p.nx + x;
  const size_t N = (size_t)p.N;
  static_for<0, Q>([&](auto I) {
    constexpr int i = I;
    if (DIR == 0)
      io[i * N + site] = L::W(i) + double(C::template decode<L, i>(f[i * N + site], p));
    else
      f[i * N + site] = C::template encode<L, i>(typename C::R(io[i * N + site] - L::W(i)), p);
  });
}

}  // namespace lbm
