// lbm_split.cuh -- the FP64 step of small D2Q37 grids, several lanes per site.
//
// What bounds the one-thread-per-site step on a small grid: a warp's FP64
// instruction takes 64 cycles on its sub-partition (19 when all four of an SM
// share the unit) whatever the number of active lanes, dependent or not, so a
// grid with fewer warps than sub-partitions takes some 420 x 64 cycles a step
// however small it is.  So several lanes share a site:
//   k_step_split: 8 lanes; lane g takes the direction pairs g, g + 8, g + 16, its
//     partial moments are summed by shuffles, every lane forms the site's
//     coefficients and stores its own pairs: some 200 operations a lane.  The
//     pairs of different lanes run the same instructions, so their directions
//     are data: small integers unpacked from immediates for the addresses,
//     doubles from a table.
//   k_step_sym: 2 lanes, which exploit that the velocity set maps onto itself
//     when x and y are swapped (see there): some 265 operations a lane.
// GB300, microseconds a step (20-step graphs), one thread per site -> here:
// 3 x 150 with thermal walls 30.0 -> 10.1, 24 x 24 22.6 -> 11.4, 64 x 64 22.7 ->
// 11.6 (17.2 with lbm_poly.cuh alone), with walls 30.0 -> 13.6, 96 x 96 22.8 ->
// 12.6.  The lanes multiply the FP64 work of a site (4.0 and 1.2 times), which
// counts when many small grids are stepped in streams of their own.  So 8 lanes
// are taken only up to one warp per multiprocessor (3 x 150: 16 lanes take 9.5
// us alone, but 21.2 for each step of eight grids at once where 8 lanes take
// 14.0 and one thread 37), and for rows of 12 sites at most, which leave most of
// a one-thread warp idle anyway: us a step and grid, 64 grids at once, one thread
// with the collision pair by pair -> 8 lanes, 12 x 50 1.85 -> 1.73, but 16 x 38 1.42 ->
// 1.75 and 32 x 19 0.76 -> 1.74 (2 lanes 0.61).  2 lanes up to one warp per
// sub-partition (eight 64 x 64 at once: 40.9 -> 34.1).
#pragma once

#include "lbm_kernels.cuh"

namespace lbm {

// Doubles of a pair slot: e, the products of its components, the weight, that of the
// collision (collision_w), |e|^2, and the factor m of the pair sum in the density (1; 1/2 for the rest
// particle, the last slot, which enters with both members equal).
struct SplitSlot {
  double x, y, xx, xy, yy, w, wg, e2, m;
};
constexpr int SPLIT_SLOTS = 19;
constexpr int SPLIT_LEAVES = 26;
struct SplitTable {
  SplitSlot s[SPLIT_SLOTS];
  // populations that leave through the low wall, one entry per wall row they
  // leave from: direction j and row r (those through the high wall: the
  // opposite directions, rows from the top)
  signed char leave_j[SPLIT_LEAVES], leave_r[SPLIT_LEAVES];
};
__host__ __device__ constexpr SplitTable make_split_table() {
  using L = D2Q37;
  SplitTable t{};
  for (int k = 0; k < SPLIT_SLOTS; ++k) {
    const int i = k < SPLIT_SLOTS - 1 ? 2 * k + 1 : 0;
    const double x = L::e[i][0], y = L::e[i][1];
    t.s[k] = SplitSlot{x, y, x * x, x * y, y * y, L::w[i], collision_w<L>(i), x * x + y * y, i ? 1.0 : 0.5};
  }
  int n = 0;
  for (int j = 0; j < L::Q; ++j)
    for (int r = 0; r < -L::e[j][1]; ++r) {
      t.leave_j[n] = (signed char)j;
      t.leave_r[n] = (signed char)r;
      ++n;
    }
  return t;
}
// e_x (2 bits) and e_y + 3 (3 bits) of the first member of each slot
__host__ __device__ constexpr unsigned long long split_ex() {
  unsigned long long v = 0;
  for (int k = 0; k < SPLIT_SLOTS - 1; ++k) v |= (unsigned long long)D2Q37::e[2 * k + 1][0] << (2 * k);
  return v;
}
__host__ __device__ constexpr unsigned long long split_ey() {
  unsigned long long v = 3ull << (3 * (SPLIT_SLOTS - 1));
  for (int k = 0; k < SPLIT_SLOTS - 1; ++k) v |= (unsigned long long)(D2Q37::e[2 * k + 1][1] + 3) << (3 * k);
  return v;
}
static __device__ const SplitTable split_table = make_split_table();

// Lanes per site of a grid of `sites` sites on nsm multiprocessors; 0: one
// thread per site.
inline int split_lanes(int nx, long long sites, int nsm) {
  if (nx <= 12 && sites * 8 <= 32LL * nsm) return 8;  // at most one warp per multiprocessor
  if (sites * 2 <= 32LL * 4 * nsm) return 2;    // at most one warp per sub-partition
  return 0;
}

template <int G>
__device__ __forceinline__ double group_sum(double v) {
#pragma unroll
  for (int o = G / 2; o > 0; o /= 2) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

constexpr int SPLIT_THREADS = 32;

template <int FO, int G>
__global__ void __launch_bounds__(SPLIT_THREADS) k_step_split(const double* __restrict__ fin, double* __restrict__ fout,
                                                              const StepParams p) {
  using L = D2Q37;
  constexpr int R = (SPLIT_SLOTS + G - 1) / G;  // slots per lane
  const int lane = threadIdx.x & (G - 1);
  const int nx = p.nx, nA = p.ny;
  const size_t N = (size_t)p.N;
  // sites of the layers a0 .. a0 + na - 1, row after row; the lanes past the end
  // repeat the last site (every lane takes part in the shuffles) and store nothing
  const int n = nx * p.na, own = (blockIdx.x * SPLIT_THREADS + threadIdx.x) / G;
  const int idx = own < n ? own : n - 1;
  const int x = idx % nx, y = p.a0 + idx / nx, site = y * nx + x;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  int leave_j[(SPLIT_LEAVES + G - 1) / G], leave_r[(SPLIT_LEAVES + G - 1) / G];
  if (p.wall == W_THERMAL) {
#pragma unroll
    for (int r = 0; r < (SPLIT_LEAVES + G - 1) / G; ++r) {
      const int t = lane + r * G < SPLIT_LEAVES ? lane + r * G : 0;
      leave_j[r] = split_table.leave_j[t];  // > 0: it moves
      leave_r[r] = split_table.leave_r[t];
    }
  }
  double g3[3];
  site_force<2>(p, x, y, 0, site, g3);
  const double g[2] = {g3[0], g3[1]};
  fin = wait_previous(fin);
  // ---- pull: the members + and - of each slot
  const int side = y < 3 ? 0 : 1;
  const bool near = near_wall(p, y, nA);
  double fp[R], fm[R];
  int beyond = 0;  // bits 2r, 2r + 1: the member of slot r comes from beyond a thermal wall
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int k = lane + r * G, i = 2 * k + 1;  // slot R - 1 may lie past the table
    const bool rest = k >= SPLIT_SLOTS - 1;
    const int ex = rest ? 0 : (int)(split_ex() >> (2 * k)) & 3, ey = rest ? 0 : ((int)(split_ey() >> (3 * k)) & 7) - 3;
    const int ip = rest ? 0 : i, im = rest ? 0 : i + 1;
    int yp = y - ey, ym = y + ey, jp = ip, jm = im;  // source rows and populations
    int xp = wrap3(x - ex, nx), xm = wrap3(x + ex, nx);
    if (p.wall == W_NONE) {
      yp = wrap3(yp, nA);
      ym = wrap3(ym, nA);
    } else if (near) {
      if (yp < 0 || yp >= nA) {  // bounced: the opposite population of the mirrored row, same column
        beyond |= 1 << (2 * r);
        yp = side == 0 ? ey - 1 - y : 2 * nA - 1 - yp;
        jp = im;
        xp = x;
      }
      if (ym < 0 || ym >= nA) {
        beyond |= 2 << (2 * r);
        ym = side == 0 ? -ey - 1 - y : 2 * nA - 1 - ym;
        jm = ip;
        xm = x;
      }
    }
    fp[r] = fin[(jp * N + (size_t)(yp * nx + xp))];
    fm[r] = fin[(jm * N + (size_t)(ym * nx + xm))];
  }
  // what leaves the column through a thermal wall, loaded with the pull: one
  // latency for both (as loops of their own they took 3 us a step)
  const bool thermal = p.wall == W_THERMAL && near;
  constexpr int LR = (SPLIT_LEAVES + G - 1) / G;
  double leave[LR] = {};
  if (thermal) {
#pragma unroll
    for (int r = 0; r < LR; ++r) {
      const int t = lane + r * G;
      if (t < SPLIT_LEAVES) {
        const int j = leave_j[r], row = side == 0 ? leave_r[r] : nA - 1 - leave_r[r];
        leave[r] = fin[((side == 0 ? j : ((j & 1) ? j + 1 : j - 1)) * N + (size_t)(row * nx + x))];
      }
    }
  }
  double rm1 = 0.0;  // rho_w - 1 of the thermal wall
  if (__any_sync(0xffffffffu, thermal)) {
    double sum = 0.0;
#pragma unroll
    for (int r = 0; r < LR; ++r)
      if (thermal && lane + r * G < SPLIT_LEAVES) sum += leave[r] - split_table.s[(leave_j[r] - 1) / 2].w;
    rm1 = (p.wallA[side] + group_sum<G>(sum)) * p.wall_inv_den[side];
  }
  // ---- pair sums and differences, moments
  double s[R], a[R];
  double m0 = 0.0, jx = 0.0, jy = 0.0, k2 = 0.0;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int k = lane + r * G;
    const int kt = k < SPLIT_SLOTS ? k : SPLIT_SLOTS - 1;
    const SplitSlot& t = split_table.s[kt];
    double dp = fp[r] - t.w, dm = fm[r] - t.w;
    if (thermal) {
      const int ip = 2 * k + 1;  // (never the rest particle)
      if (beyond & 1 << (2 * r)) dp = fma(rm1, p.fw[side][ip], p.fwd[side][ip]);
      if (beyond & 2 << (2 * r)) dm = fma(rm1, p.fw[side][ip + 1], p.fwd[side][ip + 1]);
    }
    s[r] = dp + dm;
    a[r] = dp - dm;
    if (k >= SPLIT_SLOTS) s[r] = 0.0;  // no such pair: past the rest particle
    m0 = fma(t.m, s[r], m0);
    jx = fma(t.x, a[r], jx);
    jy = fma(t.y, a[r], jy);
    k2 = fma(t.e2, s[r], k2);
  }
  m0 = group_sum<G>(m0);
  jx = group_sum<G>(jx);
  jy = group_sum<G>(jy);
  k2 = group_sum<G>(k2);
  // ---- mid-point state and coefficients, in every lane
  SiteState<double> m;
  m.drho = m0;
  m.rho = 1.0 + m0;
  const double irho = 1.0 / m.rho;
  // u and the temperature as in site_coefficients
  const double cirho = L::c * irho, hgx = 0.5 * g[0], hgy = 0.5 * g[1];
  const double ux = fma(jx, cirho, hgx), uy = fma(jy, cirho, hgy);
  const double utx = ux - hgx, uty = uy - hgy;
  const double ut2 = fma(uty, uty, utx * utx), g2 = fma(g[1], g[1], g[0] * g[0]);
  const double gu = fma(g[1], uy, g[0] * ux);
  m.u2 = fma(uy, uy, ux * ux);
  m.Th = fma(fma(fma(L::c2, k2, -2.0 * m0), irho, -ut2), 0.5, 0.125 * g2);
  m.om = site_omega<double>(p, m.rho, 1.0 + m.Th);
  m.rom = m.rho * m.om;
  const double rk = fma(-0.5, m.rom, m.rho);
  m.rkgu = FO >= 1 ? rk * gu : 0.0;
  m.T = L::c2 * m.Th;
  const double crk = L::c * rk;
  m.U[0] = L::c * ux;
  m.U[1] = L::c * uy;
  m.S[0] = crk * g[0];
  m.S[1] = crk * g[1];
  m.U[2] = m.S[2] = 0.0;
  PolyCoef2<double> c;
  poly_coef<(FO == 3 ? 2 : FO)>(m, c);
  if constexpr (FO == 3) {
    double P0 = 0.0, P1 = 0.0, P3 = 0.0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int k = lane + r * G;
      const SplitSlot& t = split_table.s[k < SPLIT_SLOTS ? k : SPLIT_SLOTS - 1];
      P0 = fma(t.xx, s[r], P0);
      P1 = fma(t.yy, s[r], P1);
      P3 = fma(t.xy, s[r], P3);
    }
    double S[6];
    const double u3[3] = {ux, uy, 0.0};
    stress_from_sums<L, double>(group_sum<G>(P0), group_sum<G>(P1), 0.0, group_sum<G>(P3), 0.0, 0.0, m0, m.rho, m.Th, u3,
                                g3, S);
    const double kf = fma(-0.5, m.om, 1.0);
    poly_add_stress(stress_terms<L, double>(S, g3, 0.5 * kf * kf), c);
  }
  // ---- relax and store: w G by its monomials
  const double hom1 = fma(-0.5, m.om, 0.5);
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int k = lane + r * G;
    const SplitSlot& t = split_table.s[k < SPLIT_SLOTS ? k : SPLIT_SLOTS - 1];
    const double ex4 = fma(t.xx, c.E40, fma(t.xy, c.E31, fma(t.yy, c.E22, c.E20)));
    const double ey4 = fma(t.yy, c.E04, fma(t.xy, c.E13, c.E02));
    const double even = fma(t.xx, ex4, fma(t.yy, ey4, fma(t.xy, c.E11, c.E00)));
    const double ox3 = fma(t.xx, c.O30, fma(t.xy, c.O21, fma(t.yy, c.O12, c.O10)));
    const double oy3 = fma(t.yy, c.O03, c.O01);
    const double odd = fma(t.x, ox3, t.y * oy3);
    const double ev = fma(hom1, s[r], t.wg * even), od = fma(hom1, a[r], t.wg * odd);
    if (own < n && k < SPLIT_SLOTS) {
      const int i = k < SPLIT_SLOTS - 1 ? 2 * k + 1 : 0;
      fout[i * N + site] = (ev + od) + t.w;
      if (k < SPLIT_SLOTS - 1) fout[(i + 1) * N + site] = (ev - od) + t.w;
    }
  }
}

// ---- two lanes per site
// The velocity set maps onto itself when x and y are swapped, so two lanes can
// run the same instructions on compile-time directions: both work in a local
// frame, x-y for lane 0 and y-x for lane 1, on the pairs
//   (1, 0) (2, 0) (3, 0) (2, +-1) (3, +-1) (q, +-q), q = 1 in lane 0, 2 in lane 1,
// which together are all eighteen; lane 0 adds the rest particle.  Of the
// coefficients a lane forms those of its local x and gets those of y from its
// partner.  Some 265 FP64 operations a lane against 420 in one thread, so a
// grid of few warps takes 0.6 of the time, for 1.2 times the FP64 work.
struct PairPath {  // population indexes and vector of a local pair's first member in global terms
  int ip, im, ex, ey;
};
__host__ __device__ constexpr int dir_of(int ex, int ey) {
  for (int i = 0; i < D2Q37::Q; ++i)
    if (D2Q37::e[i][0] == ex && D2Q37::e[i][1] == ey) return i;
  return -1;
}
constexpr int SYM_PAIRS = 9;
__host__ __device__ constexpr PairPath sym_path(int role, int k) {
  const int q = role ? 2 : 1;
  const int la[SYM_PAIRS] = {1, 2, 3, 2, 2, 3, 3, q, q}, lb[SYM_PAIRS] = {0, 0, 0, 1, -1, 1, -1, q, -q};
  const int ex = role ? lb[k] : la[k], ey = role ? la[k] : lb[k];
  return PairPath{dir_of(ex, ey), dir_of(-ex, -ey), ex, ey};
}

template <int FO>
__global__ void __launch_bounds__(SPLIT_THREADS) k_step_sym(const double* __restrict__ fin, double* __restrict__ fout,
                                                            const StepParams p) {
  using L = D2Q37;
  constexpr int NP = SYM_PAIRS;
  constexpr unsigned ALL = 0xffffffffu;
  const int role = threadIdx.x & 1;
  const int nx = p.nx, nA = p.ny;
  const size_t N = (size_t)p.N;
  // as k_step_split: the lanes past the end repeat the last site and store nothing
  const int n = nx * p.na, own = (blockIdx.x * SPLIT_THREADS + threadIdx.x) / 2;
  const int idx = own < n ? own : n - 1;
  const int x = idx % nx, y = p.a0 + idx / nx, site = y * nx + x;
  auto other = [](double v) { return __shfl_xor_sync(ALL, v, 1); };
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  double g3[3];
  site_force<2>(p, x, y, 0, site, g3);
  const double g[2] = {role ? g3[1] : g3[0], role ? g3[0] : g3[1]};  // local
  fin = wait_previous(fin);
  const int side = y < 3 ? 0 : 1;
  const bool near = near_wall(p, y, nA);
  // the weights that differ between the lanes
  constexpr double w11 = L::shell_w[2], w22 = L::shell_w[5];
  const double wq = role ? w22 : w11, q = role ? 2.0 : 1.0, qq = role ? 4.0 : 1.0;
  double fp[NP], fm[NP];
  unsigned beyond = 0;  // bits 2k, 2k + 1: the member of pair k comes from beyond a wall
  static_for<0, NP>([&](auto K) {
    constexpr int k = K;
    constexpr PairPath a0 = sym_path(0, k), a1 = sym_path(1, k);
    const int ip = role ? a1.ip : a0.ip, im = role ? a1.im : a0.im;
    const int ex = role ? a1.ex : a0.ex, ey = role ? a1.ey : a0.ey;
    int yp = y - ey, ym = y + ey, jp = ip, jm = im;
    int xp = wrap3(x - ex, nx), xm = wrap3(x + ex, nx);
    if (p.wall == W_NONE) {
      yp = wrap3(yp, nA);
      ym = wrap3(ym, nA);
    } else if (near) {
      if (yp < 0 || yp >= nA) {
        beyond |= 1u << (2 * k);
        yp = side == 0 ? ey - 1 - y : 2 * nA - 1 - yp;
        jp = im;
        xp = x;
      }
      if (ym < 0 || ym >= nA) {
        beyond |= 2u << (2 * k);
        ym = side == 0 ? -ey - 1 - y : 2 * nA - 1 - ym;
        jm = ip;
        xm = x;
      }
    }
    fp[k] = fin[(jp * N + (size_t)(yp * nx + xp))];
    fm[k] = fin[(jm * N + (size_t)(ym * nx + xm))];
  });
  const double f0 = fin[site];
  const bool thermal = p.wall == W_THERMAL && near;
  const bool any_thermal = __any_sync(ALL, thermal);  // warp-uniform
  double leave[SPLIT_LEAVES / 2] = {};  // of the column through a thermal wall: every other one
  if (thermal) {
    static_for<0, SPLIT_LEAVES / 2>([&](auto T) {
      constexpr SplitTable t = make_split_table();
      constexpr int j0 = t.leave_j[2 * T], j1 = t.leave_j[2 * T + 1], r0 = t.leave_r[2 * T], r1 = t.leave_r[2 * T + 1];
      const int j = role ? j1 : j0, r = role ? r1 : r0;
      const int js = side == 0 ? j : (j & 1 ? j + 1 : j - 1), row = side == 0 ? r : nA - 1 - r;
      leave[T] = fin[(js * N + (size_t)(row * nx + x))];
    });
  }
  double rm1 = 0.0;
  if (any_thermal) {
    double sum = 0.0;
    static_for<0, SPLIT_LEAVES / 2>([&](auto T) {
      constexpr SplitTable t = make_split_table();
      constexpr double w0 = L::W(t.leave_j[2 * T]), w1 = L::W(t.leave_j[2 * T + 1]);
      if (thermal) sum += leave[T] - (role ? w1 : w0);
    });
    rm1 = (p.wallA[side] + (sum + other(sum))) * p.wall_inv_den[side];
  }
  // ---- pair sums and differences (pair_split, or from deviations where a wall fills slots)
  constexpr double wk[NP - 2] = {L::shell_w[1], L::shell_w[3], L::shell_w[6], L::shell_w[4], L::shell_w[4], L::shell_w[7],
                                 L::shell_w[7]};
  double s[NP], a[NP];
  static_for<0, NP>([&](auto K) {
    constexpr int k = K;
    double w = wq;
    if constexpr (k < NP - 2) w = wk[k];
    const double dm = fm[k] - w;
    a[k] = fp[k] - fm[k];
    s[k] = fma(2.0, dm, a[k]);
    if (any_thermal) {
      constexpr PairPath a0 = sym_path(0, k), a1 = sym_path(1, k);
      double dp = fp[k] - w, dn = dm;
      if (thermal && (beyond & 1u << (2 * k))) {
        const int i = role ? a1.ip : a0.ip;
        dp = fma(rm1, p.fw[side][i], p.fwd[side][i]);
      }
      if (thermal && (beyond & 2u << (2 * k))) {
        const int i = role ? a1.im : a0.im;
        dn = fma(rm1, p.fw[side][i], p.fwd[side][i]);
      }
      if (thermal) {
        s[k] = dp + dn;
        a[k] = dp - dn;
      }
    }
  });
  const double d0 = f0 - L::shell_w[0];
  // ---- moments: local sums, then the partner's with x and y swapped
  const double S21 = s[3] + s[4], S31 = s[5] + s[6], SC = s[7] + s[8];
  double m0 = ((s[0] + s[1]) + (s[2] + S21)) + (S31 + SC);
  double k2 = fma(4.0, s[1], s[0]);
  k2 = fma(9.0, s[2], k2);
  k2 = fma(5.0, S21, k2);
  k2 = fma(10.0, S31, k2);
  k2 = fma(2.0 * qq, SC, k2);
  double jx = fma(2.0, a[1] + (a[3] + a[4]), a[0]);
  jx = fma(3.0, a[2] + (a[5] + a[6]), jx);
  jx = fma(q, a[7] + a[8], jx);
  double jy = fma(q, a[7] - a[8], (a[3] - a[4]) + (a[5] - a[6]));
  m0 = m0 + other(m0) + d0;
  k2 = k2 + other(k2);
  const double jxo = other(jx), jyo = other(jy);
  jx += jyo;
  jy += jxo;
  // ---- mid-point state (local frame)
  const double rho = 1.0 + m0, irho = 1.0 / rho;
  const double cirho = L::c * irho, hgx = 0.5 * g[0], hgy = 0.5 * g[1];
  const double ux = fma(jx, cirho, hgx), uy = fma(jy, cirho, hgy);
  const double utx = ux - hgx, uty = uy - hgy;
  const double ut2 = fma(uty, uty, utx * utx), g2 = fma(g[1], g[1], g[0] * g[0]);
  const double gu = fma(g[1], uy, g[0] * ux);
  const double u2 = fma(uy, uy, ux * ux);
  const double Th = fma(fma(fma(L::c2, k2, -2.0 * m0), irho, -ut2), 0.5, 0.125 * g2);
  const double om = site_omega<double>(p, rho, 1.0 + Th);
  const double rom = rho * om;
  const double rk = fma(-0.5, rom, rho);
  const double rkgu = FO >= 1 ? rk * gu : 0.0;
  const double T = L::c2 * Th;
  const double crk = L::c * rk;
  const double X = L::c * ux, Y = L::c * uy, Sx = crk * g[0], Sy = crk * g[1];
  // ---- coefficients (poly_coef): the x ones here, the y ones from the partner
  PolyCoef2<double> c;
  {
    const double xx = X * X, xy = X * Y;
    const double b0 = fma(-0.5, u2, fma(-2.0, Th, 1.0));
    const double hT = 0.5 * T, hax = fma(0.5, xx, hT), th2 = 0.5 * Th;
    const double a00 = fma(fma(0.125, u2, Th), u2, fma(Th, Th, fma(-0.5, u2, -Th)));
    c.E00 = fma(rom, a00, FO >= 1 ? fma(om, m0, -rkgu) : om * m0);
    const double rx = rom * X;
    c.E20 = rom * fma(b0, hax, -(th2 * xx));
    c.E11 = rom * (b0 - Th) * xy;
    c.E40 = rom * fma(xx, fma(1.0 / 24.0, xx, 0.25 * T), 0.5 * hT * hT);
    c.E22 = rom * hax * other(hax);
    c.O30 = rx * fma(1.0 / 6.0, xx, hT);
    c.E31 = c.O30 * Y;
    if constexpr (FO >= 1) {
      c.E20 = fma(Sx, X, c.E20);
      c.E11 = fma(Sx, Y, fma(Sy, X, c.E11));
    }
    if constexpr (FO >= 2) {
      const double px = rx + Sx;
      c.O10 = fma(b0, px, -(rkgu * X));
      c.O30 = fma(hax, Sx, c.O30);
      c.O21 = fma(hax, other(px), Sx * xy);
    } else {
      c.O10 = fma(b0, rx, Sx);
      c.O21 = hax * other(rx);
    }
  }
  if constexpr (FO == 3) {  // the sigma-bar terms (poly_add_stress), x ones
    const double Pl = fma(qq, SC, fma(9.0, s[2] + S31, fma(4.0, s[1] + S21, s[0])));  // e_x^2
    const double Ql = fma(qq, SC, S21 + S31);                                        // e_y^2
    const double Cl = fma(qq, s[7] - s[8], fma(3.0, s[5] - s[6], 2.0 * (s[3] - s[4])));
    double S[6];
    const double u3[3] = {ux, uy, 0.0}, gl[3] = {g[0], g[1], 0.0};
    stress_from_sums<L, double>(Pl + other(Ql), Ql + other(Pl), 0.0, Cl + other(Cl), 0.0, 0.0, m0, rho, Th, u3, gl, S);
    const double kf = fma(-0.5, om, 1.0);
    const StressTerms<double> st = stress_terms<L, double>(S, gl, 0.5 * kf * kf);
    c.O10 -= st.hs[0];
    c.O30 = fma(st.gs[0], st.S[0], c.O30);
    c.O21 = fma(st.gs[1], st.S[0], fma(2.0 * st.gs[0], st.S[3], c.O21));
  }
  c.E02 = other(c.E20);
  c.E04 = other(c.E40);
  c.E13 = other(c.E31);
  c.O01 = other(c.O10);
  c.O03 = other(c.O30);
  c.O12 = other(c.O21);
  // ---- relax and store
  const double om1 = 1.0 - om, hom1 = 0.5 * om1;
  const bool mine = own < n;
  double* __restrict__ fo = fout + site;
  auto put = [&](auto K, double w, double wev, double wod) {
    constexpr int k = K;
    constexpr PairPath a0 = sym_path(0, k), a1 = sym_path(1, k);
    const double ev = fma(hom1, s[k], wev), od = fma(hom1, a[k], wod);
    if (mine) {
      fo[(role ? a1.ip : a0.ip) * N] = (ev + od) + w;
      fo[(role ? a1.im : a0.im) * N] = (ev - od) + w;
    }
  };
  if (mine && role == 0) fo[0] = fma(om1, d0, L::shell_w[0] * c.E00) + L::shell_w[0];
  const double xa1 = c.E00 + (c.E20 + c.E40), xa2 = fma(4.0, fma(4.0, c.E40, c.E20), c.E00),
               xa3 = fma(9.0, fma(9.0, c.E40, c.E20), c.E00);
  const double za1 = c.O10 + c.O30, za2 = fma(4.0, c.O30, c.O10), za3 = fma(9.0, c.O30, c.O10);
  constexpr double g9 = collision_w<L>(dir_of(3, 0)), g8 = collision_w<L>(dir_of(2, 2));
  put(ic<0>{}, wk[0], wk[0] * xa1, wk[0] * za1);
  put(ic<1>{}, wk[1], wk[1] * xa2, 2.0 * wk[1] * za2);
  put(ic<2>{}, wk[2], g9 * xa3, 3.0 * g9 * za3);
  auto quad = [&](auto K, double w, double A, double xa, double xb, double ya, double za, double wa) {  // (A, +-1)
    constexpr int k = K;
    const double ee = w * (xa + (xb + c.E04)), oo = ya + c.E13, oe = w * A * (za + c.O12), eo = wa + c.O03;
    put(ic<k>{}, w, fma(w * A, oo, ee), fma(w, eo, oe));
    put(ic<k + 1>{}, w, fma(-w * A, oo, ee), fma(-w, eo, oe));
  };
  quad(ic<3>{}, wk[3], 2.0, xa2, fma(4.0, c.E22, c.E02), fma(4.0, c.E31, c.E11), za2, fma(4.0, c.O21, c.O01));
  quad(ic<5>{}, wk[5], 3.0, xa3, fma(9.0, c.E22, c.E02), fma(9.0, c.E31, c.E11), za3, fma(9.0, c.O21, c.O01));
  {  // (q, +-q)
    const double gq = role ? g8 : w11;
    const double ee = gq * fma(qq, fma(qq, (c.E40 + c.E04) + c.E22, c.E20 + c.E02), c.E00);
    const double oo = fma(qq, c.E31 + c.E13, c.E11);
    const double wqq = gq * q;
    const double oe = wqq * fma(qq, c.O30 + c.O12, c.O10), eo = fma(qq, c.O03 + c.O21, c.O01);
    const double wq2 = gq * qq;
    put(ic<7>{}, wq, fma(wq2, oo, ee), fma(wqq, eo, oe));
    put(ic<8>{}, wq, fma(-wq2, oo, ee), fma(-wqq, eo, oe));
  }
}

inline unsigned split_blocks(const StepParams& p, int G) {
  return (unsigned)(((long long)p.nx * p.na * G + SPLIT_THREADS - 1) / SPLIT_THREADS);
}

}  // namespace lbm
