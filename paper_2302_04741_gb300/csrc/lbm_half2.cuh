// lbm_half2.cuh -- the FP16-scaled step with two adjacent sites per thread.
//
// What bounds the one-site step on FP16 storage: a 2-byte warp load or store
// moves 64 bytes, so its memory pattern alone stops at 0.59 of HBM, and it
// issues some 1,100 instructions a site.  Here a thread takes sites x and x + 1
// (x even, nx even): directions with even e_x are one aligned 4-byte load, the
// odd ones two 2-byte loads, every store is 4 bytes, and the collision runs on
// both sites at once in packed FP32 (add / mul / fma.rn.f32x2: two operations
// an instruction), so a pair of sites issues about as many instructions as one
// site before.  (Two sites per thread in scalar arithmetic had twice the
// instructions and needed its outputs held for the wide store: slower.)
//
// The packed operations round as the scalar ones, and every product that the
// compiler contracts into a sum in collide_store is written as that fma here,
// so the stored values are those of the one-site kernels (batches, TMA, wave),
// bit for bit.  Where a comment says "fused", the other choice is a different
// rounding.
#pragma once

#include "lbm_kernels.cuh"

namespace lbm {

// Packed pairs of floats: one value per site of the thread.
__device__ __forceinline__ float2 vb(float k) { return make_float2(k, k); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return __ffma2_rn(b, vb(-1.f), a); }
__device__ __forceinline__ float2 vneg(float2 a) { return make_float2(-a.x, -a.y); }
template <int K>
__device__ __forceinline__ float2 vimul(float2 v) {
  if constexpr (K == 0) return vb(0.f);
  else if constexpr (K == 1) return v;
  else if constexpr (K == -1) return vneg(v);
  else return vmul(vb(float(K)), v);
}
template <int K>
__device__ __forceinline__ float2 vmac(float2 v, float2 acc) {
  if constexpr (K == 0) return acc;
  else if constexpr (K == 1) return vadd(acc, v);
  else if constexpr (K == -1) return vsub(acc, v);
  else return vfma(vb(float(K)), v, acc);
}
template <class L, int I>
__device__ __forceinline__ float2 vedot(const float2 (&v)[3]) {
  constexpr int ex = L::E(I, 0), ey = L::E(I, 1), ez = L::E(I, 2);
  float2 acc = vimul<ex>(v[0]);
  acc = vmac<ey>(v[1], acc);
  if constexpr (L::D == 3) acc = vmac<ez>(v[2], acc);
  return acc;
}
template <int D>
__device__ __forceinline__ float2 vdot(const float2 (&a)[3], const float2 (&b)[3]) {
  const float2 r = vfma(a[0], b[0], vmul(a[1], b[1]));  // the first product fused
  return D == 3 ? vfma(a[2], b[2], r) : r;
}
// both halves of v as floats
__device__ __forceinline__ float2 h2f(unsigned v) { return __half22float2(*reinterpret_cast<const __half2*>(&v)); }

// Collision of two sites from their stored values h_i (two halves each), handed
// to out(direction, values): collide_store<L, P_FP16S, FO, true>, operation for
// operation.  A shell's coefficients are formed when its first pair is reached.
template <class L, int FO, class OUT>
__device__ __forceinline__ void collide2(const unsigned (&h)[L::Q], const float2 (&g)[3], const StepParams& p, OUT&& out) {
  constexpr int NP = (L::Q - 1) / 2, D = L::D;
  const float2 half = vb(0.5f);
  float2 drho = vmul(h2f(h[0]), vb(float(L::W(0)))), j[3] = {vb(0.f), vb(0.f), vb(0.f)}, k2 = vb(0.f);
  static_for<0, NP>([&](auto K) {
    constexpr int ip = 2 * K + 1, im = ip + 1;
    constexpr int ex = L::E(ip, 0), ey = L::E(ip, 1), ez = L::E(ip, 2);
    constexpr int e2 = ex * ex + ey * ey + ez * ez;
    constexpr double w = L::W(ip);
    const float2 fp = h2f(h[ip]), fm = h2f(h[im]);
    const float2 s = vadd(fp, fm), a = vsub(fp, fm);
    drho = vfma(s, vb(float(w)), drho);
    if constexpr (ex != 0) j[0] = vfma(a, vb(float(ex * w)), j[0]);
    if constexpr (ey != 0) j[1] = vfma(a, vb(float(ey * w)), j[1]);
    if constexpr (D == 3 && ez != 0) j[2] = vfma(a, vb(float(ez * w)), j[2]);
    k2 = vfma(s, vb(float(e2 * w)), k2);
  });
  const float2 is = vb(p.h_inv_scale), sc = vb(p.h_scale);
  drho = vmul(drho, is);
  k2 = vmul(k2, is);
  const float2 rho = vadd(vb(1.f), drho);
  const float2 irho = make_float2(1.f / rho.x, 1.f / rho.y);
  constexpr float c = f2_of(L::c).hi, c2 = f2_of(L::c2).hi;
  float2 u[3], ut[3];
  for (int a = 0; a < D; ++a) {
    const float2 x = vmul(vmul(j[a], is), irho);
    u[a] = vfma(vb(c), x, vmul(half, g[a]));
    ut[a] = vfma(vb(-0.5f), g[a], u[a]);
  }
  const float2 g2 = vdot<D>(g, g);
  const float2 uts = vdot<D>(ut, ut);
  const float2 t0 = vfma(vb(c2), k2, vmul(vb(-float(D)), drho));
  const float2 t1 = vfma(t0, irho, vneg(uts));
  const float2 Th = vfma(g2, vb(float(0.25 / D)), vmul(t1, vb(float(1.0 / D))));
  const float2 u2 = vdot<D>(u, u), gu = vdot<D>(g, u);
  float2 om;
  if (p.mu_f > 0.f) {
    const float2 th = vadd(vb(1.f), Th);
    om = make_float2(site_omega<float>(p, rho.x, th.x), site_omega<float>(p, rho.y, th.y));
  } else {
    om = vb(p.omega_f);
  }
  const float2 om1 = vsub(vb(1.f), om);
  const float2 hom1 = vmul(half, om1);
  const float2 kf = vfma(vb(-0.5f), om, vb(1.f));
  const float2 rom0 = vmul(rho, om);
  const float2 rom = vmul(rom0, sc);
  const float2 rk = vmul(rho, kf);
  const float2 rkgu = FO >= 1 ? vmul(vmul(rk, gu), sc) : vb(0.f);
  const float2 rkf = vmul(rk, sc);
  float2 cu[3], cs[3];
  for (int a = 0; a < D; ++a) {
    cu[a] = vmul(vb(c), u[a]);
    cs[a] = vmul(vb(c), vmul(rkf, g[a]));
  }
  float2 a00, c1 = half, g0c = half;
  if constexpr (D == 3) {
    a00 = vfma(vb(-0.5f), u2, vmul(vb(-1.5f), Th));
  } else {
    a00 = vfma(vb(-0.5f), u2, vneg(Th));
    const float2 e = vmul(vb(0.125f), u2);
    const float2 s1 = vfma(e, u2, vmul(Th, u2));
    a00 = vadd(a00, vfma(Th, Th, s1));
    c1 = vmul(vadd(half, vfma(vb(-0.25f), u2, vneg(Th))), Th);
    g0c = vadd(half, vfma(vb(-1.5f), Th, vmul(vb(-0.25f), u2)));
  }
  const float2 b0 = vfma(vb(float(-0.5 * (D + 2))), Th, vfma(vb(-0.5f), u2, vb(1.f)));
  const float2 base = vsub(vmul(vmul(om, drho), sc), rkgu);
  const float2 rom_lo = vmul(vfma(rho, om, vneg(rom0)), sc);
  const float2 P4 = L::NEQ >= 4 ? vmul(rom, vb(float(1.0 / 24.0))) : vb(0.f);
  const float2 Q3 = vmul(rom, vb(float(1.0 / 6.0)));
  const float2 q1 = FO >= 2 ? vneg(rkgu) : vb(0.f);
  float2 P0, P2, Q1, A1;
  static_for<0, NP + 1>([&](auto K) {
    constexpr int ip = K == 0 ? 0 : 2 * K - 1;
    constexpr int sh = L::SH(ip);
    if constexpr (K == 0 || (K >= 2 && L::SH(ip) != L::SH(ip - 2)) || K == 1) {
      constexpr F2 X2f = f2_of(L::c2 * double(L::E2(sh)));
      const float2 tx = vmul(vb(X2f.hi), Th);
      float2 A0, A2;
      if constexpr (L::NEQ >= 4) {
        A0 = vfma(vmul(vb(0.125f), tx), tx, vfma(vb(X2f.hi), c1, a00));
        A2 = vfma(vb(0.25f), tx, g0c);
      } else {
        A0 = vfma(half, tx, a00);
        A2 = g0c;
      }
      A1 = vfma(half, tx, b0);
      P0 = vfma(rom, A0, vfma(rom_lo, A0, base));
      P2 = vfma(rom, A2, vmul(rom_lo, A2));
      Q1 = vfma(rom, A1, vfma(rom_lo, A1, q1));
    }
    if constexpr (K == 0) {
      out(ic<0>{}, vfma(h2f(h[0]), om1, P0));
    } else {
      constexpr int im = ip + 1;
      const float2 t = vedot<L, ip>(cu), sp = vedot<L, ip>(cs);
      const float2 t2 = vmul(t, t);
      float2 ev = vfma(t2, L::NEQ >= 4 ? vfma(t2, P4, P2) : P2, P0);
      const float2 oq = vfma(t2, Q3, Q1);
      float2 od;
      if constexpr (FO >= 1) ev = vfma(sp, t, ev);
      if constexpr (FO >= 2) od = vfma(sp, vfma(half, t2, A1), vmul(t, oq));
      else if constexpr (FO == 0 && L::D == 3 && L::E(ip, 0) == 3) od = vfma(vb(3.f), cs[0], vmul(t, oq));  // 3 cs fused
      else od = vfma(t, oq, sp);
      const float2 fp = h2f(h[ip]), fm = h2f(h[im]);
      ev = vfma(vadd(fp, fm), hom1, ev);
      od = vfma(vsub(fp, fm), hom1, od);
      out(ic<ip>{}, vadd(ev, od));
      out(ic<im>{}, vsub(ev, od));
    }
  });
}

// Resident 128-thread blocks per SM the register cap is sized for: 4 (128
// registers, 72 B of spill on D3Q39).  512 x 512 x 256 sites: 2.19 ms a step;
// 5 blocks 2.64 (296 B of spill), 3 blocks 2.43, and converting the halves a
// second time for the update, to hold fewer registers, 2.33 with 4 and 2.30
// with 5 blocks: the conversions are on the FMA pipe.
#ifndef LBM_HALF2_BLOCKS
#define LBM_HALF2_BLOCKS 4
#endif

// Whether the six rows at the ends of n layers of the wall axis take two block
// indices each, one per half of the block's sites, since they go site by site
// (and they come first, see wall_rows_first): with walls, while a launch can
// have that many rows.
__host__ __device__ constexpr bool half2_twice(int n, bool walls) { return walls && n >= 6 && n + 6 <= MAX_GRID_YZ; }
// Rows of a launch.
inline int half2_rows(int n, bool walls) { return half2_twice(n, walls) ? n + 6 : n; }

// Whether the plain step of an FP16 grid runs two sites per thread.  Needs an
// even nx (rows then start on a word).  Measured on GB300, microseconds a step
// (one site per thread -> two): 512 x 512 x 256 2860 -> 2178, 256^2 x 128 380 ->
// 299, 1024 x 512 18.7 -> 15.1, 4096 x 2048 311 -> 244, 512 x 192 5.6 -> 5.4, 256 x 256
// 4.49 -> 4.45 (eight at once 2.25 -> 1.84 each), 64^3 11.3 -> 7.3, 64 x 32 x 16 3.70 -> 3.67
// (1.33 -> 0.95).  Not taken where a warp of pairs is poorly filled, so
// that a row needs nearly as many warps as of single sites (96^3, 3 against 2 a
// row: 33.7 -> 34.5; 130 columns, 5 against 3: 32.8 -> 28.0), nor on grids so
// small that a thread's own latency counts, alone (512 x 96 4.0 -> 4.4, 256 x 192 3.95 -> 4.4,
// 128 x 128 3.1 -> 3.45, 64 x 16 x 16 3.25 -> 3.5) or with walls (256 x 192 6.1 -> 6.5).
template <int D>
inline bool half2_serves(const StepParams& p) {
  const int single = (p.nx + 31) / 32, pairs = (p.nx + 63) / 64;
  return p.nx % 2 == 0 && 5 * single >= 8 * pairs && p.N >= (D == 2 ? 65536 : 32768);
}

// Threads per block: the caller's choice up to 128, the warps that a row has
// pairs for shared evenly between its blocks (320 columns: two blocks of 96).
inline int half2_block(int nx, int bx) {
  const int warps = ((nx + 1) / 2 + 31) / 32, most = (bx < 128 ? bx : 128) / 32;
  const int blocks = (warps + most - 1) / most;
  return (warps + blocks - 1) / blocks * 32;
}

template <class L, int FO>
__global__ void __launch_bounds__(128, LBM_HALF2_BLOCKS)
    k_step_half2(const __half* __restrict__ fin, __half* __restrict__ fout, const StepParams p) {
  constexpr int D = L::D, Q = L::Q;
  const int bx = blockDim.x;
  const bool twice = half2_twice(p.na, p.wall != W_NONE);
  const int b = D == 2 ? blockIdx.y : blockIdx.z;
  const int k0 = twice && b < 12 ? b & 1 : 0, k1 = twice && b < 12 ? k0 + 1 : 2;
  const int a = p.a0 + (twice ? wall_rows_first(b < 12 ? b >> 1 : b - 6, p.na, true) : b);
  const int y = D == 2 ? a : (int)blockIdx.y;
  const int z = D == 3 ? a : 0;
  const size_t N = (size_t)p.N;
  const int row = (z * p.ny + y) * p.nx;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (near_wall(p, a, D == 2 ? p.ny : p.nz)) {  // block-uniform: a row of the wall rules, site by site
    fin = wait_previous(fin);
#pragma unroll 1
    for (int k = k0; k < k1; ++k) {
      const int x = (2 * blockIdx.x + k) * bx + threadIdx.x;
      if (x >= p.nx) break;
      float g[3], d[Q];
      site_force_r<D, float>(p, x, y, z, row + x, g);
      pull<L, P_FP16S, float, LD_PLAIN, true>(fin, p, x, y, z, d);
      collide_store<L, P_FP16S, FO, true>(d, g, row + x, fout, p);
    }
    return;
  }
  if (k0 == 1) return;  // a slab's end row that is no wall: whole in the first of its two blocks
  const int x = 2 * (blockIdx.x * bx + threadIdx.x);
  if (x >= p.nx) return;
  float2 g[3];
  if (p.gkind == G_UNIFORM) {
    for (int c = 0; c < 3; ++c) g[c] = vb(p.g0_f[c]);
  } else {
    float ga[3], gb[3];
    site_force_r<D, float>(p, x, y, z, row + x, ga);
    site_force_r<D, float>(p, x + 1, y, z, row + x + 1, gb);
    for (int c = 0; c < 3; ++c) g[c] = make_float2(ga[c], gb[c]);
  }
  fin = wait_previous(fin);
  // Byte offsets of x - 3 .. x + 4 in a row, wrapped: the address of a load is
  // then a block-uniform row pointer plus one of them.
  unsigned xs[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) xs[k] = 2u * (unsigned)wrap3(x + k - 3, p.nx);
  int ys[7], zs[7];
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    ys[k] = wrap3(y - (k - 3), p.ny) * p.nx;
    zs[k] = D == 3 ? wrap3(z - (k - 3), p.nz) * p.nx * p.ny : 0;
  }
  unsigned h[Q];
  static_for<0, Q>([&](auto I) {
    constexpr int i = I, ex = L::E(i, 0), k = 3 - ex;
    const char* src = reinterpret_cast<const char*>(fin + (i * N + (size_t)(zs[L::E(i, 2) + 3] + ys[L::E(i, 1) + 3])));
    if constexpr (ex % 2 == 0) {  // x and nx even: the two sources are one aligned word
      h[i] = *reinterpret_cast<const unsigned*>(src + xs[k]);
    } else {
      const unsigned lo = *reinterpret_cast<const unsigned short*>(src + xs[k]);
      const unsigned hi = *reinterpret_cast<const unsigned short*>(src + xs[k + 1]);
      h[i] = lo | hi << 16;
    }
  });
  __half* __restrict__ fo = fout + (row + x);
  collide2<L, FO>(h, g, p, [&](auto I, float2 v) {
    constexpr int i = I;
    *reinterpret_cast<__half2*>(fo + i * N) = __float22half2_rn(v);
  });
}

}  // namespace lbm
