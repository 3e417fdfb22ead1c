// D3Q19 fused step of the self-tuning-EOS multiphase lattice Boltzmann model
// (Huang, Wu & Adams, arXiv:1809.02390, extended to three dimensions): lattice
// constants, collision constants, the node collision and the z-marching step
// kernel.  Included by lbm3d.cu (one translation unit).
//
// One launch per time step: each block owns a 32 x 8 column of the x-y plane and
// marches through a chunk of z-planes.  The populations that a plane's nodes and
// their one-node ring pull (pull streaming, supplement Eq. 2) arrive in shared
// memory by asynchronous copies, two planes ahead; each thread turns its nodes'
// 19 into the rest population and the nine opposite pairs' sums and differences,
// keeps those in registers and puts the density into a three-plane ring buffer; the
// collision of plane z runs once the density of plane z + 1 is there, so the force
// stencil (Eq. 12) of every node reads its 18 neighbours' densities from shared
// memory.  Each population crosses DRAM once per step in each direction.
#pragma once

#include <cuda_runtime.h>

#include "lbm.h"
#include "lbm_tma.cuh"

namespace {

constexpr int Q = 19;
// Plane order: rest, +x -x, +y -y, +z -z, then six opposite pairs of edge
// velocities; plane 2P + 1 is the + member of pair P (P = 0..8) and 2P + 2 its
// opposite.  Pair directions: x, y, z, (1,1,0), (1,-1,0), (1,0,1), (1,0,-1),
// (0,1,1), (0,1,-1).
constexpr int kEX[Q] = {0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0};
constexpr int kEY[Q] = {0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1};
constexpr int kEZ[Q] = {0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1};
// The same velocities for the moments kernel.
__constant__ int cEX[Q] = {0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0};
__constant__ int cEY[Q] = {0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1};
__constant__ int cEZ[Q] = {0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1};

constexpr int TX = 32, TY = 8;  // tile of a block in x and y
constexpr int HX = TX + 2, HY = TY + 2;
constexpr int kRing = 2 * HX + 2 * TY;  // ring slots of one density plane (84)
constexpr double kSEps3 = 1.75;

// Collision constants of the initial state and of k_d3_pull (host: make_c3).
template <typename T>
struct C3 {
  int eos;
  T rho_ref, G2, lam_RT, lam_a, b, bq;
  T se, seps, sq, sp, sm, spi;
  T k_seps_ome;  // k s_eps (s_e/2 - 1): entry (e, eps) of S
  T h_sq_ome;    // h s_q (s_e/2 - 1): entry (e, q_a) of S divided by u_a
  T b_sq_omp;    // b s_q (s_p/2 - 1): scale of the (second order, q) entries of S
  T beta2;
};

// p_EOS / c^2 (times K_EOS / c^2): vdW rho R T/(1 - b rho) - a rho^2, or
// Carnahan-Starling (Eq. 20) with t = b rho / 4.
template <typename T>
__device__ __forceinline__ T p_eos(const C3<T>& c, T rho) {
  if (c.eos == LB_EOS_VDW) return c.lam_RT * rho / (T(1) - c.b * rho) - c.lam_a * rho * rho;
  const T t = c.bq * rho;
  const T om = T(1) - t;
  const T z = (T(1) + t * (T(1) + t * (T(1) - t))) / (om * om * om);
  return c.lam_RT * rho * z - c.lam_a * rho * rho;
}

// Velocity components of plane i (folded to constants in unrolled loops).
__host__ __device__ constexpr int ex3(int i) {
  return i == 1 || i == 7 || i == 9 || i == 11 || i == 13 ? 1 : (i == 2 || i == 8 || i == 10 || i == 12 || i == 14 ? -1 : 0);
}
__host__ __device__ constexpr int ey3(int i) {
  return i == 3 || i == 7 || i == 10 || i == 15 || i == 17 ? 1
                                                           : (i == 4 || i == 8 || i == 9 || i == 16 || i == 18 ? -1 : 0);
}
__host__ __device__ constexpr int ez3(int i) {
  return i == 5 || i == 11 || i == 14 || i == 15 || i == 18 ? 1
                                                            : (i == 6 || i == 12 || i == 13 || i == 16 || i == 17 ? -1 : 0);
}
constexpr bool same_velocities() {
  for (int i = 0; i < Q; ++i)
    if (ex3(i) != kEX[i] || ey3(i) != kEY[i] || ez3(i) != kEZ[i]) return false;
  return true;
}
static_assert(same_velocities(), "ex3, ey3, ez3 are kEX, kEY, kEZ");

// Value types of the step: r64 (one FP64 node) and f2 (two FP32 nodes per packed
// instruction); both round every operation as written.
using lbm::f2;
using lbm::fmav;
using lbm::r64;

__device__ __forceinline__ f2 operator-(f2 a) { return f2{make_float2(-a.v.x, -a.v.y)}; }

template <typename V>
struct Val;
template <>
struct Val<f2> {
  using real = float;
  static constexpr int lanes = 2;
  __device__ static f2 pack(const float (&a)[2]) { return f2{make_float2(a[0], a[1])}; }
  __device__ static float get(f2 v, int k) { return k ? v.v.y : v.v.x; }
  // Reciprocal: the hardware's approximation (1 ulp) and one Newton step r (2 - x r).
  __device__ static f2 rcp(f2 x) {
    const f2 r = lbm::rcp(x);
    const f2 one{make_float2(1.f, 1.f)};
    return fmav(r, fmav(-x, r, one), r);
  }
  static f2 make(double v) { return f2{make_float2(float(v), float(v))}; }
  static f2 low(double v) { return make(v - double(float(v))); }  // what make leaves of v
};
template <>
struct Val<r64> {
  using real = double;
  static constexpr int lanes = 1;
  __device__ static r64 pack(const double (&a)[1]) { return r64{a[0]}; }
  __device__ static double get(r64 v, int) { return v.v; }
  __device__ static r64 rcp(r64 x) { return r64{lbm::rcp_fp64(x.v)}; }
  static r64 make(double v) { return r64{v}; }
  static r64 low(double) { return r64{0.0}; }
};
template <typename T>
struct ValOf;
template <>
struct ValOf<float> {
  using V = f2;
};
template <>
struct ValOf<double> {
  using V = r64;
};

// Collision constants (host: make_cv3).  The stencil sums arrive as 12 s.
template <typename V>
struct CV3 {
  int eos;
  V rho_ref, nbq;                // rho_ref; -b (vdW) or -b / 4 (Carnahan-Starling)
  V lam_RT3, cA;                 // 3 lam R T, 3 G2 / 2 - 3 lam a
  V G2s, gq;                     // G2 / 12, G2 / 1728
  V lam_RT3_lo, cA_lo, G2s_lo;   // FP32: what the rounded constants leave
  V se, kse, hq;                 // s_e, k s_eps om_e / 19, h s_q om_e 5 / 57 (om_e = s_e / 2 - 1)
  V ceta, seps_a;                // -(beta_2 + 11 / 2), 2 s_eps / 21
  V sp3, spi3, bq2, bq23, nbq23;  // s_p / 3, s_pi / 3, 10 bq / 3, 10 bq / 9, its negative (bq = b s_q om_p)
  V nsp, nbq5;                   // -s_p, -5 bq / 3
  V sq6, om8;                    // s_q / 6, (1 - s_m) / 8
  V one, two, three, half, quarter, nquarter, eighth, n2, n3, n4, nhalf;
  V nthird, sixth, n12, i24, n2h, n5h, n10h, c1375, c1121;
};

// Post-collision populations of one node (two for V = f2) from the rest population f0,
// the pairs' sums s and differences d (plane 2P + 1 plus / minus plane 2P + 2), the
// density deviation delta = rho - rho_ref and 12 times the force stencil.  All are
// deviations from w_i rho_ref.  The collision is mbar = m + F_m - S (m - m_eq + F_m / 2
// - Q_m) with the 3-D S.  Its even part is worked in the variables
//   a = sum of the axis pairs, T = sum_i |c_i|^2 f_i, Xa = 3 s_0 - a, Xe, Wa, We (the
//   axis and edge parts of 3p_xx and p_ww), p_xy, p_xz, p_yz,
// in which the inverse transform is a few additions, and its odd part in d_a, j_a, m_a.
// With k = J - F (J = rho u): m - m_eq + F_m / 2 is T - delta - eta - k.u (row e),
// p - (k u) for the second-order rows, and (5 / 3)(j - 3 d) for q.  About 290 operations
// a node against 364 when every moment was formed (FP64 instructions, measured).
template <typename V>
__device__ __forceinline__ void collide3(const CV3<V>& c, V f0, const V (&s)[9], const V (&d)[9], V delta, V sx, V sy,
                                         V sz, V (&o)[Q]) {
  const V a = s[0] + (s[1] + s[2]);
  const V E12 = s[3] + s[4], E13 = s[5] + s[6], E23 = s[7] + s[8];
  const V Ed = E12 + E13 + E23;
  const V Tr = fmav(c.two, Ed, a);
  const V Xa = fmav(c.three, s[0], -a), Xe = fmav(c.n3, E23, Ed);
  const V Wa = s[1] - s[2], We = E12 - E13;
  const V pxy = s[3] - s[4], pxz = s[5] - s[6], pyz = s[7] - s[8];
  const V D12p = d[3] + d[4], D12m = d[3] - d[4], D13p = d[5] + d[6], D13m = d[5] - d[6];
  const V D23p = d[7] + d[8], D23m = d[7] - d[8];
  const V jx = d[0] + (D12p + D13p), jy = d[1] + (D12m + D23p), jz = d[2] + (D13m + D23m);

  // EOS: p_LBE = p_EOS + G^2 rho^2 / 2 (Eq. 18), eta = 3 p_LBE - rho (Eq. 9).
  const V rho = delta + c.rho_ref;
  V ir, p3;  // 1 / rho, 3 p_LBE
  // 3 p_LBE / rho = lam_RT3 z + cA rho, z the EOS's factor.  The two terms nearly cancel, and
  // the force must cancel the G^2 part of cA exactly in a flat interface, so in FP32 the
  // rounding of the three constants is the largest error of the step (two-phase 24^3 lattices,
  // 135 steps at T_r 0.857: 4.6e-7 to 6.8e-7 off 64 bits, 1.6e-7 to 2.0e-7 with the constants in
  // two floats; collide3_moments 3.9e-7 to 5.5e-7).
  constexpr bool kTwoFloats = Val<V>::lanes == 2;
  auto slope = [&](V z) { return fmav(c.cA, rho, fmav(c.lam_RT3, z, fmav(c.lam_RT3_lo, z, c.cA_lo * rho))); };
  if (c.eos == LB_EOS_VDW) {
    const V om = fmav(c.nbq, rho, c.one);
    const V r = Val<V>::rcp(rho * om);
    ir = r * om;
    if constexpr (kTwoFloats)
      p3 = rho * slope(r * rho);
    else
      p3 = rho * fmav(c.cA, rho, c.lam_RT3 * (r * rho));
  } else {
    const V om = fmav(c.nbq, rho, c.one), t = c.one - om;
    const V r = Val<V>::rcp(rho * om);
    const V io = r * rho;
    ir = r * om;
    const V z = fmav(t * t, om, c.one + t) * (io * io * io);  // (1 + t + t^2 - t^3) / (1 - t)^3
    if constexpr (kTwoFloats)
      p3 = rho * slope(z);
    else
      p3 = rho * fmav(c.lam_RT3, z, c.cA * rho);
  }
  const V eta = p3 - rho;

  // Force (Eq. 12), velocity (Eq. 5) and their products.
  V G2r;
  if constexpr (kTwoFloats)
    G2r = fmav(c.G2s, rho, c.G2s_lo * rho);
  else
    G2r = c.G2s * rho;
  const V Fx = G2r * sx, Fy = G2r * sy, Fz = G2r * sz;
  const V Jx = fmav(c.half, Fx, jx), Jy = fmav(c.half, Fy, jy), Jz = fmav(c.half, Fz, jz);
  const V ux = Jx * ir, uy = Jy * ir, uz = Jz * ir;
  const V X = (Jx - Fx) * ux, Y = (Jy - Fy) * uy, Z = (Jz - Fz) * uz;
  const V W = X + (Y + Z);
  const V FX = Fx * ux, FY = Fy * uy, FZ = Fz * uz;
  const V Fu = FX + (FY + FZ);
  const V FDxx = fmav(c.three, FX, -Fu), FDww = FY - FZ;
  // Q_m (Eq. 14 in 3-D, F~ = G s) joins the second-order equilibria: X' = k_x u_x + G^2 s_x^2 / 12.
  const V gx = c.gq * sx, gy = c.gq * sy, gz = c.gq * sz;
  const V X1 = fmav(gx, sx, X), Y1 = fmav(gy, sy, Y), Z1 = fmav(gz, sz, Z);
  const V W1 = X1 + (Y1 + Z1);
  const V dW = W1 - W;  // G^2 s.s / 12

  // q rows: G_q = (5 / 3) g.
  const V hx = fmav(c.n3, d[0], jx), hy = fmav(c.n3, d[1], jy), hz = fmav(c.n3, d[2], jz);
  const V bX = ux * hx, bY = uy * hy, bZ = uz * hz;
  const V uG = bX + (bY + bZ);
  // e and eps rows.
  const V gE = (Tr + c.rho_ref) - (p3 + W);  // T - delta - eta - k.u, delta + eta = 3 p_LBE - rho_ref
  V ge = fmav(c.n5h, gE, c.ceta * eta);
  ge = fmav(c.n10h, fmav(c.nthird, delta, a), ge);
  ge = fmav(c.c1375, dW, ge);
  const V R = fmav(c.se, fmav(c.n2h, dW, gE), fmav(c.kse, ge, c.hq * uG));
  const V Ts = fmav(c.two, Fu, Tr) - R;
  const V as = fmav(c.seps_a, ge, fmav(c.c1121, R, a));
  // 3p_xx, 3pi_xx, p_ww, pi_ww rows.
  const V Hxx = fmav(c.three, X1, -W1), Hww = Y1 - Z1;
  const V Ax = fmav(c.sp3, (Xa + Xe) - Hxx, fmav(c.bq2, bX, c.nbq23 * uG));
  const V Ix = c.spi3 * fmav(c.half, Hxx, fmav(c.n2, Xa, Xe));
  const V Xas = (Xa + FDxx) - (Ax - Ix), Xes = (Xe + FDxx) - (Ax + Ax + Ix);
  const V Aw = fmav(c.sp3, (Wa + We) - Hww, c.bq23 * (bY - bZ));
  const V Iw = c.spi3 * fmav(c.half, Hww, fmav(c.n2, Wa, We));
  const V Was = (Wa + FDww) - (Aw - Iw), Wes = (We + FDww) - (Aw + Aw + Iw);
  // Off-diagonal rows.
  auto off = [&](V p, V F1, V F2, V J1, V u1, V u2, V g1, V s2, V h1, V h2) {
    const V Fc = fmav(F1, u2, F2 * u1);
    const V H = fmav(g1, s2, fmav(c.nhalf, Fc, J1 * u2));
    return fmav(c.nbq5, fmav(u2, h1, u1 * h2), fmav(c.nsp, p - H, p + Fc));
  };
  const V xy = off(pxy, Fx, Fy, Jx, ux, uy, gx, sy, hx, hy);
  const V xz = off(pxz, Fx, Fz, Jx, ux, uz, gx, sz, hx, hz);
  const V yz = off(pyz, Fy, Fz, Jy, uy, uz, gy, sz, hy, hz);
  // Odd part: half differences of the axis pairs, and J of the edges from momentum
  // conservation (2 od + 8 J = j + F).
  const V ox = fmav(c.sq6, hx, fmav(c.sixth, Fx, c.half * d[0]));
  const V oy = fmav(c.sq6, hy, fmav(c.sixth, Fy, c.half * d[1]));
  const V oz = fmav(c.sq6, hz, fmav(c.sixth, Fz, c.half * d[2]));
  const V JX = fmav(c.nquarter, ox, c.eighth * (jx + Fx));
  const V JY = fmav(c.nquarter, oy, c.eighth * (jy + Fy));
  const V JZ = fmav(c.nquarter, oz, c.eighth * (jz + Fz));
  const V mx = c.om8 * (D12p - D13p), my = c.om8 * (D23p - D12m), mz = c.om8 * (D13m - D23m);

  // Inverse transform.
  const V a6 = c.sixth * as;
  const V ev0 = fmav(c.sixth, Xas, a6), et = fmav(c.n12, Xas, a6);
  const V ev1 = fmav(c.quarter, Was, et), ev2 = fmav(c.nquarter, Was, et);
  o[1] = ev0 + ox, o[2] = ev0 - ox;
  o[3] = ev1 + oy, o[4] = ev1 - oy;
  o[5] = ev2 + oz, o[6] = ev2 - oz;
  const V ce = c.i24 * (Ts - as);
  const V cx = fmav(c.i24, Xes, ce), eyz = fmav(c.n12, Xes, ce);
  const V w8 = c.eighth * Wes;
  const V exy = cx + w8, exz = cx - w8;
  auto edge = [&](V e, V p, V odp, V odm, V& o1, V& o2, V& o3, V& o4) {
    const V ep = fmav(c.quarter, p, e), em = fmav(c.nquarter, p, e);
    o1 = ep + odp, o2 = ep - odp;
    o3 = em + odm, o4 = em - odm;
  };
  edge(exy, xy, (JX + JY) + (mx - my), (JX - JY) + (mx + my), o[7], o[8], o[9], o[10]);
  edge(exz, xz, (JX + JZ) - (mx - mz), (JX - JZ) - (mx + mz), o[11], o[12], o[13], o[14]);
  edge(eyz, yz, (JY + JZ) + (my - mz), (JY - JZ) + (my + mz), o[15], o[16], o[17], o[18]);
  // o[0] takes what the others leave of the mass.  FP32: of the populations as they are
  // stored, one pair after the other.  Taking their even parts before the last rounding
  // (e + p + od) instead leaves that rounding out, which in quiet liquid and gas is the
  // same every step: 2e-9 of the mass lost a step, 1.3e-6 off 64 bits after 400 steps of
  // two-phase 24^3 lattices, against 2e-11 and 4e-7 with the stored ones (collide3_moments:
  // 2e-10 and 6e-7); summing the 18 first and taking them off at once leaves 1e-10 a step.
  // FP64 has no such drift to speak of (1e-18 a step) and its pipe no room for 14
  // instructions more.
  if constexpr (kTwoFloats) {
    V t = delta;
#pragma unroll
    for (int P = 0; P < 9; ++P) t = t - (o[2 * P + 1] + o[2 * P + 2]);
    o[0] = t;
  } else {
    o[0] = fmav(c.n4, fmav(c.two, cx, eyz), fmav(c.n2, fmav(c.two, et, ev0), delta));
  }
}

// 12 times the force stencil sum_i omega_i rho(x + e_i) e_i (Eq. 12) from the density
// planes of z - 1 (slot a), z (b) and z + 1 (e); at(slot, dy, dx): density of a neighbour.
template <typename V, typename At>
__device__ __forceinline__ void stencil3(const CV3<V>& c, const At& at, int a, int b, int e, V& sx, V& sy, V& sz) {
  const V u1 = at(b, 1, 1) - at(b, -1, -1), v1 = at(b, -1, 1) - at(b, 1, -1);
  const V u2 = at(e, 0, 1) - at(a, 0, -1), v2 = at(a, 0, 1) - at(e, 0, -1);
  const V u3 = at(e, 1, 0) - at(a, -1, 0), v3 = at(a, 1, 0) - at(e, -1, 0);
  sx = fmav(c.two, at(b, 0, 1) - at(b, 0, -1), (u1 + v1) + (u2 + v2));
  sy = fmav(c.two, at(b, 1, 0) - at(b, -1, 0), (u1 - v1) + (u3 + v3));
  sz = fmav(c.two, at(e, 0, 0) - at(a, 0, 0), (u2 - v2) + (u3 - v3));
}

// Window of one plane of a tile of tw x th nodes: for population i the cells that the
// pulls of the tile and of its ring read, th + 2 rows (window row r holds lattice row
// y0 - 1 - e_iy + r) of tw columns and a 16-byte run at each side (window column q =
// lattice column x0 - XO + q).  FP32 tiles are 32 x 8; FP64 tiles are chosen to fill the
// SMs (tile_plan), up to the sizes below.
template <typename T>
struct Win3 {
  static constexpr int run = 16 / int(sizeof(T));  // elements of a 16-byte run
  static constexpr int xo = run;
  static constexpr bool tensor = sizeof(T) == 4;    // tensor copies (FP32)
  static constexpr bool fixed = sizeof(T) == 4;     // 32 x 8 tiles
  static constexpr int cols = TX + 2 * run, rows = HY;
  static constexpr int cells = fixed ? cols * rows : 416;   // at most, of a window
  static constexpr int ring_cells = fixed ? HX * HY : 400;  // at most, of a density plane
  static constexpr int plane = (cells * int(sizeof(T)) + 127) / 128 * 128 / int(sizeof(T));
  static constexpr int threads = TX * TY / Val<typename ValOf<T>::V>::lanes;
  static constexpr int stages = 2;
  static constexpr unsigned smem = unsigned(stages) * Q * plane * sizeof(T) + 128;
  static_assert(rows * cols / run <= threads && kRing <= threads, "one thread per run and per ring slot");
};
static_assert(Win3<float>::plane * 4 % 128 == 0, "a tensor copy's destination is on a 128-byte boundary");

__device__ __forceinline__ int wrap(int a, int n) {
  a %= n;
  return a < 0 ? a + n : a;
}

// Resident blocks per SM: two for FP32 (128 threads of two nodes, up to 255 registers:
// at three blocks the 168 registers spill and the step is 10% slower), one for FP64
// (256 threads; its pipe is busy with two warps per scheduler).
template <typename T>
constexpr int d3_blocks() {
  return sizeof(T) == 8 ? 1 : 2;
}

__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, int x, int y, int z, int w,
                                            unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
      ::"r"(lbm::smem_addr(dst)), "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(z), "r"(w),
      "r"(lbm::smem_addr(bar))
      : "memory");
}

// Whether the windows of the tile at (x0, y0) arrive by tensor copies: nineteen a plane
// (box 40 x 10 of the map (x, y, z, plane)), issued by thread 0 and completing on the
// stage's mbarrier.  Tiles at the lattice's edge in x or y take 16-byte copies by every
// thread instead, periodic in every coordinate: the wrapped part as boxes of one 16-byte
// run was much slower (a 64^3 step, all edge tiles in x, 21 us against 13), and nineteen
// issuing lanes in place of one thread cost 7%.
template <typename T>
__host__ __device__ __forceinline__ bool tensor_tile(int x0, int y0, int nx, int ny) {
  using W = Win3<T>;
  return x0 >= W::xo && x0 + TX + W::run <= nx && y0 >= 2 && y0 + TY + 2 <= ny;
}

// The fused step.  Grid (ceil(nx/tw), ceil(ny/th), ceil(nz/tz)); each block marches a
// chunk of tz planes (tile_plan picks the three).  VEC: rows of a multiple of 16 bytes; FP32
// steps then have maps.  err is set by a bounded wait that gave up.
// have_map: the map is that of fin (else every tile is filled by runs).
// Iteration p: the window of plane p has arrived; its densities are formed and its
// populations kept; its buffer is handed to plane p + 2 (plane p + 1 is in flight); plane
// p - 1, kept from the iteration before, is collided.  Threads of ragged tiles that lie
// outside the lattice fill their density slot with the wrapped node's and store nothing.
//
// FP32 256^3: 529 us a step with the populations pulled into registers (k_d3_pull), 461 to
// 469 here.  What bounds it: the traffic between L2 and the SMs, 1.56 times the
// algorithmic reads because of the windows' halo.  Steps that moved the same windows and
// skipped the collision ran at 34.8 GLUPS with 16-byte copies by the threads whatever the
// number of blocks and stages, at 38.6 without the halo, and at 39.1 with tensor copies.
template <typename T, bool VEC>
__global__ void __launch_bounds__(Win3<T>::threads, d3_blocks<T>())
    k_d3_step(const T* fin, T* __restrict__ fout, int nx, int ny, int nz, int tw_, int th_, int tz,
              const CV3<typename ValOf<T>::V> c, const __grid_constant__ CUtensorMap map, int have_map, int* __restrict__ err) {
  using V = typename ValOf<T>::V;
  using W = Win3<T>;
  constexpr int L = Val<V>::lanes;
  constexpr bool kTensor = W::tensor && VEC;
  lbm::follow_predecessor();
  extern __shared__ __align__(128) unsigned char dyn[];
  T* win = reinterpret_cast<T*>((reinterpret_cast<uintptr_t>(dyn) + 127) & ~uintptr_t(127));
  __shared__ T rho[3][W::ring_cells];
  __shared__ __align__(8) unsigned long long bar[W::stages];
  __shared__ int gave_up;
  const int tw = W::fixed ? TX : tw_, th = W::fixed ? TY : th_;
  const int hx = tw + 2, cols = tw + 2 * W::run, runs = cols / W::run;  // pitches of a density plane and a window
  const int tid = threadIdx.x, tx = tid % tw, ty = tid / tw;
  const bool node = W::fixed || tid < tw * th;
  const int x0 = blockIdx.x * tw, y0 = blockIdx.y * th, z0 = blockIdx.z * tz;
  const int z1 = min(z0 + tz, nz);
  const size_t N = size_t(nx) * ny * nz;
  const bool tensor = kTensor && have_map && tensor_tile<T>(x0, y0, nx, ny);
  if constexpr (kTensor) {
    if (tid == 0) {
      gave_up = 0;
      for (int g = 0; g < W::stages; ++g) lbm::mbar_init(&bar[g], 1);
    }
    __syncthreads();
  }

  // Runs: thread j fills run j mod runs of window row j / runs, all planes.
  const int cr = tid / runs, cq = (tid - cr * runs) * W::run;
  const bool copier = tid < (th + 2) * runs;
  int row[3], col[VEC ? 1 : W::run];
#pragma unroll
  for (int e = 0; e < 3; ++e) row[e] = wrap(y0 - e + cr, ny) * nx;  // e_iy + 1
#pragma unroll
  for (int q = 0; q < (VEC ? 1 : W::run); ++q) col[q] = wrap(x0 - W::xo + cq + q, nx);
  auto issue = [&](int zraw, int buf) {
    const int z = zraw < 0 ? zraw + nz : (zraw >= nz ? zraw - nz : zraw);
    const int zd = z == 0 ? nz - 1 : z - 1, zu = z == nz - 1 ? 0 : z + 1;
    T* stage = win + buf * Q * W::plane;
    if constexpr (kTensor) {
      if (tensor) {
        if (tid == 0 && zraw <= z1) {
          lbm::fence_proxy_async();
          lbm::mbar_expect_tx(&bar[buf], unsigned(Q * W::rows * W::cols * sizeof(T)));
#pragma unroll
          for (int i = 0; i < Q; ++i)
            tma_load_4d(stage + i * W::plane, &map, x0 - W::xo, y0 - 1 - ey3(i),
                        ez3(i) == 0 ? z : (ez3(i) > 0 ? zd : zu), i, &bar[buf]);
        }
        return;
      }
    }
    if (copier && zraw <= z1) {
      int zo[3];  // e_iz + 1: plane z - e_iz
      zo[0] = zu * ny * nx;
      zo[1] = z * ny * nx;
      zo[2] = zd * ny * nx;
      T* dst = stage + (cr * cols + cq);
      const T* base = fin;
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const T* src = base + (zo[ez3(i) + 1] + row[ey3(i) + 1]);
        if constexpr (VEC) {
          lbm::cp_async16(dst + i * W::plane, src + col[0]);
        } else {
#pragma unroll
          for (int q = 0; q < W::run; ++q) lbm::cp_async_elem(dst + i * W::plane + q, src + col[q]);
        }
        base += N;
      }
    }
    lbm::cp_async_commit();
  };

  // Nodes of this thread: (tx, ty) and, for FP32, (tx, ty + 4).
  const int x = x0 + tx;
  constexpr int kStep = TY / L;
  // Ring slot of this thread: lower row, upper row, left and right columns.
  const bool ring = tid < 2 * hx + 2 * th;
  int hsx = 0, hsy = 0;
  if (tid < hx) {
    hsx = tid;
  } else if (tid < 2 * hx) {
    hsx = tid - hx;
    hsy = th + 1;
  } else if (ring) {
    const int r = tid - 2 * hx;
    hsx = r < th ? 0 : tw + 1;
    hsy = 1 + (r < th ? r : r - th);
  }
  // This thread's cells: of its first node in a window and in a density plane, of its ring slot.
  const int own = (ty + 1) * cols + tx + W::xo, own_rho = (ty + 1) * hx + tx + 1;
  const int ring_own = hsy * cols + hsx - 1 + W::xo, ring_rho = hsy * hx + hsx;
  struct Node {
    V f0, s[9], d[9];
  };
  // Populations of the plane staged in buf into n, and the densities of tile and ring
  // into slot.
  auto take = [&](int buf, int slot, Node& n) {
    const T* w = win + buf * Q * W::plane;
    auto pull = [&](int i) {
      T v[L];
#pragma unroll
      for (int k = 0; k < L; ++k) v[k] = w[i * W::plane + own + k * kStep * cols - ex3(i)];
      return Val<V>::pack(v);
    };
    if (node) {
      n.f0 = pull(0);
      V sum = n.f0;
#pragma unroll
      for (int P = 0; P < 9; ++P) {
        const V p = pull(2 * P + 1), m = pull(2 * P + 2);
        n.s[P] = p + m;
        n.d[P] = p - m;
        sum = sum + n.s[P];
      }
#pragma unroll
      for (int k = 0; k < L; ++k) rho[slot][own_rho + k * kStep * hx] = Val<V>::get(sum, k);
    }
    if (ring) {
      const T* r = w + ring_own;
      T a = r[0];
#pragma unroll
      for (int P = 0; P < 9; ++P)
        a += r[(2 * P + 1) * W::plane - ex3(2 * P + 1)] + r[(2 * P + 2) * W::plane - ex3(2 * P + 2)];
      rho[slot][ring_rho] = a;
    }
  };
  auto collide = [&](int z, int sp, int sc, int sn, const Node& n) {
    if (!node) return;
    auto at = [&](int slot, int dy, int dx) {
      T v[L];
#pragma unroll
      for (int k = 0; k < L; ++k) v[k] = rho[slot][own_rho + k * kStep * hx + dy * hx + dx];
      return Val<V>::pack(v);
    };
    V sx, sy, sz;
    stencil3(c, at, sp, sc, sn, sx, sy, sz);
    V o[Q];
    collide3(c, n.f0, n.s, n.d, at(sc, 0, 0), sx, sy, sz, o);
#pragma unroll
    for (int k = 0; k < L; ++k) {
      const int y = y0 + ty + k * kStep;
      if (x < nx && y < ny) {
        T* p = fout + ((z * ny + y) * nx + x);
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          *p = Val<V>::get(o[i], k);
          p += N;
        }
      }
    }
  };

  // S windows in flight: group g holds plane z0 - 1 + g and lands in buffer g mod S.
  constexpr int S = W::stages;
  int buf = 0;
  unsigned phase = 0;  // bit g: parity of the next phase of bar[g]
  // Waits for the oldest window; false (for the whole block) if that gave up, with no
  // copy of this block left in flight unless its bounded waits gave up as well.  (A flag
  // in shared memory: a barrier that also reduces a predicate cost 3% of the step.)
  auto arrive = [&]() {
    if constexpr (kTensor) {
      if (tensor) {
        if (!lbm::mbar_wait(&bar[buf], phase >> buf & 1u)) gave_up = 1;
        phase ^= 1u << buf;
      }
    }
    if (!tensor) asm volatile("cp.async.wait_group %0;" ::"n"(S - 1) : "memory");
    __syncthreads();
    if constexpr (kTensor) {
      if (gave_up) {
        if (tid == 0) {
          atomicExch(err, 1);
          for (int g = 0; g < S; ++g) lbm::mbar_wait(&bar[g], (g == buf ? phase ^ (1u << buf) : phase) >> g & 1u);
        }
        __syncthreads();
        return false;
      }
    }
    return true;
  };
  auto release = [&](int zraw) {  // its buffer, for plane zraw
    __syncthreads();
    issue(zraw, buf);
    buf = buf == S - 1 ? 0 : buf + 1;
  };
  // Plane p: taken into next; the plane before it, cur, is collided (from z0 on).
  Node A, B;
  int sp = 1, sc = 2, sn = 0;
  auto plane = [&](int p, const Node& cur, Node& next) {
    if (!arrive()) return false;
    take(buf, sn, next);
    release(p + S);
    if (p > z0) collide(p - 1, sp, sc, sn, cur);
    const int t = sp;
    sp = sc;
    sc = sn;
    sn = t;
    return true;
  };
#pragma unroll 1
  for (int g = 0; g < S; ++g) issue(z0 - 1 + g, g);
#pragma unroll 1
  for (int p = z0 - 1; p <= z1; p += 2) {
    if (!plane(p, A, B)) return;
    if (p < z1 && !plane(p + 1, B, A)) return;
  }
  lbm::cp_async_wait_all();
}

// ---------------------------------------------------------------------------
// FP32 lattices whose rows are not a multiple of 16 bytes.  Filling windows element by
// element is slower than pulling the populations straight into registers (250 x 130 x 77:
// 131 us a step against 89), and so is this kernel with collide3 (104 us: its loads then
// wait).  32 x 4 tiles, one node per thread, z-marching chunks of up to 32 planes; a
// software pipeline in registers: while plane z collides, the pulls of plane z + 2 are in
// flight, plane z + 1 is summed and held, plane z is in fc (3 blocks per SM).
constexpr int kPullTY = 4, kPullTZ = 32, kPullHY = kPullTY + 2;
constexpr int kPullRing = 2 * HX + 2 * kPullTY;
static_assert(kPullRing <= TX * kPullTY, "every ring slot needs a thread of the block");

// Post-collision populations o (deviations from w_i rho_ref) of one node from
// its post-streaming deviations f, its density deviation delta = rho - rho_ref
// and the force stencil sum s = sum_i omega_i rho(x + e_i) e_i.  Moments are the
// D3Q19 polynomials (rho, e, eps, j, q, 3p_xx, 3pi_xx, p_ww, pi_ww, p_xy, p_yz,
// p_xz, m) of the pairs' even and odd parts; the collision is
// mbar = m + F_m - S (m - m_eq + F_m/2 - Q_m) with the 3-D S, and the inverse
// uses M^-1 = M^T diag(1 / |row|^2).
template <typename T>
__device__ __forceinline__ void collide3_moments(const C3<T>& c, const T* f, T delta, T sx, T sy, T sz, T* o) {
  T s[9], d[9];
#pragma unroll
  for (int P = 0; P < 9; ++P) {
    s[P] = f[2 * P + 1] + f[2 * P + 2];
    d[P] = f[2 * P + 1] - f[2 * P + 2];
  }
  const T rho = delta + c.rho_ref;
  const T A = s[0] + s[1] + s[2];
  const T Ed = (s[3] + s[4]) + (s[5] + s[6]) + (s[7] + s[8]);
  const T m_e = T(-30) * f[0] - T(11) * A + T(8) * Ed;
  const T m_eps = T(12) * f[0] - T(4) * A + Ed;
  const T jx = d[0] + ((d[3] + d[4]) + (d[5] + d[6]));
  const T jy = d[1] + ((d[3] - d[4]) + (d[7] + d[8]));
  const T jz = d[2] + ((d[5] - d[6]) + (d[7] - d[8]));
  const T qx = jx - T(5) * d[0], qy = jy - T(5) * d[1], qz = jz - T(5) * d[2];
  const T Xa = T(2) * s[0] - s[1] - s[2];
  const T Xe = (s[3] + s[4]) + (s[5] + s[6]) - T(2) * (s[7] + s[8]);
  const T pxx = Xa + Xe, pixx = Xe - T(2) * Xa;
  const T Wa = s[1] - s[2];
  const T We = (s[3] + s[4]) - (s[5] + s[6]);
  const T pww = Wa + We, piww = We - T(2) * Wa;
  const T pxy = s[3] - s[4], pxz = s[5] - s[6], pyz = s[7] - s[8];
  const T mx = (d[3] + d[4]) - (d[5] + d[6]);
  const T my = (d[4] - d[3]) + (d[7] + d[8]);
  const T mz = (d[5] - d[6]) - (d[7] - d[8]);

  // Force (Eq. 12), velocity (Eq. 5) and eta of the self-tuning EOS:
  // p_LBE = p_EOS + G^2 rho^2 / 2 (Eq. 18) = (rho + eta) / 3 (Eq. 9).
  const T Fx = c.G2 * rho * sx, Fy = c.G2 * rho * sy, Fz = c.G2 * rho * sz;
  const T irho = T(1) / rho;
  const T ux = (jx + T(0.5) * Fx) * irho, uy = (jy + T(0.5) * Fy) * irho, uz = (jz + T(0.5) * Fz) * irho;
  const T eta = T(3) * (p_eos(c, rho) + T(0.5) * c.G2 * rho * rho) - rho;
  const T rx = rho * ux, ry = rho * uy, rz = rho * uz;
  const T rhouu = rx * ux + ry * uy + rz * uz;
  const T Fu = Fx * ux + Fy * uy + Fz * uz;

  // G = m - m_eq + F_m / 2 (the shift w_i rho_ref folded into the equilibria).
  const T Ge = m_e + T(11) * delta - T(19) * eta - T(19) * rhouu + T(19) * Fu;
  const T Geps = m_eps - T(3) * delta + T(5.5) * rhouu - c.beta2 * eta - T(5.5) * Fu;
  const T two3 = T(2.0 / 3.0);
  const T Gqx = qx + two3 * jx, Gqy = qy + two3 * jy, Gqz = qz + two3 * jz;
  const T Dxx = T(2) * rx * ux - ry * uy - rz * uz;
  const T FDxx = T(2) * Fx * ux - Fy * uy - Fz * uz;
  const T Dww = ry * uy - rz * uz;
  const T FDww = Fy * uy - Fz * uz;
  const T Fxy = Fx * uy + Fy * ux, Fyz = Fy * uz + Fz * uy, Fxz = Fx * uz + Fz * ux;
  const T Gpxx = pxx - Dxx + FDxx;
  const T Gpixx = pixx + T(0.5) * (Dxx - FDxx);
  const T Gpww = pww - Dww + FDww;
  const T Gpiww = piww + T(0.5) * (Dww - FDww);
  const T Gpxy = pxy - rx * uy + T(0.5) * Fxy;
  const T Gpyz = pyz - ry * uz + T(0.5) * Fyz;
  const T Gpxz = pxz - rx * uz + T(0.5) * Fxz;

  // Q_m (Eq. 14 in 3-D) with F~ = G s.
  const T sxx = sx * sx, syy = sy * sy, szz = sz * sz;
  const T Q2 = c.G2 * (sxx + syy + szz);
  const T Qe = T(95.0 / 24.0) * Q2, Qeps = T(-55.0 / 48.0) * Q2;
  const T g12 = c.G2 * T(1.0 / 12.0);
  const T Qxx = g12 * (T(2) * sxx - syy - szz), Qww = g12 * (syy - szz);
  const T Qxy = g12 * sx * sy, Qyz = g12 * sy * sz, Qxz = g12 * sx * sz;

  const T bq = c.b_sq_omp;
  const T Geps_Q = Geps - Qeps;
  const T me = m_e + T(38) * Fu - c.se * (Ge - Qe) - c.k_seps_ome * Geps_Q -
               c.h_sq_ome * (ux * Gqx + uy * Gqy + uz * Gqz);
  const T meps = m_eps - T(11) * Fu - c.seps * Geps_Q;
  const T jxb = jx + Fx, jyb = jy + Fy, jzb = jz + Fz;
  const T qxb = qx - two3 * Fx - c.sq * Gqx;
  const T qyb = qy - two3 * Fy - c.sq * Gqy;
  const T qzb = qz - two3 * Fz - c.sq * Gqz;
  const T pxxb = pxx + T(2) * FDxx - c.sp * (Gpxx - Qxx) - bq * (T(4) * ux * Gqx - T(2) * (uy * Gqy + uz * Gqz));
  const T pixxb = pixx - FDxx - c.spi * (Gpixx + T(0.5) * Qxx);
  const T pwwb = pww + T(2) * FDww - c.sp * (Gpww - Qww) - bq * (T(2) * (uy * Gqy - uz * Gqz));
  const T piwwb = piww - FDww - c.spi * (Gpiww + T(0.5) * Qww);
  const T pxyb = pxy + Fxy - c.sp * (Gpxy - Qxy) - bq * (uy * Gqx + ux * Gqy);
  const T pyzb = pyz + Fyz - c.sp * (Gpyz - Qyz) - bq * (uz * Gqy + uy * Gqz);
  const T pxzb = pxz + Fxz - c.sp * (Gpxz - Qxz) - bq * (uz * Gqx + ux * Gqz);
  const T om = T(1) - c.sm;
  const T mxb = om * mx, myb = om * my, mzb = om * mz;

  // Inverse transform: scaled moments, then the rest node and the nine pairs.
  const T r_ = delta * T(1.0 / 19.0);
  const T e_ = me * T(1.0 / 2394.0), p_ = meps * T(1.0 / 252.0);
  const T jx_ = jxb * T(0.1), jy_ = jyb * T(0.1), jz_ = jzb * T(0.1);
  const T qx_ = qxb * T(1.0 / 40.0), qy_ = qyb * T(1.0 / 40.0), qz_ = qzb * T(1.0 / 40.0);
  const T xx_ = pxxb * T(1.0 / 36.0), ixx_ = pixxb * T(1.0 / 72.0);
  const T ww_ = pwwb * T(1.0 / 12.0), iww_ = piwwb * T(1.0 / 24.0);
  const T xy_ = pxyb * T(0.25), yz_ = pyzb * T(0.25), xz_ = pxzb * T(0.25);
  const T mx_ = mxb * T(0.125), my_ = myb * T(0.125), mz_ = mzb * T(0.125);
  o[0] = r_ - T(30) * e_ + T(12) * p_;
  const T ax = r_ - T(11) * e_ - T(4) * p_;
  const T ayz = ax - xx_ + T(2) * ixx_;
  {
    const T ev = ax + T(2) * xx_ - T(4) * ixx_, od = jx_ - T(4) * qx_;
    o[1] = ev + od;
    o[2] = ev - od;
  }
  {
    const T ev = ayz + ww_ - T(2) * iww_, od = jy_ - T(4) * qy_;
    o[3] = ev + od;
    o[4] = ev - od;
  }
  {
    const T ev = ayz - ww_ + T(2) * iww_, od = jz_ - T(4) * qz_;
    o[5] = ev + od;
    o[6] = ev - od;
  }
  const T ce = r_ + T(8) * e_ + p_;
  const T cx = ce + xx_ + ixx_;
  const T exy = cx + ww_ + iww_, exz = cx - ww_ - iww_, eyz = ce - T(2) * (xx_ + ixx_);
  const T JX = jx_ + qx_, JY = jy_ + qy_, JZ = jz_ + qz_;
  {
    const T ev = exy + xy_, od = JX + JY + mx_ - my_;
    o[7] = ev + od;
    o[8] = ev - od;
  }
  {
    const T ev = exy - xy_, od = JX - JY + mx_ + my_;
    o[9] = ev + od;
    o[10] = ev - od;
  }
  {
    const T ev = exz + xz_, od = JX + JZ - mx_ + mz_;
    o[11] = ev + od;
    o[12] = ev - od;
  }
  {
    const T ev = exz - xz_, od = JX - JZ - mx_ - mz_;
    o[13] = ev + od;
    o[14] = ev - od;
  }
  {
    const T ev = eyz + yz_, od = JY + JZ + my_ - mz_;
    o[15] = ev + od;
    o[16] = ev - od;
  }
  {
    const T ev = eyz - yz_, od = JY - JZ + my_ + mz_;
    o[17] = ev + od;
    o[18] = ev - od;
  }
}

// Populations arriving at node (x, y, z) (pull streaming): f_i from x - e_i.
// Neighbour coordinates are precomputed with periodic wrap.  N: the node count,
// the stride between population planes, in the type S of the plane offsets (int
// when 19 N < 2^31, else long long; node indices are int).
template <typename T, typename S>
__device__ __forceinline__ void pull19(const T* f, S N, int nx, int ny, int xm, int x, int xp, int ym,
                                       int y, int yp, int zm, int z, int zp, T* v) {
  const int r00 = (z * ny + y) * nx, rm0 = (z * ny + ym) * nx, rp0 = (z * ny + yp) * nx;
  const int r0m = (zm * ny + y) * nx, r0p = (zp * ny + y) * nx;
  const int rmm = (zm * ny + ym) * nx, rpp = (zp * ny + yp) * nx;
  const int rmp = (zp * ny + ym) * nx, rpm = (zm * ny + yp) * nx;
  v[0] = lbm::ld_st(f + r00 + x);
  v[1] = lbm::ld_st(f + N + r00 + xm);
  v[2] = lbm::ld_st(f + 2 * N + r00 + xp);
  v[3] = lbm::ld_st(f + 3 * N + rm0 + x);
  v[4] = lbm::ld_st(f + 4 * N + rp0 + x);
  v[5] = lbm::ld_st(f + 5 * N + r0m + x);
  v[6] = lbm::ld_st(f + 6 * N + r0p + x);
  v[7] = lbm::ld_st(f + 7 * N + rm0 + xm);
  v[8] = lbm::ld_st(f + 8 * N + rp0 + xp);
  v[9] = lbm::ld_st(f + 9 * N + rp0 + xm);
  v[10] = lbm::ld_st(f + 10 * N + rm0 + xp);
  v[11] = lbm::ld_st(f + 11 * N + r0m + xm);
  v[12] = lbm::ld_st(f + 12 * N + r0p + xp);
  v[13] = lbm::ld_st(f + 13 * N + r0p + xm);
  v[14] = lbm::ld_st(f + 14 * N + r0m + xp);
  v[15] = lbm::ld_st(f + 15 * N + rmm + x);
  v[16] = lbm::ld_st(f + 16 * N + rpp + x);
  v[17] = lbm::ld_st(f + 17 * N + rmp + x);
  v[18] = lbm::ld_st(f + 18 * N + rpm + x);
}

template <typename T>
__device__ __forceinline__ T sum19(const T* v) {
  T a = v[0];
#pragma unroll
  for (int P = 0; P < 9; ++P) a += v[2 * P + 1] + v[2 * P + 2];
  return a;
}

__device__ __forceinline__ int dec(int a, int n) { return a == 0 ? n - 1 : a - 1; }
__device__ __forceinline__ int inc(int a, int n) { return a == n - 1 ? 0 : a + 1; }

// Force stencil of node (ly, lx) from the density planes of z - 1 (a), z (b) and
// z + 1 (e), collision and store of its 19 outputs.
template <typename T, typename S>
__device__ __forceinline__ void stencil_collide_store(const C3<T>& c, const T (*a)[HX], const T (*b)[HX],
                                                      const T (*e)[HX], int ly, int lx, const T* fc, T* __restrict__ fout,
                                                      S N, int idx) {
  const T sxv = T(1.0 / 6.0) * (b[ly][lx + 1] - b[ly][lx - 1]) +
                T(1.0 / 12.0) * ((b[ly + 1][lx + 1] - b[ly - 1][lx - 1]) + (b[ly - 1][lx + 1] - b[ly + 1][lx - 1]) +
                                 (e[ly][lx + 1] - a[ly][lx - 1]) + (a[ly][lx + 1] - e[ly][lx - 1]));
  const T syv = T(1.0 / 6.0) * (b[ly + 1][lx] - b[ly - 1][lx]) +
                T(1.0 / 12.0) * ((b[ly + 1][lx + 1] - b[ly - 1][lx - 1]) + (b[ly + 1][lx - 1] - b[ly - 1][lx + 1]) +
                                 (e[ly + 1][lx] - a[ly - 1][lx]) + (a[ly + 1][lx] - e[ly - 1][lx]));
  const T szv = T(1.0 / 6.0) * (e[ly][lx] - a[ly][lx]) +
                T(1.0 / 12.0) * ((e[ly][lx + 1] - a[ly][lx - 1]) + (e[ly][lx - 1] - a[ly][lx + 1]) +
                                 (e[ly + 1][lx] - a[ly - 1][lx]) + (e[ly - 1][lx] - a[ly + 1][lx]));
  T o[Q];
  collide3_moments(c, fc, b[ly][lx], sxv, syv, szv, o);
#pragma unroll
  for (int i = 0; i < Q; ++i) fout[i * N + idx] = o[i];
}

// S: type of the plane offsets (int when 19 nx ny nz < 2^31, else long long).
template <typename S>
__global__ void __launch_bounds__(TX* kPullTY, 3)
    k_d3_pull(const float* fin, float* __restrict__ fout, int nx, int ny, int nz, int tz, C3<float> c) {
  using T = float;
  lbm::follow_predecessor();
  __shared__ T pl[3][kPullHY][HX];
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX + tx;
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * kPullTY, z0 = blockIdx.z * tz;
  const int z1 = min(z0 + tz, nz);
  const S N = S(nx) * ny * nz;
  const int x = x0 + tx, y = y0 + ty;
  const bool active = x < nx && y < ny;
  const int xg = x % nx, yg = y % ny;
  const int xm = dec(xg, nx), xp = inc(xg, nx), ym = dec(yg, ny), yp = inc(yg, ny);
  // Ring slot of this thread (threads 0..75): top row, bottom row, left and right columns.
  const bool ring = tid < kPullRing;
  int hsx = 0, hsy = 0;
  if (tid < HX) {
    hsx = tid;
  } else if (tid < 2 * HX) {
    hsx = tid - HX;
    hsy = kPullHY - 1;
  } else if (ring) {
    const int r = tid - 2 * HX;
    hsx = r < kPullTY ? 0 : HX - 1;
    hsy = 1 + (r < kPullTY ? r : r - kPullTY);
  }
  const int hx = wrap(x0 - 1 + hsx, nx), hy = wrap(y0 - 1 + hsy, ny);
  const int hxm = dec(hx, nx), hxp = inc(hx, nx), hym = dec(hy, ny), hyp = inc(hy, ny);
  // Plane indices run from z0 - 1 to z1, at most one lattice length outside [0, nz).
  auto zwrap = [&](int zraw) { return zraw < 0 ? zraw + nz : (zraw >= nz ? zraw - nz : zraw); };
  auto pull_node = [&](int zraw, T* v) {
    const int z = zwrap(zraw), zm = dec(z, nz), zp = inc(z, nz);
    pull19(fin, N, nx, ny, xm, xg, xp, ym, yg, yp, zm, z, zp, v);
  };
  auto pull_ring = [&](int zraw, T* v) {
    const int z = zwrap(zraw), zm = dec(z, nz), zp = inc(z, nz);
    pull19(fin, N, nx, ny, hxm, hx, hxp, hym, hy, hyp, zm, z, zp, v);
  };
  auto put = [&](int slot, const T* v, const T* r) {
    pl[slot][ty + 1][tx + 1] = sum19(v);
    if (ring) pl[slot][hsy][hsx] = sum19(r);
  };

  T fc[Q], fn[Q];
  int sp = 0, sc = 1, sn = 2;
  T fr[Q], gn[Q], gr[Q];
  pull_node(z0 - 1, fn);
  if (ring) pull_ring(z0 - 1, fr);
  put(0, fn, fr);
  pull_node(z0, fc);
  if (ring) pull_ring(z0, fr);
  put(1, fc, fr);
  pull_node(z0 + 1, fn);
  if (ring) pull_ring(z0 + 1, fr);
  for (int z = z0; z < z1; ++z) {
    put(sn, fn, fr);
    if (z + 1 < z1) {
      pull_node(z + 2, gn);
      if (ring) pull_ring(z + 2, gr);
    }
    __syncthreads();
    if (active) stencil_collide_store(c, pl[sp], pl[sc], pl[sn], ty + 1, tx + 1, fc, fout, N, (z * ny + y) * nx + x);
    __syncthreads();
    const int t = sp;
    sp = sc;
    sc = sn;
    sn = t;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      fc[i] = fn[i];
      fn[i] = gn[i];
      fr[i] = gr[i];
    }
  }
}

}  // namespace
