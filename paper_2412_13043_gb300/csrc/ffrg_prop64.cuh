// FP64 integrand pieces shared by the right-hand-side kernels: per-RHS
// constants, line-form tables, lookups and propagators on the fixed-point
// functions of ffrg_fx.cuh.
#pragma once

#include "ffrg_internal.cuh"

namespace ffrg {

// Scale-dependent constants of one RHS in the kernel precision, computed once
// per RHS by the precompute kernel into a small device block (RhsArgs::kconst)
// that every CTA of the main kernel loads.  FP32 us/uo: table coordinate
// divided by n-1; plim = -2 m^2 (near-pole test).  The kernels pass
// squared momenta to the propagator as y = sy s^2 and omega^2 as som omega^2:
// FP64 sy = som = 1/k^2 with the Z table pre-scaled by k^2, so that y is the
// regulator's argument (sy = 1 for the full vertex, whose shape variables
// need s^2 itself); FP32 sy = log2(e)/k^2 (the regulator's exp2 argument)
// and som = 1/(k^2 ln 2), with the FP32 Z table pre-scaled by k^2 ln 2
// (see reg_g).
// uy1..uy4: offsets of table coordinates taken in y of S0^2 = (sum of c
// squares)/c (c = 1..4; ln(sy) and ln c folded in); twopiT = 2 pi T;
// sw2 = sum of the second-angle weights.
struct KConstPair {
  KConst<float> f;
  KConst<double> d;
};
static_assert(sizeof(KConstPair) <= kKConstBytes, "constant block too small");

// The k-dependent constants of one RHS: FP32 from kconst_f32 (or the host's
// copy of it), FP64 below; once per RHS on one thread.
template <typename T>
__device__ __forceinline__ KConst<T> make_kconst(const RhsArgs &a);
template <>
__device__ __forceinline__ KConst<float> make_kconst<float>(const RhsArgs &a) {
  // the host's copy when the scale and mass are host values (plain RHS calls)
  if (a.kc_host_ok && !a.k_dev && !a.m2_dev) return a.kc_host;
  const double kd = scale_k(a);
  return kconst_f32(a, kd, mass2(a, kd));
}
template <>
__device__ __forceinline__ KConst<double> make_kconst<double>(const RhsArgs &a) {
  const double kd = scale_k(a), m2d = mass2(a, kd);
  KConst<double> c;
  c.k2 = kd * kd;
  c.inv_k2 = 1.0 / c.k2;
  c.m2 = m2d;
  const bool full = a.model == FFRG_MODEL_D4_FULL;
  c.sy = full ? 1.0 : c.inv_k2;
  c.som = c.inv_k2;
  c.isy = full ? 1.0 : c.k2;
  c.slow = !a.fg_ok || !(kd > 0x1p-30) || !(kd < 0x1p30);
  // coordinate of y = sy s^2: u_scale ln(y) + u_off + u_scale ln(1/sy)
  int64_t off = a.fg.uo;
  if (!full && !c.slow) {
    const int hi = fx_clamp_hi(fx_bits(c.k2));
    off += fx_log(fx_scaled(a.fx->log[fx_log_index(hi)], a.fg), a.fg, hi, (uint32_t)fx_bits(c.k2));
  }
  if (!c.slow) off += (int64_t)1 << a.fg.F;   // entries of the line-form rows (tab64_entry), not nodes
  c.uy1 = {off, 1};
  c.uy2 = {off - a.fg.uc[0], 2};
  c.uy3 = {off - a.fg.uc[1], 3};
  c.uy4 = {off - a.fg.uc[2], 4};
  c.us = nullptr;
  c.twopiT = a.twopiT;
  c.sw2 = a.sum_w2;
  return c;
}

template <typename T>
__device__ __forceinline__ KConst<T> load_kconst(const RhsArgs &a);
template <>
__device__ __forceinline__ KConst<float> load_kconst<float>(const RhsArgs &a) {
  return ((const KConstPair *)a.kconst)->f;
}
template <>
__device__ __forceinline__ KConst<double> load_kconst<double>(const RhsArgs &a) {
  KConst<double> c = ((const KConstPair *)a.kconst)->d;
  c.uy1.c = 1, c.uy2.c = 2, c.uy3.c = 3, c.uy4.c = 4;
  return c;
}

// FP64 tables in line form: rows of n_pts + 1 entries, the first (T_0, 0) for
// arguments below the grid, then (T_i - d_i, d_i) per node, d_i the difference
// to the next node (0 at a row end), so that the interpolant is one FMA with
// the weight 1 + w in [1, 2) of fx_node.  Its rounding, up to |d_i| 2^-53, is
// below that of the coordinate everywhere on the grid; below the grid, where
// the coordinate is cut off, the first entry gives T_0 itself (T_0 - d_0 + d_0
// is 2e-5 off for a T_0 1e-12 of T_1).  A weight in [0, 1), with (T_i, d_i),
// would do without that entry, but takes 4 % longer to form (d=4 vertex FP64
// 3.08 -> 3.21 ms).  Layout: as the tables (D4_FULL: rows Z | lambda4 | lambda3
// rows; finite T: [row][entry][Z, lambda]).  Z rows carry k^2.  Entry i:
__device__ __forceinline__ double2 tab64_entry(const RhsArgs &a, int i, double k2) {
  const int np = a.n_pts, zn = a.n_stack * np;
  const bool ft = a.model == FFRG_MODEL_FINITE_T || a.model == FFRG_MODEL_FINITE_T_4D;
  const int j = ft ? i >> 1 : i, row = j / (np + 1), c = j - row * (np + 1), col = max(c - 1, 0);
  size_t src = (size_t)row * np;
  bool z;
  if (ft) {
    z = !(i & 1);
    if (!z) src += zn;
  } else {
    z = row < (a.model == FFRG_MODEL_D4_FULL ? 1 : a.n_stack);
    if (a.model == FFRG_MODEL_D4_FULL) src = row == 0 ? (size_t)0 : row == 1 ? (size_t)2 * zn : (size_t)zn + (size_t)(row - 2) * np;
  }
  src += col;
  const double f = z ? k2 : 1.0, v = f * a.tab[src];
  const double d = c == 0 || col == np - 1 ? 0.0 : f * a.tab[src + 1] - v;
  return make_double2(v - d, d);
}

// The function tables into shared memory, logarithms in the grid's units
// (every thread of the block; no barrier).
__device__ __forceinline__ void stage_fx(const RhsArgs &a, FxTables *s) {
  for (int j = threadIdx.x; j < kFxLog; j += blockDim.x) s->log[j] = fx_scaled(a.fx->log[j], a.fg);
  constexpr int kRest = (int)((sizeof(FxTables) - sizeof(s->log)) / 16);
  for (int j = threadIdx.x; j < kRest; j += blockDim.x)
    ((int4 *)(s->log + kFxLog))[j] = ((const int4 *)(a.fx->log + kFxLog))[j];
}

// Entry of a line-form row and weight for the coordinate of y (FP64 lookups):
// fixed point, or an FP64 logarithm when the grid or k lies outside its range.
// (y and 1/sy are passed apart: their product in the caller was computed ahead
// of the branch, three FP64 multiplications a d=4 term.)
static __device__ __noinline__ void slow_node(const RhsArgs *a, double y, double isy, int c, int &i, double &w1) {
  double w;
  lerp_pos(y * isy, a->u_scale, a->uoc[c - 1], a->n_pts, i, w);
  i = i == 0 && w == 0.0 ? 0 : i + 1;
  w1 = 1.0 + w;
}
__device__ __forceinline__ void node_of(const RhsArgs &a, const KConst<double> &kc, double y, FxOff o, int &i,
                                        double &w1) {
  if (kc.slow) slow_node(&a, y, kc.isy, o.c, i, w1);   // uniform
  else fx_node(a.fg, fx_log(kc.us->log, a.fg, y) + o.v, a.n_pts, i, w1);
}
__device__ __forceinline__ double line64(double2 t, double w1) { return fma(t.y, w1, t.x); }

// what a table lookup takes besides its row, argument and offset: the FP32
// coordinate scale, or the FP64 argument block and constants
struct Look64 {
  const RhsArgs &a;
  const KConst<double> &kc;
};
__device__ __forceinline__ float look_scale(const RhsArgs &, const KConst<float> &kc) { return kc.us; }
__device__ __forceinline__ Look64 look_scale(const RhsArgs &a, const KConst<double> &kc) { return {a, kc}; }
__device__ __forceinline__ double look(const double2 *row, double y, Look64 us, FxOff o, int) {
  int i;
  double w1;
  node_of(us.a, us.kc, y, o, i, w1);
  return line64(row[i], w1);
}

// Regulator form h(x) = x + r(x): x/(1 - e^{-x}), flat shape max(1, x).
__device__ __forceinline__ double reg_h(const RhsArgs &a, const KConst<double> &kc, double x) {
  if (a.reg == FFRG_REG_LITIM) return fx_h_flat(x);
  return fx_h(*kc.us, x);
}

// Inverse propagator from the line-form Z value (times k^2), y = sy s^2 and
// om2s = omega^2/k^2: Z (s^2 + k^2 r) = Z k^2 h(x).  OM: finite T (om2s
// counts); FULL: y = s^2.  Template arguments because the compiler computes
// both sides of such a choice, and each FP64 instruction costs a warp 16
// clocks: four of them, on the model, the shape and the sign of x, made a d=4
// term 16.4 FP64 instructions instead of 12.4 (4.05 -> 3.07 ms on the d=4
// vertex workload).
template <bool POLE = true, bool OM = false, bool FULL = false, typename Pole>
__device__ __forceinline__ double inv_prop(const RhsArgs &a, double Zk, double y, double om2s,
                                           const KConst<double> &kc, Pole &&) {
  double h = reg_h(a, kc, FULL ? y * kc.inv_k2 : y);
  if (OM) h += om2s;
  return fx_rcp(fma(Zk, h, kc.m2));
}
// Kinetic part P = k^2 h(x) (= s^2 + k^2 r), regulator derivative rd = k^2
// rdot(x) and table position of a loop momentum s^2 = x k^2.  FP64 RHS:
// rdot = 2 h^2 e^{-x} (exact also where e^{-x} is small) and the coordinate
// from the function tables in global memory.  Mixed RHS and feedback flows
// take r and rdot from expm1 and the coordinate from a logarithm: rounded to
// FP32, or seen by a step controller, their factors keep their bits, and in
// the single-launch finite-T kernel, where one warp computes them among 31
// busy ones, the fixed-point functions' many integer instructions took 2 us
// longer than FP64 ones.
__device__ __forceinline__ bool fast_factors(const RhsArgs &a) { return a.fp64 && !a.ref64; }
struct LoopNode {
  double P, rd, wl;
  int i0;
};
__device__ __forceinline__ LoopNode loop_node(const RhsArgs &a, double s2, double k2, double inv_k2) {
  LoopNode t;
  const double x = s2 * inv_k2;
  if (!fast_factors(a)) {
    double rx, rdx;
    reg_r_rdot(a.reg, x, rx, rdx);
    t.P = __dadd_rn(s2, __dmul_rn(k2, rx));
    t.rd = k2 * rdx;
  } else if (a.reg == FFRG_REG_LITIM) {
    t.P = k2 * (x < 1.0 ? 1.0 : x);
    t.rd = x < 1.0 ? 2.0 * k2 : 0.0;
  } else {
    const double h = fx_h(*a.fx, x);
    t.P = k2 * h;
    t.rd = 2.0 * k2 * h * h * exp(-x);
  }
  if (a.fg_ok && fast_factors(a)) {
    const uint64_t b = fx_bits(s2);
    const int hi = fx_clamp_hi(b);
    double w1;
    fx_node(a.fg, fx_log(fx_scaled(a.fx->log[fx_log_index(hi)], a.fg), a.fg, hi, (uint32_t)b) + a.fg.uo, t.i0, w1);
    t.wl = w1 - 1.0;
    if (t.i0 == a.n_pts - 1) {   // at and beyond the last node
      t.i0 = a.n_pts - 2;
      t.wl = 1.0;
    }
  } else {
    lerp_pos(s2, a.u_scale, a.u_off, a.n_pts, t.i0, t.wl);
  }
  return t;
}

// n-independent terms of radial node r (q = L x_r): weight x measure and the
// loop node of q^2
struct RadialNode {
  double wm;
  LoopNode n;
};
__device__ __forceinline__ RadialNode radial_node(const RhsArgs &a, int r, double L, double k2, double inv_k2) {
  RadialNode t;
  const double q = L * a.rad_x[r], w = L * a.rad_w[r], q2 = __dmul_rn(q, q);
  t.wm = w * (is_d4(a.model) ? q2 * q : q2);
  t.n = loop_node(a, q2, k2, inv_k2);
  return t;
}

// Finite T: F(n, r) = w q^2 Z rdot k^2 G^2 lambda at the loop frequency of
// stack row n (>= 0), written to both loop indices that share it: n and -n
// (bosonic) or -n-1 (fermionic); row of loop index n in radF: n + N + stat.
__device__ __forceinline__ void radial_F_finite_t(const RhsArgs &a, int n, int r, double wm, double P, double rd,
                                                  int i0, double wl, double m2) {
  const int row = min(n, a.n_stack - 1);
  const double Z = lerp_at(a.tab + (size_t)row * a.n_pts, i0, wl);
  const double Lq = lerp_at(a.tab + ((size_t)a.n_stack + row) * a.n_pts, i0, wl);
  const double om = a.stat ? (2.0 * n + 1.0) * kPi * a.T : 2.0 * kPi * a.T * n;
  const double den = fma(Z, fma(om, om, P), m2), G = fast_factors(a) ? fx_rcp(den) : 1.0 / den;
  const double F = wm * (Z * rd) * G * G * Lq;
  const int nr = a.nr, ip = (a.N + a.stat + n) * nr + r, im = (a.N - n) * nr + r;
  a.radF[ip] = F;
  a.radF[im] = F;
  if (a.radF32) {
    a.radF32[ip] = (float)F;
    a.radF32[im] = (float)F;
  }
}

}  // namespace ffrg
