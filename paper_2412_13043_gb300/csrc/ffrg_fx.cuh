// FP64-accurate scalar functions on the integer pipe.
//
// This part issues 2 FP64 results per clock and SM, one warp instruction in 16
// clocks; a 32 x 32 -> 64 bit multiply-add takes 1.3 clocks, a 64-bit high
// multiply 4.4, an integer add or shift 0.5 (throughput loops, 32 warps per
// SM).  A logarithm, an exponential or a division in FP64 is a sequence of 15
// to 40 FP64 instructions, and conversions between FP64 and other types run
// at the FP64 rate as well.  So the three functions that an integrand needs
// besides additions and products are evaluated here in 64-bit fixed point
// from the bit pattern of their argument, and hand back bit patterns:
//   fx_u    table coordinate u = u_scale ln(y) + u_off of a log grid,
//   fx_h    regulator h(x) = x / (1 - e^{-x}),
//   fx_rcp  1 / d.
// Errors: fx_h at most 0.73 ulp of a double and fx_rcp 0.50 over 4e6 arguments
// (a correctly rounded result: 0.50), fx_u below 2^-50 of a node spacing at 128
// nodes (u_scale ln(y) + u_off in FP64 is off by up to 2^-46), so the FP64
// kernels lose no accuracy.
//
// The tables are built on the host in extended precision (fx_build_tables)
// and staged in shared memory by the kernels.  The header also compiles as
// plain C++ (the CPU tests compare the functions with 40-digit values).
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define FX_FN __host__ __device__ __forceinline__
#else
#define FX_FN inline
#endif

namespace ffrg {

// ---------------------------------------------------------------------------
// Tables.  Logarithm: entry j holds r_j ~ 2^31 / (1 + j/1024), rounded up, and
// log2(2^31 / r_j) as a 64-bit fraction.  Regulator: 128 cells of x in [0, 1)
// and 128 per octave [2^e, 2^(e+1)), e = 0..5, each a polynomial of degree 5
// in the position t in [0, 1) in the cell (beyond x = 64, h = x in FP64).
// ---------------------------------------------------------------------------
constexpr int kFxLog = 1024, kFxCells = 7 * 128;
struct FxLogEntry {
  uint64_t l;   // host table: log2(2^31/r) 2^64; staged: the same times u_scale ln 2, in units of 2^-F
  uint32_t r, pad;
};
struct FxCellB {
  int64_t c2;   // 2 c_2
  int32_t c3, c4;  // c_3 / 2^7, 2 c_4 / 2^7
};
struct FxTables {
  FxLogEntry log[kFxLog];
  uint64_t c01[kFxCells][2];   // c_0, c_1 in units of 2^(e-62)
  FxCellB b[kFxCells];
  int32_t c5[kFxCells];        // 4 c_5 / 2^7
};

// Log-grid coordinate in fixed point: u 2^F = us e + l_j + zeta (b1 - zeta (b2
// - zeta (b3 - zeta b4))) + uo for y = 2^e m; us = u_scale ln 2 2^F in
// [2^53, 2^54), so that with |e| <= 200, grids within 2^+-50 and scales k
// within 2^+-30 (coordinates are taken in y = s^2/k^2) no sum leaves 64 bits.
struct FxGrid {
  int64_t us, uo, uc[3];   // uc[c-2] = us log2(c), c = 2..4: coordinate of y/c
  uint64_t b1, b2;
  uint32_t b3, b4;
  int F, nm1;              // n_pts - 1
};

FX_FN uint64_t fx_mulhi_u(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}
FX_FN int64_t fx_mulhi_s(int64_t a, int64_t b) {
#ifdef __CUDA_ARCH__
  return __mul64hi(a, b);
#else
  return (int64_t)(((__int128)a * b) >> 64);
#endif
}
FX_FN uint32_t fx_mulhi_u(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
FX_FN int32_t fx_mulhi_s(int32_t a, int32_t b) { return (int32_t)(((int64_t)a * b) >> 32); }
FX_FN uint64_t fx_bits(double v) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(v);
#else
  uint64_t u;
  memcpy(&u, &v, 8);
  return u;
#endif
}
FX_FN double fx_double(uint64_t u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)u);
#else
  double v;
  memcpy(&v, &u, 8);
  return v;
#endif
}

// us log2(y) of a positive double: us e + l_j + polynomial.  Arguments below
// 2^-200 (0 and rounding below 0 among them) count as 2^-200, above 2^200
// (infinity and NaN) as 2^200: both beyond every table.
constexpr int kFxExp = 200;
FX_FN int fx_clamp_hi(uint64_t b) {
  constexpr int kLo = (1023 - kFxExp) << 20, kHi = (1023 + kFxExp) << 20;
  const int hi = (int)(b >> 32);
  return hi < kLo ? kLo : (hi > kHi ? kHi : hi);
}
FX_FN int fx_log_index(int hi) { return (hi >> 10) & (kFxLog - 1); }
FX_FN int64_t fx_log(const FxLogEntry &t, const FxGrid &g, int hi, uint32_t lo) {
  const int e = (hi >> 20) - 1023;
  const uint32_t mh = 0x80000000u | ((uint32_t)hi << 11) | (lo >> 21), ml = lo << 11;   // mantissa in [1, 2), Q1.63
  // z = m r - 1 in [0, 2^-10 + 2^-30), units 2^-62; zeta = 2^9 z as a 64-bit fraction
  const uint64_t p = (uint64_t)mh * t.r + (((uint64_t)ml * t.r) >> 32);
  const uint64_t zeta = p << 11;   // the leading 1 of p (bit 62) is shifted out
  const uint32_t z32 = (uint32_t)(zeta >> 32);
  const uint32_t v3 = g.b3 - fx_mulhi_u(z32, g.b4);
  const uint64_t v2 = g.b2 - fx_mulhi_u(z32, v3);
  const uint64_t v1 = g.b1 - fx_mulhi_u(zeta, v2);
  return (int64_t)e * g.us + (int64_t)t.l + (int64_t)fx_mulhi_u(zeta, v1);
}
FX_FN int64_t fx_log(const FxLogEntry *tab, const FxGrid &g, double y) {
  const uint64_t b = fx_bits(y);
  const int hi = fx_clamp_hi(b);
  return fx_log(tab[fx_log_index(hi)], g, hi, (uint32_t)b);
}
// an entry of the host table with its logarithm in the grid's units
FX_FN FxLogEntry fx_scaled(FxLogEntry t, const FxGrid &g) {
  t.l = fx_mulhi_u(t.l, (uint64_t)g.us);
  return t;
}

// node and interpolation weight: i in [0, last], w1 = 1 + weight in [1, 2); at
// the last node the table's difference is 0 and the weight does not matter
FX_FN void fx_node(const FxGrid &g, int64_t u, int last, int &i, double &w1) {
  const uint64_t v = u < 0 ? 0 : (uint64_t)u;
  const int n = (int)(v >> g.F);
  i = n < last ? n : last;
  w1 = fx_double(((v << (64 - g.F)) >> 12) | 0x3FF0000000000000ull);
}
FX_FN void fx_node(const FxGrid &g, int64_t u, int &i, double &w1) { fx_node(g, u, g.nm1, i, w1); }

// h(x) = x/(1 - e^{-x}) for x >= 0 (x <= 0 and NaN below: see the callers)
FX_FN double fx_h(const FxTables &T, double x) {
  const uint64_t b = fx_bits(x);
  const int E = (int)(b >> 52) - 1023;
  // x >= 64, infinity, NaN; a negative x (rounding) counts as 0 (comparisons
  // on the bits: an FP64 one would run on the FP64 pipe, branch taken or not)
  if (E >= 6) return (b >> 63) && b <= 0xFFF0000000000000ull ? 1.0 : x;
  const uint64_t m = 0x8000000000000000ull | (b << 11);
  // position of x in [0, 1), or of x/2^E - 1, as a 64-bit fraction
  const uint64_t f = E < 0 ? (E < -64 ? 0 : m >> (-E - 1)) : m << 1;
  const int e = E < 0 ? 0 : E;
  const int c = (E < 0 ? 0 : 128 * (E + 1)) + (int)(f >> 57);
  const uint64_t t = f << 7;
  const int32_t t31 = (int32_t)(t >> 33);
  const uint64_t c0 = T.c01[c][0], c1 = T.c01[c][1];
  const FxCellB k = T.b[c];
  const int32_t q4 = k.c4 + fx_mulhi_s(t31, T.c5[c]);
  const int32_t q3 = k.c3 + fx_mulhi_s(t31, q4);
  const int64_t q2 = k.c2 + (((int64_t)q3 * t31) >> 23);
  const uint64_t q1 = c1 + (uint64_t)fx_mulhi_s(q2, (int64_t)(t >> 1));
  uint64_t H = c0 + fx_mulhi_u(t, q1);   // h 2^(62 - e), in [2^62, 1.2 2^63)
  const int s = (int)(H >> 63);
  H >>= s;
  return fx_double(((uint64_t)(e + 1022 + s) << 52) + ((H + 512) >> 10));   // the leading bit adds 1 to the exponent
}

// flat shape: max(1, x), 1 for negative x
FX_FN double fx_h_flat(double x) {
  const uint64_t b = fx_bits(x);
  return b < 0x3FF0000000000000ull || ((b >> 63) && b <= 0xFFF0000000000000ull) ? 1.0 : x;
}

// 1/d: an FP32 seed (relative error e ~ 2^-22) and 1/d = r (1 + e + e^2) + O(e^3)
FX_FN double fx_rcp(double d) {
  const uint64_t b = fx_bits(d);
  const int E = (int)((b >> 52) & 0x7FF);
  if (E < 2 || E > 2044) return 1.0 / d;   // 0, subnormal, huge, infinity, NaN
  const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b;
  const uint32_t dh = 0x80000000u | (hi << 11) | (lo >> 21), dl = lo << 11;   // mantissa, Q1.63
  uint32_t r0;   // Q1.31, in [2^30, 2^31]
#ifdef __CUDA_ARCH__
  float f = __uint_as_float(0x3F800000u | ((dh << 1) >> 9)), rf;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rf) : "f"(f));
  r0 = __float2uint_rn(rf * 2147483648.0f);
#else
  uint32_t fb = 0x3F800000u | ((dh << 1) >> 9);
  float f;
  memcpy(&f, &fb, 4);
  r0 = (uint32_t)(1.0f / f * 2147483648.0f);
#endif
  const uint64_t p = (uint64_t)dh * r0 + (((uint64_t)dl * r0) >> 32);   // d r0, units 2^-62
  const int64_t e = (int64_t)(0x4000000000000000ull - p);               // 1 - d r0, |e| < 2^42
  const int32_t es = (int32_t)(e >> 16);                                // units 2^-46
  const int64_t f1 = e + (((int64_t)es * es) >> 30);                    // e + e^2
  // r0 f1: f1 2^20 (63 bits) times r0, high part; r0 2^-31 f1 2^-62 in units 2^-62 is r0 f1 >> 31
  const int64_t fs = f1 << 20;
  const int64_t c = (int64_t)r0 * (int32_t)(fs >> 32) + (int64_t)(((uint64_t)r0 * (uint32_t)fs) >> 32);
  const uint64_t R = ((uint64_t)r0 << 31) + (uint64_t)(c >> 19);        // 1/m in units 2^-62, in [2^61, 2^62]
  // (1/m) 2^-(E - 1023): exponent field 2045 - E for R in [2^61, 2^62), its leading bit adds 1
  return fx_double((b & 0x8000000000000000ull) + ((uint64_t)(2044 - E) << 52) + ((R + 256) >> 9));
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
inline void fx_build_tables(FxTables *T) {
  for (int j = 0; j < kFxLog; ++j) {
    const uint64_t r = ((1ull << 41) + 1024 + j - 1) / (1024 + j);   // ceil(2^31 / (1 + j/1024))
    T->log[j].r = (uint32_t)r;
    T->log[j].pad = 0;
    T->log[j].l = (uint64_t)(log2l(2147483648.0L / (long double)r) * 18446744073709551616.0L);
  }
  for (int c = 0; c < kFxCells; ++c) {
    const int e = c < 128 ? 0 : c / 128 - 1;
    const long double x0 = c < 128 ? c / 128.0L : ldexpl(1.0L + (c % 128) / 128.0L, e), w = ldexpl(1.0L, e - 7);
    long double t[6], d[6], p[6] = {0, 0, 0, 0, 0, 0};
    for (int i = 0; i < 6; ++i) {   // interpolation at the Chebyshev points of the cell (divided differences)
      t[i] = 0.5L - 0.5L * cosl((2 * i + 1) * 3.14159265358979323846264338327950288L / 12.0L);
      const long double x = x0 + w * t[i];
      d[i] = ldexpl(x == 0.0L ? 1.0L : x / -expm1l(-x), 62 - e);
    }
    for (int k = 1; k < 6; ++k)
      for (int i = 5; i >= k; --i) d[i] = (d[i] - d[i - 1]) / (t[i] - t[i - k]);
    for (int i = 5; i >= 0; --i) {  // p = p (t - t_i) + d_i
      for (int k = 5; k > 0; --k) p[k] = p[k - 1] - t[i] * p[k];
      p[0] = d[i] - t[i] * p[0];
    }
    T->c01[c][0] = (uint64_t)roundl(p[0]);
    T->c01[c][1] = (uint64_t)roundl(p[1]);
    T->b[c].c2 = (int64_t)roundl(2 * p[2]);
    T->b[c].c3 = (int32_t)roundl(p[3] / 128);
    T->b[c].c4 = (int32_t)roundl(2 * p[4] / 128);
    T->c5[c] = (int32_t)roundl(4 * p[5] / 128);
  }
}

// log2(1 + z) = zeta (k1 - zeta (k2 - zeta (k3 - zeta k4))), zeta = 2^9 z in [0, 1/2 + 2^-21]: interpolation
// of log2(1 + z)/zeta at four Chebyshev points (error below 2^-60); p = k1, -k2, k3, -k4
struct FxLogPoly {
  long double p[4] = {0, 0, 0, 0};
  FxLogPoly() {
    long double t[4], d[4];
    for (int i = 0; i < 4; ++i) {
      t[i] = 0.25L - 0.25L * cosl((2 * i + 1) * 3.14159265358979323846264338327950288L / 8.0L);
      d[i] = log1pl(t[i] / 512) / t[i] / 0.693147180559945309417232121458176568L;
    }
    for (int k = 1; k < 4; ++k)
      for (int i = 3; i >= k; --i) d[i] = (d[i] - d[i - 1]) / (t[i] - t[i - k]);
    for (int i = 3; i >= 0; --i) {
      for (int k = 3; k > 0; --k) p[k] = p[k - 1] - t[i] * p[k];
      p[0] = d[i] - t[i] * p[0];
    }
  }
};

// Grid constants; false when the grid lies outside what fixed point covers.
inline bool fx_grid(int n_pts, double x_min, double x_max, FxGrid *g) {
  memset(g, 0, sizeof(*g));
  if (!(x_min > 0x1p-50) || !(x_max < 0x1p50) || !(x_max > x_min)) return false;
  const long double us = (n_pts - 1) / (2.0L * log2l((long double)x_max / x_min));
  if (!(us > 0x1p-6L) || !(us < 0x1p40L)) return false;
  int ex;
  frexpl(us, &ex);              // us in [2^(ex-1), 2^ex)
  g->F = 54 - ex;
  // F >= 32: a coordinate below 2^63 has a node number below 2^31, so fx_node
  // may cut it to 32 bits before it clamps.  Steeper grids (2^22 nodes an
  // octave and more, for instance 4096 nodes on [1, 1.0003]) are refused: a
  // momentum a few octaves away from them would not fit, and no sensible
  // momentum grid is that narrow.
  if (g->F < 32 || g->F > 60) return false;
  g->nm1 = n_pts - 1;
  const long double s = ldexpl(us, g->F);
  g->us = (int64_t)roundl(s);
  g->uo = (int64_t)roundl(-2.0L * log2l((long double)x_min) * s);
  for (int c = 2; c <= 4; ++c) g->uc[c - 2] = (int64_t)roundl(s * log2l((long double)c));
  static const FxLogPoly poly;
  const long double *p = poly.p;
  g->b1 = (uint64_t)roundl(p[0] * s);
  g->b2 = (uint64_t)roundl(-p[1] * s);
  g->b3 = (uint32_t)roundl(p[2] * s);
  g->b4 = (uint32_t)roundl(-p[3] * s);
  return true;
}

}  // namespace ffrg
