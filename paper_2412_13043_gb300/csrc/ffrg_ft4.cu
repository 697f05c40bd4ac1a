// Finite T with a 4-dimensional regulator on a frequency domain that scales
// with k (Sec. 5.3.2 "Quadraturex0" integrators, efficient with 4D
// regulators; App. G external fermion legs at p0f = pi T exp(-k/(pi T))):
//
//   I(m, p) = pref lam^2 [T sum_n | int dq0/(2 pi)] int d^3q/(2 pi)^3
//             dR(Q) G(Q)^2 L(|Q|) L(|Q+P|) G(Q+P),   Q = (q0, q), P = (p0, p),
//
// R(Q) = Z(|Q|) k^2 r(|Q|^2/k^2), G(Q) = 1/(Z(|Q|)(|Q|^2 + k^2 r) + m^2),
// Z and L on one log grid in |Q|.  The frequency set depends on k: the loop
// Matsubara frequencies with |q0| <= qmax_over_k k while there are at most
// 2N+1 (+1 fermionic) of them, Gauss-Legendre nodes of the domain beyond.
// Three launches per RHS: the frequency set, radial nodes and constants (one
// block), the loop factors F(f, r) = w_f w_r q_r^2 dR G^2 L at (q0_f, q_r) in
// FP64, and the sums of F(f, r) times the angular sum of the shifted line by
// warp-sized items (external point x rows (f, r)).  The scale k is read on the
// device (a flow's stage scale), so every step of a flow sees its own
// frequency set.
#include <math.h>

#include "ffrg_internal.cuh"
#include "ffrg_prop64.cuh"

namespace ffrg {

// kbuf layout of this model: [0, nfreq) frequencies, [nfreq, 2 nfreq) weights,
// [2 nfreq] the number of frequencies in use
__global__ void ft4_freq_kernel(RhsArgs a, int nfreq_max) {
  pdl_trigger();   // the factor kernel may start (it waits for these writes)
  if (skipped(a)) return;
  double *kb = (double *)a.kbuf, *fq = kb, *fw = kb + nfreq_max;
  const double k = scale_k(a), L0 = a.qmax_over_k * k, T = a.T;
  const int cap = 2 * a.N + 1 + (a.stat ? 1 : 0);
  int count, Nk;
  if (a.stat) {
    const double x = L0 / (kPi * T);
    Nk = x < 1.0 ? -1 : (int)floor((x - 1.0) / 2.0);
    count = 2 * Nk + 2;
  } else {
    Nk = (int)floor(L0 / (2.0 * kPi * T));
    count = 2 * Nk + 1;
  }
  const bool sum = count <= cap;
  const int nf = sum ? count : a.na2;
  for (int f = threadIdx.x; f < nf; f += blockDim.x) {
    if (sum) {
      const int n = a.stat ? f - Nk - 1 : f - Nk;
      fq[f] = a.stat ? (2.0 * n + 1.0) * kPi * T : 2.0 * kPi * T * n;
      fw[f] = T;
    } else {
      fq[f] = L0 * a.a2_x[f];
      fw[f] = L0 * a.a2_w[f] / (2.0 * kPi);
    }
  }
  const double qs = a.qmax_over_k * k;
  for (int r = threadIdx.x; r < a.nr; r += blockDim.x) a.radq[r] = qs * a.rad_x[r];
  if (threadIdx.x == 0) kb[2 * nfreq_max] = (double)nf;
  if (threadIdx.x == 32) {
    *a.work_ctr = 0u;
    if (a.fp64) ((KConstPair *)a.kconst)->d = make_kconst<double>(a);
  }
  for (int i = threadIdx.x; i < a.n_ext; i += blockDim.x) a.ext_done[i] = 0u;
  // external momenta for the items of the main kernel, on the block's last warps
  for (int i = blockDim.x - 1 - threadIdx.x; i < a.n_ext_p; i += blockDim.x) a.ext_pd[i] = ext_momentum(a, i);
}

// F(f, r) = w_f w_r q^2 dR(Q) G(Q)^2 L(|Q|), |Q|^2 = q0_f^2 + q_r^2 (FP64; FP32 copy)
__global__ void ft4_factor_kernel(RhsArgs a, int nfreq_max) {
  pdl_trigger();   // the main kernel may start staging its tables
  pdl_wait();      // frequencies, weights and q_r of the frequency kernel
  if (skipped(a)) return;
  const double *kb = (const double *)a.kbuf;
  const int nf = (int)kb[2 * nfreq_max];
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= nf * a.nr) return;
  const int f = idx / a.nr, r = idx - f * a.nr;
  const double k = scale_k(a), k2 = k * k, inv_k2 = 1.0 / k2, m2 = mass2(a, k);
  const double q = a.radq[r], q0 = kb[f];
  const LoopNode t = loop_node(a, fma(q0, q0, q * q), k2, inv_k2);
  const double Z = lerp_at(a.tab, t.i0, t.wl), L = lerp_at(a.tab + a.n_pts, t.i0, t.wl);
  const double G = fx_rcp(fma(Z, t.P, m2));
  const double wr = a.qmax_over_k * k * a.rad_w[r];
  const double F = kb[nfreq_max + f] * wr * q * q * Z * t.rd * G * G * L;
  a.radF[idx] = F;
  a.radF32[idx] = (float)F;
}

// FP32 angular sum (the mixed path) from shared memory: zl[i] = (Z_i, Z_{i+1}
// - Z_i, L_i, L_{i+1} - L_i) per node (the last node's differences 0), cw[c] =
// (c_c, v_c).  Propagator denominator Z k^2 h(x) + m^2 with h(x) = x + r(x) =
// x/(1 - e^-x) (exponential regulator; its Taylor series for x < 1/2, where
// 1 - e^-x cancels) or max(x, 1) (flat), hardware lg2/ex2/rcp.  A denominator that
// cancels more than half of its kinetic part (m^2 < 0 near the pole) is
// recomputed in FP64 from the FP64 tables.
__device__ __forceinline__ float ft4_row32(const RhsArgs &a, const float4 *zl, const float2 *cw, float sh2, float q,
                                           float p, float k2, float inv_k2, float m2, float us, float uo) {
  const int n = a.n_pts, na1 = a.na1;
  const float nm1 = (float)(n - 1);
  const float base = fmaf(q, q, fmaf(p, p, sh2)), tqp = 2.0f * q * p;
  float rs = 0.0f;
  for (int c = 0; c < na1; ++c) {
    const float2 cv = cw[c];
    const float QP2 = fmaxf(0.0f, fmaf(tqp, cv.x, base));
    float u = fminf(fmaxf(fmaf(us, hw_lg2(QP2), uo), 0.0f), nm1);   // NaN (QP2 = 0 -> -inf) saturates to 0
    const int i = min((int)u, n - 2);
    const float w = u - (float)i;
    const float4 t = zl[i];
    const float Z = fmaf(w, t.y, t.x), L = fmaf(w, t.w, t.z);
    const float x = QP2 * inv_k2;
    // G = 1/(kin + m^2), kin = Z k^2 h(x); for x >= 1/2 as d/(Z k^2 x + m^2 d),
    // d = 1 - e^-x >= 0.39 (the ex2 error, 2^-22.5, grows by at most 2.6x):
    // one reciprocal for regulator and propagator
    float num = 1.0f, kin, den;
    if (a.reg == FFRG_REG_LITIM) {
      kin = Z * k2 * fmaxf(x, 1.0f);
      den = kin + m2;
    } else if (x < 0.5f) {   // x/(1 - e^-x) = 1 + x/2 + x^2/12 - x^4/720 + x^6/30240 - ..., remainder < 4e-9
      const float x2 = x * x;
      kin = Z * k2 * fmaf(x2, fmaf(x2, fmaf(x2, 1.0f / 30240.0f, -1.0f / 720.0f), 1.0f / 12.0f), fmaf(x, 0.5f, 1.0f));
      den = kin + m2;
    } else {
      num = 1.0f - hw_ex2(-1.4426950408889634f * x);
      kin = Z * k2 * x;          // = the kinetic part times d
      den = fmaf(m2, num, kin);  // = d (kinetic part + m^2)
    }
    float g;
    if (m2 < 0.0f && den < 0.5f * kin) {
      const double QPd = (double)QP2;
      const double Zd = look(a.tab, QPd, a.u_scale, a.u_off, n);
      g = (float)(1.0 / prop_den(a.reg, Zd, 0.0, QPd, (double)m2, (double)k2, 1.0 / (double)k2));
    } else {
      g = num * hw_rcp(den);
    }
    rs = fmaf(cv.y * L, g, rs);
  }
  return rs;
}

// Warp items: external point e = (p, m) x `cr` rows (f, r), f major (cr and
// the item order depend only on the shape and the frequency set); a lane's
// rows and the items of an external point are added in a fixed order, FP64.
// The warp that completes an external point writes its output.  Each CTA
// first stages the tables and the angle rule: FP64 (one 512-thread CTA per SM)
// the function tables and line-form tables of ffrg_prop64.cuh, FP32 node
// quadruples.  Bound: FP64 six FP64 instructions and the integer work of one
// logarithm, regulator and reciprocal per term.  64 momenta x 9 frequencies,
// 96 x 48 nodes, k = 1 (25 loop frequencies): FP64 10.60 ms with FP64
// functions and one block per external point, 0.74 ms so; mixed 0.162, 0.123 ms so.
template <typename T>
__global__ void __launch_bounds__(sizeof(T) == 8 ? kThreads64 : kThreads)
    ft4_main_kernel(RhsArgs a, int nfreq_max) {
  if (skipped(a)) {   // wait all the same: this kernel completes after the two before it
    pdl_wait();
    return;
  }
  extern __shared__ __align__(16) unsigned char ft4_smem[];
  const int lane = threadIdx.x & 31, nm = a.n_ext_ang;
  const double *kb = (const double *)a.kbuf;
  const double k = scale_k(a), k2 = k * k, m2 = mass2(a, k);
  // FP64: function tables | (Z, L) line-form pairs | (node, weight)
  FxTables *fx = (FxTables *)ft4_smem;
  double2 *zl64 = (double2 *)(ft4_smem + sizeof(FxTables)), *cw64 = zl64 + 2 * (a.n_pts + 1);
  float4 *zl = reinterpret_cast<float4 *>(ft4_smem);
  float2 *cw = reinterpret_cast<float2 *>(zl + a.n_pts);
  if constexpr (sizeof(T) == 8) {
    stage_fx(a, fx);
    for (int i = threadIdx.x; i < 2 * (a.n_pts + 1); i += blockDim.x) zl64[i] = tab64_entry(a, i, k2);
    for (int c = threadIdx.x; c < a.na1; c += blockDim.x) cw64[c] = make_double2(a.a1_x[c], a.a1_w[c]);
  } else {
    const double *Zt = a.tab, *Lt = a.tab + a.n_pts;
    for (int i = threadIdx.x; i < a.n_pts; i += blockDim.x) {
      const bool last = i + 1 >= a.n_pts;
      const double z0 = Zt[i], l0 = Lt[i];
      zl[i] = make_float4((float)z0, last ? 0.0f : (float)(Zt[i + 1] - z0), (float)l0,
                          last ? 0.0f : (float)(Lt[i + 1] - l0));
    }
    for (int c = threadIdx.x; c < a.na1; c += blockDim.x) cw[c] = make_float2((float)a.a1_x[c], (float)a.a1_w[c]);
  }
  // an FP64 exponential per item held small problems back (15 x 9 external
  // points, 5 x 96 rows, 12 angles, mixed: 38.9 us, 26.5 so): p0 here and |p| from
  // the frequency kernel
  const double p0f = a.stat ? kPi * a.T * exp(-k / (kPi * a.T)) : 0.0;
  const float k2f = (float)k2, ik2f = (float)(1.0 / k2), m2f = (float)m2;
  __syncthreads();
  pdl_wait();   // the factor kernel's F(f, r) (and through it the frequency set, constants and counters)
  const int rows = (int)kb[2 * nfreq_max] * a.nr, cr = a.cr, nc = max(1, (rows + cr - 1) / cr);
  const float us = (float)(a.u_scale * 0.69314718055994530942), uo = (float)a.u_off;
  KConst<double> kc;
  if constexpr (sizeof(T) == 8) {
    kc = load_kconst<double>(a);
    kc.us = fx;
  }
  ItemQueue items(a.work_ctr);
  for (;;) {
    const int d = items.pop(a.n_ext * nc);
    if (d >= a.n_ext * nc) break;
    const int e = d / nc, c0 = d - e * nc, ip = e / nm, m = e - ip * nm;
    const double p = a.ext_pd[ip];
    const double p0 = a.stat ? p0f : 2.0 * kPi * a.T * m;
    double acc = 0.0;
    for (int i = c0 * cr + lane; i < min((c0 + 1) * cr, rows); i += 32) {
      const int f = i / a.nr, r = i - f * a.nr;
      const double sh = kb[f] + p0, q = a.radq[r];
      if constexpr (sizeof(T) == 8) {
        // sum_c v_c L(|Q+P|) G(Q+P) at y = |Q+P|^2 / k^2 = by + ty c
        const double by = fma(sh, sh, fma(q, q, p * p)) * kc.sy, ty = 2.0 * q * p * kc.sy;
        double rs = 0.0;
        for (int c = 0; c < a.na1; ++c) {
          const double2 cv = cw64[c];
          const double y = fma(ty, cv.x, by);
          int n;
          double w1;
          node_of(a, kc, y, kc.uy1, n, w1);
          const double Z = line64(zl64[2 * n], w1), L = line64(zl64[2 * n + 1], w1);
          rs = fma(cv.y * L, inv_prop<false>(a, Z, y, 0.0, kc, 0), rs);
        }
        acc = fma(a.radF[i], rs, acc);
      } else {
        const float rs = ft4_row32(a, zl, cw, (float)(sh * sh), (float)q, (float)p, k2f, ik2f, m2f, us, uo);
        acc = fma(a.radF[i], (double)rs, acc);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    unsigned done = 0;
    if (lane == 0) {
      a.partial[(size_t)e * nc + c0] = acc;
      __threadfence();
      done = atomicAdd(a.ext_done + e, 1u);
    }
    done = __shfl_sync(0xffffffffu, done, 0);
    if (done == (unsigned)nc - 1u) {
      __threadfence();
      double t = 0.0;
      for (int j = lane; j < nc; j += 32) t += __ldcg(a.partial + (size_t)e * nc + j);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
      if (lane == 0) {
        const double v = a.norm * t;
        a.out[e] = v;
        if (!isfinite(v)) raise_status(a.status, kStatusNonFinite);
      }
    }
  }
}

int launch_ft4(ffrg_ctx *ctx, const Plan *pl_c, const RhsArgs &a_in, int precision, cudaStream_t s) {
  Plan *pl = const_cast<Plan *>(pl_c);
  RhsArgs a = a_in;
  a.fp64 = precision != FFRG_MIXED;
  if (!a.kbuf || !a.radq || !a.radF || !a.radF32 || !a.a2_x || !a.work_ctr || !a.ext_done || !a.kconst) {
    ctx->last_error = "plan without the frequency buffer, radial factors or counters";
    return FFRG_EINVAL;
  }
  const size_t smem = a.fp64 ? sizeof(FxTables) + (size_t)(2 * (pl->n_pts + 1) + pl->na1) * sizeof(double2)
                             : (size_t)pl->n_pts * sizeof(float4) + (size_t)pl->na1 * sizeof(float2);
  void (*kern)(RhsArgs, int) = a.fp64 ? ft4_main_kernel<double> : ft4_main_kernel<float>;
  const int threads = a.fp64 ? kThreads64 : kThreads;
  int &grid = a.fp64 ? pl->grid64 : pl->grid32;
  if (grid == 0) {   // (external points) x (rows of the largest frequency set) in warp items
    const int st = persistent_grid(ctx, (const void *)kern, smem, a.n_items, &grid, threads);
    if (st) return st;
  }
  const int nfreq = pl->nfreq;
  ft4_freq_kernel<<<1, kThreads, 0, s>>>(a, nfreq);
  const int terms = nfreq * pl->nr;
  cudaError_t e = launch_dependent(ft4_factor_kernel, dim3((terms + kThreads - 1) / kThreads), dim3(kThreads), 0, s,
                                   true, a, nfreq);
  if (e != cudaSuccess) return set_cuda_error(ctx, e, "finite-T 4D factor launch");
  const bool prof = ctx->profiling && ctx->prof_used * 2 + 1 < (int)ctx->prof_events.size();
  if (prof) cudaEventRecord(ctx->prof_events[2 * ctx->prof_used], s);
  e = launch_dependent(kern, dim3(grid), dim3(threads), smem, s, true, a, nfreq);
  if (e != cudaSuccess) return set_cuda_error(ctx, e, "finite-T 4D launch");
  if (prof) {
    cudaEventRecord(ctx->prof_events[2 * ctx->prof_used + 1], s);
    ctx->prof_used++;
  }
  return set_cuda_error(ctx, cudaGetLastError(), "finite-T 4D launch");
}

}  // namespace ffrg
