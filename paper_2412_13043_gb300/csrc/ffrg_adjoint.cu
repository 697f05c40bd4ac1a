// Vector-Jacobian product of the momentum-loop RHS with respect to the
// dressing-table values (reverse-mode counterpart of the paper's forward-mode
// Jacobians, Sec. 5.2.2):  tbar_j = sum_e gbar_e d out_e / d T_j.
//
// Every lookup is a lerp between two table nodes, so each integrand
// evaluation scatters (1-w) c and w c into two entries of the gradient, where
// c is the derivative of the term with respect to the looked-up value.  The
// Z(q) dependence of the per-radial factor F (regulator derivative and
// G(q)^2) enters through dF/dZ(q) times the angular row sum.
//
// Determinism: no floating-point atomics.  Each warp owns C copies of the
// gradient in shared memory, one per group of 32/C lanes' turn (C a power of
// two that the launch picks, adjoint_setup): lanes of one turn add to
// different copies at once, the 32/C turns follow in a fixed order.  The
// copies are then summed in a fixed order into one partial per CTA, and a
// second kernel sums the CTA partials in a fixed order.  Results are
// reproducible run to run for a given GPU (the persistent grid size fixes
// which rows each warp owns).
//
// Bound: the FP64 pipe (16 clocks a warp instruction).  A d=4 inner term has
// 17 FP64 instructions of value and derivatives, with the fixed-point
// functions of ffrg_prop64.cuh, and three lookups to scatter, 2 + 4 x 16/C
// each.  A turn costs a warp's two FP64 adds however few lanes take part, so
// one lane per turn (C = 1) took longer than the evaluation.  96 points x 4
// angles, 96 x 48 x 16 nodes: 25.05 ms a VJP with FP64 functions and C = 1,
// 3.1 ms so (C = 16).
#include <math.h>

#include <algorithm>

#include "ffrg_internal.cuh"
#include "ffrg_prop64.cuh"

namespace ffrg {

constexpr int kAdjMaxWarps = 8;
constexpr int kLam4Copies = 1;   // lambda4 takes part in the one-loop rows of the d=4 blocks only

struct AdjArgs {
  RhsArgs a;
  const double *gbar;  // [n_ext]
  double *gpart;       // [grid][tab_count]
  double *jrows;       // Jacobian mode: one gradient row per work item [n_items][tab_count]
  int lc;              // log2 of the copies of Z and lambda3
  int n_wide;          // gradient entries with 2^lc copies (the rest: kLam4Copies)
};

// doubles of one warp's gradient copies
__host__ __device__ inline int adj_warp_doubles(const AdjArgs &A) {
  return (A.n_wide << A.lc) + (A.a.tab_count - A.n_wide) * kLam4Copies;
}

// shared memory: function tables | line-form tables | angle rules | per-warp gradient copies
struct AdjSmem {
  FxTables *fx;
  double2 *tab, *cw2;
  double *c1, *s1, *w1, *grad;
  __device__ AdjSmem(unsigned char *base, const RhsArgs &a) {
    fx = (FxTables *)base;
    tab = (double2 *)(base + sizeof(FxTables));
    cw2 = tab + a.tab64_count;
    c1 = (double *)(cw2 + a.na2);
    s1 = c1 + a.na1;
    w1 = s1 + a.na1;
    grad = w1 + a.na1;
  }
};

__device__ __forceinline__ void adj_prologue(const AdjArgs &A, AdjSmem &S) {
  const RhsArgs &a = A.a;
  const double k = scale_k(a), k2 = k * k;
  stage_fx(a, S.fx);
  for (int i = threadIdx.x; i < a.tab64_count; i += blockDim.x) S.tab[i] = tab64_entry(a, i, k2);
  for (int i = threadIdx.x; i < a.na1; i += blockDim.x) {
    double c = a.a1_x[i];
    S.c1[i] = c;
    S.s1[i] = sqrt(fmax(0.0, 1.0 - c * c));
    S.w1[i] = a.a1_w[i];
  }
  for (int i = threadIdx.x; i < a.na2; i += blockDim.x) S.cw2[i] = make_double2(a.a2_x[i], a.a2_w[i]);
  const int all = (int)(blockDim.x >> 5) * adj_warp_doubles(A);
  for (int i = threadIdx.x; i < all; i += blockDim.x) S.grad[i] = 0.0;
  __syncthreads();
}

// Block-wide: the sum of all warps' copies per table value (fixed order:
// warps, then copies starting at the value's own index, which spreads the
// threads over banks) into dst; the copies are cleared.  Z values carry k^2.
__device__ __forceinline__ void adj_collect(const AdjArgs &A, AdjSmem &S, double k2, double *dst) {
  const RhsArgs &a = A.a;
  __syncthreads();
  const int nw = blockDim.x >> 5, per = adj_warp_doubles(A), C = 1 << A.lc;
  for (int i = threadIdx.x; i < a.tab_count; i += blockDim.x) {
    const bool wide = i < A.n_wide;
    const int n = wide ? C : kLam4Copies;
    double *g = S.grad + (wide ? i << A.lc : (A.n_wide << A.lc) + (i - A.n_wide) * kLam4Copies);
    double s = 0.0;
    for (int w = 0; w < nw; ++w)
      for (int c = 0; c < n; ++c) {
        double &v = g[(size_t)w * per + ((c + i) & (n - 1))];
        s += v;
        v = 0.0;
      }
    dst[i] = i < a.n_pts ? k2 * s : s;
  }
  __syncthreads();
}

// A lookup's entry in a line-form row, and its cell of the gradient: the cell's
// first node (the last node counts as weight 1 of the cell before it) and 1 +
// weight; and its value
struct AdjPos {
  int e, i;
  double w1;
};
__device__ __forceinline__ AdjPos adj_pos(const RhsArgs &a, const KConst<double> &kc, double y, FxOff o) {
  AdjPos p;
  node_of(a, kc, y, o, p.e, p.w1);
  p.i = min(max(p.e - 1, 0), a.n_pts - 2);
  if (p.e == 0) p.w1 = 1.0;
  if (p.e == a.n_pts) p.w1 = 2.0;
  return p;
}
__device__ __forceinline__ double adj_val(const double2 *row, AdjPos p) { return line64(row[p.e], p.w1); }

// add c (1 - w) and c w to entries j + p.i and + 1, in turns of 2^lc lanes
__device__ __forceinline__ void adj_scatter(double *g, int lc, int j, AdjPos p, double c, bool valid, int lane) {
  const double v1 = fma(c, p.w1, -c), v0 = c - v1;
  double *e = g + (((j + p.i) << lc) + (lane & ((1 << lc) - 1)));
  const int turn = lane >> lc;
  for (int t = 0; t < (32 >> lc); ++t) {
    if (t == turn && valid) {
      e[0] += v0;
      e[1 << lc] += v1;
    }
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------
// d = 3:  term = F_r w_j G(s); row = (radial node, block of jb angle nodes)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void d3_adjoint_rows(const AdjArgs &A, const AdjSmem &S, const KConst<double> &kc, double *g,
                                                int e, int row, bool valid, int lane) {
  const RhsArgs &a = A.a;
  const int nblk = (a.na1 + a.jb - 1) / a.jb;
  const double p = (e < a.n_ext_p) ? a.ext_pd[e] : 0.0;
  const double gn = (A.jrows ? 1.0 : A.gbar[e]) * a.norm;
  if (!valid) row = 0;
  const int o = row / nblk, j0 = (row - o * nblk) * a.jb;
  const double q = a.radq[o], gF = gn * a.radF[o], dF = a.radD[o];
  const double by = fma(q, q, p * p) * kc.sy, ty = 2.0 * q * p * kc.sy;
  double vrow = 0.0;
  for (int jj = 0; jj < a.jb; ++jj) {
    const bool on = valid && j0 + jj < a.na1;
    const int j = on ? j0 + jj : 0;
    const double y = fma(ty, S.c1[j], by);
    const AdjPos ps = adj_pos(a, kc, y, kc.uy1);
    const double h = reg_h(a, kc, y), G = fx_rcp(fma(adj_val(S.tab, ps), h, kc.m2));
    const double wG = on ? S.w1[j] * G : 0.0;
    vrow += wG;
    adj_scatter(g, A.lc, 0, ps, -gF * wG * (G * h), on, lane);
  }
  adj_scatter(g, A.lc, 0, adj_pos(a, kc, q * q * kc.sy, kc.uy1), gn * dF * vrow * kc.inv_k2, valid, lane);
}

// ---------------------------------------------------------------------------
// d = 4 vertex expansion (tables Z | lambda3 | lambda4 at offsets 0 | n | 2n);
// row = (radial node, first-angle node)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void d4_adjoint_rows(const AdjArgs &A, const AdjSmem &S, const KConst<double> &kc, double *g,
                                                int e, int row, bool valid, int lane) {
  const RhsArgs &a = A.a;
  const int np = a.n_pts, np_ = a.n_ext_p, npsi = a.n_ext_ang, lc = A.lc;
  const double2 *Zt = S.tab, *L3 = S.tab + (np + 1), *L4 = S.tab + 2 * (np + 1);
  double *g4 = g + (A.n_wide << lc);
  int block, ip, jp = 0;
  if (e <= np_) {
    block = 0;
    ip = e;
  } else if (e < np_ + 1 + np_ * npsi) {
    block = 1;
    ip = (e - np_ - 1) / npsi;
    jp = (e - np_ - 1) - ip * npsi;
  } else {
    block = 2;
    ip = e - np_ - 1 - np_ * npsi;
  }
  const double p = (block == 0 && ip == np_) ? 0.0 : a.ext_pd[ip], p2 = p * p, sy = kc.sy, sw2 = kc.sw2;
  const double coef = block == 1 ? 3.0 : (block == 2 ? 1.5 : 1.0);
  const double gn = (A.jrows ? 1.0 : A.gbar[e]) * a.norm * coef;
  if (!valid) row = 0;
  const int r = row / a.na1, ia = row - r * a.na1;
  const double q = a.radq[r], dF = a.radD[r], q2 = q * q, qp = q * p, c1 = S.c1[ia], w1 = S.w1[ia];
  const double A2 = fma(2.0 * qp, c1, q2 + p2), Ay = A2 * sy;
  const AdjPos pA = adj_pos(a, kc, Ay, kc.uy1);
  const double hA = reg_h(a, kc, Ay), GA = fx_rcp(fma(adj_val(Zt, pA), hA, kc.m2));
  const double GPA = -GA * (GA * hA);        // d GA / d Z(A) / k^2
  const double gF = gn * a.radF[r] * w1;     // d(out)/d(row value) x gbar
  double v;                                  // row value (without F w1)
  if (block == 0) {
    const AdjPos p4 = adj_pos(a, kc, (q2 + p2) * sy, kc.uy2), p3 = adj_pos(a, kc, (q2 + A2 + p2) * sy, kc.uy3);
    const double l4 = adj_val(L4, p4), l3 = adj_val(L3, p3), gs = gF * sw2;
    v = sw2 * fma(l3 * l3, GA, -0.5 * l4);
    adj_scatter(g4, 0, 0, p4, -0.5 * gs, valid, lane);
    adj_scatter(g, lc, np, p3, gs * 2.0 * l3 * GA, valid, lane);
    adj_scatter(g, lc, 0, pA, gs * l3 * l3 * GPA, valid, lane);
  } else if (block == 2) {
    const AdjPos p4 = adj_pos(a, kc, (q2 + A2 + 2.0 * p2) * sy, kc.uy4);
    const double l4 = adj_val(L4, p4), gs = gF * sw2;
    v = sw2 * GA * l4 * l4;
    adj_scatter(g4, 0, 0, p4, gs * 2.0 * GA * l4, valid, lane);
    adj_scatter(g, lc, 0, pA, gs * l4 * l4 * GPA, valid, lane);
  } else {
    const double cpsi = a.psi_x[jp], spsi = a.psi_s[jp], C2 = 2.0 * p2 * (1.0 + cpsi);
    const AdjPos pa = adj_pos(a, kc, (q2 + A2 + p2) * sy, kc.uy3);
    const double la = adj_val(L3, pa);
    const double base = q2 + p2, t1 = 2.0 * qp * cpsi * c1, t2 = 2.0 * qp * spsi * S.s1[ia];
    const double by = base * sy, b0 = (base - t1) * sy, t2y = t2 * sy, sab = (A2 + C2) * sy;
    const double gFA = gF * GA * la;         // common factor of the inner terms
    double rs = 0.0;
    for (int b = 0; b < a.na2; ++b) {
      const double2 cw = S.cw2[b];
      const double By = fma(-t2y, cw.x, b0);
      const AdjPos pB = adj_pos(a, kc, By, kc.uy1), pb = adj_pos(a, kc, by + By, kc.uy3),
                   pc = adj_pos(a, kc, sab + By, kc.uy3);
      const double h = reg_h(a, kc, By), GB = fx_rcp(fma(adj_val(Zt, pB), h, kc.m2));
      const double lb = adj_val(L3, pb), lc_ = adj_val(L3, pc);
      const double wG = cw.y * GB, t = gFA * wG, cb = t * lc_;
      rs = fma(wG * lb, lc_, rs);
      adj_scatter(g, lc, np, pb, cb, valid, lane);
      adj_scatter(g, lc, np, pc, t * lb, valid, lane);
      adj_scatter(g, lc, 0, pB, -(cb * lb) * (GB * h), valid, lane);
    }
    v = GA * la * rs;
    adj_scatter(g, lc, 0, pA, gF * GPA * la * rs, valid, lane);
    adj_scatter(g, lc, np, pa, gF * GA * rs, valid, lane);
  }
  // Z(q) through F = w q^3 dR(q) G(q)^2
  adj_scatter(g, lc, 0, adj_pos(a, kc, q2 * sy, kc.uy1), gn * dF * w1 * v * kc.inv_k2, valid, lane);
}

// VJP: warps take units of 32 rows of an external point (d=4: three-point
// block first) in a fixed stride.  Jacobian: CTAs take items (external point x
// chunk), the warps of a CTA its units, and each item's gradient is collected
// into its row.
template <int MODEL>
__global__ void __launch_bounds__(32 * kAdjMaxWarps) adjoint_kernel(AdjArgs A) {
  const RhsArgs &a = A.a;
  extern __shared__ __align__(128) unsigned char smem[];
  AdjSmem S(smem, a);
  adj_prologue(A, S);
  KConst<double> kc = load_kconst<double>(a);
  kc.us = S.fx;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  double *g = S.grad + (size_t)warp * adj_warp_doubles(A);
  const int rows = MODEL == FFRG_MODEL_D3 ? a.nr * ((a.na1 + a.jb - 1) / a.jb) : a.nr * a.na1;
  auto unit = [&](int e, int row, int end) {
    if constexpr (MODEL == FFRG_MODEL_D3) d3_adjoint_rows(A, S, kc, g, e, row, row < end, lane);
    else d4_adjoint_rows(A, S, kc, g, e, row, row < end, lane);
  };
  if (!A.jrows) {
    const int per = (rows + 31) / 32, rot = MODEL == FFRG_MODEL_D3 ? 0 : a.n_ext_p + 1;
    // unit u = e per + j, kept as (e, j): u itself exceeds 32 bits for problems
    // whose 512-row items fit
    const int u0 = warp * gridDim.x + blockIdx.x, step = nw * gridDim.x, de = step / per, dj = step % per;
    for (int e = u0 / per, j = u0 % per; e < a.n_ext;) {
      unit((e + rot) % a.n_ext, j * 32 + lane, rows);
      e += de;
      j += dj;
      if (j >= per) {
        j -= per;
        ++e;
      }
    }
    adj_collect(A, S, kc.k2, A.gpart + (size_t)blockIdx.x * a.tab_count);
    return;
  }
  const int irows = rows / a.nr * a.cr;
  for (int item = blockIdx.x; item < a.n_items; item += gridDim.x) {
    const int e = item / a.n_chunks, c = item - e * a.n_chunks, end = min((c + 1) * irows, rows);
    for (int row = c * irows + warp * 32; row < end; row += nw * 32) unit(e, row + lane, end);
    adj_collect(A, S, kc.k2, A.jrows + (size_t)item * a.tab_count);
  }
}

// fixed-order sum of the CTA partials: a warp per table value, lanes strided, then the warp tree
__global__ void adj_reduce_kernel(const double *gpart, int grid, int count, double *tbar) {
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (i >= count) return;
  double s = 0.0;
  for (int b = lane; b < grid; b += 32) s += gpart[(size_t)b * count + i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if (lane == 0) tbar[i] = s;
}

}  // namespace ffrg

using namespace ffrg;

namespace ffrg {

// fixed-order sum of the chunk rows of each external point: J[e][j]
__global__ void jac_reduce_kernel(const double *jrows, int n_ext, int n_chunks, int T, double *J) {
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (size_t)n_ext * T) return;
  const int e = (int)(idx / T), j = (int)(idx % T);
  double s = 0.0;
  for (int c = 0; c < n_chunks; ++c) s += jrows[((size_t)e * n_chunks + c) * T + j];
  J[idx] = s;
}

// Launch geometry, shared memory and scratch of the adjoint kernels of a plan,
// and A's share of it.  Copies C and warps: the pair with the least FP64 work
// per inner term, 17 + 3 (2 + 4 x 16/C) instructions of 16 clocks on one pipe
// that one warp per SMSP keeps about half busy and two almost full, among
// those whose gradients fit (96 points: C = 16 with 6 warps).
static int adjoint_setup(ffrg_ctx *ctx, Plan *pl, AdjArgs &A, void (**kern_out)(AdjArgs)) {
  void (*kern)(AdjArgs) =
      pl->model == FFRG_MODEL_D3 ? adjoint_kernel<FFRG_MODEL_D3> : adjoint_kernel<FFRG_MODEL_D4_VERTEX>;
  *kern_out = kern;
  // tables up to what eight warps with one copy each hold in 200 KB
  const size_t limit = (((size_t)pl->tab_count * 8 + 15) & ~(size_t)15) +
                       ((((size_t)(3 * pl->na1 + 2 * pl->na2)) * 8 + 15) & ~(size_t)15) +
                       (size_t)kAdjMaxWarps * pl->tab_count * 8;
  if (limit > 200 * 1024) {
    ctx->last_error = "adjoint: tables too large for per-warp shared-memory gradients";
    return FFRG_EINVAL;
  }
  A.a.tab_count = pl->tab_count;
  A.n_wide = (pl->model == FFRG_MODEL_D3 ? 1 : 2) * pl->n_pts;
  if (pl->adj_grid) {
    A.lc = pl->adj_lc;
    return FFRG_OK;
  }
  const size_t fixed = sizeof(FxTables) + (size_t)pl->tab64_count * 16 + ((size_t)3 * pl->na1 + 2 * (size_t)pl->na2) * 8;
  int lc = 0, nw = 0;
  double best = 0.0;
  for (int l = 0; l <= 5; ++l) {
    A.lc = l;
    const size_t per = (size_t)adj_warp_doubles(A) * 8;
    const int w = fixed + per > kMaxDynSmemBytes ? 0 : (int)std::min<size_t>(kAdjMaxWarps, (kMaxDynSmemBytes - fixed) / per);
    const double rate = std::min(1.0, 0.13 * w) / (17.0 + 3.0 * (2.0 + 64.0 / (1 << l)));
    if (w >= 1 && rate > best) {
      best = rate;
      lc = l;
      nw = w;
    }
  }
  if (nw == 0) {
    ctx->last_error = "adjoint: tables too large for per-warp shared-memory gradients";
    return FFRG_EINVAL;
  }
  A.lc = lc;
  const size_t smem = fixed + (size_t)nw * adj_warp_doubles(A) * 8;
  int st = ensure_smem_limit(ctx, (const void *)kern, smem);
  if (st) return st;
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * nw, smem);
  if (e != cudaSuccess || per_sm < 1) return set_cuda_error(ctx, e ? e : cudaErrorInvalidConfiguration, "occupancy");
  const int grid = std::max(1, std::min(pl->n_items, per_sm * ctx->num_sms));
  st = dev_alloc(ctx, (void **)&pl->radD, (size_t)pl->nr * pl->nfreq * sizeof(double));
  if (!st) st = dev_alloc(ctx, (void **)&pl->gpart, (size_t)grid * pl->tab_count * sizeof(double));
  if (st) return st;
  pl->adj_smem = smem;
  pl->adj_grid = grid;
  pl->adj_lc = lc;
  pl->adj_threads = 32 * nw;
  return FFRG_OK;
}

// Full Jacobian d out_e / d T_j (row-major n_ext x table values) at scale k.
int launch_jacobian(ffrg_ctx *ctx, const ffrg_problem *pb, const ffrg_table_desc *td, const double *tab, double k,
                    double *J, cudaStream_t s) {
  if (pb->model != FFRG_MODEL_D3 && pb->model != FFRG_MODEL_D4_VERTEX) return FFRG_EINVAL;
  int st = validate_problem(pb, td);
  if (st) return st;
  Plan *pl = nullptr;
  st = get_plan(ctx, pb, td, &pl);
  if (st) return st;
  AdjArgs A;
  memset(&A, 0, sizeof(A));
  void (*kern)(AdjArgs) = nullptr;
  st = adjoint_setup(ctx, pl, A, &kern);
  if (st) return st;
  if (!pl->jrows) {
    st = dev_alloc(ctx, (void **)&pl->jrows, (size_t)pl->n_items * pl->tab_count * sizeof(double));
    if (st) return st;
  }
  fill_args(pl, pb, td, tab, k, A.a);
  A.a.status = ctx->status_dev;
  A.a.cr = pl->cr;  // block-sized work items
  A.a.jb = pl->jb;
  A.a.n_chunks = pl->n_chunks;
  A.a.n_items = pl->n_items;
  A.a.radD = pl->radD;
  A.jrows = pl->jrows;
  st = launch_precompute(ctx, A.a, s);
  if (st) return st;
  kern<<<pl->adj_grid, pl->adj_threads, pl->adj_smem, s>>>(A);
  const size_t tot = (size_t)pl->n_ext * pl->tab_count;
  jac_reduce_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(pl->jrows, pl->n_ext, pl->n_chunks, pl->tab_count, J);
  return set_cuda_error(ctx, cudaGetLastError(), "jacobian launch");
}

}  // namespace ffrg

extern "C" int ffrg_rhs_jacobian(ffrg_ctx *ctx, const ffrg_problem *pb, const ffrg_tables *tables, double k,
                                 double *J_dev, void *stream) {
  if (!ctx || !pb || !tables || !J_dev || !(k > 0.0) || !isfinite(k)) return FFRG_EINVAL;
  cudaSetDevice(ctx->device);
  return launch_jacobian(ctx, pb, &tables->desc, tables->dev, k, J_dev, (cudaStream_t)stream);
}

extern "C" int ffrg_rhs_adjoint(ffrg_ctx *ctx, const ffrg_problem *pb, const ffrg_tables *tables, double k,
                                const double *gbar_dev, double *tbar_dev, int precision, void *stream) {
  if (!ctx || !pb || !tables || !gbar_dev || !tbar_dev) return FFRG_EINVAL;
  if (!(k > 0.0) || !isfinite(k)) return FFRG_EINVAL;
  if (precision != FFRG_FP64) return FFRG_EINVAL;
  if (pb->model != FFRG_MODEL_D3 && pb->model != FFRG_MODEL_D4_VERTEX) return FFRG_EINVAL;
  int st = validate_problem(pb, &tables->desc);
  if (st) return st;
  cudaSetDevice(ctx->device);
  Plan *pl = nullptr;
  st = get_plan(ctx, pb, &tables->desc, &pl);
  if (st) return st;
  cudaStream_t s = (cudaStream_t)stream;
  AdjArgs A;
  memset(&A, 0, sizeof(A));
  void (*kern)(AdjArgs) = nullptr;
  st = adjoint_setup(ctx, pl, A, &kern);
  if (st) return st;
  fill_args(pl, pb, &tables->desc, tables->dev, k, A.a);
  A.a.status = ctx->status_dev;
  A.a.cr = pl->cr;  // block-sized work items
  A.a.jb = pl->jb;
  A.a.n_chunks = pl->n_chunks;
  A.a.n_items = pl->n_items;
  A.a.radD = pl->radD;
  A.gbar = gbar_dev;
  A.gpart = pl->gpart;
  st = launch_precompute(ctx, A.a, s);
  if (st) return st;
  kern<<<pl->adj_grid, pl->adj_threads, pl->adj_smem, s>>>(A);
  adj_reduce_kernel<<<(pl->tab_count + 7) / 8, 256, 0, s>>>(pl->gpart, pl->adj_grid, pl->tab_count, tbar_dev);
  return set_cuda_error(ctx, cudaGetLastError(), "adjoint launch");
}
