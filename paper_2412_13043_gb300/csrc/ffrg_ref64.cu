// FP64 right-hand side of adaptive feedback flows (d=3 and d=4 vertex
// expansion), with logarithms, exponentials and divisions as FP64 functions.
//
// The feedback map divides (I(p) - I(0)) by p^2, which lifts the last bits of
// an RHS by up to (k/p)^2 ~ 1e8 into the state, and the step controller sees
// them: results that differ in the last bit take other steps, and endpoints
// then differ by the flow's tolerance.  So these flows keep one arithmetic, to
// the bit, apart from the faster one of ffrg_prop64.cuh: every lane's terms,
// the order of its rows, the shuffle tree of an item and the order of the
// items are fixed by the problem shape; products and sums that the compiler
// could contract are written out.
//
// What the launch chooses is where the rows are computed.  The terms are bound
// by the FP64 pipe (134 FP64 instructions, 16 clocks each per warp and SM), so
// a problem with fewer items than resident warps leaves SMs idle.  Then
// (ROWS) any warp computes 32 rows of an item into a row buffer, and the warp
// that completes an item adds its rows in the item's own order.  193 external
// points x 32 x 16 x 8 nodes: 386 items on 49 SMs 0.78 ms a RHS, 3088 row
// groups on 152 SMs 0.22 ms.
#include <math.h>

#include <algorithm>

#include "ffrg_internal.cuh"

namespace ffrg {

struct RefSmem {
  double *tab, *c2, *c1, *s1, *w1;   // tables | second-angle (node, weight) pairs | first-angle nodes, sines, weights
  __device__ RefSmem(unsigned char *base, const RhsArgs &a) {
    tab = (double *)base;
    c2 = tab + ((a.tab_count + 1) & ~1);
    c1 = c2 + 2 * a.na2;
    s1 = c1 + a.na1;
    w1 = s1 + a.na1;
  }
  static size_t bytes(const Plan *pl) {
    return ((size_t)((pl->tab_count + 1) & ~1) + 2 * (size_t)pl->na2 + 3 * (size_t)pl->na1) * sizeof(double);
  }
};

struct RefConst {
  double k2, inv_k2, m2;
};

__device__ __forceinline__ double ref_prop(const RhsArgs &a, double Z, double s2, const RefConst &kc) {
  return 1.0 / prop_den(a.reg, Z, 0.0, s2, kc.m2, kc.k2, kc.inv_k2);
}

// rows of one item
template <int MODEL>
__device__ __forceinline__ int ref_item_rows(const RhsArgs &a) {
  return MODEL == FFRG_MODEL_D3 ? a.cr : a.cr * a.na1;
}

// value of row R of external point e, to be multiplied by the radial factor of node r
template <int MODEL>
__device__ __forceinline__ double ref_row(const RhsArgs &a, const RefSmem &S, const RefConst &kc, int e, int R, int &r) {
  const int np = a.n_pts, na1 = a.na1;
  const double us = a.u_scale;
  const double *Zt = S.tab;
  if constexpr (MODEL == FFRG_MODEL_D3) {
    const int jb = a.jb, nblk = (na1 + jb - 1) / jb;
    const double p = (e < a.n_ext_p) ? a.ext_pd[e] : 0.0;
    r = R / nblk;
    const int j0 = (R - r * nblk) * jb, j1 = min(j0 + jb, na1);
    const double q = a.radq[r];
    const double by = fma(q, q, __dmul_rn(p, p)), ty = 2.0 * q * p;
    double rs = 0.0;
    for (int j = j0; j < j1; ++j) {
      const double y = fma(ty, S.c1[j], by);
      const double Z = lerp(Zt, y, us, a.uoc[0], np);
      rs = fma(S.w1[j], ref_prop(a, Z, y, kc), rs);
    }
    return rs;
  } else {
    const double *L3 = S.tab + np, *L4 = S.tab + 2 * np;
    const int np_ = a.n_ext_p, npsi = a.n_ext_ang;
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
    const double p = (block == 0 && ip == np_) ? 0.0 : a.ext_pd[ip], p2 = __dmul_rn(p, p);
    const double cpsi = block == 1 ? a.psi_x[jp] : 1.0, spsi = block == 1 ? a.psi_s[jp] : 0.0;
    const double C2 = __dmul_rn(2.0 * p2, 1.0 + cpsi);
    r = R / na1;
    const int ia = R - r * na1;
    const double q = a.radq[r], q2 = __dmul_rn(q, q), qp = __dmul_rn(q, p), c1 = S.c1[ia];
    const double qq = __dadd_rn(q2, p2);
    const double A2 = fma(2.0 * qp, c1, qq);   // >= 0 up to rounding; lookups clamp
    const double GA = ref_prop(a, lerp(Zt, A2, us, a.uoc[0], np), A2, kc);
    double v;
    if (block == 0) {
      const double l4 = lerp(L4, qq, us, a.uoc[1], np);
      const double l3 = lerp(L3, __dadd_rn(__dadd_rn(q2, A2), p2), us, a.uoc[2], np);
      v = a.sum_w2 * fma(__dmul_rn(l3, l3), GA, -0.5 * l4);
    } else if (block == 2) {
      const double l4 = lerp(L4, fma(2.0, p2, __dadd_rn(q2, A2)), us, a.uoc[3], np);
      v = __dmul_rn(__dmul_rn(__dmul_rn(a.sum_w2, GA), l4), l4);
    } else {
      const double la = lerp(L3, __dadd_rn(__dadd_rn(q2, A2), p2), us, a.uoc[2], np);
      const double base = qq, t2 = 2.0 * qp * spsi * S.s1[ia];
      const double b0 = fma(-(2.0 * qp * cpsi), c1, base), sab = __dadd_rn(A2, C2);
      double rs = 0.0;
      for (int b = 0; b < a.na2; ++b) {
        const double x2 = S.c2[2 * b], w2 = S.c2[2 * b + 1];
        const double B2 = fma(-t2, x2, b0);
        const double GB = ref_prop(a, lerp(Zt, B2, us, a.uoc[0], np), B2, kc);
        const double lb = lerp(L3, __dadd_rn(base, B2), us, a.uoc[2], np);
        const double lc = lerp(L3, __dadd_rn(sab, B2), us, a.uoc[2], np);
        rs = fma(__dmul_rn(__dmul_rn(w2, GB), lb), lc, rs);
      }
      v = __dmul_rn(__dmul_rn(GA, la), rs);
    }
    return __dmul_rn(S.w1[ia], v);
  }
}

__device__ __forceinline__ double ref_tree(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Item sum acc (lane 0) of item (e, c) into the partials; the warp that
// completes the external point adds them in order and writes the output.
template <int MODEL>
__device__ __forceinline__ void ref_item_done(const RhsArgs &a, int e, int c, double acc, int lane) {
  unsigned done = 0;
  if (lane == 0) {
    a.partial[(size_t)e * a.n_chunks + c] = acc;
    __threadfence();
    done = atomicAdd(a.ext_done + e, 1u);
  }
  done = __shfl_sync(0xffffffffu, done, 0);
  if (done != (unsigned)a.n_chunks - 1u) return;
  __threadfence();
  double t = 0.0;
  for (int j = lane; j < a.n_chunks; j += 32) t += __ldcg(a.partial + (size_t)e * a.n_chunks + j);
  t = ref_tree(t);
  if (lane == 0) {
    double coef = 1.0;
    if (MODEL != FFRG_MODEL_D3) {
      const int np_ = a.n_ext_p;
      if (e > np_ && e < np_ + 1 + np_ * a.n_ext_ang) coef = 3.0;
      else if (e >= np_ + 1 + np_ * a.n_ext_ang) coef = 1.5;
    }
    const double v = a.norm * coef * t;
    a.out[e] = v;
    if (!isfinite(v)) raise_status(a.status, kStatusNonFinite);
  }
}

template <int MODEL, bool ROWS>
__global__ void __launch_bounds__(kThreads) ref64_kernel(RhsArgs a) {
  if (a.skip && *(volatile const int *)a.skip) {
    pdl_wait();   // completes after its precompute
    return;
  }
  extern __shared__ __align__(128) unsigned char smem[];
  RefSmem S(smem, a);
  for (int i = threadIdx.x; i < a.na1; i += blockDim.x) {
    const double c = a.a1_x[i];
    S.c1[i] = c;
    S.s1[i] = sqrt(fmax(0.0, 1.0 - c * c));
    S.w1[i] = a.a1_w[i];
  }
  for (int i = threadIdx.x; i < a.na2; i += blockDim.x) {
    S.c2[2 * i] = a.a2_x[i];
    S.c2[2 * i + 1] = a.a2_w[i];
  }
  pdl_wait();
  for (int i = threadIdx.x; i < a.tab_count; i += blockDim.x) S.tab[i] = a.tab[i];
  __syncthreads();
  RefConst kc;
  const double k = scale_k(a);
  kc.k2 = k * k;
  kc.inv_k2 = 1.0 / kc.k2;
  kc.m2 = fma(a.m2_over_k2 * k, k, a.m2_dev ? *a.m2_dev : a.m2_shift);
  const int lane = threadIdx.x & 31;
  // d=4: the three-point block, with the second-angle loop, first
  const int rot = MODEL == FFRG_MODEL_D3 ? 0 : a.n_ext_p + 1;
  const int rows = ref64_rows(MODEL, a.nr, a.na1, a.jb), irows = ref_item_rows<MODEL>(a), nseg = ROWS ? (irows + 31) / 32 : 1;
  ItemQueue items(a.work_ctr);
  for (;;) {
    const int d = items.pop(a.n_items * nseg);
    if (d >= a.n_items * nseg) break;
    const int s = d % nseg, item = d / nseg, c = item % a.n_chunks, e = (item / a.n_chunks + rot) % a.n_ext;
    const int R0 = c * irows, R1 = min(R0 + irows, rows);
    if (!ROWS) {
      double acc = 0.0;
      for (int R = R0 + lane; R < R1; R += 32) {
        int r;
        const double x = ref_row<MODEL>(a, S, kc, e, R, r);
        acc = fma(a.radF[r], x, acc);
      }
      ref_item_done<MODEL>(a, e, c, ref_tree(acc), lane);
      continue;
    }
    const int segs = (R1 - R0 + 31) / 32;
    if (s >= segs) continue;   // the last item of an external point may be shorter
    const int R = R0 + 32 * s + lane;
    double *buf = a.rowbuf + (size_t)e * rows;
    if (R < R1) {
      int r;
      __stcg(buf + R, ref_row<MODEL>(a, S, kc, e, R, r));
    }
    unsigned done = 0;
    __threadfence();
    __syncwarp();
    if (lane == 0) done = atomicAdd(ref64_item_done(a) + (size_t)e * a.n_chunks + c, 1u);
    done = __shfl_sync(0xffffffffu, done, 0);
    if (done != (unsigned)segs - 1u) continue;
    __threadfence();
    double acc = 0.0;
    const int per_r = rows / a.nr;
    for (int i = R0 + lane; i < R1; i += 32) acc = fma(a.radF[i / per_r], __ldcg(buf + i), acc);
    ref_item_done<MODEL>(a, e, c, ref_tree(acc), lane);
  }
}

size_t ref64_smem(const Plan *pl) { return RefSmem::bytes(pl); }

// Row buffer and item counters (in one allocation) of a plan whose items are fewer than the
// resident warps (optional, not taken in a context with a memory budget:
// without them the items run whole).
void ref64_setup(ffrg_ctx *ctx, Plan *pl) {
  const int items = pl->model == FFRG_MODEL_D3 ? pl->fn_items64 : pl->fn_items;
  if (pl->rowbuf || ctx->budget || items >= 152 * 16) return;
  const int rows = ref64_rows(pl->model, pl->nr, pl->na1, pl->fjb64);
  if (dev_alloc(ctx, (void **)&pl->rowbuf, (size_t)pl->n_ext * rows * sizeof(double) + (size_t)items * sizeof(unsigned)))
    pl->rowbuf = nullptr;
}

// The main kernel after the precompute kernel (which resets the counters).
int launch_ref64(ffrg_ctx *ctx, Plan *pl, const RhsArgs &a, cudaStream_t s) {
  const bool d3 = a.model == FFRG_MODEL_D3;
  void (*kern)(RhsArgs) = a.rowbuf ? (d3 ? ref64_kernel<FFRG_MODEL_D3, true> : ref64_kernel<FFRG_MODEL_D4_VERTEX, true>)
                                   : (d3 ? ref64_kernel<FFRG_MODEL_D3, false> : ref64_kernel<FFRG_MODEL_D4_VERTEX, false>);
  const size_t smem = ref64_smem(pl);
  if (pl->grid_ref == 0) {
    const int irows = d3 ? a.cr : a.cr * a.na1;
    const int st = persistent_grid(ctx, (const void *)kern, smem, a.n_items * (a.rowbuf ? (irows + 31) / 32 : 1),
                                   &pl->grid_ref, kThreads);
    if (st) return st;
  }
  return set_cuda_error(ctx, launch_dependent(kern, dim3(pl->grid_ref), dim3(kThreads), smem, s, true, a),
                        "feedback-flow rhs launch");
}

}  // namespace ffrg
