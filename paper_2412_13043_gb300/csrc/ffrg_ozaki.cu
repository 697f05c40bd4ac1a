// Finite-T sums over many loop-side states sharing one angle-integrated
// kernel K(p, q) (Sec. 5.3.2 momentum integrals; the finite-T RHS is the sum
// over loop frequencies n and radial nodes r of a loop-side factor F(n, r)
// times the angular sum of the shifted line, K[j(n+m)][p][r]):
//
//   out[s][e] = norm sum_{n, r} w_r q_r^2 F_s(n, r) K[j(n + m_e)][p_e][r]
//
// For S states this is one dense product A B^T with A[(m, p)][(n, r)] =
// K[j(n+m)][p][r] (n_ext x nfreq n_rad) and B[s][(n, r)] = w_r q_r^2 F_s(n, r).
// It runs on the tensor cores, FP64-faithful, by an Ozaki-type split:
//   - each row of A and of B is scaled by a power of two 2^-e so that its
//     largest magnitude is below 1, then cut into kSlices fixed-point slices
//     of kBits bits, x = sum_i x_i 2^(-kBits (i+1)), x_0 integer in
//     [-32, 32], x_i in [-16, 16]; the integers are exact in BF16;
//   - up to four slice pairs (i, j) of one level i + j summed over at most 2^13
//     K-elements are an integer below 2^24 in magnitude, exact in the FP32
//     tensor-memory accumulator (ffrg_umma.cuh): one pass; the pairs with i + j
//     < kSlices are kept;
//   - per output, the passes of one level i + j are added as integers
//     (exact), the levels in FP64 from the smallest, and the result scaled by
//     norm 2^(e_row + e_state - 2 kBits).
// The neglected levels and slice residuals are below ~2^-48 of
// max|A_row| max|B_s| per term.
#include <math.h>

#include <algorithm>

#include "ffrg_internal.cuh"
#include "ffrg_umma.cuh"

namespace ffrg {

using umma::kGroups;
using umma::kSlices;
using umma::level_groups;
constexpr int kBits = 5;

struct StatesScratch {
  uint16_t *A, *B;
  float *part;
  int *e_row, *e_col;
};

// |v| as an ordered integer (IEEE bit pattern without the sign)
__device__ __forceinline__ unsigned long long mag_bits(double v) {
  return (unsigned long long)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFull;
}

// exponent e with |x| < 2^e for every |x| whose bit pattern is at most m (0 for m = 0)
__device__ __forceinline__ int scale_exp_bits(unsigned long long m) {
  return m ? (int)(m >> 52) - 1022 : 0;
}

__device__ __forceinline__ unsigned long long block_max_bits(unsigned long long v, unsigned long long *red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
    v = w > v ? w : v;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) red[warp] = v;
  __syncthreads();
  unsigned long long m = 0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = red[w] > m ? red[w] : m;
  __syncthreads();
  return m;
}

// X = round(v 2^(50 - e)) as an integer, |X| <= 2^50 for |v| < 2^e (integer
// operations on the IEEE fields; subnormal v gives 0)
__device__ __forceinline__ long long fixed50(double v, int e) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(v);
  const int E = (int)((u >> 52) & 0x7FF);
  if (E == 0) return 0;
  const long long M = (long long)((u & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull);
  const int sh = E - 1025 - e;           // v 2^(50-e) = M 2^sh
  long long X;
  if (sh >= 0) X = M << sh;
  else if (sh > -54) X = (M + (1ll << (-sh - 1))) >> (-sh);
  else X = 0;
  return (u >> 63) ? -X : X;
}

// slices of the 8 values v[0..7] (scale 2^-e) at K-elements 8g .. 8g + 7 of
// row `row` of a panel with tiles `th` rows high: x = sum_i a_i 2^(-5(i+1)),
// a_0 in [-32, 32], the other digits in [-16, 15]; one
// 16-byte core-matrix row per slice, slice arrays `slice_elems` apart
__device__ __forceinline__ void write_slices8(uint16_t *dst, size_t slice_elems, int k_tiles, int row, int th, int g,
                                              const double (&v)[8], int e) {
  const int col = 8 * g;
  const size_t off = ((size_t)(row / th) * k_tiles + col / umma::kBK) * (size_t)(th * umma::kBK) +
                     umma::tile_offset(row % th, col % umma::kBK, th);
  // Digits by one biased shift: with 16 added at the weight of every slice
  // but the first, the 5-bit fields of X are the digits plus 16.  The integer
  // k - 16 in FP32 is (2^23 + k) - (2^23 + 16), its upper half the BF16 bits.
  constexpr long long kBias = 16ll * (((1ll << (kBits * (kSlices - 1))) - 1) / 31);
  long long X[8];
#pragma unroll
  for (int h = 0; h < 8; ++h) X[h] = fixed50(v[h], e) + kBias;
#pragma unroll
  for (int i = 0; i < kSlices; ++i) {
    const int w = kBits * (kSlices - 1 - i);
    uint32_t pk[4];
#pragma unroll
    for (int h = 0; h < 8; h += 2) {
      float lo, hi;
      if (i == 0) {   // the first slice, in [-32, 32]
        lo = __uint_as_float(0x4B000000u + (uint32_t)((int)(X[h] >> w) + 64)) - 8388672.0f;
        hi = __uint_as_float(0x4B000000u + (uint32_t)((int)(X[h + 1] >> w) + 64)) - 8388672.0f;
      } else {
        lo = __uint_as_float(0x4B000000u | ((uint32_t)(X[h] >> w) & 31u)) - 8388624.0f;
        hi = __uint_as_float(0x4B000000u | ((uint32_t)(X[h + 1] >> w) & 31u)) - 8388624.0f;
      }
      pk[h >> 1] = __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632);
    }
    *reinterpret_cast<uint4 *>(dst + (size_t)i * slice_elems + off) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
  }
}

struct SplitArgs {
  const void *K;          // angle-integrated kernel [N + M][n_p][n_rad], double or float
  int k_double;
  const double *F;        // states [S][nfreq][n_rad] (B split)
  const double *rad_x, *rad_w;  // unit radial rule on [0, 1]
  double qscale;          // k qmax: q_r = qscale x_r
  int n_p, nm, nr, nfreq, n_lo, stat, n_rows, n_cols, kdim, k_tiles;
  uint16_t *A, *B;
  int *e_row, *e_col;
  size_t a_slice, b_slice;  // elements per slice array
};

// one block per row of A (external point e = (p, m); padded rows are zero)
__global__ void __launch_bounds__(256) split_A_kernel(SplitArgs g) {
  __shared__ unsigned long long red[8];
  const int row = blockIdx.x;
  const int kpad = g.k_tiles * umma::kBK;
  const bool live = row < g.n_rows;
  const int ip = live ? row / g.nm : 0, m = live ? row % g.nm : 0;
  auto val = [&](int col) -> double {
    if (!live || col >= g.kdim) return 0.0;
    const int nrow = col / g.nr, r = col - nrow * g.nr;
    const int n = nrow + g.n_lo + m;
    const int j = g.stat ? (n >= 0 ? n : -n - 1) : abs(n);
    const size_t o = ((size_t)j * g.n_p + ip) * g.nr + r;
    return g.k_double ? ((const double *)g.K)[o] : (double)((const float *)g.K)[o];
  };
  unsigned long long mx = 0;
  for (int c = threadIdx.x; c < kpad; c += blockDim.x) {
    const unsigned long long b = mag_bits(val(c));
    mx = b > mx ? b : mx;
  }
  const int e = scale_exp_bits(block_max_bits(mx, red));
  if (threadIdx.x == 0) g.e_row[row] = e;
  for (int q = threadIdx.x; q < kpad / 8; q += blockDim.x) {
    double v[8];
#pragma unroll
    for (int h = 0; h < 8; ++h) v[h] = val(8 * q + h);
    write_slices8(g.A, g.a_slice, g.k_tiles, row, umma::kBM, q, v, e);
  }
}

// one block per 8 states (padded states are zero), four warps a state for its
// largest value, then eight lanes side by side for the eight states' slices of
// the same K-elements: 128 contiguous bytes of a core matrix (a block per
// state wrote 16 bytes here and there: 64 us for 1024 states of 3168 terms,
// 37 so).  Few states leave SMs idle: there the K-elements are shared out over
// gridDim.y blocks, each of which finds the largest values itself.  The state carries the radial weight and measure w_r q_r^2 (from
// the unit rule, staged per block).
constexpr int kStatesPerBlock = 8;
__global__ void __launch_bounds__(1024) split_B_kernel(SplitArgs g) {
  __shared__ unsigned long long red[32];
  extern __shared__ double wq[];   // [n_rad]: (k qmax)^3 w_r x_r^2
  const int kpad = g.k_tiles * umma::kBK, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double q3 = g.qscale * g.qscale * g.qscale;
  for (int r = threadIdx.x; r < g.nr; r += blockDim.x) wq[r] = q3 * g.rad_w[r] * g.rad_x[r] * g.rad_x[r];
  __syncthreads();
  {
    const int s = blockIdx.x * kStatesPerBlock + (warp >> 2);
    unsigned long long mx = 0;
    if (s < g.n_cols)
      for (int c = (warp & 3) * 32 + lane; c < g.kdim; c += 128) {
        const unsigned long long b = mag_bits(wq[c % g.nr] * g.F[(size_t)s * g.kdim + c]);
        mx = b > mx ? b : mx;
      }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long w = __shfl_xor_sync(0xffffffffu, mx, o);
      mx = w > mx ? w : mx;
    }
    if (lane == 0) red[warp] = mx;
  }
  __syncthreads();
  const int row = lane & 7, s = blockIdx.x * kStatesPerBlock + row;
  unsigned long long mx = 0;
  for (int w = 0; w < 4; ++w) mx = red[4 * row + w] > mx ? red[4 * row + w] : mx;
  const int e = scale_exp_bits(mx);
  if (blockIdx.y == 0 && threadIdx.x < kStatesPerBlock) g.e_col[s] = e;
  const double *F = g.F + (size_t)s * g.kdim;
  for (int q = (blockIdx.y * 32 + warp) * 4 + (lane >> 3); q < kpad / 8; q += gridDim.y * 128) {
    double v[8];
    int r = 8 * q % g.nr;
#pragma unroll
    for (int h = 0; h < 8; ++h) {
      v[h] = s < g.n_cols && 8 * q + h < g.kdim ? wq[r] * F[8 * q + h] : 0.0;
      if (++r == g.nr) r = 0;
    }
    write_slices8(g.B, g.b_slice, g.k_tiles, s, umma::kBN, q, v, e);
  }
}

struct CombineArgs {
  const float *part;     // [passes][rows_pad][cols_pad]
  const int *e_row, *e_col;
  double *out;           // [S][n_ext]
  unsigned *status;
  double norm;
  int n_rows, n_cols, rows_pad, cols_pad, n_chunks;
};

// thread per output (state fastest): the passes of a level are exact
// integers (level sums below 3072 x 196608 < 2^31 in all); levels 0..6 and 7..9
// are combined exactly in two 64-bit integers, which one FP64 FMA adds; the
// scale goes into the exponent (FP64 levels and ldexp: 39 us for 576 x 1024
// outputs, 12 so)
__global__ void __launch_bounds__(256) combine_kernel(CombineArgs g) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)g.n_rows * g.n_cols) return;
  const int e = (int)(t / g.n_cols), s = (int)(t % g.n_cols);
  const size_t plane = (size_t)g.rows_pad * g.cols_pad, at = (size_t)e * g.cols_pad + s;
  // the passes in level order: all loads independent
  int lsum[kSlices];
#pragma unroll
  for (int l = 0; l < kSlices; ++l) lsum[l] = 0;
  for (int c = 0; c < g.n_chunks; ++c) {
    float v[kGroups];
#pragma unroll
    for (int p = 0; p < kGroups; ++p) v[p] = g.part[(size_t)(p * g.n_chunks + c) * plane + at];
#pragma unroll
    for (int l = 0, p = 0; l < kSlices; ++l)
#pragma unroll
      for (int i = 0; i < level_groups(l); ++i, ++p) lsum[l] += __float2int_rn(v[p]);
  }
  long long hi = 0, lo = 0;
#pragma unroll
  for (int l = 0; l < kSlices; ++l) {
    if (l > 6) lo += (long long)lsum[l] << (kBits * (9 - l));
    else hi += (long long)lsum[l] << (kBits * (6 - l));
  }
  // (hi 2^15 + lo) 2^-45, scaled by its exponent bits while the result is normal
  const double acc = fma((double)hi, 32768.0, (double)lo);
  const int x = g.e_row[e] + g.e_col[s] - 2 * kBits - 45;
  const long long bits = __double_as_longlong(acc);
  const int be = (int)(bits >> 52) & 0x7FF;
  const double sc = be > 0 && be + x > 0 && be + x < 0x7FF ? __longlong_as_double(bits + ((long long)x << 52)) : ldexp(acc, x);
  const double v = g.norm * sc;
  g.out[(size_t)s * g.n_rows + e] = v;
  if (!isfinite(v)) atomicOr(g.status, kStatusNonFinite);
}

}  // namespace ffrg

using namespace ffrg;

extern "C" int ffrg_ft_states(ffrg_ctx *ctx, const ffrg_problem *pb, const ffrg_tables *tables, double k,
                              int n_states, const double *F_dev, double *out_dev, int precision, void *stream) {
  if (!ctx || !pb || !tables || !F_dev || !out_dev) return FFRG_EINVAL;
  if (pb->model != FFRG_MODEL_FINITE_T || n_states < 1) return FFRG_EINVAL;
  if (!(k > 0.0) || !isfinite(k)) return FFRG_EINVAL;
  if (precision != FFRG_FP64 && precision != FFRG_MIXED) return FFRG_EINVAL;
  int st = validate_problem(pb, &tables->desc);
  if (st) return st;
  cudaSetDevice(ctx->device);
  cudaStream_t s = (cudaStream_t)stream;
  Plan *pl = nullptr;
  st = get_plan(ctx, pb, &tables->desc, &pl);
  if (st) return st;

  // geometry of the product
  const int n_rows = pl->n_ext, kdim = pl->nfreq * pl->nr;
  const int m_tiles = (n_rows + umma::kBM - 1) / umma::kBM;
  const int n_tiles = (n_states + umma::kBN - 1) / umma::kBN;
  const int k_tiles = (kdim + umma::kBK - 1) / umma::kBK;
  // K ranges: as many as exactness needs, and where the tiles are too few for
  // two blocks on each SM up to 16, of 128 elements or more (34 states, 725 terms:
  // 512 69 us, 256 59, 128 57) (the sums are
  // integers: any cut gives the same bits).  576 external points x 3168 terms:
  // 256 states 305 us for the call with one range, 242 with four; 512 states
  // 319, with two 287; 1024 states need no more than one.  Their sums are
  // optional scratch, so one range in a context with a memory budget.
  const int fill = ctx->budget ? 1 : std::min((2 * ctx->num_sms - 1) / (m_tiles * n_tiles * kGroups) + 1, 16);
  const int kt_chunk = std::min({k_tiles, umma::kMaxExactK / umma::kBK, std::max(4, (k_tiles + fill - 1) / fill)});
  const int n_chunks = (k_tiles + kt_chunk - 1) / kt_chunk;
  if (k_tiles > 196608 / umma::kBK) {   // level sums must fit 32-bit integers
    ctx->last_error = "ffrg_ft_states: more than 196608 (loop frequency, radial node) terms";
    return FFRG_EINVAL;
  }
  const int passes = kGroups * n_chunks;
  const int rows_pad = m_tiles * umma::kBM, cols_pad = n_tiles * umma::kBN;
  const size_t a_slice = (size_t)rows_pad * k_tiles * umma::kBK, b_slice = (size_t)cols_pad * k_tiles * umma::kBK;

  // K in the requested precision (the finite-T RHS up to, not including, its contraction)
  RhsArgs a;
  fill_args(pl, pb, &tables->desc, tables->dev, k, a);
  a.out = out_dev;   // not written: no contraction
  a.status = ctx->status_dev;
  const int prof_on = ctx->profiling;   // the profiling events time the tensor-core kernel only
  ctx->profiling = 0;
  st = launch_rhs_stages(ctx, pl, a, precision, s, false);
  ctx->profiling = prof_on;
  if (st) return st;

  // scratch, kept by the context and grown on demand (256-byte segments):
  // A slices | B slices | pass sums | scales
  auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
  const size_t o_B = al(kSlices * a_slice * 2), o_part = o_B + al(kSlices * b_slice * 2);
  const size_t o_er = o_part + al((size_t)passes * rows_pad * cols_pad * 4);
  const size_t o_ec = o_er + al((size_t)rows_pad * 4);
  const size_t need = o_ec + al((size_t)cols_pad * 4);
  if (ctx->states_cap < need) {
    dev_free(ctx, ctx->states_dev, ctx->states_cap);
    ctx->states_dev = nullptr;
    ctx->states_cap = 0;
    st = dev_alloc(ctx, &ctx->states_dev, need);
    if (st) return st;
    ctx->states_cap = need;
  }
  unsigned char *base = (unsigned char *)ctx->states_dev;
  StatesScratch sc{(uint16_t *)base, (uint16_t *)(base + o_B), (float *)(base + o_part), (int *)(base + o_er),
                   (int *)(base + o_ec)};

  SplitArgs sg;
  sg.K = pl->kbuf;
  sg.k_double = precision == FFRG_FP64;
  sg.F = F_dev;
  sg.rad_x = pl->rad_x;
  sg.rad_w = pl->rad_w;
  sg.qscale = k * pb->qmax_over_k;
  sg.n_p = pl->n_ext_p;
  sg.nm = pl->n_ext_ang;
  sg.nr = pl->nr;
  sg.nfreq = pl->nfreq;
  sg.n_lo = -pl->N - pl->stat;
  sg.stat = pl->stat;
  sg.n_rows = n_rows;
  sg.n_cols = n_states;
  sg.kdim = kdim;
  sg.k_tiles = k_tiles;
  sg.A = sc.A;
  sg.B = sc.B;
  sg.e_row = sc.e_row;
  sg.e_col = sc.e_col;
  sg.a_slice = a_slice;
  sg.b_slice = b_slice;
  split_A_kernel<<<rows_pad, 256, 0, s>>>(sg);
  const int b_blocks = cols_pad / kStatesPerBlock;
  split_B_kernel<<<dim3(b_blocks, std::max(1, ctx->num_sms / b_blocks)), 1024, (size_t)pl->nr * sizeof(double), s>>>(sg);

  st = ensure_smem_limit(ctx, (const void *)umma::slice_pair_gemm, umma::kSmemBytes);
  if (st) return st;
  constexpr umma::PairGroups kPairGroups = umma::pair_groups();
  umma::GemmArgs gg{sc.A, sc.B, sc.part, m_tiles, n_tiles, k_tiles, kt_chunk, n_chunks, ctx->status_dev, kPairGroups};
  const bool prof = ctx->profiling && ctx->prof_used * 2 + 1 < (int)ctx->prof_events.size();
  if (prof) cudaEventRecord(ctx->prof_events[2 * ctx->prof_used], s);
  umma::slice_pair_gemm<<<dim3(n_tiles, m_tiles, passes), umma::kThreadsGemm, umma::kSmemBytes, s>>>(gg);
  if (prof) {
    cudaEventRecord(ctx->prof_events[2 * ctx->prof_used + 1], s);
    ctx->prof_used++;
  }

  CombineArgs cg{sc.part, sc.e_row, sc.e_col, out_dev, ctx->status_dev, a.norm, n_rows, n_states, rows_pad,
                 cols_pad, n_chunks};
  const long long n_out = (long long)n_rows * n_states;
  combine_kernel<<<(unsigned)((n_out + 255) / 256), 256, 0, s>>>(cg);
  return set_cuda_error(ctx, cudaGetLastError(), "ffrg_ft_states launch");
}
