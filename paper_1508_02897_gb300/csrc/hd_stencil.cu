// Medium and PML tables (setup) and the global complex 5-point operator.
//
// Discretisation (Sec. 2, Eq. (pml); Sec. 3 "second order finite difference"):
// the operator J^{-1} div(A grad u) + k^2 u, A = diag(alpha2/alpha1,
// alpha1/alpha2), J = alpha1 alpha2, is multiplied by J h^2 and discretised in
// conservative form, giving the complex-symmetric row
//   west  alpha2(y_j) / alpha1(x_{i-1/2})     east  alpha2(y_j) / alpha1(x_{i+1/2})
//   south alpha1(x_i) / alpha2(y_{j-1/2})     north alpha1(x_i) / alpha2(y_{j+1/2})
//   centre -(sum of the four) + h^2 alpha1(x_i) alpha2(y_j) k^2(x_i, y_j)
// with zero (Dirichlet) values outside the box.  The same row builder serves
// the global operator and, in the factorisation, the local operators of
// Eq. (pmlij) with the box's own PML tables.
#include <algorithm>

#include "hd_internal.cuh"

namespace hd {

// alpha = 1 + i s0 (xi / npml)^p at position `pos` (cell units) of a segment
// of `ncell` cells whose first and last `npml` cells are PML (Sec. 2: sigma = 0
// inside, > 0 in the layer; xi = distance into the layer).
__device__ __forceinline__ double2 pml_alpha(double pos, int ncell, int npml, double s0, int power) {
  if (npml <= 0) return make_double2(1.0, 0.0);
  double lo = (double)npml, hi = (double)(ncell - npml);
  double xi = pos < lo ? lo - pos : (pos > hi ? pos - hi : 0.0);
  double t = xi / (double)npml, p = 1.0;
  for (int e = 0; e < power; ++e) p *= t;
  return make_double2(1.0, s0 * p);
}

// Fills, for a segment of ncell cells: centre alphas a_c[ncell] and the
// reciprocals of the face alphas ia_f[ncell+1].
__device__ void fill_segment(double2 *a_c, double2 *ia_f, int ncell, int npml, double s0, int power, int t, int nt) {
  for (int l = t; l < ncell; l += nt) a_c[l] = pml_alpha(l + 0.5, ncell, npml, s0, power);
  for (int f = t; f <= ncell; f += nt) ia_f[f] = cinv(pml_alpha((double)f, ncell, npml, s0, power));
}

__global__ void k_global_tables(double2 *ax_c, double2 *iax_f, double2 *ay_c, double2 *iay_f, int NX, int NY,
                                int npml, double s0, int power) {
  int t = threadIdx.x, nt = blockDim.x;
  if (blockIdx.x == 0) fill_segment(ax_c, iax_f, NX, npml, s0, power, t, nt);
  else fill_segment(ay_c, iay_f, NY, npml, s0, power, t, nt);
}

// Per box: the PML of Omega_ij itself (its outer npml cells on every side).
__global__ void k_local_tables(const SubDev *subs, double2 *pool, float2 *poolf, int npml, double s0, int power) {
  const SubDev s = subs[blockIdx.x];
  double2 *a1c = pool + s.aoff;
  double2 *ia1f = a1c + s.ex;
  double2 *a2c = ia1f + s.ex + 1;
  double2 *ia2f = a2c + s.ey;
  fill_segment(a1c, ia1f, s.ex, npml, s0, power, threadIdx.x, blockDim.x);
  fill_segment(a2c, ia2f, s.ey, npml, s0, power, threadIdx.x, blockDim.x);
  __syncthreads();
  for (int i = threadIdx.x; i < 2 * s.ex + 2 * s.ey + 2; i += blockDim.x)
    poolf[s.aoff + i] = make_float2((float)a1c[i].x, (float)a1c[i].y);
}

// k^2 = (omega / c)^2 per cell, and the centre coefficient h^2 k^2 - 4 that A has
// wherever both alphas are 1 (outside the PML).
__global__ void k_wavenumber(const double *__restrict__ c, double *__restrict__ k2, double *__restrict__ cc,
                             int64_t n, double omega, double h2, int32_t *status) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  double ci = c[i];
  double k = omega / ci;
  if (!(ci > 0.0) || !isfinite(k)) atomicOr(status, ST_NONFINITE);
  const double kk = k * k;
  k2[i] = kk;
  cc[i] = add_rn(mul_rn(h2, kk), -4.0);
}

cudaError_t launch_setup_tables(hd_ctx *ctx, const double *c_dev, cudaStream_t st) {
  k_global_tables<<<2, 256, 0, st>>>(ctx->d_gax_c, ctx->d_giax_f, ctx->d_gay_c, ctx->d_giay_f, ctx->NX, ctx->NY,
                                     ctx->npml, ctx->s0, ctx->power);
  k_local_tables<<<ctx->nsub, 256, 0, st>>>(ctx->d_subs, ctx->d_lpool, ctx->d_lpoolf, ctx->npml, ctx->s0, ctx->power);
  int64_t n = (int64_t)ctx->NX * ctx->NY;
  k_wavenumber<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(c_dev, ctx->d_k2, ctx->d_cc, n, ctx->omega,
                                                             ctx->h * ctx->h, ctx->d_status);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- operator
struct OpArgs {
  const double2 *ax_c, *iax_f, *ay_c, *iay_f;
  const double *k2, *cc;
  int NX, NY, npml;
  double h2;
};

// y = A x (MODE 0) or y = b - A x (MODE 1), one grid per blockIdx.z.
//
// Outside the PML every alpha is 1 and a row is x_W + x_E + x_S + x_N + cc x_C with the stored
// centre cc = h^2 k^2 - 4: few bytes per cell, and FP64 runs at 1/64 of FP32, so the FP64 pipe
// bounds it (two thirds above the time of its bytes).  The sum is taken as
// (x_S + x_E + cc x_C) + (x_W + x_N): x_S + x_E of cell (i, j) is x_W + x_N of cell (i + 1, j - 1),
// so a warp that walks down the grid forms each pair once and passes it to the lane on its left,
// and a cell costs two additions and one FMA per component instead of three and one.  The centre
// joins one pair before the pairs meet: for a wave the two halves nearly cancel, and their sum
// is exact or close to it, where x_W + x_N + x_S + x_E would be rounded at four times the wave's size
// first.  (Error against extended precision on waves of 10 to 20 cells, relative to the four
// neighbours added one by one to cc x_C: 0.96 to 1.08, with the four summed first 1.31 to 1.5;
// on white noise 0.77.)
// A warp takes ST_COLS columns (its last lane only forms pairs) and `R` rows; every entry of x is
// loaded once per tile.  The tiles fill the part outside the PML from its lower corner; the frame
// around them (the PML and what is left of a tile) takes the general form, a thread per cell.
// 4096^2: 300 -> 225 us (FP64 pipe 78 % busy); 1024^2: 36 -> 25 us.
constexpr int ST_COLS = 31, ST_WARPS = 8;

// p = x_S + x_E, q = x_W + x_N (in a tile p is there a row before q)
template <int MODE> __device__ __forceinline__ double2 stencil_end(double cc, double2 xc, double2 p, double2 q, double2 b) {
  const double2 y = cadd(make_double2(__fma_rn(cc, xc.x, p.x), __fma_rn(cc, xc.y, p.y)), q);
  return MODE == 1 ? csub(b, y) : y;
}

// One cell anywhere in the grid.
template <int MODE>
__device__ __forceinline__ void stencil_cell(const OpArgs &a, const double2 *__restrict__ x, const double2 *__restrict__ b,
                                             double2 *__restrict__ y, int i, int j) {
  const int64_t idx = (int64_t)j * a.NX + i;
  const double2 zero = make_double2(0.0, 0.0);
  const double2 xc = x[idx];
  const double2 xw = i > 0 ? x[idx - 1] : zero, xe = i + 1 < a.NX ? x[idx + 1] : zero;
  const double2 xs = j > 0 ? x[idx - a.NX] : zero, xn = j + 1 < a.NY ? x[idx + a.NX] : zero;
  if (i >= a.npml && i < a.NX - a.npml && j >= a.npml && j < a.NY - a.npml) {
    y[idx] = stencil_end<MODE>(a.cc[idx], xc, cadd(xs, xe), cadd(xw, xn), MODE == 1 ? b[idx] : zero);
    return;
  }
  const double2 a1 = a.ax_c[i], a2 = a.ay_c[j];
  double2 cw = a.iax_f[i], ce = a.iax_f[i + 1], cs = a.iay_f[j], cn = a.iay_f[j + 1], j12;
  if (j >= a.npml && j < a.NY - a.npml) {          // only x in the PML: the alphas of y are 1
    cs = cn = j12 = a1;
  } else if (i >= a.npml && i < a.NX - a.npml) {   // only y
    cw = ce = j12 = a2;
  } else {
    cw = cmul(a2, cw);
    ce = cmul(a2, ce);
    cs = cmul(a1, cs);
    cn = cmul(a1, cn);
    j12 = cmul(a1, a2);
  }
  const double hk = mul_rn(a.h2, a.k2[idx]);
  const double2 cc = make_double2(-(cw.x + ce.x + cs.x + cn.x) + hk * j12.x, -(cw.y + ce.y + cs.y + cn.y) + hk * j12.y);
  double2 acc = cmul(cc, xc);
  acc = cfma(cw, xw, acc);
  acc = cfma(ce, xe, acc);
  acc = cfma(cs, xs, acc);
  acc = cfma(cn, xn, acc);
  if (MODE == 1) acc = csub(b[idx], acc);
  y[idx] = acc;
}

__device__ __forceinline__ double2 shfl_up1(double2 v) {
  return make_double2(__shfl_up_sync(0xffffffffu, v.x, 1), __shfl_up_sync(0xffffffffu, v.y, 1));
}
__device__ __forceinline__ double2 shfl_down1(double2 v) {
  return make_double2(__shfl_down_sync(0xffffffffu, v.x, 1), __shfl_down_sync(0xffffffffu, v.y, 1));
}

// The tiled part [x0, x0 + ST_COLS ntx) x [y0, y0 + R nty), and the cells around it.
struct StencilTiles {
  int x0, y0, ntx, nty, x1, y1;
  int64_t low, high;     // frame cells below y0 (whole rows), from y1 on
  int side, nframe;      // frame cells per row between, blocks of the frame
};

template <int MODE, int R>
__global__ void __launch_bounds__(32 * ST_WARPS) k_stencil(OpArgs a, StencilTiles q, const double2 *__restrict__ x_all,
                                                           int64_t xs_, const double2 *__restrict__ b_all, int64_t bs_,
                                                           double2 *__restrict__ y_all, int64_t ys_) {
  const double2 *x = x_all + (int64_t)blockIdx.z * xs_;
  const double2 *b = MODE == 1 ? b_all + (int64_t)blockIdx.z * bs_ : nullptr;
  double2 *y = y_all + (int64_t)blockIdx.z * ys_;
  const int lane = threadIdx.x;
  if ((int)blockIdx.x < q.nframe) {
    int64_t t = (int64_t)blockIdx.x * (32 * ST_WARPS) + threadIdx.y * 32 + lane;
    int i, j;
    if (t < q.low + q.high) {
      const int64_t u = t < q.low ? t : t - q.low;
      j = (int)(u / a.NX);
      i = (int)(u - (int64_t)j * a.NX);
      if (t >= q.low) j += q.y1;
    } else {
      t -= q.low + q.high;
      if (q.side == 0) return;
      j = (int)(t / q.side);
      i = (int)(t - (int64_t)j * q.side);
      j += q.y0;
      if (i >= q.x0) i += q.x1 - q.x0;
      if (j >= q.y1) return;
    }
    stencil_cell<MODE>(a, x, b, y, i, j);
    return;
  }
  const int tile = ((int)blockIdx.x - q.nframe) * ST_WARPS + threadIdx.y;
  if (tile >= q.ntx * q.nty) return;
  const int ty = tile / q.ntx, c0 = q.x0 + ST_COLS * (tile - ty * q.ntx), j0 = q.y0 + R * ty;
  const int i = c0 + lane;
  // lane 0 also loads the column on its left
  auto west = [&](const double2 *p, double2 v) {
    double2 u = shfl_up1(v);
    if (lane == 0) u = p[-1];
    return u;
  };
  const double2 *p = x + (int64_t)(j0 - 1) * a.NX + i;
  const double *pc = a.cc + (int64_t)j0 * a.NX + i;
  const double2 *pb = MODE == 1 ? b + (int64_t)j0 * a.NX + i : nullptr;
  double2 *py = y + (int64_t)j0 * a.NX + i;
  const double2 x0 = p[0];
  p += a.NX;
  double2 xc = p[0];
  double2 d = cadd(west(p - a.NX, x0), xc);   // x_W + x_N of the row above the tile
#pragma unroll 4
  for (int r = 0; r < R; ++r) {
    const double2 xn = p[a.NX];
    const double cc = pc[0];
    const double2 bv = MODE == 1 ? pb[0] : make_double2(0.0, 0.0);
    const double2 e = shfl_down1(d);   // x_S + x_E of this cell
    d = cadd(west(p, xc), xn);
    if (lane < ST_COLS) py[0] = stencil_end<MODE>(cc, xc, e, d, bv);
    xc = xn;
    p += a.NX;
    pc += a.NX;
    py += a.NX;
    if (MODE == 1) pb += a.NX;
  }
}

static OpArgs op_args(hd_ctx *ctx) {
  OpArgs a;
  a.ax_c = ctx->d_gax_c; a.iax_f = ctx->d_giax_f; a.ay_c = ctx->d_gay_c; a.iay_f = ctx->d_giay_f;
  a.k2 = ctx->d_k2; a.cc = ctx->d_cc; a.NX = ctx->NX; a.NY = ctx->NY; a.npml = ctx->npml; a.h2 = ctx->h * ctx->h;
  return a;
}

template <int MODE>
static cudaError_t launch_stencil(hd_ctx *ctx, const double2 *x, int64_t xs, const double2 *b, int64_t bs, double2 *y,
                                  int64_t ys, int nrhs, cudaStream_t st) {
  // 16 rows per warp re-read an eighth of x and form a sixteenth of the pairs twice; smaller grids
  // take 8 or 4 rows to have enough warps (1024^2: 26 / 29 us with 8 / 16)
  const int64_t cells = (int64_t)ctx->NX * ctx->NY * nrhs;
  const int R = cells < 1 << 20 ? 4 : (cells < 1 << 23 ? 8 : 16), p = std::max(ctx->npml, 1);   // a tile's neighbours are cells of the grid
  StencilTiles q;
  q.x0 = q.y0 = p;
  q.ntx = std::max(0, (ctx->NX - 2 * p) / ST_COLS);
  q.nty = std::max(0, (ctx->NY - 2 * p) / R);
  if (q.ntx == 0 || q.nty == 0) { q.ntx = q.nty = 0; q.x0 = 0; q.y0 = 0; }
  q.x1 = q.x0 + ST_COLS * q.ntx;
  q.y1 = q.y0 + R * q.nty;
  q.low = (int64_t)q.y0 * ctx->NX;
  q.high = (int64_t)(ctx->NY - q.y1) * ctx->NX;
  q.side = ctx->NX - (q.x1 - q.x0);
  const int per = 32 * ST_WARPS;
  q.nframe = (int)((q.low + q.high + (int64_t)(q.y1 - q.y0) * q.side + per - 1) / per);
  const dim3 grid(q.nframe + (q.ntx * q.nty + ST_WARPS - 1) / ST_WARPS, 1, nrhs), block(32, ST_WARPS);
  if (R == 4) k_stencil<MODE, 4><<<grid, block, 0, st>>>(op_args(ctx), q, x, xs, b, bs, y, ys);
  else if (R == 8) k_stencil<MODE, 8><<<grid, block, 0, st>>>(op_args(ctx), q, x, xs, b, bs, y, ys);
  else k_stencil<MODE, 16><<<grid, block, 0, st>>>(op_args(ctx), q, x, xs, b, bs, y, ys);
  return cudaGetLastError();
}

cudaError_t launch_matvec(hd_ctx *ctx, const double2 *x, int64_t xs, double2 *y, int64_t ys, int nrhs,
                          cudaStream_t st) {
  return launch_stencil<0>(ctx, x, xs, nullptr, 0, y, ys, nrhs, st);
}

cudaError_t launch_residual(hd_ctx *ctx, const double2 *b, const double2 *x, double2 *r, int nrhs, cudaStream_t st) {
  const int64_t n = (int64_t)ctx->NX * ctx->NY;
  return launch_stencil<1>(ctx, x, n, b, n, r, n, nrhs, st);
}

cudaError_t launch_residual_strided(hd_ctx *ctx, const double2 *b, int64_t bs, const double2 *x, int64_t xs,
                                    double2 *r, int64_t rs, int nrhs, cudaStream_t st) {
  return launch_stencil<1>(ctx, x, xs, b, bs, r, rs, nrhs, st);
}

__global__ void k_rhs(OpArgs a, const double2 *f, double2 *b) {  // b may alias f
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int j = blockIdx.y;
  if (i >= a.NX) return;
  int64_t idx = (int64_t)j * a.NX + i;
  double2 jac = cmul(a.ax_c[i], a.ay_c[j]);
  double2 v = cmul(jac, f[idx]);
  b[idx] = make_double2(a.h2 * v.x, a.h2 * v.y);
}

cudaError_t launch_rhs(hd_ctx *ctx, const double2 *f, double2 *b, cudaStream_t st) {
  dim3 grid((ctx->NX + 255) / 256, ctx->NY);
  k_rhs<<<grid, 256, 0, st>>>(op_args(ctx), f, b);
  return cudaGetLastError();
}

}  // namespace hd
