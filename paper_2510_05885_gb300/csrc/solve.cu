// FP64 residual, refinement vectors, adjoint, slack-form and Newton-step
// kernels (sm_103a).  The residual r = b - K x is computed on the FP64 KKT
// values for iterative refinement (Section 4.3).
#include "runtime.h"
#include "reduce.cuh"

#include <algorithm>

namespace ncl {

static unsigned grid_for(int64_t n, int per = 256) {
  int64_t b = (n + per - 1) / per;
  if (b > 152 * 16) b = 152 * 16;
  if (b < 1) b = 1;
  return (unsigned)b;
}

// ---------------------------------------------------------------------------
// FP64 residual R = B - K X on the FP64 KKT values, with per-instance
// ||R||_inf and ||X||_inf (bit patterns, atomicMax).  Kf holds the values of
// the full pattern in its row order (written before ||K||), so the entries
// and column indices are read contiguously and only X is gathered.  Each warp
// takes a contiguous run of rows, so that its running maxima change instance
// (and go to the atomics) only at an instance boundary.
//
// One right-hand side: 4 lanes per row, 8 rows per warp trip; every load of a
// trip that does not depend on another (row bounds, B, the row's own X) is
// issued before the products.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_residual(DevPlan P, const double* __restrict__ Kf,
                                                  const double* __restrict__ B, const double* __restrict__ X,
                                                  double* __restrict__ R, unsigned long long* rnorm,
                                                  unsigned long long* xnorm, int64_t rows_per_warp) {
  constexpr int LPR = 4;   // lanes per row
  const int lane = threadIdx.x & 31, sub = lane & (LPR - 1);
  const int64_t gwarp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t r_begin = gwarp * rows_per_warp;
  const int64_t r_end = min(P.dim, r_begin + rows_per_warp);
  // running maxima of |r| and |x| for the instance of this lane's rows
  int cur = -1;
  unsigned long long rmx = 0ull, xmx = 0ull;
  // the trip count is uniform across the warp so that the full-mask
  // shuffles are safe
  for (int64_t rb = r_begin; rb < r_end; rb += 32 / LPR) {
    const int64_t row = rb + lane / LPR;
    const bool valid = row < r_end;
    const int64_t q0 = valid ? P.F_rowptr[row] : 0, q1 = valid ? P.F_rowptr[row + 1] : 0;
    const int inst = valid ? P.row_inst[row] : -1;
    const bool use = valid && sub == 0;
    const double bv = use ? B[row] : 0.0, xv = use ? X[row] : 0.0;
    double acc = 0.0;
    int64_t q = q0 + sub;
    for (; q + LPR < q1; q += 2 * LPR) {
      const double k0 = Kf[q], k1 = Kf[q + LPR];
      const int64_t c0 = P.F_col[q], c1 = P.F_col[q + LPR];
      acc = fma(k1, X[c1], fma(k0, X[c0], acc));
    }
    if (q < q1) acc = fma(Kf[q], X[P.F_col[q]], acc);
    if (use && inst != cur) {
      if (cur >= 0) {
        atomicMax(&rnorm[cur], rmx);
        atomicMax(&xnorm[cur], xmx);
      }
      rmx = xmx = 0ull;
      cur = inst;
    }
    acc += __shfl_xor_sync(FULL_MASK, acc, 2);
    acc += __shfl_xor_sync(FULL_MASK, acc, 1);
    if (use) {
      const double res = bv - acc;
      R[row] = res;
      const unsigned long long u = dbits(fabs(res)), v = dbits(fabs(xv));
      rmx = u > rmx ? u : rmx;
      xmx = v > xmx ? v : xmx;
    }
  }
  warp_flush_max(rnorm, cur, rmx);
  warp_flush_max(xnorm, cur, xmx);
}

// Several right-hand sides: one lane per (row, right-hand side), 32 / NR rows
// per warp trip.  FP64 runs at two products per clock and SM here, so what
// counts is the number of FP64 warp instructions: a lane that owns its sum
// needs no additions across lanes and no idle lanes at the end of a row.
// With 4 lanes per row that each carried all right-hand sides: 64 scenarios
// of 100 buses, 4 of them: 1.42 -> 0.91 ms; 300x300, 8 of them: 0.45 ->
// 0.29 ms (0.7 TFLOP/s).  Gathering X from an interleaved copy instead gave
// nothing (0.96 and 0.28 ms with the copy): the gathers are not the bound.
template <int NR>
__global__ void __launch_bounds__(256) k_residual_rhs(DevPlan P, const double* __restrict__ Kf,
                                                      const double* __restrict__ B, int64_t ldb,
                                                      const double* __restrict__ X, int64_t ldx,
                                                      double* __restrict__ R, int64_t ldr, int nrhs,
                                                      unsigned long long* rnorm, unsigned long long* xnorm,
                                                      int64_t rows_per_warp) {
  constexpr int U = 4;   // entries in flight
  const int lane = threadIdx.x & 31, r = lane & (NR - 1);
  const int64_t gwarp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t r_begin = gwarp * rows_per_warp;
  const int64_t r_end = min(P.dim, r_begin + rows_per_warp);
  const double* Xr = X + min(r, nrhs - 1) * ldx;
  int key = -1;   // instance * nrhs + right-hand side of the running maxima
  unsigned long long rmx = 0ull, xmx = 0ull;
  if (r < nrhs)
    for (int64_t row = r_begin + lane / NR; row < r_end; row += 32 / NR) {
      const int64_t q0 = P.F_rowptr[row], q1 = P.F_rowptr[row + 1];
      const int k = P.row_inst[row] * nrhs + r;
      const double bv = B[r * ldb + row], xv = Xr[row];
      double a0 = 0.0, a1 = 0.0;
      for (int64_t q = q0; q < q1; q += U) {
        double kv[U], x[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
          kv[u] = q + u < q1 ? Kf[q + u] : 0.0;
          x[u] = q + u < q1 ? Xr[P.F_col[q + u]] : 0.0;
        }
        a0 = fma(kv[0], x[0], a0);
#pragma unroll
        for (int u = 1; u < U; u++)
          if (q + u < q1) {
            if (u & 1) a1 = fma(kv[u], x[u], a1);
            else a0 = fma(kv[u], x[u], a0);
          }
      }
      if (k != key) {
        if (key >= 0) {
          atomicMax(&rnorm[key], rmx);
          atomicMax(&xnorm[key], xmx);
        }
        rmx = xmx = 0ull;
        key = k;
      }
      const double res = bv - (a0 + a1);
      R[r * ldr + row] = res;
      const unsigned long long u = dbits(fabs(res)), v = dbits(fabs(xv));
      rmx = u > rmx ? u : rmx;
      xmx = v > xmx ? v : xmx;
    }
  // lanes of one right-hand side and one instance go to memory together
  const int k0 = __shfl_sync(FULL_MASK, key, r);
  const bool same = key == k0;
  unsigned long long rw = same ? rmx : 0ull, xw = same ? xmx : 0ull;
#pragma unroll
  for (int o = 16; o >= NR; o >>= 1) {
    const unsigned long long u = __shfl_xor_sync(FULL_MASK, rw, o), v = __shfl_xor_sync(FULL_MASK, xw, o);
    rw = u > rw ? u : rw;
    xw = v > xw ? v : xw;
  }
  if (key >= 0 && (lane < NR || !same)) {
    atomicMax(&rnorm[key], same ? rw : rmx);
    atomicMax(&xnorm[key], same ? xw : xmx);
  }
}

void launch_residual(const DevPlan& P, const double* Kf, const double* B, int64_t ldb, const double* X,
                     int64_t ldx, double* R, int64_t ldr, int nrhs, unsigned long long* rnorm,
                     unsigned long long* xnorm, cudaStream_t st) {
  if (P.dim == 0) return;
  const unsigned grid = grid_for(P.dim * 8);
  const int64_t nwarp = (int64_t)grid * 8;
  const int64_t rpw = ((P.dim + nwarp - 1) / nwarp + 7) / 8 * 8;
  if (nrhs <= 1) {
    k_residual<<<grid, 256, 0, st>>>(P, Kf, B, X, R, rnorm, xnorm, rpw);
    return;
  }
  const auto k = nrhs <= 2 ? k_residual_rhs<2> : nrhs <= 4 ? k_residual_rhs<4> : k_residual_rhs<8>;
  k<<<grid, 256, 0, st>>>(P, Kf, B, ldb, X, ldx, R, ldr, nrhs, rnorm, xnorm, rpw);
}

// per-instance ||B||_inf; each CTA takes a contiguous run of rows (see k_knorm)
__global__ void k_vec_norm(DevPlan P, const double* __restrict__ B, int64_t ldb, int nrhs, unsigned long long* out,
                           int64_t rows_per_cta) {
  const int64_t i_begin = blockIdx.x * rows_per_cta, i_end = min(P.dim, i_begin + rows_per_cta);
  for (int r = 0; r < nrhs; r++) {
    int cur = -1;
    unsigned long long mx = 0ull;
    for (int64_t i = i_begin + threadIdx.x; i < i_end; i += blockDim.x) {
      const int inst = P.row_inst[i];
      const unsigned long long v = dbits(fabs(B[r * ldb + i]));
      if (inst != cur) {
        if (cur >= 0) atomicMax(&out[cur * nrhs + r], mx);
        cur = inst;
        mx = 0ull;
      }
      mx = v > mx ? v : mx;
    }
    warp_flush_max(out + r, cur < 0 ? -1 : cur * nrhs, mx);
  }
}

void launch_vec_norm(const DevPlan& P, const double* B, int64_t ldb, int nrhs, unsigned long long* out,
                     cudaStream_t st) {
  if (P.dim == 0) return;
  const unsigned grid = grid_for(P.dim);
  k_vec_norm<<<grid, 256, 0, st>>>(P, B, ldb, nrhs, out, (P.dim + grid - 1) / grid);
}

__global__ void k_axpy(double* X, int64_t ldx, const double* Y, int64_t ldy, double a, int64_t dim, int nrhs) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < dim; i += (int64_t)gridDim.x * blockDim.x)
    for (int r = 0; r < nrhs; r++) X[r * ldx + i] += a * Y[r * ldy + i];
}

void launch_axpy_inplace(double* X, int64_t ldx, const double* Y, int64_t ldy, double a, int64_t dim, int nrhs,
                         cudaStream_t st) {
  if (dim) k_axpy<<<grid_for(dim), 256, 0, st>>>(X, ldx, Y, ldy, a, dim, nrhs);
}

// ---------------------------------------------------------------------------
// FP64 vector kernels of the FGMRES refinement (single instance).
// Reductions are two-pass with a fixed grid: per-block partial sums here,
// summed on the host in block order (bitwise reproducible).
// ---------------------------------------------------------------------------
constexpr int VGRID = 256;

// Y = K X (full FP64 CSR)
__global__ void k_spmv(DevPlan P, const double* __restrict__ Klow, const double* __restrict__ X,
                       double* __restrict__ Y) {
  const int lane = threadIdx.x & 31, sub = lane & 7;
  const int64_t gwarp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t rb = gwarp * 4; rb < P.dim; rb += nwarp * 4) {
    const int64_t row = rb + (lane >> 3);
    const bool valid = row < P.dim;
    const int64_t q0 = valid ? P.F_rowptr[row] : 0, q1 = valid ? P.F_rowptr[row + 1] : 0;
    double acc = 0.0;
    for (int64_t q = q0 + sub; q < q1; q += 8) acc = fma(Klow[P.F_src[q]], X[P.F_col[q]], acc);
    acc += __shfl_xor_sync(0xffffffffu, acc, 4);
    acc += __shfl_xor_sync(0xffffffffu, acc, 2);
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    if (valid && sub == 0) Y[row] = acc;
  }
}

// partial[i * VGRID + block] = sum over the block's slice of V_i . w  (i < nv)
__global__ void __launch_bounds__(256) k_multidot(int64_t n, const double* __restrict__ V, int64_t ldv, int nv,
                                                  const double* __restrict__ w, double* __restrict__ partial) {
  __shared__ double red[256];
  const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
  const int64_t lo = blockIdx.x * chunk, hi = min(n, lo + chunk);
  for (int i = 0; i < nv; i++) {
    double acc = 0.0;
    for (int64_t e = lo + threadIdx.x; e < hi; e += blockDim.x) acc = fma(V[i * ldv + e], w[e], acc);
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
      if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
      __syncthreads();
    }
    if (threadIdx.x == 0) partial[i * VGRID + blockIdx.x] = red[0];
    __syncthreads();
  }
}

// w = a * w + sum_i c[i] V_i   (c on the device)
__global__ void k_multi_axpy(int64_t n, const double* __restrict__ V, int64_t ldv, int nv,
                             const double* __restrict__ c, double a, double* __restrict__ w) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    double acc = a != 0.0 ? a * w[e] : 0.0;
    for (int i = 0; i < nv; i++) acc = fma(c[i], V[i * ldv + e], acc);
    w[e] = acc;
  }
}

void launch_spmv(const DevPlan& P, const double* Klow, const double* X, double* Y, cudaStream_t st) {
  if (P.dim) k_spmv<<<grid_for(P.dim * 8), 256, 0, st>>>(P, Klow, X, Y);
}
void launch_multidot(int64_t n, const double* V, int64_t ldv, int nv, const double* w, double* partial,
                     cudaStream_t st) {
  if (nv > 0) k_multidot<<<VGRID, 256, 0, st>>>(n, V, ldv, nv, w, partial);
}
void launch_multi_axpy(int64_t n, const double* V, int64_t ldv, int nv, const double* c, double a, double* w,
                       cudaStream_t st) {
  k_multi_axpy<<<grid_for(n), 256, 0, st>>>(n, V, ldv, nv, c, a, w);
}
int vec_grid() { return VGRID; }

// ---------------------------------------------------------------------------
// Adjoint: dl/dK = -GB X^T folded onto the stored values (see ncl_kkt.h).
// ---------------------------------------------------------------------------
__global__ void k_adj_H(DevPlan P, const double* X, int64_t ldx, const double* GB, int64_t ldgb, int nrhs,
                        double* G_H) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < P.nnzH; q += (int64_t)gridDim.x * blockDim.x) {
    const int32_t i = P.H_row[q], j = P.H_col[q];
    double g = 0.0;
    for (int r = 0; r < nrhs; r++) {
      g -= GB[r * ldgb + i] * X[r * ldx + j];
      if (i != j) g -= GB[r * ldgb + j] * X[r * ldx + i];
    }
    G_H[q] = g;
  }
}

__global__ void k_adj_S(DevPlan P, const double* X, int64_t ldx, const double* GB, int64_t ldgb, int nrhs,
                        double* G_S) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < P.nvar; v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t i = P.var_row[v];
    double g = 0.0;
    for (int r = 0; r < nrhs; r++) g -= GB[r * ldgb + i] * X[r * ldx + i];
    G_S[v] = g;
  }
}

// (J x)_con and (J gb)_con for the condensed form
__global__ void k_jmul(DevPlan P, const double* Jv, const double* X, int64_t ldx, const double* GB, int64_t ldgb,
                       int nrhs, double* jx, double* jg) {
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < P.ncon; c += (int64_t)gridDim.x * blockDim.x) {
    for (int r = 0; r < nrhs; r++) {
      double a = 0.0, b = 0.0;
      for (int64_t q = P.J_rowptr[c]; q < P.J_rowptr[c + 1]; q++) {
        a = fma(Jv[q], X[r * ldx + P.J_col[q]], a);
        b = fma(Jv[q], GB[r * ldgb + P.J_col[q]], b);
      }
      jx[r * P.ncon + c] = a;
      jg[r * P.ncon + c] = b;
    }
  }
}

// dl/dJ: K2r from the (2,1) block; K from the product sum_r w_r J_r^T J_r
// (w_r = rho, or rho Omega_r with slacks, Eq. K1s)
__global__ void k_adj_J(DevPlan P, const double* w, const double* X, int64_t ldx, const double* GB, int64_t ldgb,
                        int nrhs, const double* jx, const double* jg, double* G_J) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < P.nnzJ; q += (int64_t)gridDim.x * blockDim.x) {
    const int32_t con = P.J_con[q], c = P.J_col[q];
    double g = 0.0;
    if (P.form == 0) {
      const int32_t rr = P.con_row[con];
      for (int r = 0; r < nrhs; r++) g -= GB[r * ldgb + rr] * X[r * ldx + c] + GB[r * ldgb + c] * X[r * ldx + rr];
    } else {
      const double rh = w[con];
      for (int r = 0; r < nrhs; r++)
        g -= rh * (jg[r * P.ncon + con] * X[r * ldx + c] + jx[r * P.ncon + con] * GB[r * ldgb + c]);
    }
    G_J[q] = g;
  }
}

// per-instance scalar gradients (one CTA per instance, fixed reduction order)
// (dl/drho of K uses dw_r/drho: 1 without slacks, Sigma_s^2/(rho+Sigma_s)^2 with)
__global__ void __launch_bounds__(256) k_adj_scal(DevPlan P, const int64_t* inst_n, const int64_t* inst_con_off,
                                                  const double* rho, const double* dw, const double* X,
                                                  int64_t ldx, const double* GB, int64_t ldgb, int nrhs,
                                                  const double* jx, const double* jg, double* G_scal) {
  __shared__ double red[2][256];
  const int inst = blockIdx.x;
  const int64_t r0 = P.inst_row_off[inst], r1 = P.inst_row_off[inst + 1];
  const int64_t n = inst_n[inst];
  double gd = 0.0, gr = 0.0;
  for (int64_t i = r0 + threadIdx.x; i < r1; i += blockDim.x) {
    double s = 0.0;
    for (int r = 0; r < nrhs; r++) s += GB[r * ldgb + i] * X[r * ldx + i];
    if (i - r0 < n) gd -= s;
    else gr -= s;  // dual rows (K2r only)
  }
  if (P.form == 0) {
    const double rh = rho[inst];
    gr = gr / (rh * rh);
  } else {
    gr = 0.0;
    for (int64_t c = inst_con_off[inst] + threadIdx.x; c < inst_con_off[inst + 1]; c += blockDim.x)
      for (int r = 0; r < nrhs; r++) gr -= dw[c] * jg[r * P.ncon + c] * jx[r * P.ncon + c];
  }
  red[0][threadIdx.x] = gd;
  red[1][threadIdx.x] = gr;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      red[0][threadIdx.x] += red[0][threadIdx.x + o];
      red[1][threadIdx.x] += red[1][threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    G_scal[2 * inst] = red[0][0];
    G_scal[2 * inst + 1] = red[1][0];
  }
}

void launch_adjoint_values(const DevPlan& P, const double* Jv, const double* w, const double* X, int64_t ldx,
                           const double* GB, int64_t ldgb, int nrhs, double* G_H, double* G_J, double* G_S,
                           double* G_scal, double* jx, double* jg, cudaStream_t st) {
  if (G_H && P.nnzH) k_adj_H<<<grid_for(P.nnzH), 256, 0, st>>>(P, X, ldx, GB, ldgb, nrhs, G_H);
  if (G_S && P.nvar) k_adj_S<<<grid_for(P.nvar), 256, 0, st>>>(P, X, ldx, GB, ldgb, nrhs, G_S);
  const bool need_j = P.form == 1 && P.ncon && (G_J || G_scal);
  if (need_j) k_jmul<<<grid_for(P.ncon), 256, 0, st>>>(P, Jv, X, ldx, GB, ldgb, nrhs, jx, jg);
  if (G_J && P.nnzJ) k_adj_J<<<grid_for(P.nnzJ), 256, 0, st>>>(P, w, X, ldx, GB, ldgb, nrhs, jx, jg, G_J);
  (void)G_scal;
}

void launch_adjoint_scalars(const DevPlan& P, const int64_t* inst_n, const int64_t* inst_con_off, const double* rho,
                            const double* dw, const double* X, int64_t ldx, const double* GB, int64_t ldgb,
                            int nrhs, const double* jx, const double* jg, double* G_scal, cudaStream_t st) {
  k_adj_scal<<<P.ninst, 256, 0, st>>>(P, inst_n, inst_con_off, rho, dw, X, ldx, GB, ldgb, nrhs, jx, jg, G_scal);
}

// Slack step of the condensed form with slacks (Section 3.3, proof of the
// proposition on Eq. K1s):  Delta s_r = (rho (J Delta t)_r + r_s,r) /
// (Sigma_s,r + rho) for an inequality row; 0 for a row without slack
// (Sigma_s = +inf).  rho is the penalty of the factored matrix (rho-hat).
// One thread per (row, right-hand side).
__global__ void k_slack_step(DevPlan P, const double* __restrict__ Jv, const double* __restrict__ rho,
                             const double* __restrict__ ss, int nrhs, const double* __restrict__ DT, int64_t ldt,
                             const double* __restrict__ RS, int64_t ldr, double* __restrict__ DS, int64_t lds) {
  const int64_t total = P.ncon * (int64_t)nrhs;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t c = idx % P.ncon;
    const int r = (int)(idx / P.ncon);
    const double s = ss[c];
    if (isinf(s) && s > 0) {
      DS[r * lds + c] = 0.0;
      continue;
    }
    double jt = 0.0;
    for (int64_t q = P.J_rowptr[c]; q < P.J_rowptr[c + 1]; q++) jt = fma(Jv[q], DT[r * ldt + P.J_col[q]], jt);
    const double rh = rho[P.con_inst[c]];
    DS[r * lds + c] = fma(rh, jt, RS[r * ldr + c]) / (s + rh);
  }
}

// Right-hand side of Eq. K1s as the proof's elimination of Delta s gives it:
//   OUT = RT + rho J_I^T (Sigma_s + rho I)^{-1} RS,
// one thread per (variable, right-hand side), the variable's J values in
// constraint order (deterministic; OUT may alias RT).
__global__ void k_k1s_rhs(DevPlan P, const double* __restrict__ Jv, const double* __restrict__ rho,
                          const double* __restrict__ ss, int nrhs, const double* RT, int64_t ldt,
                          const double* __restrict__ RS, int64_t ldr, double* OUT, int64_t ldo) {
  const int64_t total = P.dim * (int64_t)nrhs;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = idx % P.dim;
    const int r = (int)(idx / P.dim);
    double acc = 0.0;
    for (int64_t q = P.JT_ptr[v]; q < P.JT_ptr[v + 1]; q++) {
      const int32_t e = P.JT_idx[q];
      const int32_t c = P.J_con[e];
      const double s = ss[c];
      if (isinf(s) && s > 0) continue;
      const double rh = rho[P.con_inst[c]];
      acc = fma(rh * Jv[e], RS[r * ldr + c] / (s + rh), acc);
    }
    OUT[r * ldo + v] = RT[r * ldt + v] + acc;
  }
}

void launch_k1s_rhs(const DevPlan& P, const double* Jv, const double* rho, const double* ss, int nrhs,
                    const double* RT, int64_t ldt, const double* RS, int64_t ldr, double* OUT, int64_t ldo,
                    cudaStream_t st) {
  const int64_t total = P.dim * (int64_t)nrhs;
  if (total == 0) return;
  k_k1s_rhs<<<grid_for(total), 256, 0, st>>>(P, Jv, rho, ss, nrhs, RT, ldt, RS, ldr, OUT, ldo);
}

// ---------------------------------------------------------------------------
// Newton step of Algorithm NCL around the factorisation (Section 3.1-3.3):
// the right-hand side of Eq. K2r (unknown [Delta x; -Delta y]) or Eq. K1
// (unknown Delta x), and the recovery of the other components from Eq. K3:
//   Delta y   = -(second block of the K2r solution), or
//             = -rho (J Delta x + c) + y_k - y          (Eq. K1, elimination)
//   Delta r   = (Delta y - y_k + y) / rho - r            (Eq. K2, elimination)
//   Delta z_l = -(X - L)^{-1} (Z_l Delta x - mu e) - z_l (eliminated from Eq. K3)
//   Delta z_u =  (U - X)^{-1} (Z_u Delta x + mu e) - z_u
// rho is the penalty of the factored matrix (rho-hat).  An infinite bound
// gives (x - l)^{-1} = 0 (IEEE), so its barrier terms vanish.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double barrier_grad(const NewtonDev& pt, int64_t v, double mu) {
  // -(X - L)^{-1} mu e + (U - X)^{-1} mu e, component v
  return -mu / (pt.x[v] - pt.lo[v]) + mu / (pt.up[v] - pt.x[v]);
}

__global__ void k_newton_rhs(DevPlan P, const double* __restrict__ Jv, const double* __restrict__ rho,
                             const double* __restrict__ mu, NewtonDev pt, double* __restrict__ B) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < P.dim;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int32_t inst = P.row_inst[k];
    const double rh = rho[inst], m = mu[inst];
    const int32_t v = P.row_var[k];
    if (v >= 0) {
      // J^T y (K2r) or J^T (y_k - rho c) (K), the variable's J values in constraint order
      double jt = 0.0;
      for (int64_t q = P.JT_ptr[k]; q < P.JT_ptr[k + 1]; q++) {
        const int32_t e = P.JT_idx[q], c = P.J_con[e];
        const double wv = P.form == 0 ? pt.y[c] : pt.yk[c] - rh * pt.c[c];
        jt = fma(Jv[e], wv, jt);
      }
      const double gb = pt.g[v] + barrier_grad(pt, v, m);
      B[k] = P.form == 0 ? -(gb - jt) : jt - gb;
    } else {
      const int32_t c = P.row_con[k];
      B[k] = -(pt.c[c] - (pt.yk[c] - pt.y[c]) / rh);
    }
  }
}

__global__ void k_newton_recover_var(DevPlan P, const double* __restrict__ mu, NewtonDev pt,
                                     const double* __restrict__ X, double* __restrict__ dx,
                                     double* __restrict__ dzl, double* __restrict__ dzu) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < P.nvar;
       v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t k = P.var_row[v];
    const double m = mu[P.row_inst[k]];
    const double d = X[k];
    if (dx) dx[v] = d;
    if (dzl) dzl[v] = -(pt.zl[v] * d - m) / (pt.x[v] - pt.lo[v]) - pt.zl[v];
    if (dzu) dzu[v] = (pt.zu[v] * d + m) / (pt.up[v] - pt.x[v]) - pt.zu[v];
  }
}

__global__ void k_newton_recover_con(DevPlan P, const double* __restrict__ Jv, const double* __restrict__ rho,
                                     NewtonDev pt, const double* __restrict__ X, double* __restrict__ dy,
                                     double* __restrict__ dr) {
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < P.ncon;
       c += (int64_t)gridDim.x * blockDim.x) {
    const double rh = rho[P.con_inst[c]];
    double d;
    if (P.form == 0) {
      d = -X[P.con_row[c]];
    } else {
      double jx = 0.0;
      for (int64_t q = P.J_rowptr[c]; q < P.J_rowptr[c + 1]; q++) jx = fma(Jv[q], X[P.J_col[q]], jx);
      d = -rh * (jx + pt.c[c]) + pt.yk[c] - pt.y[c];
    }
    if (dy) dy[c] = d;
    if (dr) dr[c] = (d - pt.yk[c] + pt.y[c]) / rh - pt.r[c];
  }
}

void launch_newton_rhs(const DevPlan& P, const double* Jv, const double* rho, const double* mu, NewtonDev pt,
                       double* B, cudaStream_t st) {
  if (P.dim) k_newton_rhs<<<grid_for(P.dim), 256, 0, st>>>(P, Jv, rho, mu, pt, B);
}

void launch_newton_recover(const DevPlan& P, const double* Jv, const double* rho, const double* mu, NewtonDev pt,
                           const double* X, double* dx, double* dy, double* dr, double* dzl, double* dzu,
                           cudaStream_t st) {
  if (P.nvar) k_newton_recover_var<<<grid_for(P.nvar), 256, 0, st>>>(P, mu, pt, X, dx, dzl, dzu);
  if (P.ncon && (dy || dr)) k_newton_recover_con<<<grid_for(P.ncon), 256, 0, st>>>(P, Jv, rho, pt, X, dy, dr);
}

void launch_slack_step(const DevPlan& P, const double* Jv, const double* rho, const double* ss, int nrhs,
                       const double* DT, int64_t ldt, const double* RS, int64_t ldr, double* DS, int64_t lds,
                       cudaStream_t st) {
  const int64_t total = P.ncon * (int64_t)nrhs;
  if (total == 0) return;
  k_slack_step<<<grid_for(total), 256, 0, st>>>(P, Jv, rho, ss, nrhs, DT, ldt, RS, ldr, DS, lds);
}

}  // namespace ncl
