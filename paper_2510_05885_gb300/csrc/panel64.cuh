// FP64 pivot blocks and panels of large fronts (internal).
//
// A double-precision warp instruction keeps its scheduler for 64 cycles here,
// whatever its active lanes (measured: 16 independent FMAs of one warp, 1027
// cycles; with all four schedulers at it an SM does 1.7 to 2 FMAs per clock).
// So a 128-column panel, whose diagonal block is 0.35 million FMAs for one
// CTA, held one SM for 0.2 ms while the others waited.  A panel is 32 columns
// instead, nearly all of the work is left to update tiles that spread over the
// chip, and the panel runs beside them: one launch per panel holds the panel's
// own update and factorisation and the rest of the previous panel's update.
// FP64 factorisation and solve of the condensed 100 x 100 grid: panels 10.4 ->
// 4.2 ms with their updates (which took 3.7 ms besides), whole call 21.5 ->
// 11.3 ms (13.0 with 32-column panels and their updates in launches of their
// own).  Small fronts by the same pieces: 1.61 -> 0.62 ms.
#pragma once
#include "panel_roles.cuh"
#include "simt_tile.cuh"

namespace ncl {

// 1 / d by the hardware's seed (measured: 2^-19.9) and one step of third order,
// r (1 + e + e^2) with e = 1 - d r: three dependent FMAs instead of a
// division's longer chain.  Differs from the division in 3 of 10^4 random
// arguments, by the last bit.  Pivots near the ends of the exponent range take
// the division.  (Compared as integers: a double compare costs an FMA's time.)
__device__ __forceinline__ double pivot_rcp64(double d) {
  const unsigned ex = ((unsigned)__double2hiint(d) >> 20) & 0x7ffu;
  if (ex - 64u > 1918u) return 1.0 / d;
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
  const double e = fma(-d, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// static_pivot with the common case decided on the bit patterns
__device__ __forceinline__ double static_pivot64(double d, int sign, double eps, int policy, int8_t& st) {
  const unsigned long long b = __double_as_longlong(d) & 0x7fffffffffffffffull;
  if (b > (unsigned long long)__double_as_longlong(eps) && b < 0x7ff0000000000000ull) {
    st = 0;
    return d;
  }
  return static_pivot(d, sign, eps, policy, st);
}

constexpr int P64_WARPS = 7;   // of a CTA's eight; the last one publishes
__device__ __forceinline__ void p64_bar() { asm volatile("bar.sync 1, 224;" ::: "memory"); }

// LDL^T of a block of w <= 32 columns in shared memory (A, row stride lda, the
// lower part) by the warps 0..6 of a CTA; L and the pivots (dsh, status in
// pst) in place.  The block is dealt out in 20 tiles of 8 x 4 over the warps (a
// lane holds one entry of up to three tiles), and only tiles with columns left
// are touched.  Per column: its entries go to shared memory, warp 0 takes the
// pivot's reciprocal and forms the column of L, every warp updates its tiles.
// done(k) is called after column k is in A.  ws: 64 entries.  (One warp with a
// row per lane and shuffles: 47k cycles for 32 columns.)
template <typename Done>
__device__ __forceinline__ void factor_block64(double* A, int lda, int w, const int8_t* sg, double eps, int policy,
                                               double* ws, double* dsh, int8_t* pst, Done done) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  double a[3];
  int row[3], cb[3];
#pragma unroll
  for (int s = 0; s < 3; s++) {
    // tiles column by column: 4, 4, 3, 3, 2, 2, 1, 1 of them
    const int id = warp + P64_WARPS * s;
    int rb = 3;
    if (id < 8) { cb[s] = id >> 2; rb = id & 3; }
    else if (id < 14) { cb[s] = 2 + (id - 8) / 3; rb = 1 + (id - 8) % 3; }
    else if (id < 18) { cb[s] = 4 + (id - 14) / 2; rb = 2 + (id - 14) % 2; }
    else cb[s] = id < 20 ? id - 12 : -1;
    row[s] = 8 * rb + g;
    a[s] = (cb[s] >= 0 && row[s] < w && 4 * cb[s] + t <= row[s]) ? A[row[s] * lda + 4 * cb[s] + t] : 0.0;
  }
#pragma unroll 1
  for (int k = 0; k < w; k++) {
    double* wk = ws + 32 * (k & 1);
#pragma unroll
    for (int s = 0; s < 3; s++)
      if (cb[s] == k >> 2 && t == (k & 3)) wk[row[s]] = a[s];
    p64_bar();
    if (warp == 0) {
      int8_t st;
      const double d = static_pivot64(wk[k], sg[k], eps, policy, st);
      const double r = pivot_rcp64(d);
      if (lane >= k && lane < w) A[lane * lda + k] = lane == k ? d : wk[lane] * r;
      if (lane == k) {
        dsh[k] = d;
        pst[k] = st;
      }
    }
    p64_bar();
    done(k);
#pragma unroll
    for (int s = 0; s < 3; s++)
      if (4 * cb[s] + 3 > k) {   // (-1: never)
        const int c = 4 * cb[s] + t;
        if (c > k && c <= row[s] && row[s] < w) a[s] -= A[row[s] * lda + k] * wk[c];
      }
  }
}

// X = R L^-T for eight rows of a warp, four lanes to a row, each holding every
// fourth of its 32 columns in x, so that a warp instruction has all its lanes
// at work: the columns k0 .. k0 + 7 of the unit lower L (shared, row stride
// LDS, zero on and above the diagonal), the finished value of a column handed
// to the row's lanes by a shuffle.
__device__ __forceinline__ void rows_step64(double (&x)[8], const double* L, int k0, int lane) {
  const int t = lane & 3;
#pragma unroll
  for (int k = k0; k < k0 + 8; k++) {
    const double v = __shfl_sync(0xffffffffu, x[k >> 2], (lane & ~3) | (k & 3));
#pragma unroll
    for (int m = 0; m < 8; m++)
      if (m > (k >> 2) || (m == (k >> 2) && t > (k & 3))) x[m] -= L[(t + 4 * m) * LDS + k] * v;
  }
}

// Pivot columns of a whole front in shared memory (F, row stride ldf, ncol <=
// 64): per 32 columns the pivot block, then the rows below eight to a warp,
// L21 = F21 L_jj^-T D^-1, then the next columns' update.  The inverse of a
// front's only sub-block comes out as 32 more rows, I L^-T, to Iv (row stride
// LDS).  L, rd, ws, d: 32 x LDS, 32, 64 and 64 entries.  Called by 256 threads.
__device__ __forceinline__ void factor_front64(const DevPlan& P, const DevNum<double>& N, double* F, int ldf, int nrow,
                                               int ncol, int col0, double* L, double* Iv, double* rd, double* ws,
                                               double* d, int8_t* sg, int8_t* pst, double eps, int policy) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, t = lane & 3;
  if (tid < 64) sg[tid] = tid < ncol ? P.col_sign[col0 + tid] : 1;
  __syncthreads();
  for (int c0 = 0; c0 < ncol; c0 += 32) {
    const int cw = min(32, ncol - c0), rb = c0 + cw;
    if (warp < P64_WARPS)
      factor_block64(F + c0 * ldf + c0, ldf, cw, sg + c0, eps, policy, ws, d + c0, pst + c0, [](int) {});
    __syncthreads();
    for (int idx = tid; idx < 1024; idx += 256) {
      const int r = idx >> 5, c = idx & 31;
      L[r * LDS + c] = (c < r && r < cw) ? F[(c0 + r) * ldf + c0 + c] : 0.0;
    }
    if (tid < cw) {
      rd[tid] = pivot_rcp64(d[c0 + tid]);
      N.D[col0 + c0 + tid] = d[c0 + tid];
      N.piv[col0 + c0 + tid] = pst[c0 + tid];
    }
    __syncthreads();
    const int nrg = (nrow - rb + 7) / 8, ng = nrg + (ncol <= 32 ? (cw + 7) / 8 : 0);
    for (int gr = warp; gr < ng; gr += 8) {
      const int i = 8 * (gr < nrg ? gr : gr - nrg) + (lane >> 2);
      const bool act = gr < nrg && rb + i < nrow;
      double* Fr = F + (act ? rb + i : 0) * ldf + c0;
      double x[8];
#pragma unroll
      for (int m = 0; m < 8; m++) {
        const int c = t + 4 * m;
        x[m] = gr < nrg ? (act && c < cw ? Fr[c] : 0.0) : (c == i ? 1.0 : 0.0);
      }
#pragma unroll
      for (int j = 0; j < 4; j++)
        if (8 * j < cw) rows_step64(x, L, 8 * j, lane);
#pragma unroll
      for (int m = 0; m < 8; m++) {
        const int c = t + 4 * m;
        if (gr >= nrg) Iv[c * LDS + i] = x[m];
        else if (act && c < cw) Fr[c] = x[m] * rd[c];
      }
    }
    __syncthreads();
    if (rb < ncol) {
      // F[r][c] -= sum_u L[r][u] d_u L[c][u], lane = column, eight rows of a warp at a time
      const int c = rb + lane;
      for (int r0 = rb + 8 * warp; r0 < nrow; r0 += 64) {
        double acc[8];
#pragma unroll
        for (int m = 0; m < 8; m++) acc[m] = 0.0;
#pragma unroll 4
        for (int u = 0; u < 32; u++) {
          const double b = F[min(c, ncol - 1) * ldf + c0 + u] * d[c0 + u];
#pragma unroll
          for (int m = 0; m < 8; m++) acc[m] += F[min(r0 + m, nrow - 1) * ldf + c0 + u] * b;
        }
#pragma unroll
        for (int m = 0; m < 8; m++)
          if (c < ncol && r0 + m < nrow && c <= r0 + m) F[(r0 + m) * ldf + c] -= acc[m];
      }
      __syncthreads();
    }
  }
}

struct Panel64Smem {
  double C[32 * LDS];         // the CTA's 32 x 32 tile of the panel
  union {
    struct {
      double A[32 * LDS], B[32 * LDS];   // previous panel's columns, k-major
    } up;
    double L[32 * LDS];       // row role: L11, zero on and above the diagonal and past w
  };
  double ws[64], d[32];
  int8_t sg[32], pst[32];
};

// C (shared) = the tile of rows r0.. and columns q0.. of the front, less the
// previous panel's contribution (columns q0 - 32 .. q0 - 1; none for the first
// panel).  DIAG: r0 = q0, the lower part only.  Called by 256 threads.
template <bool DIAG>
__device__ __forceinline__ void panel64_tile(const DevNum<double>& N, const double* Lb, int ncp, int nrow, int col0,
                                             int q0, int w, int r0, Panel64Smem& sh) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  double c4[4];
#pragma unroll
  for (int q = 0; q < 4; q++) {
    const int r = warp + 8 * q;
    const bool in = r0 + r < nrow && lane < w && (!DIAG || (r < w && lane <= r));
    c4[q] = in ? Lb[(int64_t)(r0 + r) * ncp + q0 + lane] : 0.0;
  }
  if (q0 > 0) {
    double a4[4], b4[4];
    const double dk = N.D[col0 + q0 - 32 + lane];
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int r = warp + 8 * q;
      a4[q] = r0 + r < nrow ? Lb[(int64_t)(r0 + r) * ncp + q0 - 32 + lane] : 0.0;
      b4[q] = r < w ? Lb[(int64_t)(q0 + r) * ncp + q0 - 32 + lane] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int r = warp + 8 * q;
      sh.up.A[lane * LDS + r] = a4[q];
      sh.up.B[lane * LDS + r] = b4[q] * dk;
    }
    __syncthreads();
    // rows 2 ty, 2 ty + 1, columns tx, tx + 16
    const int tx = tid & 15, ty = tid >> 4;
    double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
    const bool right = !DIAG || warp >= 4;   // columns 16.. of rows below 16 are above the diagonal
#pragma unroll 4
    for (int k = 0; k < 32; k++) {
      const double x0 = sh.up.A[k * LDS + 2 * ty], x1 = sh.up.A[k * LDS + 2 * ty + 1];
      const double y0 = sh.up.B[k * LDS + tx];
      acc[0][0] += x0 * y0;
      acc[1][0] += x1 * y0;
      if (right) {
        const double y1 = sh.up.B[k * LDS + tx + 16];
        acc[0][1] += x0 * y1;
        acc[1][1] += x1 * y1;
      }
    }
#pragma unroll
    for (int a = 0; a < 2; a++)
#pragma unroll
      for (int b = 0; b < 2; b++) sh.C[(2 * ty + a) * LDS + tx + 16 * b] = acc[a][b];
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; q++) c4[q] -= sh.C[(warp + 8 * q) * LDS + lane];
  }
#pragma unroll
  for (int q = 0; q < 4; q++) sh.C[(warp + 8 * q) * LDS + lane] = c4[q];
  __syncthreads();
}

// Diagonal role: warp 7 publishes the block eight columns at a time (fence,
// release flag) while the others go on.
__device__ __forceinline__ void panel_diag_role64(const DevPlan& P, const DevNum<double>& N, int s, int q0, int* flags,
                                                  double eps, int policy, Panel64Smem& sh) {
  const int ncol = P.sn_ncol[s], ncp = P.sn_ncolp[s], col0 = P.sn_col0[s];
  const int w = min(32, ncol - q0), tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  double* Lf = N.L + P.sn_Loff[s];
  if (tid < 32) sh.sg[tid] = tid < w ? P.col_sign[col0 + q0 + tid] : 1;
  panel64_tile<true>(N, Lf, ncp, P.sn_nrow[s], col0, q0, w, q0, sh);
  if (warp < P64_WARPS) {
    factor_block64(sh.C, LDS, w, sh.sg, eps, policy, sh.ws, sh.d, sh.pst, [&](int k) {
      // a barrier of its own for each group: warp 7 may be a group behind
      if ((k & 7) == 7 || k == w - 1) asm volatile("bar.arrive %0, 256;" ::"r"(2 + (k >> 3)) : "memory");
    });
    return;
  }
  double* Lb = Lf + (int64_t)q0 * ncp + q0;
  for (int j = 0; 8 * j < w; j++) {
    asm volatile("bar.sync %0, 256;" ::"r"(2 + j) : "memory");
    const int c = 8 * j + (lane & 7);
    for (int r = 8 * j + (lane >> 3); r < w; r += 4)
      if (c <= r) Lb[(int64_t)r * ncp + c] = sh.C[r * LDS + c];
    if (lane < 8 && c < w) {
      N.D[col0 + q0 + c] = sh.d[c];
      N.piv[col0 + q0 + c] = sh.pst[c];
    }
    __syncwarp();
    if (lane == 0) {
      __threadfence();
      st_release_i32(flags + j, 1);
    }
  }
}

// Row role (one CTA per 32 rows, four warps with a scheduler each): X = R L^-T
// as the columns of L11 are published, L21 = X D^-1.
__device__ __forceinline__ void panel_rows_role64(const DevPlan& P, const DevNum<double>& N, int s, int q0, int r0,
                                                  const int* flags, int* err, long long wait, Panel64Smem& sh) {
  const int ncol = P.sn_ncol[s], nrow = P.sn_nrow[s], ncp = P.sn_ncolp[s], col0 = P.sn_col0[s];
  const int w = min(32, ncol - q0);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, t = lane & 3;
  double* Lb = N.L + P.sn_Loff[s];
  panel64_tile<false>(N, Lb, ncp, nrow, col0, q0, w, r0, sh);
  const int lr = 8 * (warp & 3) + (lane >> 2);
  double x[8];
#pragma unroll
  for (int m = 0; m < 8; m++) x[m] = sh.C[lr * LDS + t + 4 * m];
#pragma unroll
  for (int j = 0; j < 4; j++) {
    if (8 * j >= w) break;
    if (tid == 0) panel_wait(flags + j, err, wait);
    __syncthreads();   // (also: the update's operands, which L shares, are done with)
    {
      const int r = tid >> 3, c = 8 * j + (tid & 7);
      const double v = r < w && c < r ? __ldcg(Lb + (int64_t)(q0 + r) * ncp + q0 + c) : 0.0;
      const double dv = tid < 8 && c < w ? __ldcg(N.D + col0 + q0 + c) : 1.0;
      sh.L[r * LDS + c] = v;
      if (tid < 8) sh.d[c] = pivot_rcp64(dv);
    }
    __syncthreads();
    if (warp < 4) rows_step64(x, sh.L, 8 * j, lane);
  }
  if (warp >= 4 || r0 + lr >= nrow) return;
  const int cend = q0 + w == ncol ? ncp - q0 : w;   // the last panel also clears the padding columns
  double* Lr = Lb + (int64_t)(r0 + lr) * ncp + q0;
#pragma unroll
  for (int m = 0; m < 8; m++) {
    const int c = t + 4 * m;
    if (c < cend) Lr[c] = c < w ? x[m] * sh.d[c] : 0.0;
  }
  for (int c = 32 + t; c < cend; c += 4) Lr[c] = 0.0;
}

}  // namespace ncl
