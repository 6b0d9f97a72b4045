// Dense front kernels (sm_103a): the per-step macro-panel kernel of large
// fronts (the roles are in panel_roles.cuh), and whole small fronts.
#include "panel_roles.cuh"
#include "panel8.cuh"
#include "panel64.cuh"

#include <algorithm>

namespace ncl {

// One launch per macro panel step of a level: for each large front, one
// CTA in the diagonal role and one per RB rows below the panel in the row
// role.  A CTA's role comes from the front's ticket counter (the first CTA
// to arrive takes the diagonal), so every CTA that waits waits for a CTA
// that is already running: the waits cannot deadlock, whatever the order
// in which CTAs are scheduled.  Waits are bounded (the factor's error flag
// is set past the limit).
// items: (front, q0, sync slot); sync[slot] = ticket counter, sync[slot + 1
// + j] = flag of sub-block j.
template <typename T, int NB>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 2 : 1) k_macro_panel(DevPlan P, DevNum<T> N, const int4* __restrict__ items,
                                                        int* sync, int* err, double eps, int policy,
                                                        long long wait) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int ticket;
  const int4 it = items[blockIdx.x];
  const int s = it.x, q0 = it.y;
  int* slot = sync + it.z;
  if (threadIdx.x == 0) ticket = atomicAdd(slot, 1);
  __syncthreads();
  if (ticket == 0) {
    panel_diag_role<T, NB>(P, N, s, q0, slot + 1, eps, policy, smem_raw);
  } else {
    const int qe = min(q0 + NB, P.sn_ncol[s]);
    panel_rows_role<T, NB>(P, N, s, q0, qe + RB * (ticket - 1), slot + 1, err, wait, smem_raw);
  }
}

// FP64: one launch per 32-column panel (panel64.cuh).  The first npanel CTAs
// take the panels' roles as above, each with its own tile's share of the
// previous panel's update; the other CTAs are the tiles of that update to the
// right of the panel.  (One to four CTAs per SM, by the shared memory asked
// for: 11.48, 11.29, 11.29 and 11.30 ms for the whole call, so no more is
// asked for than is used.)
__global__ void __launch_bounds__(256) k_panel64(DevPlan P, DevNum<double> N, const int4* __restrict__ items,
                                                 int npanel, int* sync, int* err, double eps, int policy,
                                                 long long wait, const GemmProb* __restrict__ probs,
                                                 const int32_t* __restrict__ tile_prob) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int ticket;
  if ((int)blockIdx.x >= npanel) {
    simt_tile<double>(N, probs, tile_prob, blockIdx.x - npanel, *reinterpret_cast<SimtTile<double>*>(smem_raw));
    return;
  }
  Panel64Smem& sh = *reinterpret_cast<Panel64Smem*>(smem_raw);
  const int4 it = items[blockIdx.x];
  const int s = it.x, q0 = it.y;
  int* slot = sync + it.z;
  if (threadIdx.x == 0) ticket = atomicAdd(slot, 1);
  __syncthreads();
  if (ticket == 0)
    panel_diag_role64(P, N, s, q0, slot + 1, eps, policy, sh);
  else
    panel_rows_role64(P, N, s, q0, min(q0 + 32, P.sn_ncol[s]) + 32 * (ticket - 1), slot + 1, err, wait, sh);
}

void launch_panel64(const DevPlan& P, const DevNum<double>& N, const int4* items, int count, int* sync, int* err,
                    double eps, int policy, long long wait, const GemmProb* probs, const int32_t* tile_prob,
                    int64_t tiles, cudaStream_t st) {
  if (count <= 0) return;
  static_assert(sizeof(SimtTile<double>) <= sizeof(Panel64Smem), "one size for both");
  static_assert(sizeof(Panel64Smem) <= 48 * 1024, "no opt-in needed");
  k_panel64<<<(unsigned)(count + tiles), 256, sizeof(Panel64Smem), st>>>(P, N, items, count, sync, err, eps, policy,
                                                                         wait, probs, tile_prob);
}

// Small fronts (ncol <= 64): one CTA factors the pivot columns of the whole
// front in shared memory, FP32 eight columns at a time (panel8.cuh), FP64 by
// 32-column sub-blocks (panel64.cuh); a front's only sub-block is inverted too,
// for the triangular sweeps.  The update block F22 -= L21 D1 L21^T is left to
// the SIMT update kernel, which spreads it over many CTAs.
int small_front_smem(int nrow, int ncp, int esz) {
  if (esz == 4)   // front, panel rows, pivot block and its inverse, pivots, signs and statuses
    return (nrow * panel8_ld(ncp) + (64 + nrow) * P8_LD + 2 * 32 * LDS + 64) * 4 + 128;
  return (nrow * (ncp + 1) + 2 * 32 * LDS + 32 + 64 + 64) * esz + 128;
}

// the subtree factorisation's front, pivot block, its inverse, pivots
int subtree_front_smem(int nrow, int ncp, int esz) { return (nrow * (ncp + 1) + 2 * 32 * LDS + 32) * esz; }

// Write a shared-memory front back.  A pivot block of one sub-block (at most 32
// columns) is written as its inverse Iv, which the sweeps apply; wider ones
// are inverted after the factorisation (invert.cu).
template <typename T>
__device__ __forceinline__ void store_front(T* Lg, const T* F, const T* Iv, int nrow, int ncol, int ncp, int ldf) {
  for (int idx = threadIdx.x; idx < nrow * ncp; idx += blockDim.x) {
    const int r = idx / ncp, c = idx - r * ncp;
    Lg[idx] = (r < ncol && c < r && ncol <= 32) ? Iv[r * LDS + c] : F[r * ldf + c];
  }
}

// FP32: the pivot columns of a shared-memory front (rows x ncol, stride
// panel8_ld(ncp)), eight at a time, the pivots and statuses to global memory
// and, for a front of one 32-column sub-block, the inverse of its pivot block
// to Iv (by warp 0; the other warps go on).  256 threads.
__device__ __forceinline__ void factor_front32(const DevPlan& P, const DevNum<float>& N, float* F, int ldf, int nrow,
                                               int ncol, int col0, float* Ls, float* Xs, float* Lu, float* Iv,
                                               float* dsh, int8_t* sg, double eps, int policy) {
  int8_t* pst = sg + 64;
  const int tid = threadIdx.x;
  if (tid < 64) sg[tid] = tid < ncol ? P.col_sign[col0 + tid] : 1;
  __syncthreads();
  int c = 0;
  auto put = [&](int row, float (&l)[8]) { panel8_put(F + row * ldf + c, l, min(8, ncol - c)); };
  if (nrow <= 256) {
#pragma unroll 1
    for (; c + 8 <= ncol; c += 8)
      panel8_step<256, 1, true>(F, ldf, c, ncol, nrow, sg, (float)eps, policy, Ls, Xs, dsh, pst, put);
  } else {
#pragma unroll 1
    for (; c + 8 <= ncol; c += 8)
      panel8_step<256, 2, true>(F, ldf, c, ncol, nrow, sg, (float)eps, policy, Ls, Xs, dsh, pst, put);
  }
  if (c < ncol) panel8_step<256, 2, false>(F, ldf, c, ncol, nrow, sg, (float)eps, policy, Ls, Xs, dsh, pst, put);
  if (tid < ncol) {
    N.D[col0 + tid] = dsh[tid];
    N.piv[col0 + tid] = pst[tid];
  }
  if (ncol <= 32 && tid < 32) {
#pragma unroll 4
    for (int u = 0; u < 32; u++) Lu[tid * LDS + u] = (u < tid && tid < ncol) ? F[tid * ldf + u] : 0.f;
    __syncwarp();
    invert_sub32<float>(Lu, Iv, ncol, tid);
  }
}

// 256 threads per CTA (128 was measured slower on the 20 x 25, 300 x 300 and
// 700 x 700 systems: the rows below the sub-block take twice the passes)
constexpr int SMALL_THREADS = 256;

template <typename T>
__global__ void __launch_bounds__(SMALL_THREADS) k_factor_small(DevPlan P, DevNum<T> N,
                                                                const int32_t* __restrict__ list, double eps,
                                                                int policy) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int s = list[blockIdx.x];
  const int ncol = P.sn_ncol[s], nrow = P.sn_nrow[s], ncp = P.sn_ncolp[s], col0 = P.sn_col0[s];
  if constexpr (sizeof(T) == 4) {
    const int ldf = panel8_ld(ncp);
    float* F = reinterpret_cast<float*>(smem_raw);
    float* Ls = F + nrow * ldf;
    float* Xs = Ls + 64 * P8_LD;
    float* Lu = Xs + nrow * P8_LD;
    float* Iv = Lu + 32 * LDS;
    float* dsh = Iv + 32 * LDS;
    float* Lg = N.L + P.sn_Loff[s];
    load_tile(F, ldf, Lg, ncp, nrow, ncp, [](int, int) { return true; });
    factor_front32(P, N, F, ldf, nrow, ncol, col0, Ls, Xs, Lu, Iv, dsh, reinterpret_cast<int8_t*>(dsh + 64), eps, policy);
    // rows below first: warp 0 may still be inverting the pivot block
    const int nw = ncol <= 32 ? 7 : 8, w0 = 8 - nw;
    const int warp = threadIdx.x >> 5;
    if (warp >= w0)
      for (int idx = (warp - w0) * 32 + (threadIdx.x & 31) + ncol * ncp; idx < nrow * ncp; idx += 32 * nw)
        Lg[idx] = F[(idx / ncp) * ldf + idx % ncp];
    __syncthreads();
    store_front<T>(Lg, F, Iv, ncol, ncol, ncp, ldf);
    return;
  }
  if constexpr (sizeof(T) == 8) {
    const int ldf = ncp + 1;   // odd: column accesses by lanes are conflict-free
    double* F = reinterpret_cast<double*>(smem_raw);
    double* L = F + nrow * ldf;
    double* Iv = L + 32 * LDS;
    double* rd = Iv + 32 * LDS;
    double* ws = rd + 32;
    double* d = ws + 64;
    int8_t* sg = reinterpret_cast<int8_t*>(d + 64);
    double* Lg = N.L + P.sn_Loff[s];
    load_tile(F, ldf, Lg, ncp, nrow, ncp, [](int, int) { return true; });
    factor_front64(P, N, F, ldf, nrow, ncol, col0, L, Iv, rd, ws, d, sg, sg + 64, eps, policy);
    store_front<T>(Lg, F, Iv, nrow, ncol, ncp, ldf);
  }
}

template <typename T>
void launch_factor_small(const DevPlan& P, const DevNum<T>& N, const int32_t* list, int count, int smem_bytes,
                         double eps, int policy, cudaStream_t st) {
  if (count <= 0) return;
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_factor_small<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMALL_SMEM_MAX);
    attr = true;
  }
  k_factor_small<T><<<count, SMALL_THREADS, smem_bytes, st>>>(P, N, list, eps, policy);
}

// ---------------------------------------------------------------------------
// Factorisation of the subtrees of small fronts.
//
// The fronts of the small-subtree region (at most 32 pivots, small enough
// for the shared-memory front, and only such fronts below them) are
// factored by one CTA per maximal subtree, in one launch for the whole region;
// the level launches of the assembly, the small-front factorisation and the
// update blocks skip them.  A subtree's fronts are listed level by level: the
// leaves that fit a warp's share of the shared memory first, a warp each (see
// below), then the others one after the other by the whole CTA.  Per front:
//   the front is assembled straight into shared memory (original entries,
//   then the children's update blocks child by child; a child's entries
//   that land below the pivot columns go to this front's update block in
//   global memory, zeroed first), the 32-column pivot block is factored by
//   one warp, the rows below by the blocked substitution, L21 = F21 L11^-T
//   D1^-1 (one warp inverts the pivot block meanwhile), the factor block
//   written back, and the update block F22 -= L21 D1 L21^T formed from the
//   shared-memory front.
// The children's update blocks were written by the same CTA earlier, so a
// barrier orders them; nothing waits across CTAs.
// What bounds it is each front's chain of small steps: half of a warp's time
// goes to barriers behind the pivot block's warp and to instruction fetches
// (37 % of the issue slots used, 530 GB/s).  So many fronts run side by side:
// CTAs of four warps, six to an SM, which the region's limit on a front's size
// allows (api.cu), and no chain of dependent trips to memory within a front.
// 700 x 700 7.9 -> 6.2 ms, 64 scenarios 9.1 -> 8.3 ms, 64 uneven instances
// 1.96 -> 1.49 ms (before leaves were done by a warp each, see below).  (256 threads: 700 x 700 1.4 ms slower, scenarios 2.0 ms.)
// ---------------------------------------------------------------------------
constexpr int SUBTREE_THREADS = 128;

template <typename T>
__device__ __forceinline__ void subtree_front(const DevPlan& P, const DevNum<T>& N, int s, double eps, int policy,
                                              unsigned char* smem_raw) {
  const int ncol = P.sn_ncol[s], nrow = P.sn_nrow[s], ncp = P.sn_ncolp[s], col0 = P.sn_col0[s];
  const int nb = nrow - ncol;
  const int ldf = ncp + 1;
  T* F = reinterpret_cast<T*>(smem_raw);
  T* Ls = F + nrow * ldf;
  T* Iv = Ls + 32 * LDS;
  T* dsh = Iv + 32 * LDS;
  T* Lg = N.L + P.sn_Loff[s];
  T* Ub = N.U + P.sn_Uoff[s];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = blockDim.x >> 5;
  // zero the front and, where children add to it, the update block
  const int ch0 = P.child_ptr[s], ch1 = P.child_ptr[s + 1];
  for (int idx = tid; idx < nrow * ldf; idx += blockDim.x) F[idx] = T(0);
  if (ch1 > ch0)
    for (int idx = tid; idx < nb * nb; idx += blockDim.x) Ub[idx] = T(0);
  __syncthreads();
  // original entries (each lands in its own position): the front's entries
  // spread over all threads, four at a time
  const int64_t rbase = P.sn_rows_off[s];
  {
    const int64_t q0 = P.amap_ptr[rbase], q1 = P.amap_ptr[rbase + nrow];
    for (int64_t q = q0 + tid; q < q1; q += 4 * blockDim.x) {
      T v[4];
      int at[4];
#pragma unroll
      for (int i = 0; i < 4; i++) {
        const int64_t e = q + i * blockDim.x;
        at[i] = -1;
        if (e < q1) {
          at[i] = P.amap_row[e] * ldf + P.amap_col[e];
          v[i] = (T)N.Klow[P.amap_src[e]];
        }
      }
#pragma unroll
      for (int i = 0; i < 4; i++)
        if (at[i] >= 0) F[at[i]] = v[i];
    }
  }
  // the children's update blocks, child by child (the targets of one child
  // are distinct: its relative map is increasing): four rows of a child to a
  // warp, its loads before its stores (the compiler has to take a store for a
  // possible change of the next load, and one by one each is a trip to L2)
  for (int k = ch0; k < ch1; k++) {
    __syncthreads();
    const int c = P.child_list[k];
    const int nbc = P.sn_nrow[c] - P.sn_ncol[c];
    const int32_t* rel = P.relmap + P.relmap_off[c];
    const T* Uc = N.U + P.sn_Uoff[c];
    for (int a0 = warp; a0 < nbc; a0 += 4 * nw) {
      int ra[4];
#pragma unroll
      for (int i = 0; i < 4; i++) ra[i] = rel[min(a0 + i * nw, nbc - 1)];
      for (int b = lane; b <= min(a0 + 3 * nw, nbc - 1); b += 32) {
        const int rb = rel[b];
        T v[4], t[4];
#pragma unroll
        for (int i = 0; i < 4; i++) {
          const int a = a0 + i * nw;
          const bool ok = a < nbc && b <= a;
          v[i] = ok ? Uc[(int64_t)a * nbc + b] : T(0);
          t[i] = !ok ? T(0) : rb < ncol ? F[ra[i] * ldf + rb] : Ub[(int64_t)(ra[i] - ncol) * nb + (rb - ncol)];
        }
#pragma unroll
        for (int i = 0; i < 4; i++) {
          const int a = a0 + i * nw;
          if (a < nbc && b <= a) {
            if (rb < ncol) F[ra[i] * ldf + rb] = t[i] + v[i];
            else Ub[(int64_t)(ra[i] - ncol) * nb + (rb - ncol)] = t[i] + v[i];
          }
        }
      }
    }
  }
  __syncthreads();
  // the pivot block (one 32-column sub-block) by warp 0: LDL^T, pivots,
  // statuses and the zero-padded unit lower block
  if (warp == 0) {
    int8_t st;
    const T d = factor_sub32<T, true>(F, ldf, ncol, lane < ncol ? P.col_sign[col0 + lane] : 1, eps, policy, lane, st);
    dsh[lane] = d;
    if (lane < ncol) {
      N.D[col0 + lane] = d;
      N.piv[col0 + lane] = st;
    }
#pragma unroll 4
    for (int u = 0; u < 32; u++) Ls[lane * LDS + u] = (u < lane && lane < ncol) ? F[lane * ldf + u] : T(0);
  }
  __syncthreads();
  // warp 0: the pivot block's inverse; the others, the rows below: L21 = F21
  // L11^-T D1^-1
  if (warp == 0) {
    invert_sub32<T>(Ls, Iv, ncol, lane);
  } else {
    block_trsm32<T>(F + ncol * ldf, ldf, nb, ncol, Ls, LDS, 32, blockDim.x - 32);
    asm volatile("bar.sync 1, %0;" ::"r"(blockDim.x - 32) : "memory");
    const T rd = pivot_rcp(dsh[lane]);
    if (lane < ncol)
      for (int r = warp - 1; r < nb; r += nw - 1) F[(ncol + r) * ldf + lane] *= rd;
  }
  __syncthreads();
  // write the factor block back, and form the update block from it:
  // 4 x 4 register tiles of its lower triangle spread over all threads
  // (9 shared loads per 16 products), F22[a][b] -= sum_k (L[a][k] d_k) L[b][k]
  for (int r = warp; r < nrow; r += nw)
    if (lane < ncp) Lg[(int64_t)r * ncp + lane] = (r < ncol && lane < r) ? Iv[r * LDS + lane] : F[r * ldf + lane];
  const int T4 = (nb + 3) / 4;
  const int ntl = T4 * (T4 + 1) / 2;
  for (int e = tid; e < ntl; e += blockDim.x) {
    int ti = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
    while (ti * (ti + 1) / 2 > e) ti--;
    while ((ti + 1) * (ti + 2) / 2 <= e) ti++;
    const int tj = e - ti * (ti + 1) / 2;
    const int a0 = 4 * ti, b0 = 4 * tj;
    const T* fa = F + (ncol + a0) * ldf;
    const T* fb = F + (ncol + b0) * ldf;
    T acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
      for (int j = 0; j < 4; j++) acc[i][j] = T(0);
#pragma unroll 4
    for (int k = 0; k < ncol; k++) {
      const T dk = dsh[k];
      T av[4], bv[4];
#pragma unroll
      for (int i = 0; i < 4; i++) av[i] = a0 + i < nb ? fa[i * ldf + k] * dk : T(0);
#pragma unroll
      for (int j = 0; j < 4; j++) bv[j] = b0 + j < nb ? fb[j * ldf + k] : T(0);
#pragma unroll
      for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[i][j] += av[i] * bv[j];
    }
    // (all loads, then all stores)
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const int a = a0 + i, b = b0 + j;
        acc[i][j] = (ch1 > ch0 && a < nb && b <= a ? Ub[(int64_t)a * nb + b] : T(0)) - acc[i][j];
      }
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const int a = a0 + i, b = b0 + j;
        if (a < nb && b <= a) Ub[(int64_t)a * nb + b] = acc[i][j];
      }
  }
}

// A leaf of a subtree by one warp: the front in shared memory, right-looking with
// a lane to a row, the pivot block's inverse with a lane to a column, the update
// block row by row.  Half of the region's fronts are leaves, of 6 pivots and 30
// rows in the middle: too small for a CTA's barriers, and four at a time wait for
// memory together (subtree factorisation of 64 scenarios 8.3 -> 5.9 ms, of 64
// uneven instances 1.49 -> 1.17 ms).  Short loops instead of a 32-column block in
// registers, whose code would not stay in the instruction cache beside the rest.
__host__ __device__ inline int leaf_words(int nrow, int ncol, int ncp) {
  return nrow * (ncp + 1) + ncol * (ncol + 1) + ncol;   // front, inverse, pivots
}
template <typename T>
__device__ __forceinline__ void subtree_leaf(const DevPlan& P, const DevNum<T>& N, int s, double eps, int policy, T* F) {
  const int ncol = P.sn_ncol[s], nrow = P.sn_nrow[s], ncp = P.sn_ncolp[s], col0 = P.sn_col0[s];
  const int nb = nrow - ncol, ldf = ncp + 1, ldi = ncol + 1, lane = threadIdx.x & 31;
  T* Iv = F + nrow * ldf;
  T* ds = Iv + ncol * ldi;
  T* Lg = N.L + P.sn_Loff[s];
  T* Ub = N.U + P.sn_Uoff[s];
  const int64_t rbase = P.sn_rows_off[s];
  const int64_t q0 = P.amap_ptr[rbase], q1 = P.amap_ptr[rbase + nrow];
  for (int idx = lane; idx < nrow * ldf; idx += 32) F[idx] = T(0);
  __syncwarp();
  for (int64_t q = q0 + lane; q < q1; q += 4 * 32) {
    T v[4];
    int at[4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
      const int64_t e = q + 32 * i;
      at[i] = -1;
      if (e < q1) {
        at[i] = P.amap_row[e] * ldf + P.amap_col[e];
        v[i] = (T)N.Klow[P.amap_src[e]];
      }
    }
#pragma unroll
    for (int i = 0; i < 4; i++)
      if (at[i] >= 0) F[at[i]] = v[i];
  }
  const int sign = lane < ncol ? P.col_sign[col0 + lane] : 1;
  int8_t my_st = 0;
  T my_d = T(1);
  __syncwarp();
#pragma unroll 1
  for (int k = 0; k < ncol; k++) {
    int8_t st;
    const T d = static_pivot(F[k * ldf + k], __shfl_sync(0xffffffffu, sign, k), eps, policy, st);
    const T rd = pivot_rcp(d);
    if (lane == k) {
      my_d = d;
      my_st = st;
    }
    // the rows' later columns, with the pivot rows' entries of column k before they are scaled
    for (int r = k + 1 + lane; r < nrow; r += 32) {
      const T l = F[r * ldf + k] * rd;
      const int ce = min(r + 1, ncol);
#pragma unroll 4
      for (int c = k + 1; c < ce; c++) F[r * ldf + c] -= l * F[c * ldf + k];
    }
    __syncwarp();
    for (int r = k + 1 + lane; r < nrow; r += 32) F[r * ldf + k] *= rd;
    __syncwarp();
  }
  if (lane < ncol) {
    ds[lane] = my_d;
    N.D[col0 + lane] = my_d;
    N.piv[col0 + lane] = my_st;
    for (int i = lane + 1; i < ncol; i++) {
      T a = F[i * ldf + lane];
      for (int k = lane + 1; k < i; k++) a += F[i * ldf + k] * Iv[k * ldi + lane];
      Iv[i * ldi + lane] = -a;
    }
  }
  __syncwarp();
  for (int r = 0; r < nrow; r++)
    if (lane < ncp)
      Lg[(int64_t)r * ncp + lane] =
          r < ncol ? (lane < r ? Iv[r * ldi + lane] : lane == r ? ds[r] : T(0)) : F[r * ldf + lane];
  for (int a = 0; a < nb; a++)
    for (int b = lane; b <= a; b += 32) {
      T acc = T(0);
#pragma unroll 4
      for (int k = 0; k < ncol; k++) acc += (F[(ncol + a) * ldf + k] * ds[k]) * F[(ncol + b) * ldf + k];
      Ub[(int64_t)a * nb + b] = -acc;
    }
  __syncwarp();
}

// items: (first node, nodes, first level bound, levels); the nodes of level 0
// (leaves) come first, and those that fit a warp's share of the shared memory
// are done four at a time
template <typename T>
__global__ void __launch_bounds__(SUBTREE_THREADS, sizeof(T) == 4 ? 6 : 4) k_subtree_factor(DevPlan P, DevNum<T> N, const int4* __restrict__ items,
                                                        int count, const int32_t* __restrict__ nodes,
                                                        const int32_t* __restrict__ bounds, int* counter, int words,
                                                        double eps, int policy) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_item;
  constexpr int NW = SUBTREE_THREADS / 32;
  const int warp = threadIdx.x >> 5, share = words / NW;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_item = atomicAdd(counter, 1);
    __syncthreads();
    const int it = s_item;
    if (it >= count) break;
    const int4 item = items[it];
    const int leaves = bounds[item.z + 1];
    auto fits = [&](int s) { return leaf_words(P.sn_nrow[s], P.sn_ncol[s], P.sn_ncolp[s]) <= share; };
    for (int q = warp; q < leaves; q += NW) {
      const int s = nodes[item.x + q];
      if (fits(s)) subtree_leaf<T>(P, N, s, eps, policy, reinterpret_cast<T*>(smem_raw) + warp * share);
    }
    __syncthreads();
    for (int q = 0; q < item.y; q++) {
      const int s = nodes[item.x + q];
      if (q < leaves && fits(s)) continue;
      subtree_front<T>(P, N, s, eps, policy, smem_raw);
      __syncthreads();
    }
  }
}

template <typename T>
void launch_subtree_factor(const DevPlan& P, const DevNum<T>& N, const int4* items, int count, const int32_t* nodes,
                           const int32_t* bounds, int* counter, int smem, int nsm, double eps, int policy, cudaStream_t st) {
  if (count <= 0) return;
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_subtree_factor<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMALL_SMEM_MAX);
    attr = true;
  }
  // as many CTAs as fit on the device at once (they take subtrees from a counter)
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_subtree_factor<T>, SUBTREE_THREADS, smem) != cudaSuccess)
    per_sm = 4;
  const int grid = std::min(count, nsm * std::max(per_sm, 1));
  k_subtree_factor<T><<<grid, SUBTREE_THREADS, smem, st>>>(P, N, items, count, nodes, bounds, counter, smem / (int)sizeof(T), eps,
                                                          policy);
}

template void launch_subtree_factor<float>(const DevPlan&, const DevNum<float>&, const int4*, int, const int32_t*,
                                           const int32_t*, int*, int, int, double, int, cudaStream_t);
template void launch_subtree_factor<double>(const DevPlan&, const DevNum<double>&, const int4*, int, const int32_t*,
                                            const int32_t*, int*, int, int, double, int, cudaStream_t);

template void launch_factor_small<float>(const DevPlan&, const DevNum<float>&, const int32_t*, int, int, double,
                                         int, cudaStream_t);
template void launch_factor_small<double>(const DevPlan&, const DevNum<double>&, const int32_t*, int, int, double,
                                          int, cudaStream_t);

// (a 192-column FP32 panel was measured slower than 128 columns on the
// condensed 300 x 300 and stabilized 700 x 700 grids: the diagonal role's
// serial chain of 32-column factorisations grows with the width)
void launch_macro_panel(const DevPlan& P, const DevNum<float>& N, const int4* items, int count, int* sync, int* err,
                        double eps, int policy, long long wait, cudaStream_t st) {
  if (count <= 0) return;
  static bool attr = false;
  const int smem = macro_panel_smem(4, MACRO_NB);
  if (!attr) {
    cudaFuncSetAttribute(k_macro_panel<float, MACRO_NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    attr = true;
  }
  k_macro_panel<float, MACRO_NB><<<count, 256, smem, st>>>(P, N, items, sync, err, eps, policy, wait);
}

}  // namespace ncl
