// Inverses of the unit lower pivot blocks, after the factorisation (sm_103a).
//
// The triangular sweeps apply L11^-1 as a product (sweep.cu), so once all
// fronts are factored the strictly lower part of L11 is replaced by that of
// its inverse, in place:
//   - the 128 x 128 diagonal blocks by one CTA each, in shared memory: the
//     32 x 32 sub-blocks by a warp each, then pairs of inverted blocks A, C
//     with B below A merged, [A 0; B C]^-1 = [A^-1 0; -C^-1 B A^-1  C^-1];
//   - FP32: pairs of inverted blocks of 128, 256, ... columns merged by two
//     products, T = B A^-1 and X = -C^-1 T, over the tiles of all fronts in
//     one launch each.  T goes (transposed) to the upper triangle of the
//     pivot block, which nothing else uses.
// (The pivot blocks of at most 32 columns of the fronts kept in shared memory
// are inverted where they are factored.)  The factorisation itself uses
// substitution throughout; an error of the inverse only enters the solve's
// preconditioner, which the FP64 refinement corrects.  A product with an inverse
// leaves a larger residual than substitution where L11 is badly conditioned:
// against block-rows substituted with 32-column inverses, over condensed and
// stabilized grids and penalties 1e2 to 1e6 (12 to 20 draws each, both
// precisions), the error of an unrefined solution is 0.8 to 1.25 times as large
// (geometric means), its backward error 0.65 to 1.5 times, at the condensed
// form's penalty 1e5 2.2 to 2.6 times (at most 8); 775 refinement steps in all
// instead of 767.
#include "runtime.h"

namespace ncl {

namespace {

// merge the pairs of inverted h x h diagonal blocks of the WB x WB block A
// (unit diagonal stored, zero above it): 256 threads, TR x TC outputs each
template <typename T, int WB, int h, int TR, int TC>
__device__ __forceinline__ void merge_pairs(T* A, T* Tm) {
  constexpr int LDA = WB + 1, LDT = h + 1;
  constexpr int PT = (h / TR) * (h / TC);   // threads per pair
  static_assert(PT * (WB / (2 * h)) == 256, "one output tile per thread");
  const int p = threadIdx.x / PT, t = threadIdx.x % PT;
  const int i0 = (t / (h / TC)) * TR, n0 = (t % (h / TC)) * TC;
  const T* Ai = A + (2 * p * h) * LDA + 2 * p * h;
  T* Bp = A + ((2 * p + 1) * h) * LDA + 2 * p * h;
  const T* Ci = Bp + h;
  T* Tp = Tm + p * h * LDT;
  T acc[TR][TC];
#pragma unroll
  for (int a = 0; a < TR; a++)
#pragma unroll
    for (int b = 0; b < TC; b++) acc[a][b] = T(0);
#pragma unroll 4
  for (int k = n0; k < h; k++) {
    T x[TR], y[TC];
#pragma unroll
    for (int a = 0; a < TR; a++) x[a] = Bp[(i0 + a) * LDA + k];
#pragma unroll
    for (int b = 0; b < TC; b++) y[b] = Ai[k * LDA + n0 + b];
#pragma unroll
    for (int a = 0; a < TR; a++)
#pragma unroll
      for (int b = 0; b < TC; b++) acc[a][b] += x[a] * y[b];
  }
#pragma unroll
  for (int a = 0; a < TR; a++)
#pragma unroll
    for (int b = 0; b < TC; b++) {
      Tp[(i0 + a) * LDT + n0 + b] = acc[a][b];
      acc[a][b] = T(0);
    }
  __syncthreads();
#pragma unroll 4
  for (int k = 0; k < i0 + TR; k++) {
    T x[TR], y[TC];
#pragma unroll
    for (int a = 0; a < TR; a++) x[a] = Ci[(i0 + a) * LDA + k];
#pragma unroll
    for (int b = 0; b < TC; b++) y[b] = Tp[k * LDT + n0 + b];
#pragma unroll
    for (int a = 0; a < TR; a++)
#pragma unroll
      for (int b = 0; b < TC; b++) acc[a][b] += x[a] * y[b];
  }
#pragma unroll
  for (int a = 0; a < TR; a++)
#pragma unroll
    for (int b = 0; b < TC; b++) Bp[(i0 + a) * LDA + n0 + b] = -acc[a][b];
  __syncthreads();
}

}  // namespace

// items: (supernode, first column), a block of at most WB columns each
template <typename T, int WB>
__global__ void __launch_bounds__(256) k_invert_diag(DevPlan P, DevNum<T> N, const int2* __restrict__ items) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int LDA = WB + 1;
  T* A = reinterpret_cast<T*>(smem_raw);
  T* Tm = A + WB * LDA;
  const int2 it = items[blockIdx.x];
  const int ncp = P.sn_ncolp[it.x], w = min(WB, P.sn_ncol[it.x] - it.y);
  T* Lb = N.L + P.sn_Loff[it.x] + (int64_t)it.y * ncp + it.y;
  // the strictly lower part (only its own rows: a root's block may end the
  // factor's storage), unit diagonal
  for (int base = threadIdx.x; base < WB * WB; base += 8 * 256) {
    T v[8];
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const int idx = base + 256 * k, r = idx / WB, c = idx % WB;
      v[k] = (c < r && r < w) ? Lb[(int64_t)r * ncp + c] : (c == r ? T(1) : T(0));
    }
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const int idx = base + 256 * k;
      A[(idx / WB) * LDA + idx % WB] = v[k];
    }
  }
  __syncthreads();
  // the 32 x 32 sub-blocks: lane j forms column j of the inverse
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp < WB / 32) {
    T* D = A + (32 * warp) * LDA + 32 * warp;
    T x[32];
#pragma unroll
    for (int i = 0; i < 32; i++) {
      T a0 = T(0), a1 = T(0);
#pragma unroll
      for (int k = 0; k + 1 < i; k += 2) {
        a0 += D[i * LDA + k] * x[k];
        a1 += D[i * LDA + k + 1] * x[k + 1];
      }
      if (i & 1) a0 += D[i * LDA + i - 1] * x[i - 1];
      x[i] = (i == lane) ? T(1) : (i > lane ? -(a0 + a1) : T(0));
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 32; i++) D[i * LDA + lane] = x[i];
  }
  __syncthreads();
  if constexpr (WB == 64) {
    merge_pairs<T, WB, 32, 2, 2>(A, Tm);
  } else {
    merge_pairs<T, WB, 32, 2, 4>(A, Tm);
    merge_pairs<T, WB, 64, 4, 4>(A, Tm);
  }
  for (int idx = threadIdx.x; idx < w * WB; idx += 256) {
    const int r = idx / WB, c = idx % WB;
    if (c < r) Lb[(int64_t)r * ncp + c] = A[r * LDA + c];
  }
}

template <typename T>
void launch_invert_diag(const DevPlan& P, const DevNum<T>& N, const int2* items, int count, int width,
                        cudaStream_t st) {
  if (count <= 0) return;
  auto go = [&](auto k, int smem) {
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    k<<<count, 256, smem, st>>>(P, N, items);
  };
  if (width <= 64) go(k_invert_diag<T, 64>, (64 * 65 + 32 * 33) * (int)sizeof(T));
  else go(k_invert_diag<T, 128>, (128 * 129 + 64 * 65) * (int)sizeof(T));
}
template void launch_invert_diag<float>(const DevPlan&, const DevNum<float>&, const int2*, int, int, cudaStream_t);
template void launch_invert_diag<double>(const DevPlan&, const DevNum<double>&, const int2*, int, int, cudaStream_t);

// ---------------------------------------------------------------------------
// FP32 merges of wider blocks.  Item (supernode, q0, row tile, column tile):
// A^-1 is the h x h block at (q0, q0), C^-1 the m x m one at (q0 + h, q0 + h)
// (m <= h), B the m x h block below A.  A CTA of 256 threads forms a 128 x 64
// tile of T (SECOND = false, stored transposed above the diagonal) or of X,
// 8 x 4 outputs per thread, the operands' next 16 columns fetched while the
// current ones are multiplied; the triangular operand's zero part is skipped.
// FINE: 64 x 32 tiles, 4 x 2 outputs per thread, 32 columns at a time, four
// CTAs to an item: a launch that does not fill the chip lasts as long as a
// tile, and a 128 x 64 tile lasts as long as its multiplications, a 64 x 32 one
// as half as many load latencies (condensed 100 x 100 2.75 -> 2.66 ms per step,
// stabilized 150 x 150 3.47 -> 3.38 ms).  The products of an entry are summed
// in the same order either way.
// ---------------------------------------------------------------------------
template <bool SECOND, bool FINE>
__global__ void __launch_bounds__(256) k_invert_merge(DevPlan P, DevNum<float> N, const int4* __restrict__ items,
                                                      int h) {
  constexpr int TM = FINE ? 64 : 128, TN = FINE ? 32 : 64, KC = FINE ? 32 : 16, RA = TM / 16, RB = TN / 16;
  __shared__ __align__(16) float As[KC][TM + 4];
  __shared__ __align__(16) float Bs[KC][TN + 4];
  const int4 it = items[FINE ? blockIdx.x >> 2 : blockIdx.x];
  const int sub = FINE ? blockIdx.x & 3 : 0;
  const int ncol = P.sn_ncol[it.x], ncp = P.sn_ncolp[it.x];
  const int q0 = it.y, i0 = 128 * it.z + TM * (sub & 1), n0 = 64 * it.w + TN * (sub >> 1);
  const int m = min(h, ncol - q0 - h);
  if (FINE && i0 >= m) return;
  float* Lb = N.L + P.sn_Loff[it.x];
  float* low = Lb + (int64_t)(q0 + h) * ncp + q0;        // B, then X
  float* up = Lb + (int64_t)q0 * ncp + q0 + h;           // T transposed: up[n][i]
  const float* Ai = Lb + (int64_t)q0 * ncp + q0;
  const float* Ci = Lb + (int64_t)(q0 + h) * ncp + q0 + h;
  // T[i][n] = sum_{k >= n} B[i][k] Ai[k][n];  X[i][n] = -sum_{k <= i} Ci[i][k] T[k][n]
  const int kbeg = SECOND ? 0 : n0, kend = SECOND ? min(m, i0 + TM) : h;
  const int t = threadIdx.x, ar = t / (KC / 8), ak = t % (KC / 8) * 8;
  float4 fa[2], fb;
  auto fetch = [&](int k0) {
    const int i = i0 + ar;
#pragma unroll
    for (int q = 0; q < 2; q++) {
      const int k = k0 + ak + 4 * q;
      fa[q] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (i < m && k < kend) {   // (a vector past the pivots stays within the padded row)
        fa[q] = __ldg(reinterpret_cast<const float4*>((SECOND ? Ci : low) + (int64_t)i * ncp + k));
        float* f = reinterpret_cast<float*>(&fa[q]);
#pragma unroll
        for (int e = 0; e < 4; e++)
          if (SECOND) f[e] = k + e < i ? f[e] : (k + e == i ? 1.f : 0.f);
      }
    }
    fb = make_float4(0.f, 0.f, 0.f, 0.f);
    if (!SECOND) {
      const int k = k0 + t / (TN / 4), n = n0 + t % (TN / 4) * 4;
      if (k < kend) {
        fb = __ldg(reinterpret_cast<const float4*>(Ai + (int64_t)k * ncp + n));
        float* f = reinterpret_cast<float*>(&fb);
#pragma unroll
        for (int e = 0; e < 4; e++) f[e] = n + e < k ? f[e] : (n + e == k ? 1.f : 0.f);
      }
    } else {
      const int n = n0 + t / (KC / 4), k = k0 + t % (KC / 4) * 4;
      if (k < kend) {
        fb = __ldg(reinterpret_cast<const float4*>(up + (int64_t)n * ncp + k));
        float* f = reinterpret_cast<float*>(&fb);
#pragma unroll
        for (int e = 0; e < 4; e++) f[e] = k + e < m ? f[e] : 0.f;
      }
    }
  };
  const int tx = t & 15, ty = t >> 4;   // outputs: rows RA ty.., columns RB tx..
  float acc[RA][RB];
#pragma unroll
  for (int a = 0; a < RA; a++)
#pragma unroll
    for (int b = 0; b < RB; b++) acc[a][b] = 0.f;
  fetch(kbeg);
  for (int k0 = kbeg; k0 < kend; k0 += KC) {
#pragma unroll
    for (int q = 0; q < 2; q++)
#pragma unroll
      for (int e = 0; e < 4; e++) As[ak + 4 * q + e][ar] = reinterpret_cast<const float*>(&fa[q])[e];
    if (!SECOND) {
      *reinterpret_cast<float4*>(&Bs[t / (TN / 4)][t % (TN / 4) * 4]) = fb;
    } else {
#pragma unroll
      for (int e = 0; e < 4; e++) Bs[t % (KC / 4) * 4 + e][t / (KC / 4)] = reinterpret_cast<const float*>(&fb)[e];
    }
    __syncthreads();
    if (k0 + KC < kend) fetch(k0 + KC);
#pragma unroll
    for (int k = 0; k < KC; k++) {
      float xs[RA], ys[RB];
#pragma unroll
      for (int a = 0; a < RA; a += 4) *reinterpret_cast<float4*>(xs + a) = *reinterpret_cast<const float4*>(&As[k][RA * ty + a]);
      if constexpr (RB == 4) *reinterpret_cast<float4*>(ys) = *reinterpret_cast<const float4*>(&Bs[k][RB * tx]);
      else *reinterpret_cast<float2*>(ys) = *reinterpret_cast<const float2*>(&Bs[k][RB * tx]);
#pragma unroll
      for (int a = 0; a < RA; a++)
#pragma unroll
        for (int b = 0; b < RB; b++) acc[a][b] = fmaf(xs[a], ys[b], acc[a][b]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int a = 0; a < RA; a++) {
    const int i = i0 + RA * ty + a;
    if (i >= m) break;
#pragma unroll
    for (int b = 0; b < RB; b++) {
      const int n = n0 + RB * tx + b;
      if (SECOND) low[(int64_t)i * ncp + n] = -acc[a][b];
      else up[(int64_t)n * ncp + i] = acc[a][b];
    }
  }
}

void launch_invert_merge(const DevPlan& P, const DevNum<float>& N, const int4* items, int count, int h, bool second,
                         cudaStream_t st) {
  if (count <= 0) return;
  // four CTAs to an SM (76, 152, 304, 608 items: slack 200 6.16, 6.11, 6.09, 6.09 ms, condensed 300 12.91, 12.91, 12.87,
  // 12.85 ms, the others alike)
  const bool fine = count <= 608;
  const auto k = second ? (fine ? k_invert_merge<true, true> : k_invert_merge<true, false>)
                        : (fine ? k_invert_merge<false, true> : k_invert_merge<false, false>);
  k<<<fine ? 4 * count : count, 256, 0, st>>>(P, N, items, h);
}

}  // namespace ncl
