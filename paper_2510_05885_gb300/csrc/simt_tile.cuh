// FP32 and FP64 trailing updates on the CUDA cores (internal).
#pragma once
#include "runtime.h"

namespace ncl {

// ---------------------------------------------------------------------------
// SIMT update C -= A diag(d) B^T (lower part), 256 threads, TM x TM outputs
// per thread: rows TM ty .. TM ty + TM - 1 (16-byte shared loads of A per k)
// and columns tx + 16 b (conflict-free loads of B, and coalesced row segments
// of C).  FP32: FFMA, 64 x 64 tiles.  FP64: DFMA, 32 x 32 tiles: an SM does
// 1.7 to 2 of them per clock, so that a 64 x 64 tile 128 deep keeps its SM
// busy for 0.15 ms while the others have run out of tiles; at that rate the
// smaller tile's additional shared and global loads cost nothing.
// ---------------------------------------------------------------------------
// a thread's entries of a 16-byte aligned shared array
__device__ __forceinline__ void ld_shared(const float* p, float (&v)[4]) {
  const float4 x = *reinterpret_cast<const float4*>(p);
  v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
}
__device__ __forceinline__ void ld_shared(const double* p, double (&v)[2]) {
  const double2 x = *reinterpret_cast<const double2*>(p);
  v[0] = x.x; v[1] = x.y;
}

__device__ __forceinline__ void decode_tile(int64_t t, int Nt, int& ti, int& tj) {
  const int64_t tri = (int64_t)Nt * (Nt + 1) / 2;
  if (t < tri) {
    int a = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
    while ((int64_t)a * (a + 1) / 2 > t) a--;
    while ((int64_t)(a + 1) * (a + 2) / 2 <= t) a++;
    ti = a;
    tj = (int)(t - (int64_t)a * (a + 1) / 2);
  } else {
    const int64_t u = t - tri;
    ti = Nt + (int)(u / Nt);
    tj = (int)(u % Nt);
  }
}

template <typename T>
struct SimtTile {
  static constexpr int TB = gemm_tile(sizeof(T)), KC = 16, TM = TB / 16;
  T As[KC][TB + 4];   // rows 16-byte aligned
  T Bs[KC][TB + 1];
};

// tile gt of the launch's problems; called by 256 threads
template <typename T>
__device__ __forceinline__ void simt_tile(const DevNum<T>& N, const GemmProb* __restrict__ probs,
                                          const int32_t* __restrict__ tile_prob, int64_t gt, SimtTile<T>& sh) {
  constexpr int TB = SimtTile<T>::TB, KC = SimtTile<T>::KC, TM = SimtTile<T>::TM;
  auto& As = sh.As;
  auto& Bs = sh.Bs;
  const GemmProb pb = probs[tile_prob[gt]];
  int ti, tj;
  decode_tile(gt - pb.tile0, pb.Nt, ti, tj);
  const int i0 = ti * TB, j0 = tj * TB;
  const T* A = N.L + pb.a_off;
  const T* B = N.L + pb.b_off;
  const T* d = N.D + pb.d_off;
  T* C = (pb.c_in_u ? N.U : N.L) + pb.c_off;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  T acc[TM][TM];
#pragma unroll
  for (int a = 0; a < TM; a++)
#pragma unroll
    for (int b = 0; b < TM; b++) acc[a][b] = T(0);
  // the next K chunk is fetched into registers while the current one is
  // multiplied (thread: k = kk, rows rr + 16 q of A and of B)
  const int kk = threadIdx.x & 15, rr = threadIdx.x >> 4;
  T fa[TM], fb[TM];
  auto fetch = [&](int k0) {
    const int k = k0 + kk;
    const bool kin = k < pb.K;
    const T dk = kin ? d[k] : T(0);
#pragma unroll
    for (int q = 0; q < TM; q++) {
      const int ia = i0 + rr + 16 * q, jb = j0 + rr + 16 * q;
      fa[q] = (ia < pb.M && kin) ? A[(int64_t)ia * pb.lda + k] : T(0);
      fb[q] = (jb < pb.N && kin) ? B[(int64_t)jb * pb.lda + k] * dk : T(0);
    }
  };
  fetch(0);
  for (int k0 = 0; k0 < pb.K; k0 += KC) {
#pragma unroll
    for (int q = 0; q < TM; q++) {
      As[kk][rr + 16 * q] = fa[q];
      Bs[kk][rr + 16 * q] = fb[q];
    }
    __syncthreads();
    if (k0 + KC < pb.K) fetch(k0 + KC);
    // (FP64: the last chunk only as far as it goes, in fours)
    const int kc = sizeof(T) == 8 ? min(KC, (pb.K - k0 + 3) & ~3) : KC;
#pragma unroll (sizeof(T) == 8 ? 4 : KC)
    for (int k2 = 0; k2 < kc; k2++) {
      T av[TM], bv[TM];
      ld_shared(&As[k2][TM * ty], av);
#pragma unroll
      for (int b = 0; b < TM; b++) bv[b] = Bs[k2][tx + 16 * b];
#pragma unroll
      for (int a = 0; a < TM; a++)
#pragma unroll
        for (int b = 0; b < TM; b++) acc[a][b] += av[a] * bv[b];
    }
    __syncthreads();
  }
  // all loads of C first, then the stores
  T cv[TM][TM];
#pragma unroll
  for (int a = 0; a < TM; a++) {
    const int i = i0 + TM * ty + a;
#pragma unroll
    for (int b = 0; b < TM; b++) {
      const int j = j0 + tx + 16 * b;
      cv[a][b] = (i < pb.M && j < pb.N && j <= i) ? C[(int64_t)i * pb.ldc + j] : T(0);
    }
  }
#pragma unroll
  for (int a = 0; a < TM; a++) {
    const int i = i0 + TM * ty + a;
#pragma unroll
    for (int b = 0; b < TM; b++) {
      const int j = j0 + tx + 16 * b;
      if (i < pb.M && j < pb.N && j <= i) C[(int64_t)i * pb.ldc + j] = cv[a][b] - acc[a][b];
    }
  }
}

}  // namespace ncl
