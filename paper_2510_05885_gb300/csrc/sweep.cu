// Triangular sweeps with the supernodal factors of P K P^T = L D L^T (sm_103a):
//   forward  L y = P b   leaves to root, level by level,
//   backward L^T x = D^-1 y   root to leaves,   then P^T x.
// After the factorisation the pivot blocks L11 hold their own inverses
// (invert.cu), so a pivot block is applied as a product, and a level of the
// tree takes one launch per direction (two where it has large supernodes):
//   forward   y1 = L11^-1 t1,  W = (children's updates) - L21 y1,
//             t1 = the supernode's right-hand side plus the children's updates;
//   backward  z1 = D^-1 y1 - L21^T x2,  x1 = L11^-T z1.
// Every front row pulls its children's updates itself, through a list of the
// entries of W that land on it (children in a fixed order): no atomics, and
// bitwise the same result every time.
//
// Roles (a block's role follows from its index):
//   narrow   at most 32 pivots and a small front: one warp per supernode;
//   block    at most 128 pivots and, on a level with little work, a front of at
//            most SWEEP_BLOCK_BYTES: one CTA of 256 threads per supernode, both
//            steps in one launch; forward, a large front's rows below are dealt
//            out to several CTAs, each forming y for itself;
//   strips   larger ones: runs of rows of [L11^-1; L21] (forward) or 16
//            columns of them (backward) per CTA, one launch for each of the
//            two steps.
// The vectors hold a pivot's right-hand sides next to each other (entry
// k * nrhs + r): a gathered row of up to 8 right-hand sides is one sector.
// y and z live in a vector of their own, so that no CTA overwrites what
// another one still reads.
//
// What bounds a sweep is the depth of the tree: some twenty dependent levels
// of a few microseconds each, while the factor itself would stream in 70 us
// (300 x 300 condensed) or 0.4 ms (700 x 700).  So a role reads what it needs
// with as few dependent loads as it can (one record per supernode, one per
// front row, factor entries as 16-byte vectors with several in flight), and
// a level's launch overlaps the end of the one before it.  Measured against
// chained 128-row block-rows with a launch each for the pivot blocks and the
// rows below: a refined solve of the stabilized 93 x 107 grid 2.54 -> 0.66 ms,
// of the condensed 300 x 300 grid with 8 right-hand sides 37.3 -> 10.8 ms (with
// one role per size of front and interleaved vectors in shared memory: 1.12 and
// 15.6 ms); the small subtrees' sweep 0.68 -> 0.41 (forward) and 0.71 -> 0.34 ms
// (backward) at 700 x 700, where one warp used to walk a subtree supernode by
// supernode.
#include "runtime.h"

#include <algorithm>
#include <type_traits>

namespace ncl {

namespace {

// 16-byte vectors of factor entries (rows of L start 16-byte aligned: the
// blocks start at multiples of 32 elements and the row stride is a multiple
// of 4 elements)
template <typename T> struct Vec16;
template <> struct Vec16<float> {
  using type = float4;
  static constexpr int n = 4;
};
template <> struct Vec16<double> {
  using type = double2;
  static constexpr int n = 2;
};
template <typename T> struct Vec2 { using type = float2; };
template <> struct Vec2<double> { using type = double2; };

__device__ __forceinline__ SnMeta load_meta(const SnMeta* p) {
  union {
    int4 v[3];
    SnMeta m;
  } u;
  const int4* q = reinterpret_cast<const int4*>(p);
#pragma unroll
  for (int i = 0; i < 3; i++) u.v[i] = __ldg(q + i);
  return u.m;
}

// Programmatic dependent launch: a level's kernel starts while the previous
// one drains, reads what the factorisation left (records, factor entries,
// index lists) and waits here before it touches xp, yv or W.  (Those pointers
// carry no __restrict__: a load the compiler knows to be read-only may be
// moved up across the wait.)
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void start_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename T, int NR>
__device__ __forceinline__ void load_rhs(const T* v, int64_t k, int nrhs, T (&out)[NR]) {
#pragma unroll
  for (int r = 0; r < NR; r++) out[r] = r < nrhs ? v[k * nrhs + r] : T(0);
}
template <typename T, int NR>
__device__ __forceinline__ void store_rhs(T* v, int64_t k, int nrhs, const T (&in)[NR]) {
#pragma unroll
  for (int r = 0; r < NR; r++)
    if (r < nrhs) v[k * nrhs + r] = in[r];
}

// The entries of W (children's updates) that land on K front rows of this
// thread.  A row's record holds its first two sources (most rows have one or
// two); further ones are in a list the second one then names.  index() reads
// the records, load() the values of the first two, add() sums in the
// children's order.
constexpr uint32_t WM_NONE = 0x7fffffffu, WM_LIST = 0x80000000u;

template <typename T, int NR, int K>
struct Pulls {
  uint2 s[K];
  T v0[K][NR], v1[K][NR];
  // frow(k): the front row, or a negative number for none
  template <typename F>
  __device__ __forceinline__ void index(const DevPlan& P, F frow) {
#pragma unroll
    for (int k = 0; k < K; k++) {
      const int64_t f = frow(k);
      s[k] = f >= 0 ? __ldg(P.wm + f) : make_uint2(WM_NONE, WM_NONE);
    }
  }
  __device__ __forceinline__ void load(const T* W, int nrhs) {
#pragma unroll
    for (int k = 0; k < K; k++)
#pragma unroll
      for (int r = 0; r < NR; r++) {
        v0[k][r] = (s[k].x != WM_NONE && r < nrhs) ? W[(int64_t)s[k].x * nrhs + r] : T(0);
        v1[k][r] = (s[k].y < WM_NONE && r < nrhs) ? W[(int64_t)s[k].y * nrhs + r] : T(0);
      }
  }
  __device__ __forceinline__ void add(const DevPlan& P, const T* W, int nrhs, T (&acc)[K][NR]) {
#pragma unroll
    for (int k = 0; k < K; k++) {
#pragma unroll
      for (int r = 0; r < NR; r++) acc[k][r] = acc[k][r] + v0[k][r] + v1[k][r];
      if (s[k].y & WM_LIST) {
        const uint32_t* l = P.wm_list + (s[k].y & WM_NONE);
        const uint32_t n = __ldg(l);
        for (uint32_t q = 1; q <= n; q++) {
          const uint32_t src = __ldg(l + q);
#pragma unroll
          for (int r = 0; r < NR; r++)
            if (r < nrhs) acc[k][r] += W[(int64_t)src * nrhs + r];
        }
      }
    }
  }
};

// ---------------------------------------------------------------------------
// narrow supernodes (at most 32 pivots): one warp
// ---------------------------------------------------------------------------
// vpr = the row's vectors rounded up to a power of two: vpr lanes read a row,
// the warp 32 / vpr rows at a time.
// U loads in flight per lane and 32 K rows below staged at a time: many in the
// level launches, whose time is one warp's; few in the subtree launches, which
// have more warps than fit and gain more from registers saved.
// Sums over the lanes go step by step for eight values together: one after the
// other, each a chain of shuffles, they took longer than the products (a block
// of 34 pivots 1.7 us for either product, backward 0.65 us; the refined solve
// of the stabilized 93 x 107 grid 1.06 -> 0.99 ms).
constexpr int SUMS(int nr, int n) { return nr >= 8 ? 1 : n < 8 / nr ? n : 8 / nr; }
constexpr int NARROW_K(int nr) { return nr >= 8 ? 2 : 4; }
constexpr int NARROW_SMEM(int nr, int k) { return (64 + 32 * k) * nr; }   // values per warp

template <typename T, int NR, int U, int K>
__device__ __forceinline__ void warp_fwd(const DevPlan& P, const DevNum<T>& N, int s, const T* xp, T* yv, T* W,
                                         int nrhs, int lane, T* tb) {
  using V = typename Vec16<T>::type;
  constexpr int VW = Vec16<T>::n, CR = 32 * K;
  T* ty = tb + 32 * NR;      // y
  T* gs = ty + 32 * NR;      // the children's updates of the rows below
  const SnMeta m = load_meta(P.sn_meta + s);
  const int nb = m.nrow - m.ncol;
  int vpr = 1;
  while (vpr * VW < m.ncol) vpr *= 2;
  const int G = 32 / vpr, g = lane / vpr, v = lane & (vpr - 1);
  const bool vok = v * VW < m.ncp;
  const T* Lb = N.L + m.L + v * VW;
  auto row_vec = [&](int row, int end) {
    if (vok && row < end) return __ldg(reinterpret_cast<const V*>(Lb + (int64_t)row * m.ncp));
    return V{};
  };
  V li[U], lb[U];
#pragma unroll
  for (int u = 0; u < U; u++) li[u] = row_vec(u * G + g, m.ncol);
#pragma unroll
  for (int u = 0; u < U; u++) lb[u] = row_vec(m.ncol + u * G + g, m.nrow);
  Pulls<T, NR, 1> pt;
  Pulls<T, NR, K> pb;
  pt.index(P, [&](int) { return lane < m.ncol ? m.rows + lane : (int64_t)-1; });
  pb.index(P, [&](int k) { return lane + 32 * k < nb ? m.rows + m.ncol + lane + 32 * k : (int64_t)-1; });
  wait_previous();
  T t[1][NR];
#pragma unroll
  for (int r = 0; r < NR; r++) t[0][r] = T(0);
  if (lane < m.ncol) load_rhs<T, NR>(xp, m.col0 + lane, nrhs, t[0]);
  pt.load(W, nrhs);
  pb.load(W, nrhs);
  pt.add(P, W, nrhs, t);
#pragma unroll
  for (int r = 0; r < NR; r++) {
    tb[lane * NR + r] = t[0][r];
    ty[lane * NR + r] = T(0);
  }
  auto stage = [&] {
    T a[K][NR];
#pragma unroll
    for (int k = 0; k < K; k++)
#pragma unroll
      for (int r = 0; r < NR; r++) a[k][r] = T(0);
    pb.add(P, W, nrhs, a);
#pragma unroll
    for (int k = 0; k < K; k++)
#pragma unroll
      for (int r = 0; r < NR; r++) gs[(lane + 32 * k) * NR + r] = a[k][r];
  };
  stage();
  __syncwarp();
  T x[VW][NR];
  auto lane_vec = [&](const T* src) {
#pragma unroll
    for (int e = 0; e < VW; e++)
#pragma unroll
      for (int r = 0; r < NR; r++) x[e][r] = src[(v * VW + e) * NR + r];
  };
  constexpr int B = SUMS(NR, U);
  static_assert(U % B == 0, "whole batches");
  auto row_sums = [&](T (&a)[B][NR]) {
    for (int o = vpr >> 1; o > 0; o >>= 1)
#pragma unroll
      for (int u = 0; u < B; u++)
#pragma unroll
        for (int r = 0; r < NR; r++) a[u][r] += __shfl_xor_sync(0xffffffffu, a[u][r], o);
  };
  // y = L11^-1 t
  lane_vec(tb);
  for (int u0 = 0; u0 * G < m.ncol; u0 += U) {
    if (u0 > 0)
#pragma unroll
      for (int u = 0; u < U; u++) li[u] = row_vec((u0 + u) * G + g, m.ncol);
#pragma unroll
    for (int ub = 0; ub < U; ub += B) {
      if ((u0 + ub) * G >= m.ncol) break;
      T a[B][NR];
#pragma unroll
      for (int u = 0; u < B; u++) {
        const int i = (u0 + ub + u) * G + g;
#pragma unroll
        for (int r = 0; r < NR; r++) a[u][r] = T(0);
#pragma unroll
        for (int e = 0; e < VW; e++) {
          const T l = v * VW + e < i ? reinterpret_cast<const T*>(&li[ub + u])[e] : T(0);
#pragma unroll
          for (int r = 0; r < NR; r++) a[u][r] += l * x[e][r];
        }
      }
      row_sums(a);
#pragma unroll
      for (int u = 0; u < B; u++) {
        const int i = (u0 + ub + u) * G + g;
        if (v != 0 || i >= m.ncol) continue;
#pragma unroll
        for (int r = 0; r < NR; r++) ty[i * NR + r] = a[u][r] += tb[i * NR + r];
        store_rhs<T, NR>(yv, m.col0 + i, nrhs, a[u]);
      }
    }
  }
  __syncwarp();
  // W = children's updates - L21 y
  lane_vec(ty);
  for (int c0 = 0; c0 < nb; c0 += CR) {
    const int n = min(CR, nb - c0);
    if (c0 > 0) {
      pb.index(P, [&](int k) {
        return c0 + lane + 32 * k < nb ? m.rows + m.ncol + c0 + lane + 32 * k : (int64_t)-1;
      });
      pb.load(W, nrhs);
      __syncwarp();
      stage();
      __syncwarp();
    }
    for (int u0 = 0; u0 * G < n; u0 += U) {
      if (c0 + u0 > 0)
#pragma unroll
        for (int u = 0; u < U; u++) lb[u] = row_vec(m.ncol + c0 + (u0 + u) * G + g, m.nrow);
#pragma unroll
      for (int ub = 0; ub < U; ub += B) {
        if ((u0 + ub) * G >= n) break;
        T a[B][NR];
#pragma unroll
        for (int u = 0; u < B; u++) {
#pragma unroll
          for (int r = 0; r < NR; r++) a[u][r] = T(0);
#pragma unroll
          for (int e = 0; e < VW; e++)   // (the padding columns of L are zero, and so is y there)
#pragma unroll
            for (int r = 0; r < NR; r++) a[u][r] += reinterpret_cast<const T*>(&lb[ub + u])[e] * x[e][r];
        }
        row_sums(a);
#pragma unroll
        for (int u = 0; u < B; u++) {
          const int a0 = (u0 + ub + u) * G + g;
          if (v != 0 || a0 >= n) continue;
#pragma unroll
          for (int r = 0; r < NR; r++) a[u][r] = gs[a0 * NR + r] - a[u][r];
          store_rhs<T, NR>(W, (int64_t)m.W + c0 + a0, nrhs, a[u]);
        }
      }
    }
  }
  __syncwarp();
}

template <typename T, int NR, int U, int K>
__device__ __forceinline__ void warp_bwd(const DevPlan& P, const DevNum<T>& N, int s, T* xp, const T* yv, int nrhs,
                                         int lane, T* tb) {
  using V = typename Vec16<T>::type;
  constexpr int VW = Vec16<T>::n, CR = 32 * K;
  T* tx = tb + 32 * NR;      // column sums
  T* xs = tx + 32 * NR;      // x of the rows below
  const SnMeta m = load_meta(P.sn_meta + s);
  const int nb = m.nrow - m.ncol;
  int vpr = 1;
  while (vpr * VW < m.ncol) vpr *= 2;
  const int G = 32 / vpr, g = lane / vpr, v = lane & (vpr - 1);
  const bool vok = v * VW < m.ncp;
  const T* Lb = N.L + m.L + v * VW;
  auto row_vec = [&](int row, int end) {
    if (vok && row < end) return __ldg(reinterpret_cast<const V*>(Lb + (int64_t)row * m.ncp));
    return V{};
  };
  V l[U];
#pragma unroll
  for (int u = 0; u < U; u++) l[u] = row_vec(m.ncol + u * G + g, m.ncol + min(nb, CR));   // (the staged rows only)
  const int32_t* rows = P.sn_rows + m.rows + m.ncol;
  int idx[K];
#pragma unroll
  for (int k = 0; k < K; k++) idx[k] = lane + 32 * k < nb ? __ldg(rows + lane + 32 * k) : -1;
  const T d = lane < m.ncol ? N.D[m.col0 + lane] : T(1);
  wait_previous();
  T z[NR];
#pragma unroll
  for (int r = 0; r < NR; r++) z[r] = T(0);
  if (lane < m.ncol) load_rhs<T, NR>(yv, m.col0 + lane, nrhs, z);
  T acc[VW][NR];
#pragma unroll
  for (int e = 0; e < VW; e++)
#pragma unroll
    for (int r = 0; r < NR; r++) acc[e][r] = T(0);
  for (int c0 = 0; c0 < nb; c0 += CR) {
    const int n = min(CR, nb - c0);
    if (c0 > 0)
#pragma unroll
      for (int k = 0; k < K; k++) idx[k] = c0 + lane + 32 * k < nb ? __ldg(rows + c0 + lane + 32 * k) : -1;
    __syncwarp();
    {
      T x[K][NR];
#pragma unroll
      for (int k = 0; k < K; k++)
#pragma unroll
        for (int r = 0; r < NR; r++) x[k][r] = (idx[k] >= 0 && r < nrhs) ? xp[(int64_t)idx[k] * nrhs + r] : T(0);
#pragma unroll
      for (int k = 0; k < K; k++)
#pragma unroll
        for (int r = 0; r < NR; r++) xs[(lane + 32 * k) * NR + r] = x[k][r];
    }
    __syncwarp();
    for (int u0 = 0; u0 * G < n; u0 += U) {
      if (c0 + u0 > 0)
#pragma unroll
        for (int u = 0; u < U; u++) l[u] = row_vec(m.ncol + c0 + (u0 + u) * G + g, m.ncol + c0 + n);
#pragma unroll
      for (int u = 0; u < U; u++) {
        const int a = min((u0 + u) * G + g, CR - 1);   // (rows past the end have l = 0)
#pragma unroll
        for (int e = 0; e < VW; e++)
#pragma unroll
          for (int r = 0; r < NR; r++) acc[e][r] += reinterpret_cast<const T*>(&l[u])[e] * xs[a * NR + r];
      }
    }
  }
  // the inverse's rows, in flight during the reductions
#pragma unroll
  for (int u = 0; u < U; u++) l[u] = row_vec(u * G + g, m.ncol);
  auto col_sum = [&] {   // over the groups, to tx
    for (int o = vpr; o < 32; o *= 2)
#pragma unroll
      for (int e = 0; e < VW; e++)
#pragma unroll
        for (int r = 0; r < NR; r++) acc[e][r] += __shfl_xor_sync(0xffffffffu, acc[e][r], o);
    __syncwarp();
    if (g == 0)
#pragma unroll
      for (int e = 0; e < VW; e++)
#pragma unroll
        for (int r = 0; r < NR; r++) tx[(v * VW + e) * NR + r] = acc[e][r];
    __syncwarp();
  };
  col_sum();
  // z = D^-1 y - L21^T x2, x = L11^-T z
#pragma unroll
  for (int r = 0; r < NR; r++)
    tb[lane * NR + r] = z[r] = lane < m.ncol ? z[r] / d - tx[lane * NR + r] : T(0);
  __syncwarp();
#pragma unroll
  for (int e = 0; e < VW; e++)
#pragma unroll
    for (int r = 0; r < NR; r++) acc[e][r] = T(0);
  for (int u0 = 0; u0 * G < m.ncol; u0 += U) {
    if (u0 > 0)
#pragma unroll
      for (int u = 0; u < U; u++) l[u] = row_vec((u0 + u) * G + g, m.ncol);
#pragma unroll
    for (int u = 0; u < U; u++) {
      const int i = (u0 + u) * G + g;
#pragma unroll
      for (int e = 0; e < VW; e++) {
        const T le = i > v * VW + e ? reinterpret_cast<const T*>(&l[u])[e] : T(0);
#pragma unroll
        for (int r = 0; r < NR; r++) acc[e][r] += le * tb[min(i, 31) * NR + r];
      }
    }
  }
  col_sum();
  if (lane < m.ncol) {
#pragma unroll
    for (int r = 0; r < NR; r++) z[r] += tx[lane * NR + r];
    store_rhs<T, NR>(xp, m.col0 + lane, nrhs, z);
  }
  __syncwarp();
}

// ---------------------------------------------------------------------------
// one CTA of 256 threads per supernode (at most 128 pivots, at most
// SWEEP_BLOCK_BELOW rows below)
// ---------------------------------------------------------------------------
// rows in flight per group of lanes
constexpr int BLOCK_RPT(int nr) { return nr >= 4 ? 4 : 8; }

template <typename T, int NR>
__device__ __forceinline__ void block_fwd(const DevPlan& P, const DevNum<T>& N, const int4 it, const T* xp, T* yv, T* W,
                                          int nrhs, T* smem) {
  using V = typename Vec16<T>::type;
  constexpr int VW = Vec16<T>::n, RPT = BLOCK_RPT(NR), PK = NR >= 4 ? 1 : 2;   // pulled rows per thread at a time
  // t and y by right-hand side: a lane reads a vector of them in one conflict-free 16-byte load.  Interleaved, the
  // lanes of a warp met in the same banks; eight right-hand sides on the 300x300 system: 15.5 -> 12.9 ms per solve.
  T* ts = smem;              // [NR][128]
  T* ys = ts + 128 * NR;     // [NR][128]
  T* gs = ys + 128 * NR;     // rows below * NR
  const SnMeta m = load_meta(P.sn_meta + it.x);
  const T* Lb = N.L + m.L;
  const int rlo = it.y, nb = it.z - it.y, tid = threadIdx.x;
  const int nv = (m.ncol + VW - 1) / VW;
  int tpr = 4;
  while (tpr < 32 && tpr < nv) tpr *= 2;
  const int v0 = tid & (tpr - 1), slots = 256 / tpr, slot = tid / tpr;
  Pulls<T, NR, 1> pt;
  Pulls<T, NR, PK> pb;
  pt.index(P, [&](int) { return tid < m.ncol ? m.rows + tid : (int64_t)-1; });
  auto below = [&](int k) { return tid + 256 * k < nb ? m.rows + rlo + tid + 256 * k : (int64_t)-1; };
  pb.index(P, below);
  // the pivot rows' first vectors (FP32: the row's only one for each lane)
  V l[RPT];
  auto fetch = [&](int row0, int end, int v, bool tri) {
#pragma unroll
    for (int k = 0; k < RPT; k++) {
      const int row = row0 + k * slots + slot;
      if (row < end && v < nv && (!tri || v * VW < row))
        l[k] = __ldg(reinterpret_cast<const V*>(Lb + (int64_t)row * m.ncp) + v);
      else
        l[k] = V{};
    }
  };
  fetch(0, m.ncol, v0, true);
  wait_previous();
  {
    T t[1][NR];
#pragma unroll
    for (int r = 0; r < NR; r++) t[0][r] = T(0);
    if (tid < m.ncol) load_rhs<T, NR>(xp, m.col0 + tid, nrhs, t[0]);
    pt.load(W, nrhs);
    pb.load(W, nrhs);
    pt.add(P, W, nrhs, t);
    if (tid < 128)
#pragma unroll
      for (int r = 0; r < NR; r++) {
        ts[r * 128 + tid] = t[0][r];
        ys[r * 128 + tid] = T(0);
      }
    for (int k0 = 0; 256 * k0 < nb; k0 += PK) {
      if (k0 > 0) {
        pb.index(P, [&](int k) { return below(k0 + k); });
        pb.load(W, nrhs);
      }
      T a[PK][NR];
#pragma unroll
      for (int k = 0; k < PK; k++)
#pragma unroll
        for (int r = 0; r < NR; r++) a[k][r] = T(0);
      pb.add(P, W, nrhs, a);
#pragma unroll
      for (int k = 0; k < PK; k++)
        if (tid + 256 * (k0 + k) < nb)
#pragma unroll
          for (int r = 0; r < NR; r++) gs[(tid + 256 * (k0 + k)) * NR + r] = a[k][r];
    }
  }
  __syncthreads();
  // rows [0, ncol): y = t + (row left of the diagonal) t; then the rows below:
  // W = children's updates - row y
  auto pass = [&](int row0, int end, const T* x, bool tri, bool fetched) {
    T acc[RPT][NR];
#pragma unroll
    for (int k = 0; k < RPT; k++)
#pragma unroll
      for (int r = 0; r < NR; r++) acc[k][r] = T(0);
    for (int v = v0; v < tpr || v < nv; v += tpr) {
      if (v != v0 || !fetched) fetch(row0, end, v, tri);
#pragma unroll
      for (int r = 0; r < NR; r++) {
        const V x4 = *reinterpret_cast<const V*>(x + r * 128 + v * VW);   // zero past the pivots
#pragma unroll
        for (int e = 0; e < VW; e++)
#pragma unroll
          for (int k = 0; k < RPT; k++)
            acc[k][r] += ((!tri || v * VW + e < row0 + k * slots + slot) ? reinterpret_cast<const T*>(&l[k])[e] : T(0)) *
                         reinterpret_cast<const T*>(&x4)[e];
      }
    }
#pragma unroll
    for (int k0 = 0; k0 < RPT; k0 += SUMS(NR, RPT))
      for (int o = tpr >> 1; o > 0; o >>= 1)
#pragma unroll
        for (int k = k0; k < k0 + SUMS(NR, RPT); k++)
#pragma unroll
          for (int r = 0; r < NR; r++) acc[k][r] += __shfl_xor_sync(0xffffffffu, acc[k][r], o);
#pragma unroll
    for (int k = 0; k < RPT; k++) {
      const int row = row0 + k * slots + slot;
      if (v0 == 0 && row < end) {
        if (tri) {
#pragma unroll
          for (int r = 0; r < NR; r++) ys[r * 128 + row] = acc[k][r] += ts[r * 128 + row];
          if (rlo == m.ncol) store_rhs<T, NR>(yv, m.col0 + row, nrhs, acc[k]);
        } else {
#pragma unroll
          for (int r = 0; r < NR; r++) acc[k][r] = gs[(row - rlo) * NR + r] - acc[k][r];
          store_rhs<T, NR>(W, (int64_t)m.W + row - m.ncol, nrhs, acc[k]);
        }
      }
    }
  };
  for (int r0 = 0; r0 < m.ncol; r0 += RPT * slots) pass(r0, m.ncol, ts, true, r0 == 0);
  fetch(rlo, it.z, v0, false);   // (in flight across the barrier)
  __syncthreads();
  for (int r0 = rlo; r0 < it.z; r0 += RPT * slots) pass(r0, it.z, ys, false, r0 == rlo);
}

template <typename T, int NR>
__device__ __forceinline__ void block_bwd(const DevPlan& P, const DevNum<T>& N, int s, T* xp, const T* yv, int nrhs,
                                          T* smem) {
  using V = typename Vec16<T>::type;
  constexpr int VW = Vec16<T>::n, K = SWEEP_BLOCK_BELOW / 256;
  T* zs = smem;                    // 128 * NR
  T* red = zs + 128 * NR;          // 8 warps * 32 * VW * NR
  T* xs = red + 256 * VW * NR;     // rows below * NR
  const SnMeta m = load_meta(P.sn_meta + s);
  const int nb = m.nrow - m.ncol, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // vpr lanes (a power of two; FP64: up to two warps) read a row, the CTA
  // 256 / vpr rows at a time, eight loads in flight per lane
  int vpr = 1;
  while (vpr * VW < m.ncol) vpr *= 2;
  const int v = tid & (vpr - 1), rg = tid / vpr, RG = 256 / vpr;
  const bool vok = v * VW < m.ncp;
  const T* Lb = N.L + m.L + v * VW;
  V l[8];
  auto fetch = [&](int row0, int end) {
#pragma unroll
    for (int u = 0; u < 8; u++) {
      const int row = row0 + u * RG + rg;
      if (vok && row < end) l[u] = __ldg(reinterpret_cast<const V*>(Lb + (int64_t)row * m.ncp));
      else l[u] = V{};
    }
  };
  fetch(m.ncol, m.nrow);
  int idx[K];
#pragma unroll
  for (int k = 0; k < K; k++) idx[k] = tid + 256 * k < nb ? __ldg(P.sn_rows + m.rows + m.ncol + tid + 256 * k) : -1;
  const T d = tid < m.ncol ? N.D[m.col0 + tid] : T(1);
  wait_previous();
  T z[NR], acc[VW][NR];
#pragma unroll
  for (int r = 0; r < NR; r++) z[r] = T(0);
  if (tid < m.ncol) load_rhs<T, NR>(yv, m.col0 + tid, nrhs, z);
#pragma unroll
  for (int k = 0; k < K; k++)
    if (idx[k] >= 0) {
      T x[NR];
      load_rhs<T, NR>(xp, idx[k], nrhs, x);
#pragma unroll
      for (int r = 0; r < NR; r++) xs[(tid + 256 * k) * NR + r] = x[r];
    }
  auto zero = [&] {
#pragma unroll
    for (int e = 0; e < VW; e++)
#pragma unroll
      for (int r = 0; r < NR; r++) acc[e][r] = T(0);
  };
  // the CTA's sums of this thread's column (threads below ncol), after a barrier
  auto col_sum = [&](T (&out)[NR]) {
    for (int o = vpr; o < 32; o *= 2)
#pragma unroll
      for (int e = 0; e < VW; e++)
#pragma unroll
        for (int r = 0; r < NR; r++) acc[e][r] += __shfl_xor_sync(0xffffffffu, acc[e][r], o);
    if (lane < vpr)
#pragma unroll
      for (int e = 0; e < VW; e++)
#pragma unroll
        for (int r = 0; r < NR; r++) red[((warp * 32 + lane) * VW + e) * NR + r] = acc[e][r];
    __syncthreads();
#pragma unroll
    for (int r = 0; r < NR; r++) out[r] = T(0);
    if (tid < m.ncol) {
      const int cv = tid / VW, step = vpr > 32 ? vpr / 32 : 1;   // warps that hold this vector
      for (int w = cv >> 5; w < 8; w += step)
#pragma unroll
        for (int r = 0; r < NR; r++) out[r] += red[((w * 32 + (cv & 31)) * VW + tid % VW) * NR + r];
    }
  };
  zero();
  __syncthreads();
  for (int r0 = 0; r0 < nb; r0 += 8 * RG) {
    if (r0 > 0) fetch(m.ncol + r0, m.nrow);
#pragma unroll
    for (int u = 0; u < 8; u++) {
      const int a = min(r0 + u * RG + rg, nb - 1);   // (rows past the end have l = 0)
#pragma unroll
      for (int e = 0; e < VW; e++)
#pragma unroll
        for (int r = 0; r < NR; r++) acc[e][r] += reinterpret_cast<const T*>(&l[u])[e] * xs[a * NR + r];
    }
  }
  fetch(0, m.ncol);   // the inverse's rows, in flight during the reduction
  T sum[NR];
  col_sum(sum);
  if (tid < m.ncol)
#pragma unroll
    for (int r = 0; r < NR; r++) zs[tid * NR + r] = z[r] = z[r] / d - sum[r];
  zero();
  __syncthreads();
  for (int r0 = 0; r0 < m.ncol; r0 += 8 * RG) {
    if (r0 > 0) fetch(r0, m.ncol);
#pragma unroll
    for (int u = 0; u < 8; u++) {
      const int i = r0 + u * RG + rg, ic = min(i, m.ncol - 1);
#pragma unroll
      for (int e = 0; e < VW; e++) {
        const T le = i > v * VW + e ? reinterpret_cast<const T*>(&l[u])[e] : T(0);
#pragma unroll
        for (int r = 0; r < NR; r++) acc[e][r] += le * zs[ic * NR + r];
      }
    }
  }
  col_sum(sum);
  if (tid < m.ncol) {
#pragma unroll
    for (int r = 0; r < NR; r++) z[r] += sum[r];
    store_rhs<T, NR>(xp, m.col0 + tid, nrhs, z);
  }
}

// ---------------------------------------------------------------------------
// strips of large supernodes
// ---------------------------------------------------------------------------
// Rows [it.y, it.z) of [L11^-1; L21], all of them pivot rows or all below:
// each warp two rows at a time, their vectors read by the 32 lanes.  A pivot
// row i gives y_i = t_i + (row left of the diagonal) . t, a row below W =
// (children's updates) - row . y.  The vector is staged in shared memory in
// chunks of CH entries (a supernode wider than a chunk has 16 rows to a CTA,
// so that each warp has one pair of rows).
template <typename T, int NR>
__device__ __forceinline__ void strip_fwd(const DevPlan& P, const DevNum<T>& N, const int4 it, const T* xp, T* yv,
                                          T* W, int nrhs, T* vec, int ldv) {
  using V = typename Vec16<T>::type;
  constexpr int VW = Vec16<T>::n, CH = SWEEP_CHUNK_BYTES / (NR * (int)sizeof(T)), U = 4;
  const SnMeta m = load_meta(P.sn_meta + it.x);
  const T* Lb = N.L + m.L;
  const bool piv = it.y < m.ncol;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int K = piv ? it.z : m.ncol;   // entries of the vector that matter
  int held = -1;                       // the chunk in shared memory
  for (int p0 = it.y; p0 < it.z; p0 += 16) {
    const int ra = p0 + 2 * warp, rb = ra + 1;
    const int ka = piv ? ra : m.ncol, kb = piv ? rb : m.ncol;   // row lengths
    const T* la = Lb + (int64_t)min(ra, m.nrow - 1) * m.ncp;
    const T* lb = Lb + (int64_t)min(rb, m.nrow - 1) * m.ncp;
    V va[U], vb[U];
    auto fetch = [&](int c0, int k0, int lim) {
#pragma unroll
      for (int u = 0; u < U; u++) {
        const int k = k0 + (32 * u + lane) * VW;
        const bool ok = k < lim;
        va[u] = ok ? __ldg(reinterpret_cast<const V*>(la + c0 + k)) : V{};
        vb[u] = ok ? __ldg(reinterpret_cast<const V*>(lb + c0 + k)) : V{};
      }
    };
    fetch(0, 0, min(min(CH, K), kb));
    // lane 0 finishes row ra, lane 1 row rb
    Pulls<T, NR, 1> pg;
    const bool mine = lane < 2 && ra + lane < it.z;
    pg.index(P, [&](int) { return mine ? m.rows + ra + lane : (int64_t)-1; });
    T g[1][NR];
    T a0[NR], a1[NR];
#pragma unroll
    for (int r = 0; r < NR; r++) g[0][r] = a0[r] = a1[r] = T(0);
    for (int c0 = 0; c0 < K; c0 += CH) {
      const int len = min(CH, K - c0), plen = (len + 3) & ~3;
      if (held != c0) {
        if (held >= 0) __syncthreads();
        // SK entries per thread at a time, their loads in flight together
        constexpr int SK = NR >= 8 ? 1 : (NR >= 4 ? 2 : 4);
        Pulls<T, NR, SK> pv;
        auto frow = [&](int j) { return piv && j < len ? m.rows + c0 + j : (int64_t)-1; };
        pv.index(P, [&](int k) { return frow(threadIdx.x + 256 * k); });
        if (held < 0) wait_previous();
        for (int j0 = threadIdx.x; j0 < plen; j0 += 256 * SK) {
          T t[SK][NR];
          if (j0 >= 256 * SK) pv.index(P, [&](int k) { return frow(j0 + 256 * k); });
#pragma unroll
          for (int k = 0; k < SK; k++)
#pragma unroll
            for (int r = 0; r < NR; r++)
              t[k][r] = (j0 + 256 * k < len && r < nrhs)
                            ? (piv ? xp : yv)[(int64_t)(m.col0 + c0 + j0 + 256 * k) * nrhs + r]
                            : T(0);
          pv.load(W, nrhs);
          pv.add(P, W, nrhs, t);
#pragma unroll
          for (int k = 0; k < SK; k++)
            if (j0 + 256 * k < plen)
#pragma unroll
              for (int r = 0; r < NR; r++) vec[r * ldv + j0 + 256 * k] = t[k][r];
        }
        held = c0;
        if (c0 == 0) pg.load(W, nrhs);
        __syncthreads();
      } else if (c0 == 0) {
        pg.load(W, nrhs);
      }
      if (c0 == 0 && mine && piv) load_rhs<T, NR>(xp, m.col0 + ra + lane, nrhs, g[0]);
      const int lim = min(len, kb - c0);   // both rows end here at most
      for (int k0 = 0; k0 < lim; k0 += 32 * U * VW) {
        if (c0 + k0 > 0) fetch(c0, k0, lim);
#pragma unroll
        for (int u = 0; u < U; u++) {
          const int k = k0 + (32 * u + lane) * VW;
          if (k < lim) {
            T xa[VW], xb[VW];
#pragma unroll
            for (int e = 0; e < VW; e++) {
              xa[e] = c0 + k + e < ka ? reinterpret_cast<const T*>(&va[u])[e] : T(0);
              xb[e] = c0 + k + e < kb ? reinterpret_cast<const T*>(&vb[u])[e] : T(0);
            }
#pragma unroll
            for (int r = 0; r < NR; r++) {
              const V x4 = *reinterpret_cast<const V*>(vec + r * ldv + k);
#pragma unroll
              for (int e = 0; e < VW; e++) {
                a0[r] += xa[e] * reinterpret_cast<const T*>(&x4)[e];
                a1[r] += xb[e] * reinterpret_cast<const T*>(&x4)[e];
              }
            }
          }
        }
      }
    }
#pragma unroll
    for (int r = 0; r < NR; r++)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        a0[r] += __shfl_xor_sync(0xffffffffu, a0[r], o);
        a1[r] += __shfl_xor_sync(0xffffffffu, a1[r], o);
      }
    if (mine) {
      pg.add(P, W, nrhs, g);
#pragma unroll
      for (int r = 0; r < NR; r++) {
        const T a = lane ? a1[r] : a0[r];
        g[0][r] = piv ? g[0][r] + a : g[0][r] - a;
      }
      if (piv) store_rhs<T, NR>(yv, m.col0 + ra + lane, nrhs, g[0]);
      else store_rhs<T, NR>(W, (int64_t)m.W + ra + lane - m.ncol, nrhs, g[0]);
    }
  }
}

// Columns [it.y, it.y + 16) of L21 (PIV = false: z = D^-1 y - L21^T x2, kept
// in yv) or of L11^-1 (PIV: x = z + the entries below the diagonal times z):
// a row's 16 columns are one 64-byte (FP64: 128-byte) segment, read by 4 (8)
// lanes, the CTA's 64 (32) groups of lanes striding over the rows.
template <typename T, int NR, bool PIV>
__device__ __forceinline__ void strip_bwd(const DevPlan& P, const DevNum<T>& N, const int4 it, T* xp, T* yv, int nrhs,
                                          T* smem) {
  using V = typename Vec16<T>::type;
  constexpr int VW = Vec16<T>::n, LPR = 16 / VW, CH = SWEEP_CHUNK_BYTES / (NR * (int)sizeof(T));
  T* red = smem;                    // 8 warps * 16 columns * NR
  T* vec = smem + 8 * 16 * NR;
  const SnMeta m = load_meta(P.sn_meta + it.x);
  const int j0 = it.y, cl = threadIdx.x & (LPR - 1), rg = threadIdx.x / LPR, RG = blockDim.x / LPR;
  const int jc = j0 + cl * VW;      // this lane's first column
  const int n = PIV ? m.ncol - j0 : m.nrow - m.ncol;   // rows (PIV: from row j0)
  const bool root = m.nrow == m.ncol;                  // nothing below: z = D^-1 y has not been formed
  const T* base = N.L + m.L + (int64_t)(PIV ? j0 : m.ncol) * m.ncp + jc;
  T acc[VW][NR];
#pragma unroll
  for (int e = 0; e < VW; e++)
#pragma unroll
    for (int r = 0; r < NR; r++) acc[e][r] = T(0);
  V l[8];
  auto fetch = [&](int i0, int end) {
#pragma unroll
    for (int u = 0; u < 8; u++) {
      const int i = i0 + u * RG + rg;
      if (jc < m.ncp && i < end) l[u] = __ldg(reinterpret_cast<const V*>(base + (int64_t)i * m.ncp));
      else l[u] = V{};
    }
  };
  fetch(0, min(n, CH));
  for (int c0 = 0; c0 < n; c0 += CH) {
    const int len = min(CH, n - c0);
    __syncthreads();
    for (int i0 = threadIdx.x; i0 < len; i0 += 4 * 256) {
      // four entries per thread, their loads in flight together
      int64_t k[4];
      T d[4], x[4][NR];
#pragma unroll
      for (int q = 0; q < 4; q++) {
        const int i = c0 + i0 + 256 * q;
        k[q] = c0 + len <= i ? -1 : (PIV ? m.col0 + j0 + i : __ldg(P.sn_rows + m.rows + m.ncol + i));
        d[q] = (PIV && root && k[q] >= 0) ? N.D[k[q]] : T(1);
      }
      wait_previous();   // (only the first call waits)
#pragma unroll
      for (int q = 0; q < 4; q++)
#pragma unroll
        for (int r = 0; r < NR; r++)
          x[q][r] = (k[q] >= 0 && r < nrhs) ? (PIV ? yv : xp)[k[q] * nrhs + r] / d[q] : T(0);
#pragma unroll
      for (int q = 0; q < 4; q++)
        if (k[q] >= 0)
#pragma unroll
          for (int r = 0; r < NR; r++) vec[(i0 + 256 * q) * NR + r] = x[q][r];
    }
    __syncthreads();
    for (int i0 = 0; i0 < len; i0 += 8 * RG) {
      if (c0 + i0 > 0) fetch(c0 + i0, c0 + len);
#pragma unroll
      for (int u = 0; u < 8; u++) {
        const int i = i0 + u * RG + rg, ic = min(i, len - 1);   // (rows past the end have l = 0)
#pragma unroll
        for (int e = 0; e < VW; e++) {
          const T le = (!PIV || c0 + i > cl * VW + e) ? reinterpret_cast<const T*>(&l[u])[e] : T(0);
#pragma unroll
          for (int r = 0; r < NR; r++) acc[e][r] += le * vec[ic * NR + r];
        }
      }
    }
  }
  wait_previous();   // (threads that staged nothing)
#pragma unroll
  for (int e = 0; e < VW; e++)
#pragma unroll
    for (int r = 0; r < NR; r++) {
#pragma unroll
      for (int o = 16; o >= LPR; o >>= 1) acc[e][r] += __shfl_xor_sync(0xffffffffu, acc[e][r], o);
    }
  const int warp = threadIdx.x >> 5;
  if ((threadIdx.x & 31) < LPR)
#pragma unroll
    for (int e = 0; e < VW; e++)
#pragma unroll
      for (int r = 0; r < NR; r++) red[(warp * 16 + cl * VW + e) * NR + r] = acc[e][r];
  __syncthreads();
  const int c = threadIdx.x / NR, r = threadIdx.x % NR;
  if (c < 16 && j0 + c < m.ncol && r < nrhs) {
    T sum = T(0);
#pragma unroll
    for (int w = 0; w < 8; w++) sum += red[(w * 16 + c) * NR + r];
    const int64_t k = m.col0 + j0 + c;
    T v = yv[k * nrhs + r];
    if (!PIV || root) v /= N.D[k];
    if (PIV) xp[k * nrhs + r] = v + sum;
    else yv[k * nrhs + r] = v - sum;
  }
}

}  // namespace

// ---------------------------------------------------------------------------
// level launches
// ---------------------------------------------------------------------------
// blocks [0, nnarrow / 8): narrow supernodes, eight to a CTA; then one block
// supernode per CTA; then one strip per CTA
template <typename T, int NR>
__global__ void __launch_bounds__(256) k_fwd_level(DevPlan P, DevNum<T> N, SweepItems I, const T* xp,
                                                   T* yv, T* W, int nrhs) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* smem = reinterpret_cast<T*>(smem_raw);
  start_next();
  int b = blockIdx.x;
  const int nw = (I.nnarrow + 7) / 8;
  if (b < nw) {
    const int w = threadIdx.x >> 5, i = 8 * b + w;
    if (i < I.nnarrow) warp_fwd<T, NR, 8, NARROW_K(NR)>(P, N, I.narrow[i], xp, yv, W, nrhs, threadIdx.x & 31, smem + w * NARROW_SMEM(NR, NARROW_K(NR)));
    return;
  }
  b -= nw;
  if (b < I.nblock) {
    block_fwd<T, NR>(P, N, I.fblock[b], xp, yv, W, nrhs, smem);
    return;
  }
  strip_fwd<T, NR>(P, N, I.strips[b - I.nblock], xp, yv, W, nrhs, smem,
                   min((I.vec + 3) & ~3, SWEEP_CHUNK_BYTES / (NR * (int)sizeof(T))));
}

template <typename T, int NR, bool PIV>
__global__ void __launch_bounds__(256) k_bwd_level(DevPlan P, DevNum<T> N, SweepItems I, T* xp, T* yv, int nrhs) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* smem = reinterpret_cast<T*>(smem_raw);
  start_next();
  int b = blockIdx.x;
  const int nw = (I.nnarrow + 7) / 8;
  if (b < nw) {
    const int w = threadIdx.x >> 5, i = 8 * b + w;
    if (i < I.nnarrow) warp_bwd<T, NR, 8, NARROW_K(NR)>(P, N, I.narrow[i], xp, yv, nrhs, threadIdx.x & 31, smem + w * NARROW_SMEM(NR, NARROW_K(NR)));
    return;
  }
  b -= nw;
  if (b < I.nblock) {
    block_bwd<T, NR>(P, N, I.block[b], xp, yv, nrhs, smem);
    return;
  }
  strip_bwd<T, NR, PIV>(P, N, I.strips[b - I.nblock], xp, yv, nrhs, smem);
}

// ---------------------------------------------------------------------------
// The region of small subtrees (at most 32 pivots per supernode, see the
// subtree factorisation): one CTA of 4 warps per maximal subtree, its
// supernodes level by level (a warp each), one launch per direction for the
// whole region.  items: (first node, nodes, first level bound, levels); the
// bounds of an item's levels are offsets into its nodes.
// ---------------------------------------------------------------------------
template <typename T, int NR>
__global__ void __launch_bounds__(128, NR >= 4 ? 5 : 8) k_region_fwd(DevPlan P, DevNum<T> N, const int4* __restrict__ items,
                                                    const int32_t* __restrict__ nodes,
                                                    const int32_t* __restrict__ bounds, const T* xp,
                                                    T* yv, T* W, int nrhs) {
  __shared__ T tb[4][NARROW_SMEM(NR, 1)];
  const int4 it = items[blockIdx.x];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int l = 0; l < it.w; l++) {
    const int q1 = bounds[it.z + l + 1];
    for (int q = bounds[it.z + l] + warp; q < q1; q += 4)
      warp_fwd<T, NR, 4, 1>(P, N, nodes[it.x + q], xp, yv, W, nrhs, lane, tb[warp]);
    if (l + 1 < it.w) __syncthreads();
  }
}

template <typename T, int NR>
__global__ void __launch_bounds__(128, NR >= 4 ? 5 : 8) k_region_bwd(DevPlan P, DevNum<T> N, const int4* __restrict__ items,
                                                    const int32_t* __restrict__ nodes,
                                                    const int32_t* __restrict__ bounds, T* xp, const T* yv,
                                                    int nrhs) {
  __shared__ T tb[4][NARROW_SMEM(NR, 1)];
  const int4 it = items[blockIdx.x];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int l = it.w - 1; l >= 0; l--) {
    const int q1 = bounds[it.z + l + 1];
    for (int q = bounds[it.z + l] + warp; q < q1; q += 4)
      warp_bwd<T, NR, 4, 1>(P, N, nodes[it.x + q], xp, yv, nrhs, lane, tb[warp]);
    if (l > 0) __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// FP64 factors: pivot blocks wider than 128, chained over 128-row block-rows
// (inverting them whole would cost n^3 / 3 operations at the FP64 rate, more
// than the one or two sweeps of an FP64 solve gain; the 128 x 128 diagonal
// blocks are inverted).  One CTA per block-row, which takes its block-row
// from the supernode's ticket counter, in order, so every block-row it waits
// for belongs to a CTA that is already running: the waits cannot deadlock,
// whatever the order in which CTAs are scheduled.  Waits are bounded: past
// the limit the CTA sets the sweep's error flag, goes on with what it has
// and still publishes, so that nobody waits on it; the host then reports the
// sweep as failed.
//   forward:  y_B = L_BB^-1 (t_B - sum_{J<B} L_BJ y_J)
//   backward: x_B = L_BB^-T (z_B - sum_{I>B} L_IB^T x_I)
// ---------------------------------------------------------------------------
namespace {

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(int* p, int v) {
  asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// thread 0 waits (bounded by `limit` clock cycles) for the flag; err is the
// sweep's error flag: once set, nobody waits any more
__device__ __forceinline__ void chain_wait(const int* flag, int* err, long long limit) {
  if (ld_acquire(flag) || ld_acquire(err)) return;
  const long long t0 = clock64();
  while (!ld_acquire(flag)) {
    if (clock64() - t0 > limit || ld_acquire(err)) {
      atomicExch(err, 1);
      break;
    }
    __nanosleep(32);
  }
}

constexpr int CHAIN_THREADS = 512;

}  // namespace

// items: (supernode, first block-row flag)
template <typename T, int NR>
__global__ void __launch_bounds__(CHAIN_THREADS) k_fwd_chain(DevPlan P, DevNum<T> N, const int2* __restrict__ items,
                                                             const T* __restrict__ xp, T* yv,
                                                             const T* __restrict__ W, int nrhs, int* tickets,
                                                             int* flags, int* err, long long wait) {
  __shared__ T ts[CHAIN_ROWS * NR], ys[CHAIN_ROWS * NR];
  __shared__ int sb;
  const int2 it = items[blockIdx.x];
  if (threadIdx.x == 0) sb = atomicAdd(&tickets[it.x], 1);
  __syncthreads();
  const int B = sb;
  const SnMeta m = load_meta(P.sn_meta + it.x);
  const int R0 = CHAIN_ROWS * B, nr = min(CHAIN_ROWS, m.ncol - R0);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const T* Lb = N.L + m.L + (int64_t)R0 * m.ncp;
  if (threadIdx.x < CHAIN_ROWS) {
    const int i = threadIdx.x;
    Pulls<T, NR, 1> p;
    p.index(P, [&](int) { return i < nr ? m.rows + R0 + i : (int64_t)-1; });
    T t[1][NR];
#pragma unroll
    for (int r = 0; r < NR; r++) t[0][r] = T(0);
    if (i < nr) load_rhs<T, NR>(xp, m.col0 + R0 + i, nrhs, t[0]);
    p.load(W, nrhs);
    p.add(P, W, nrhs, t);
#pragma unroll
    for (int r = 0; r < NR; r++) ts[i * NR + r] = t[0][r];
  }
  // four lanes to a row: a lane sums the columns 8 j + 2 t, 8 j + 2 t + 1 of
  // its row (t = lane % 4), so that two additions across lanes end a sum.  (A
  // warp over a row needs five, at 64 cycles each in FP64, for every row; that
  // was more than the products: 88 -> 37 us for the levels with more than 128 pivots of the condensed
  // 100 x 100 grid's root.)  A block's entries are loaded before the wait for
  // the vector they meet.
  static_assert(CHAIN_THREADS == 4 * CHAIN_ROWS, "four lanes to a row");
  const int row = threadIdx.x >> 2, t2 = 2 * (threadIdx.x & 3);
  const T* Lr = Lb + (int64_t)(row < nr ? row : 0) * m.ncp + t2;
  using V2 = typename Vec2<T>::type;
  constexpr int NV = CHAIN_ROWS / 8;
  V2 l[NV];
  auto fetch = [&](int c0, bool tri) {
#pragma unroll
    for (int j = 0; j < NV; j++) {
      l[j] = V2{T(0), T(0)};
      if (row < nr && (!tri || 8 * j + t2 < row)) l[j] = __ldg(reinterpret_cast<const V2*>(Lr + c0 + 8 * j));
    }
  };
  T acc[NR];
#pragma unroll
  for (int r = 0; r < NR; r++) acc[r] = T(0);
  auto product = [&](const T* v, bool tri) {
#pragma unroll
    for (int j = 0; j < NV; j++) {
      const int c = 8 * j + t2;
      const T l1 = !tri || c + 1 < row ? l[j].y : T(0);
#pragma unroll
      for (int r = 0; r < NR; r++) {
        acc[r] += l[j].x * v[c * NR + r];
        acc[r] += l1 * v[(c + 1) * NR + r];
      }
    }
  };
  auto reduce = [&] {
#pragma unroll
    for (int r = 0; r < NR; r++) {
      acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], 1);
      acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], 2);
    }
  };
  for (int J = 0; J < B; J++) {
    fetch(CHAIN_ROWS * J, false);
    if (threadIdx.x == 0) chain_wait(flags + it.y + J, err, wait);
    __syncthreads();
    for (int i = threadIdx.x; i < CHAIN_ROWS * NR; i += blockDim.x) {
      const int c = i / NR, r = i % NR;
      ys[i] = r < nrhs ? __ldcg(yv + (int64_t)(m.col0 + CHAIN_ROWS * J + c) * nrhs + r) : T(0);
    }
    __syncthreads();
    product(ys, false);
  }
  fetch(R0, true);
  reduce();
  __syncthreads();
  if (t2 == 0)
#pragma unroll
    for (int r = 0; r < NR; r++) ts[row * NR + r] -= acc[r];
  __syncthreads();
#pragma unroll
  for (int r = 0; r < NR; r++) acc[r] = T(0);
  product(ts, true);
  reduce();
  if (t2 == 0) {
#pragma unroll
    for (int r = 0; r < NR; r++) acc[r] += ts[row * NR + r];
    if (row < nr) store_rhs<T, NR>(yv, m.col0 + R0 + row, nrhs, acc);
  }
  __syncthreads();
  if (threadIdx.x == 0) st_release(flags + it.y + B, 1);
}

template <typename T, int NR>
__global__ void __launch_bounds__(CHAIN_THREADS) k_bwd_chain(DevPlan P, DevNum<T> N, const int2* __restrict__ items,
                                                             T* xp, const T* __restrict__ yv, int nrhs, int* tickets,
                                                             int* flags, int* err, long long wait) {
  __shared__ T zs[CHAIN_ROWS * NR], xs[CHAIN_ROWS * NR], red[(CHAIN_THREADS - CHAIN_ROWS) * NR];
  __shared__ int sb;
  const int2 it = items[blockIdx.x];
  const SnMeta m = load_meta(P.sn_meta + it.x);
  const int nbr = (m.ncol + CHAIN_ROWS - 1) / CHAIN_ROWS;
  if (threadIdx.x == 0) sb = nbr - 1 - atomicAdd(&tickets[it.x], 1);
  __syncthreads();
  const int B = sb;
  const int R0 = CHAIN_ROWS * B, nr = min(CHAIN_ROWS, m.ncol - R0);
  constexpr int G = CHAIN_THREADS / CHAIN_ROWS;
  const int c = threadIdx.x & (CHAIN_ROWS - 1), g = threadIdx.x / CHAIN_ROWS;   // column, row group
  const T* Lc = N.L + m.L + R0 + min(c, nr - 1);
  for (int i = threadIdx.x; i < CHAIN_ROWS; i += blockDim.x) {
    T z[NR];
#pragma unroll
    for (int r = 0; r < NR; r++) z[r] = T(0);
    if (i < nr) {
      load_rhs<T, NR>(yv, m.col0 + R0 + i, nrhs, z);
      if (m.nrow == m.ncol) {   // nothing below: z = D^-1 y has not been formed
        const T d = N.D[m.col0 + R0 + i];
#pragma unroll
        for (int r = 0; r < NR; r++) z[r] /= d;
      }
    }
#pragma unroll
    for (int r = 0; r < NR; r++) zs[i * NR + r] = z[r];
  }
  T acc[NR];
#pragma unroll
  for (int r = 0; r < NR; r++) acc[r] = T(0);
  auto reduce = [&] {   // the groups' sums to group 0's threads
    if (g > 0)
#pragma unroll
      for (int r = 0; r < NR; r++) red[((g - 1) * CHAIN_ROWS + c) * NR + r] = acc[r];
    __syncthreads();
    if (g == 0)
#pragma unroll
      for (int q = 0; q < G - 1; q++)
#pragma unroll
        for (int r = 0; r < NR; r++) acc[r] += red[(q * CHAIN_ROWS + c) * NR + r];
  };
  for (int I = nbr - 1; I > B; I--) {
    const int I0 = CHAIN_ROWS * I, ni = min(CHAIN_ROWS, m.ncol - I0);
    if (threadIdx.x == 0) chain_wait(flags + it.y + I, err, wait);
    __syncthreads();
    for (int i = threadIdx.x; i < CHAIN_ROWS * NR; i += blockDim.x) {
      const int k = i / NR, r = i % NR;
      xs[i] = (r < nrhs && k < ni) ? __ldcg(xp + (int64_t)(m.col0 + I0 + k) * nrhs + r) : T(0);
    }
    __syncthreads();
#pragma unroll 8
    for (int i = g; i < ni; i += G) {
      const T l = __ldg(Lc + (int64_t)(I0 + i) * m.ncp);
#pragma unroll
      for (int r = 0; r < NR; r++) acc[r] += l * xs[i * NR + r];
    }
  }
  __syncthreads();
  reduce();
  if (g == 0)
#pragma unroll
    for (int r = 0; r < NR; r++) zs[c * NR + r] -= acc[r];
  __syncthreads();
#pragma unroll
  for (int r = 0; r < NR; r++) acc[r] = T(0);
#pragma unroll 8
  for (int i = g; i < nr; i += G) {
    const T l = i > c ? __ldg(Lc + (int64_t)(R0 + i) * m.ncp) : T(0);
#pragma unroll
    for (int r = 0; r < NR; r++) acc[r] += l * zs[i * NR + r];
  }
  reduce();
  if (g == 0 && c < nr) {
#pragma unroll
    for (int r = 0; r < NR; r++) acc[r] += zs[c * NR + r];
    store_rhs<T, NR>(xp, m.col0 + R0 + c, nrhs, acc);
  }
  __syncthreads();
  if (threadIdx.x == 0) st_release(flags + it.y + B, 1);
}

// ---------------------------------------------------------------------------
// permutations between the caller's columns and the interleaved vector
// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_perm_in(DevPlan P, T* __restrict__ xp, const double* __restrict__ B, int64_t ldb, int nrhs) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < P.dim; k += (int64_t)gridDim.x * blockDim.x) {
    const int32_t src = P.perm[k];
    for (int r = 0; r < nrhs; r++) xp[k * nrhs + r] = (T)B[r * ldb + src];
  }
}

template <typename T>
__global__ void k_perm_out(DevPlan P, const T* __restrict__ xp, double* __restrict__ X, int64_t ldx, int nrhs,
                           int accumulate) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < P.dim; k += (int64_t)gridDim.x * blockDim.x) {
    const int32_t dst = P.perm[k];
    for (int r = 0; r < nrhs; r++) {
      const double v = (double)xp[k * nrhs + r];
      if (accumulate) X[r * ldx + dst] += v;
      else X[r * ldx + dst] = v;
    }
  }
}

static unsigned perm_grid(int64_t n) { return (unsigned)std::min<int64_t>((n + 255) / 256, 152 * 16); }

template <typename T>
void launch_perm_in(const DevPlan& P, T* xp, const double* B, int64_t ldb, int nrhs, cudaStream_t st) {
  if (P.dim) k_perm_in<T><<<perm_grid(P.dim), 256, 0, st>>>(P, xp, B, ldb, nrhs);
}
template <typename T>
void launch_perm_out(const DevPlan& P, const T* xp, double* X, int64_t ldx, int nrhs, int acc, cudaStream_t st) {
  if (P.dim) k_perm_out<T><<<perm_grid(P.dim), 256, 0, st>>>(P, xp, X, ldx, nrhs, acc);
}

// ---------------------------------------------------------------------------
// launchers: the kernels are compiled for 1, 2, 4 and 8 right-hand sides
// ---------------------------------------------------------------------------
template <typename F>
static void by_nrhs(int nrhs, F&& f) {
  if (nrhs <= 1) f(std::integral_constant<int, 1>{});
  else if (nrhs <= 2) f(std::integral_constant<int, 2>{});
  else if (nrhs <= 4) f(std::integral_constant<int, 4>{});
  else f(std::integral_constant<int, 8>{});
}

// a launch that may start before the previous kernel of the stream has ended
// (the kernel waits itself, see wait_previous); overlap = false: after a
// memset, an ordinary launch.  The limit on a kernel's dynamic shared memory
// belongs to the kernel and the device, not to the launch or the handle: every
// launch asks for the same one, the most that any launch of the kernel takes,
// so that threads with a handle each cannot lower it for one another between
// the request and the launch.  (Errors of either call stay with the thread
// until the sweeps' cudaGetLastError.)
template <int SMEM_MAX, typename... KA, typename... A>
static void launch_overlapped(bool overlap, void (*k)(KA...), int grid, int block, int smem, cudaStream_t st, A... args) {
  static_assert(SMEM_MAX <= 227 * 1024, "a CTA's shared memory");
  if (smem > 48 * 1024) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX);
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = overlap ? 1 : 0;
  cudaLaunchKernelEx(&cfg, k, KA(args)...);
}

static int level_blocks(const SweepItems& I) { return (I.nnarrow + 7) / 8 + I.nblock + I.nstrips; }

// dynamic shared memory of a level launch: the roles' needs, the staged vector
// of `vec` entries at most a chunk
static constexpr int level_smem(bool narrow, bool block, bool strips, int block_below, int vec, int nr, int esz, bool bwd) {
  int v = narrow ? 8 * NARROW_SMEM(nr, NARROW_K(nr)) / nr : 0;   // values per right-hand side
  if (block) v = std::max(v, (bwd ? 128 + 256 * (16 / esz) : 256) + block_below);
  if (strips) v = std::max(v, std::min((vec + 3) & ~3, SWEEP_CHUNK_BYTES / (nr * esz)) + (bwd ? 8 * 16 : 0));
  return v * nr * esz;
}
static int level_smem(const SweepItems& I, int nr, int esz, bool bwd) {
  return level_smem(I.nnarrow > 0, I.nblock > 0, I.nstrips > 0, I.block_below, I.vec, nr, esz, bwd);
}
// the most a launch takes: every role, a full chunk
static constexpr int level_smem_max(int nr, int esz, bool bwd) {
  return level_smem(true, true, true, SWEEP_BLOCK_BELOW, SWEEP_CHUNK_BYTES, nr, esz, bwd);
}

template <typename T>
void launch_fwd_level(const DevPlan& P, const DevNum<T>& N, const SweepItems& I, const T* xp, T* yv, T* W, int nrhs,
                      bool overlap, cudaStream_t st) {
  const int grid = level_blocks(I);
  if (grid <= 0) return;
  by_nrhs(nrhs, [&](auto nr) {
    constexpr int NR = decltype(nr)::value;
    const int smem = level_smem(I, NR, sizeof(T), false);
    launch_overlapped<level_smem_max(NR, sizeof(T), false)>(overlap, k_fwd_level<T, NR>, grid, 256, smem, st, P, N, I, xp, yv, W, nrhs);
  });
}

template <typename T>
void launch_bwd_level(const DevPlan& P, const DevNum<T>& N, const SweepItems& I, bool piv, T* xp, T* yv, int nrhs,
                      cudaStream_t st) {
  const int grid = level_blocks(I);
  if (grid <= 0) return;
  by_nrhs(nrhs, [&](auto nr) {
    constexpr int NR = decltype(nr)::value;
    const int smem = level_smem(I, NR, sizeof(T), true);
    constexpr int most = level_smem_max(NR, sizeof(T), true);
    if (piv) launch_overlapped<most>(true, k_bwd_level<T, NR, true>, grid, 256, smem, st, P, N, I, xp, yv, nrhs);
    else launch_overlapped<most>(true, k_bwd_level<T, NR, false>, grid, 256, smem, st, P, N, I, xp, yv, nrhs);
  });
}

template <typename T>
void launch_region_fwd(const DevPlan& P, const DevNum<T>& N, const int4* items, int count, const int32_t* nodes,
                       const int32_t* bounds, const T* xp, T* yv, T* W, int nrhs, cudaStream_t st) {
  if (count <= 0) return;
  by_nrhs(nrhs, [&](auto nr) {
    k_region_fwd<T, decltype(nr)::value><<<count, 128, 0, st>>>(P, N, items, nodes, bounds, xp, yv, W, nrhs);
  });
}

template <typename T>
void launch_region_bwd(const DevPlan& P, const DevNum<T>& N, const int4* items, int count, const int32_t* nodes,
                       const int32_t* bounds, T* xp, const T* yv, int nrhs, cudaStream_t st) {
  if (count <= 0) return;
  by_nrhs(nrhs, [&](auto nr) {
    k_region_bwd<T, decltype(nr)::value><<<count, 128, 0, st>>>(P, N, items, nodes, bounds, xp, yv, nrhs);
  });
}

// FP32 sweeps have no chains; the FP32 kernel is there for the self-test of a
// wait that runs out, which has one right-hand side
template <typename T>
void launch_fwd_chain(const DevPlan& P, const DevNum<T>& N, const int2* items, int count, const T* xp, T* yv,
                      const T* W, int nrhs, int* tickets, int* flags, int* err, long long wait, cudaStream_t st) {
  if (count <= 0) return;
  auto go = [&](auto nr) {
    k_fwd_chain<T, decltype(nr)::value><<<count, CHAIN_THREADS, 0, st>>>(P, N, items, xp, yv, W, nrhs, tickets, flags,
                                                                         err, wait);
  };
  if constexpr (sizeof(T) == 8) by_nrhs(nrhs, go);
  else go(std::integral_constant<int, 1>{});
}

void launch_bwd_chain(const DevPlan& P, const DevNum<double>& N, const int2* items, int count, double* xp,
                      const double* yv, int nrhs, int* tickets, int* flags, int* err, long long wait, cudaStream_t st) {
  if (count <= 0) return;
  by_nrhs(nrhs, [&](auto nr) {
    k_bwd_chain<double, decltype(nr)::value><<<count, CHAIN_THREADS, 0, st>>>(P, N, items, xp, yv, nrhs, tickets, flags,
                                                                              err, wait);
  });
}

#define NCL_INST(T)                                                                                               \
  template void launch_perm_in<T>(const DevPlan&, T*, const double*, int64_t, int, cudaStream_t);                 \
  template void launch_perm_out<T>(const DevPlan&, const T*, double*, int64_t, int, int, cudaStream_t);           \
  template void launch_fwd_level<T>(const DevPlan&, const DevNum<T>&, const SweepItems&, const T*, T*, T*, int,   \
                                    bool, cudaStream_t);                                                                \
  template void launch_bwd_level<T>(const DevPlan&, const DevNum<T>&, const SweepItems&, bool, T*, T*, int,       \
                                    cudaStream_t);                                                                \
  template void launch_region_fwd<T>(const DevPlan&, const DevNum<T>&, const int4*, int, const int32_t*,          \
                                     const int32_t*, const T*, T*, T*, int, cudaStream_t);                        \
  template void launch_region_bwd<T>(const DevPlan&, const DevNum<T>&, const int4*, int, const int32_t*,          \
                                     const int32_t*, T*, const T*, int, cudaStream_t);                            \
  template void launch_fwd_chain<T>(const DevPlan&, const DevNum<T>&, const int2*, int, const T*, T*, const T*,   \
                                    int, int*, int*, int*, long long, cudaStream_t);
NCL_INST(float)
NCL_INST(double)
#undef NCL_INST

}  // namespace ncl
