// Batched inverses and solves of dense complex matrices by blocked in-place
// Gauss-Jordan elimination with partial pivoting (setup of the leaf maps and of
// the preconditioner's cluster blocks, recovery of the leaf solutions).
//
// One panel of NB columns at a time, two launches each:
//
//  * panel   one CTA per matrix, the N x NB panel in registers (a thread owns
//            whole rows).  Unblocked in-place Gauss-Jordan on the panel with the
//            pivots searched among the rows not yet used; afterwards the panel
//            holds Z with  Z_K = P^{-1},  Z_i = -A_iK P^{-1}  (K the NB pivot
//            rows after the interchanges, P = A_KK).  The CTA then makes the
//            interchanges in the other columns and copies their rows K to U.
//  * update  A_ij <- (i in K ? 0 : A_ij) + (Z U)_ij for the columns outside the
//            panel, 64 x 32 tiles over all matrices of the batch.
//
// Inverse: X = A^{-1} up to the interchanges, A^{-1}[:, perm[i]] = X[:, i].
// Solve: only the columns right of the panel are updated; the columns
// [N, ncols) end as A^{-1} times their input.
//
// What bounds it: in complex double the FP64 pipe (4 fused multiply-adds per
// entry and panel column, two per SM and clock on GB300); the update has 8 NB
// of them per 32 bytes moved, so narrow panels (NB = 8) already keep memory out
// of the way and the panel launches short.  In complex float the batches are
// small and the panels' chain of N pivot searches dominates; wider panels
// (NB = 16) halve the launches and the passes over the matrices.
#include <algorithm>

#include "common.cuh"
#include "hps_internal.h"

namespace hps {

namespace {

template <class T>
struct GjArgs {
  T* A;
  long long stride;  // elements between matrices
  int ld, N, ncols;  // ncols > N: right-hand sides (solve)
  int solve;
  T* U;              // [matrix][NB][ncols]
  long long ustride;
  int* perm;         // [matrix][pstride]
  int pstride;
  const int* ids;    // matrix of each CTA (nullptr: 0, 1, ...)
  int* status;
};

// Pivot key: grows with |re| + |im| (sign-free high words of the number).
__device__ __forceinline__ unsigned pivot_key(double2 v) { return (unsigned)__double2hiint(fabs(v.x) + fabs(v.y)); }
__device__ __forceinline__ unsigned pivot_key(float2 v) { return __float_as_uint(fabsf(v.x) + fabsf(v.y)); }

// v -= m * u
__device__ __forceinline__ void cfms(double2& v, double2 m, double2 u) {
  v.x = fma(-m.x, u.x, fma(m.y, u.y, v.x));
  v.y = fma(-m.x, u.y, fma(-m.y, u.x, v.y));
}

// NT threads, RP rows per thread: N <= NT * RP.
template <class T, int NB, int NT, int RP>
__global__ void __launch_bounds__(NT) gj_panel_kernel(const GjArgs<T> a, int k0, int nb) {
  constexpr int kNone = 0x7fffffff;
  __shared__ T ps[NB], ks[NB], pinv_s;
  __shared__ unsigned wkey[NT / 32];
  __shared__ int widx[NT / 32];
  __shared__ int piv[NB];
  __shared__ int mv_row[2 * NB], mv_src[2 * NB], mv_n;
  const int b = a.ids ? a.ids[blockIdx.x] : (int)blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  T* M = a.A + b * a.stride;
  const int N = a.N;
  T row[RP][NB];
#pragma unroll
  for (int i = 0; i < RP; ++i) {
    const int r = tid + i * NT;
#pragma unroll
    for (int j = 0; j < NB; ++j) row[i][j] = (r < N && j < nb) ? M[(long long)r * a.ld + k0 + j] : czero<T>();
  }
#pragma unroll
  for (int c = 0; c < NB; ++c) {
    if (c >= nb) break;
    const int k = k0 + c;
    // pivot: the largest entry of column k among the rows >= k, the first one on a tie
    unsigned key = 0;
    int idx = kNone;
#pragma unroll
    for (int i = 0; i < RP; ++i) {
      const int r = tid + i * NT;
      if (r >= k && r < N) {
        const unsigned kk = pivot_key(row[i][c]);
        if (idx == kNone || kk > key) {
          key = kk;
          idx = r;
        }
      }
    }
    unsigned wm = __reduce_max_sync(0xffffffffu, key);
    int p = __reduce_min_sync(0xffffffffu, key == wm ? idx : kNone);
    if (lane == 0) {
      wkey[warp] = wm;
      widx[warp] = p;
    }
    __syncthreads();
    key = lane < NT / 32 ? wkey[lane] : 0u;
    idx = lane < NT / 32 ? widx[lane] : kNone;
    wm = __reduce_max_sync(0xffffffffu, key);
    p = __reduce_min_sync(0xffffffffu, key == wm ? idx : kNone);
    // the owners of rows p and k publish them (and the pivot's inverse)
#pragma unroll
    for (int i = 0; i < RP; ++i) {
      const int r = tid + i * NT;
      if (r == p) {
        const T pv = row[i][c];
        const bool ok = pv.x != 0 || pv.y != 0;
        if (!ok || pv.x != pv.x || pv.y != pv.y) atomicExch(a.status, 1);
        pinv_s = ok ? cinv(pv) : czero<T>();
#pragma unroll
        for (int j = 0; j < NB; ++j) ps[j] = row[i][j];
        piv[c] = p;
      }
      if (r == k)
#pragma unroll
        for (int j = 0; j < NB; ++j) ks[j] = row[i][j];
    }
    __syncthreads();
    const T inv = pinv_s;
#pragma unroll
    for (int i = 0; i < RP; ++i) {
      const int r = tid + i * NT;
      if (r >= N) continue;
      if (r == k) {  // the pivot row, divided by the pivot
#pragma unroll
        for (int j = 0; j < NB; ++j) row[i][j] = j == c ? inv : cmul(ps[j], inv);
        continue;
      }
      if (r == p)  // row k moved to the pivot's place
#pragma unroll
        for (int j = 0; j < NB; ++j) row[i][j] = ks[j];
      const T m = cmul(row[i][c], inv);
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        if (j == c) {
          row[i][j].x = -m.x;
          row[i][j].y = -m.y;
        } else {
          cfms(row[i][j], m, ps[j]);
        }
      }
    }
  }
#pragma unroll
  for (int i = 0; i < RP; ++i) {
    const int r = tid + i * NT;
    if (r >= N) continue;
#pragma unroll
    for (int j = 0; j < NB; ++j)
      if (j < nb) M[(long long)r * a.ld + k0 + j] = row[i][j];
  }
  // The interchanges of the panel as one move of at most 2 NB rows: lane l of warp 0 holds a row
  // involved (lanes < nb: the rows k0 + l) and which lane's old content ends there.
  if (warp == 0) {
    int rid = lane < nb ? k0 + lane : -1, src = lane, n = nb;
    for (int c = 0; c < nb; ++c) {
      const int p = piv[c];
      unsigned hit = __ballot_sync(0xffffffffu, rid == p);
      if (!hit) {
        if (lane == n) rid = p;
        hit = 1u << n;
        ++n;
      }
      const int l = __ffs(hit) - 1;
      const int sc = __shfl_sync(0xffffffffu, src, c), sl = __shfl_sync(0xffffffffu, src, l);
      if (lane == c) src = sl;
      if (lane == l) src = sc;
    }
    const int from = __shfl_sync(0xffffffffu, rid, src);
    if (lane < n) {
      mv_row[lane] = rid;
      mv_src[lane] = from;
    }
    if (lane == 0) mv_n = n;
  }
  int* perm = a.perm + (long long)b * a.pstride;
  if (k0 == 0)
    for (int r = tid; r < N; r += NT) perm[r] = r;
  __syncthreads();
  const int n = mv_n;
  if (warp == 0) {
    const int v = lane < n ? perm[mv_src[lane]] : 0;
    __syncwarp();
    if (lane < n) perm[mv_row[lane]] = v;
  }
  T* U = a.U + b * a.ustride;
  const int jbeg = a.solve ? k0 + nb : 0;
  for (int j = jbeg + tid; j < a.ncols; j += NT) {
    if (j >= k0 && j < k0 + nb) continue;
    T v[2 * NB];
#pragma unroll
    for (int i = 0; i < 2 * NB; ++i)
      if (i < n) v[i] = M[(long long)mv_src[i] * a.ld + j];
#pragma unroll
    for (int i = 0; i < 2 * NB; ++i)
      if (i < n) {
        if (i < nb) U[(long long)i * a.ncols + j] = v[i];
        else M[(long long)mv_row[i] * a.ld + j] = v[i];
      }
  }
}

constexpr int kUpRows = 64, kUpCols = 32;

// One 64 x 32 tile of A <- (K rows zeroed) A + Z U: a thread owns 4 consecutive rows and 2
// columns 16 apart (row and column accesses of a half warp are 16 consecutive entries).
template <class T, int NB>
__global__ void __launch_bounds__(256) gj_update_kernel(const GjArgs<T> a, int k0, int nb, int ctiles) {
  const int b = a.ids ? a.ids[blockIdx.y] : (int)blockIdx.y;
  const int jbeg = a.solve ? k0 + nb : 0;
  const int r0 = ((int)blockIdx.x / ctiles) * kUpRows + (threadIdx.x >> 4) * 4;
  const int j0 = jbeg + ((int)blockIdx.x % ctiles) * kUpCols + (threadIdx.x & 15);
  const int N = a.N;
  if (r0 >= N) return;
  T* M = a.A + b * a.stride;
  const T* U = a.U + b * a.ustride;
  bool on[2];
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int j = j0 + 16 * e;
    on[e] = j < a.ncols && !(j >= k0 && j < k0 + nb);
  }
  T acc[4][2];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int r = r0 + i;
      acc[i][e] = (on[e] && r < N && !(r >= k0 && r < k0 + nb)) ? M[(long long)r * a.ld + j0 + 16 * e] : czero<T>();
    }
#pragma unroll
  for (int c = 0; c < NB; ++c) {
    if (c >= nb) break;
    T u[2], z[4];
#pragma unroll
    for (int e = 0; e < 2; ++e) u[e] = on[e] ? U[(long long)c * a.ncols + j0 + 16 * e] : czero<T>();
#pragma unroll
    for (int i = 0; i < 4; ++i) z[i] = (r0 + i < N) ? M[(long long)(r0 + i) * a.ld + k0 + c] : czero<T>();
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int e = 0; e < 2; ++e) cfma(acc[i][e], z[i], u[e]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int e = 0; e < 2; ++e)
      if (on[e] && r0 + i < N) M[(long long)(r0 + i) * a.ld + j0 + 16 * e] = acc[i][e];
}

template <class T, int NB, int NT, int RP>
cudaError_t run(const GjArgs<T>& a, int nbatch, cudaStream_t st) {
  for (int k0 = 0; k0 < a.N; k0 += NB) {
    const int nb = std::min(NB, a.N - k0);
    gj_panel_kernel<T, NB, NT, RP><<<nbatch, NT, 0, st>>>(a, k0, nb);
    const int cols = a.ncols - (a.solve ? k0 + nb : 0);
    const int ctiles = (cols + kUpCols - 1) / kUpCols, rtiles = (a.N + kUpRows - 1) / kUpRows;
    if (ctiles > 0) gj_update_kernel<T, NB><<<dim3(ctiles * rtiles, nbatch), 256, 0, st>>>(a, k0, nb, ctiles);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// ---------------------------------------------------------------------------
// The same blocking for an augmented matrix [A | E] in complex float (leaf systems and cluster
// systems of a mixed-only preconditioner).  Every entry gets exactly the operations, in the same
// order, of eliminating one column at a time: v -= m_k u_k for k = 0, 1, ..., with u_k the pivot
// row divided by its pivot, because the results are rounded to FP16 afterwards and another order
// of summation (1e-7) would move entries across the rounding boundaries of 2^-11.  The panel keeps
// the multipliers m in place of the eliminated columns; a thread per column makes the panel's
// interchanges and the NB pivot rows' own recurrences; the update is a 64 x 64 tiled sweep over
// the columns right of the panel.  Columns of E whose pivot rows are still zero are skipped.
// Measured, setup of 8^3 leaves at p = 8 with 45 distinct cluster systems of 864 rows: the cluster
// part 250 ms with one CTA streaming its matrix from L2 once per column, 21 ms here.
// ---------------------------------------------------------------------------
struct AugArgs {
  float2* A;
  long long stride;
  int ld, n, ncols, gj0;
  float2* U;  // [matrix][NB][ncols]
  long long ustride;
  const int* ids;
  int* status;
};

// v -= m u and a b, their roundings spelled out: the panel, the pivot rows and the update have to
// round alike wherever an entry happens to be processed.
__device__ __forceinline__ void aug_update(float2& v, const float2 m, const float2 u) {
  v.x = __fsub_rn(v.x, __fmaf_rn(m.x, u.x, -__fmul_rn(m.y, u.y)));
  v.y = __fsub_rn(v.y, __fmaf_rn(m.y, u.x, __fmul_rn(m.x, u.y)));
}
__device__ __forceinline__ float2 aug_mul(const float2 a, const float2 b) {
  return make_float2(__fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y)), __fmaf_rn(a.x, b.y, __fmul_rn(a.y, b.x)));
}

template <int NB, int NT, int RP>
__global__ void __launch_bounds__(NT) aug_panel_kernel(const AugArgs a, int k0, int nb) {
  constexpr int kNone = 0x7fffffff;
  __shared__ float2 us[NB], ks[NB], inv_s[NB], mk[NB][NB];
  __shared__ unsigned wkey[NT / 32];
  __shared__ int widx[NT / 32];
  __shared__ int piv[NB];
  __shared__ int mv_row[2 * NB], mv_src[2 * NB], mv_n;
  const int b = a.ids ? a.ids[blockIdx.x] : (int)blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = a.n;
  float2* M = a.A + b * a.stride;
  const bool gj = k0 >= a.gj0;           // panels do not cross gj0
  const int lo = gj ? a.gj0 : k0;        // rows the panel touches
  float2 row[RP][NB];
#pragma unroll
  for (int i = 0; i < RP; ++i) {
    const int r = tid + i * NT;
#pragma unroll
    for (int j = 0; j < NB; ++j)
      row[i][j] = (r >= lo && r < n && j < nb) ? M[(long long)r * a.ld + k0 + j] : czero<float2>();
  }
#pragma unroll
  for (int c = 0; c < NB; ++c) {
    if (c >= nb) break;
    const int k = k0 + c;
    unsigned key = 0;
    int idx = kNone;
#pragma unroll
    for (int i = 0; i < RP; ++i) {
      const int r = tid + i * NT;
      if (r >= k && r < n) {
        const unsigned kk = pivot_key(row[i][c]);
        if (idx == kNone || kk > key) {
          key = kk;
          idx = r;
        }
      }
    }
    unsigned wm = __reduce_max_sync(0xffffffffu, key);
    int p = __reduce_min_sync(0xffffffffu, key == wm ? idx : kNone);
    if (lane == 0) {
      wkey[warp] = wm;
      widx[warp] = p;
    }
    __syncthreads();
    key = lane < NT / 32 ? wkey[lane] : 0u;
    idx = lane < NT / 32 ? widx[lane] : kNone;
    wm = __reduce_max_sync(0xffffffffu, key);
    p = __reduce_min_sync(0xffffffffu, key == wm ? idx : kNone);
#pragma unroll
    for (int i = 0; i < RP; ++i) {
      const int r = tid + i * NT;
      if (r == p) {
        const float2 pv = row[i][c];
        const bool ok = pv.x != 0 || pv.y != 0;
        if (!ok || pv.x != pv.x || pv.y != pv.y) atomicExch(a.status, 1);
        const float2 inv = ok ? cinv(pv) : czero<float2>();
        inv_s[c] = inv;
        // multipliers of the earlier columns, then the pivot row divided by the pivot
#pragma unroll
        for (int j = 0; j < NB; ++j) us[j] = j <= c ? row[i][j] : aug_mul(row[i][j], inv);
        piv[c] = p;
      }
      if (r == k)
#pragma unroll
        for (int j = 0; j < NB; ++j) ks[j] = row[i][j];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < RP; ++i) {
      const int r = tid + i * NT;
      if (r >= n || r < lo) continue;
      if (r == k) {
#pragma unroll
        for (int j = 0; j < NB; ++j) row[i][j] = us[j];
        continue;
      }
      if (r == p)
#pragma unroll
        for (int j = 0; j < NB; ++j) row[i][j] = ks[j];
      if (r < k && !gj) continue;
      const float2 m = row[i][c];
#pragma unroll
      for (int j = 0; j < NB; ++j)
        if (j > c) aug_update(row[i][j], m, us[j]);
    }
  }
  // multipliers in place of the panel; those of the pivot rows also in shared memory
#pragma unroll
  for (int i = 0; i < RP; ++i) {
    const int r = tid + i * NT;
    if (r >= n || r < lo) continue;
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      if (j < nb) M[(long long)r * a.ld + k0 + j] = row[i][j];
      if (r >= k0 && r < k0 + nb) mk[r - k0][j] = row[i][j];
    }
  }
  if (warp == 0) {  // the interchanges as one move, as in gj_panel_kernel
    int rid = lane < nb ? k0 + lane : -1, src = lane, cnt = nb;
    for (int c = 0; c < nb; ++c) {
      const int p = piv[c];
      unsigned hit = __ballot_sync(0xffffffffu, rid == p);
      if (!hit) {
        if (lane == cnt) rid = p;
        hit = 1u << cnt;
        ++cnt;
      }
      const int l = __ffs(hit) - 1;
      const int sc = __shfl_sync(0xffffffffu, src, c), sl = __shfl_sync(0xffffffffu, src, l);
      if (lane == c) src = sl;
      if (lane == l) src = sc;
    }
    const int from = __shfl_sync(0xffffffffu, rid, src);
    if (lane < cnt) {
      mv_row[lane] = rid;
      mv_src[lane] = from;
    }
    if (lane == 0) mv_n = cnt;
  }
  __syncthreads();
  const int cnt = mv_n;
  float2* U = a.U + b * a.ustride;
  for (int j = k0 + nb + tid; j < a.ncols; j += NT) {
    float2 v[2 * NB];
#pragma unroll
    for (int i = 0; i < 2 * NB; ++i) v[i] = i < cnt ? M[(long long)mv_src[i] * a.ld + j] : czero<float2>();
#pragma unroll
    for (int i = 0; i < 2 * NB; ++i)
      if (i >= nb && i < cnt) M[(long long)mv_row[i] * a.ld + j] = v[i];
#pragma unroll
    for (int c = 0; c < NB; ++c) {
      if (c >= nb) break;
      // row c has had the updates of the earlier columns: now its division, then its use
      v[c] = aug_mul(v[c], inv_s[c]);
      const float2 u = v[c];
      U[(long long)c * a.ncols + j] = u;
#pragma unroll
      for (int i = 0; i < NB; ++i)
        if (i < nb && (i > c || (i < c && gj))) aug_update(v[i], mk[i][c], u);
    }
#pragma unroll
    for (int c = 0; c < NB; ++c)
      if (c < nb) M[(long long)(k0 + c) * a.ld + j] = v[c];
  }
}

template <int NB>
__global__ void __launch_bounds__(256) aug_update_kernel(const AugArgs a, int k0, int nb, int ctiles) {
  __shared__ __align__(16) float2 sm[NB][64], su[NB][64];
  const int b = a.ids ? a.ids[blockIdx.y] : (int)blockIdx.y, n = a.n, tid = threadIdx.x;
  const int lo = k0 >= a.gj0 ? a.gj0 : k0 + nb;
  const int r0 = lo + ((int)blockIdx.x / ctiles) * 64, j0 = k0 + nb + ((int)blockIdx.x % ctiles) * 64;
  float2* M = a.A + b * a.stride;
  const float2* U = a.U + b * a.ustride;
  int any = 0;
  for (int t = tid; t < NB * 64; t += 256) {
    const int c = t / 64, j = j0 + t % 64;
    const float2 u = (c < nb && j < a.ncols) ? U[(long long)c * a.ncols + j] : czero<float2>();
    su[c][t % 64] = u;
    any |= u.x != 0.f || u.y != 0.f;
    const int c2 = t % NB, r = r0 + t / NB;
    sm[c2][t / NB] = (c2 < nb && r < n) ? M[(long long)r * a.ld + k0 + c2] : czero<float2>();
  }
  if (!__syncthreads_or(any)) return;  // the pivot rows are zero in all these columns
  const int tx = (tid & 15) * 4, ty = (tid >> 4) * 4;
  float2 acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int e = 0; e < 4; ++e)
      acc[i][e] = (r0 + ty + i < n && j0 + tx + e < a.ncols) ? M[(long long)(r0 + ty + i) * a.ld + j0 + tx + e]
                                                             : czero<float2>();
#pragma unroll
  for (int c = 0; c < NB; ++c) {
    if (c >= nb) break;
    float2 m[4], u[4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float4 x = *reinterpret_cast<const float4*>(&sm[c][ty + 2 * h]);
      const float4 y = *reinterpret_cast<const float4*>(&su[c][tx + 2 * h]);
      m[2 * h] = make_float2(x.x, x.y);
      m[2 * h + 1] = make_float2(x.z, x.w);
      u[2 * h] = make_float2(y.x, y.y);
      u[2 * h + 1] = make_float2(y.z, y.w);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) aug_update(acc[i][e], m[i], u[e]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + ty + i;
    if (r >= n || (r >= k0 && r < k0 + nb)) continue;  // the pivot rows are done
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (j0 + tx + e < a.ncols) M[(long long)r * a.ld + j0 + tx + e] = acc[i][e];
  }
}

template <int NB, int NT, int RP>
cudaError_t run_aug(const AugArgs& a, int nbatch, cudaStream_t st) {
  for (int k0 = 0; k0 < a.n;) {
    const int end = k0 < a.gj0 ? a.gj0 : a.n;
    const int nb = std::min(NB, end - k0);
    aug_panel_kernel<NB, NT, RP><<<nbatch, NT, 0, st>>>(a, k0, nb);
    const int lo = k0 >= a.gj0 ? a.gj0 : k0 + nb;
    const int ctiles = (a.ncols - k0 - nb + 63) / 64, rtiles = (a.n - lo + 63) / 64;
    if (ctiles * rtiles > 0) aug_update_kernel<NB><<<dim3(ctiles * rtiles, nbatch), 256, 0, st>>>(a, k0, nb, ctiles);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k0 += nb;
  }
  return cudaSuccess;
}

constexpr int kAugNb = 16;

// panel width: rows of a panel live in registers, NB * RP complex values per thread
template <class T> constexpr int kNbSmall = 8;
constexpr int kSmallN = 1024;   // NT * RP of the widest small shape
constexpr int kLargeN = 3072;   // 512 threads x 6 rows

}  // namespace

template <class T>
size_t gj_scratch_elems(int ncols) {
  return (size_t)kNbSmall<T> * ncols;
}
template size_t gj_scratch_elems<double2>(int);

template <class T>
cudaError_t batched_gj(T* A, long long stride, int ld, int N, int ncols, int nbatch, T* U, long long ustride, int* perm,
                       int pstride, int* status, cudaStream_t st, const int* ids) {
  if (N <= 0 || nbatch <= 0) return cudaSuccess;
  if (N > kLargeN || ncols < N) return cudaErrorInvalidValue;
  GjArgs<T> a;
  a.A = A;
  a.stride = stride;
  a.ld = ld;
  a.N = N;
  a.ncols = ncols;
  a.solve = ncols > N ? 1 : 0;
  a.U = U;
  a.ustride = ustride;
  a.perm = perm;
  a.pstride = pstride;
  a.ids = ids;
  a.status = status;
  constexpr int NB = kNbSmall<T>;
  if (N <= 128) return run<T, NB, 128, 1>(a, nbatch, st);
  if (N <= 256) return run<T, NB, 256, 1>(a, nbatch, st);
  if (N <= 512) return run<T, NB, 512, 1>(a, nbatch, st);
  if (N <= kSmallN) return run<T, NB, 512, 2>(a, nbatch, st);
  return run<T, NB / 2, 512, 6>(a, nbatch, st);
}
template cudaError_t batched_gj<double2>(double2*, long long, int, int, int, int, double2*, long long, int*, int, int*,
                                         cudaStream_t, const int*);

size_t gj_augmented_scratch_elems(int ncols) { return (size_t)kAugNb * ncols; }

cudaError_t batched_gj_augmented(float2* A, long long stride, int ld, int n, int ncols, int gj0, int nbatch, float2* U,
                                 long long ustride, int* status, cudaStream_t st, const int* ids) {
  if (n <= 0 || nbatch <= 0) return cudaSuccess;
  if (n > 5120 || ncols < n || gj0 < 0 || gj0 > n) return cudaErrorInvalidValue;
  AugArgs a;
  a.A = A;
  a.stride = stride;
  a.ld = ld;
  a.n = n;
  a.ncols = ncols;
  a.gj0 = gj0;
  a.U = U;
  a.ustride = ustride;
  a.ids = ids;
  a.status = status;
  if (n <= 256) return run_aug<kAugNb, 256, 1>(a, nbatch, st);
  if (n <= 512) return run_aug<kAugNb, 512, 1>(a, nbatch, st);
  if (n <= 1024) return run_aug<kAugNb, 512, 2>(a, nbatch, st);
  if (n <= 2048) return run_aug<kAugNb / 2, 512, 4>(a, nbatch, st);
  return run_aug<kAugNb / 4, 512, 10>(a, nbatch, st);
}

}  // namespace hps
