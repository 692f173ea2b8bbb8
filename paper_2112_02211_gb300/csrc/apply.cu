// Per-iteration operators of the HPS face system, as one family of
// HBM-streaming batched GEMV kernels ("items" of q^2 matrix rows each):
//
//  * apply     y = f + Pi (R f)           (leaf ItI maps, Sec. 2.2, eq. (inter))
//  * residual  y = b - (f + Pi (R f))
//  * rhs       b = tbar - Pi (H s)        (body-load response of each leaf)
//  * precond   z = J^{-1} r on 2x2x2 clusters (Sec. 4, Algorithm 4 in face form):
//      stage B  z_ext = r_ext,  t = r_int - B r_ext   (B = internal rows of R~;
//               its own kernel, one thread per row, B stored transposed)
//      stage K  z_int = K_c t                          (K_c = (I + D)^{-1})
//
// An item is (leaf, part) for apply/rhs (a part of the rows of its faces with a neighbour), a leaf
// or a part of its rows for B, and for K a part of one slot of a distinct K block against up to 8
// vectors: clusters sharing that block and right-hand sides, so that a block shared by many is read
// once per 8 or 4 of them.  The swap Pi is fused into the store: the rows
// of leaf tau's face k produce the incoming data of the neighbour across k,
// so every output slot has exactly one writer and no atomics are needed.
// Faces on the boundary of the cube only copy (their rows of R are never
// read).  A CTA stages the item's input vector in shared memory; each warp
// streams RPW matrix rows with 16-byte loads (1 complex double or 2 complex
// floats per lane per load), accumulates in the matrix's precision and
// reduces with warp shuffles that halve the values in flight at every step.
//
// What bounds it: HBM for one right-hand side in complex float; the FP64 pipe (4 fused
// multiply-adds per entry, two per SM and clock) in complex double, where the warp reductions
// used to cost another third; shared-memory reads of the staged vectors for many right-hand
// sides, which several rows per warp share.  Measured, 9^3 leaves, p = 8, complex double: 331 -> 263
// us.  (Complex-float vectors take stream_apply.cu where that is faster, see stream_apply_better.)
#include <algorithm>
#include <array>
#include <map>
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "hps_internal.h"

namespace hps {

// Returns the CUDA error of expr from a function that returns cudaError_t.
#define HPS_TRY_CUDA_E(expr)          \
  do {                                \
    const cudaError_t e_ = (expr);    \
    if (e_ != cudaSuccess) return e_; \
  } while (0)

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

// One 16-byte load per lane: VPL complex entries of the matrix type, widened to
// the accumulation type.
template <class TM> struct MT;
template <> struct MT<double2> {
  static constexpr int VPL = 1;
  using Acc = double2;
  __device__ static __forceinline__ void load(const double2* p, double2 (&v)[1]) { v[0] = __ldg(p); }
};
template <> struct MT<float2> {
  static constexpr int VPL = 2;
  using Acc = float2;
  __device__ static __forceinline__ void load(const float2* p, float2 (&v)[2]) {
    const float4 t = __ldg(reinterpret_cast<const float4*>(p));
    v[0] = make_float2(t.x, t.y);
    v[1] = make_float2(t.z, t.w);
  }
};
template <> struct MT<__half2> {
  static constexpr int VPL = 4;
  using Acc = float2;
  __device__ static __forceinline__ void load(const __half2* p, float2 (&v)[4]) {
    const uint4 t = __ldg(reinterpret_cast<const uint4*>(p));
    v[0] = __half22float2(*reinterpret_cast<const __half2*>(&t.x));
    v[1] = __half22float2(*reinterpret_cast<const __half2*>(&t.y));
    v[2] = __half22float2(*reinterpret_cast<const __half2*>(&t.z));
    v[3] = __half22float2(*reinterpret_cast<const __half2*>(&t.w));
  }
};
__device__ __forceinline__ float2 rscale(float2 v, const float* s, long long i) {
  if (!s) return v;
  const float f = s[i];
  return make_float2(v.x * f, v.y * f);
}
__device__ __forceinline__ double2 rscale(double2 v, const float*, long long) { return v; }

// Staged vectors in shared memory, VPL entries per lane and load: column c of a vector lies at
// staged(c), so that a warp's 16-byte reads take consecutive addresses (4 entries per lane in two
// halves of a 128-column chunk; read 8 bytes at a time they conflict four ways).
template <int VPL> __device__ __forceinline__ int staged(int c) {
  return VPL == 4 ? (c & ~127) + ((c & 2) << 5) + ((c & 124) >> 1) + (c & 1) : c;
}
__device__ __forceinline__ void load_staged(const float2* x, int c, float2 (&v)[4]) {  // c a multiple of 4
  const float2* p = x + staged<4>(c);
  const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 64);
  v[0] = make_float2(a.x, a.y);
  v[1] = make_float2(a.z, a.w);
  v[2] = make_float2(b.x, b.y);
  v[3] = make_float2(b.z, b.w);
}

struct ItemInfo {
  const void* mat;
  long long xoff;  // base offset of the input vector (per rhs)
  long long ooff;  // base offset of the output (per rhs)
  long long aoff;  // auxiliary offset (neighbour input / residual base)
  int ld, ncols;
  int nrows;       // matrix rows of the item (q^2, or all internal-face rows of a leaf)
  int leaf, face, nbr;
  int mask;        // apply, rhs: faces with a neighbour; stage K: members
  int row0;        // apply, rhs: first row of the item among the rows of those faces
  unsigned flist;  // apply, rhs: those faces, 4 bits each
};

// Rows of a leaf's faces with a neighbour, cut into `parts` items: row l of an item belongs to the
// (row0 + l) / q2 -th of those faces.
__device__ __forceinline__ void leaf_rows(const GridDims& g, int q2, int parts, long long item, ItemInfo& it) {
  it.leaf = (int)(item / parts);
  const int part = (int)(item % parts);
  it.mask = 0;
  it.flist = 0;
  int n = 0;
#pragma unroll
  for (int f = 0; f < 6; ++f)
    if (g.neighbor(it.leaf, f) >= 0) {
      it.mask |= 1 << f;
      it.flist |= (unsigned)f << (4 * n++);
    }
  const int rows = n * q2;
  it.row0 = rows * part / parts;
  it.nrows = rows * (part + 1) / parts - it.row0;
}
// The leaf across a face that has one (for the stores of single rows; GridDims::neighbor divides).
__device__ __forceinline__ int across(const GridDims& g, int leaf, int face) {
  const int step = face >> 1 == 0 ? 1 : face >> 1 == 1 ? g.nx : g.nx * g.ny;
  return leaf + (face & 1 ? step : -step);
}
// inv: row_inv(q2)
__device__ __forceinline__ void leaf_row(const ItemInfo& it, int q2, unsigned inv, int l, int& face, int& j) {
  const unsigned r = it.row0 + l, k = (r * inv) >> 20;
  j = (int)(r - k * q2);
  face = (it.flist >> (4 * k)) & 7u;
}
// Most right-hand sides x rows of accumulators per thread (complex values).
template <class TM> constexpr int kMaxAcc = sizeof(TM) == 16 ? 16 : 32;

// ---------------------------------------------------------------------------
// y = f + g (apply) in the output's precision.  Double-float outputs (float4)
// keep f + g exactly (TwoSum), so the identity part of I + Pi R loses nothing.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void sum_out(double2& y, double2 f, double2 g) { y = cadd(f, g); }
__device__ __forceinline__ void sum_out(double2& y, float2 f, float2 g) {
  y = make_double2((double)f.x + (double)g.x, (double)f.y + (double)g.y);
}
__device__ __forceinline__ void sum_out(double2& y, double2 f, float2 g) {
  y = make_double2(f.x + (double)g.x, f.y + (double)g.y);
}
__device__ __forceinline__ void sum_out(float2& y, float2 f, float2 g) { y = cadd(f, g); }
__device__ __forceinline__ void sum_out(float4& y, float2 f, float2 g) {
  const dfr re = df_two_sum(f.x, g.x), im = df_two_sum(f.y, g.y);
  y = make_float4(re.h, im.h, re.l, im.l);
}
__device__ __forceinline__ void sum_out(float4& y, float4 f, float2 g) {
  y = dfc_store(dfc_add(dfc_load(f), dfc{{g.x, 0.f}, {g.y, 0.f}}));
}
// residual form y = b - (f + g): only produced in complex double
__device__ __forceinline__ void residual_out(double2& y, double2 b) { y = csub(b, y); }
template <class T> __device__ __forceinline__ void residual_out(T&, double2) {}

// ---------------------------------------------------------------------------
// Policies
// ---------------------------------------------------------------------------
template <class TM_, class TIN, class TOUT>
struct ApplyP {
  using TM = TM_;
  using Acc = typename MT<TM>::Acc;
  struct Args {
    const TM* R;
    int ldR, nb, q2;
    GridDims g;
    const TIN* f;
    TOUT* y;
    const double2* bvec;  // residual mode: y = b - (I + Pi R) f
    long long nf;
    int nrhs, parts;
    unsigned inv;
    long long nitems;
  };
  __device__ static bool decode(const Args& A, long long item, ItemInfo& it) {
    leaf_rows(A.g, A.q2, A.parts, item, it);
    it.face = (int)(item % A.parts);
    it.xoff = (long long)it.leaf * A.nb;
    it.mat = A.R + (long long)it.leaf * A.nb * A.ldR;
    it.ld = A.ldR;
    it.ncols = A.nb;
    return true;
  }
  __device__ static long long row_off(const Args& A, const ItemInfo& it, int l) {
    if (it.mask == 63) return (long long)(it.row0 + l) * A.ldR;
    int face, j;
    leaf_row(it, A.q2, A.inv, l, face, j);
    return (long long)(face * A.q2 + j) * A.ldR;
  }
  __device__ static Acc load_x(const Args& A, const ItemInfo& it, int rhs, int c) {
    return cvt<Acc>(A.f[rhs * A.nf + it.xoff + c]);
  }
  __device__ static void finish(const Args& A, long long o, Acc g) {
    TOUT v;
    sum_out(v, A.f[o], g);
    if (A.bvec) residual_out(v, A.bvec[o]);
    A.y[o] = v;
  }
  __device__ static void store(const Args& A, const ItemInfo& it, const Acc* outs, int nr, int tid) {
    for (int l = tid; l < it.nrows; l += kThreads) {
      int face, j;
      leaf_row(it, A.q2, A.inv, l, face, j);
      const long long o = (long long)across(A.g, it.leaf, face) * A.nb + (long long)(face ^ 1) * A.q2 + j;
      for (int rhs = 0; rhs < nr; ++rhs) finish(A, rhs * A.nf + o, outs[rhs * it.nrows + l]);
    }
    if (it.face != 0 || it.mask == 63) return;
    // the leaf's first item: faces on the boundary of the cube only copy
    for (int idx = tid; idx < 6 * A.q2; idx += kThreads)
      if (!((it.mask >> (idx / A.q2)) & 1))
        for (int rhs = 0; rhs < nr; ++rhs) finish(A, rhs * A.nf + it.xoff + idx, czero<Acc>());
  }
};

template <class TM_>
struct RhsP {
  using TM = TM_;
  using Acc = typename MT<TM>::Acc;
  struct Args {
    const TM* H;
    int ldH, ni, nb, q2;
    GridDims g;
    const double2* s;
    const double2* t;
    double2* out;
    long long nf, nint;
    int nrhs, parts;
    unsigned inv;
    long long nitems;
  };
  __device__ static bool decode(const Args& A, long long item, ItemInfo& it) {
    leaf_rows(A.g, A.q2, A.parts, item, it);
    it.face = (int)(item % A.parts);
    it.mat = A.H + (long long)it.leaf * A.nb * A.ldH;
    it.ld = A.ldH;
    it.ncols = A.ni;
    it.xoff = (long long)it.leaf * A.ni;
    return A.s != nullptr;  // no body load: h = 0
  }
  __device__ static long long row_off(const Args& A, const ItemInfo& it, int l) {
    int face, j;
    leaf_row(it, A.q2, A.inv, l, face, j);
    return (long long)(face * A.q2 + j) * A.ldH;
  }
  __device__ static Acc load_x(const Args& A, const ItemInfo& it, int rhs, int c) {
    return cvt<Acc>(A.s[rhs * A.nint + it.xoff + c]);
  }
  __device__ static void store(const Args& A, const ItemInfo& it, const Acc* outs, int nr, int tid) {
    for (int l = tid; l < it.nrows; l += kThreads) {
      int face, j;
      leaf_row(it, A.q2, A.inv, l, face, j);
      const long long o = (long long)across(A.g, it.leaf, face) * A.nb + (long long)(face ^ 1) * A.q2 + j;
      for (int rhs = 0; rhs < nr; ++rhs) {
        const double2 v = outs ? cvt<double2>(outs[rhs * it.nrows + l]) : make_double2(-0.0, -0.0);
        A.out[rhs * A.nf + o] = make_double2(-v.x, -v.y);
      }
    }
    if (it.face != 0 || it.mask == 63) return;
    // the leaf's first item: boundary faces take t (or 0)
    for (int idx = tid; idx < 6 * A.q2; idx += kThreads)
      if (!((it.mask >> (idx / A.q2)) & 1))
        for (int rhs = 0; rhs < nr; ++rhs) {
          const long long o = rhs * A.nf + (long long)it.leaf * A.nb + idx;
          A.out[o] = A.t ? A.t[o] : make_double2(0.0, 0.0);
        }
  }
};

// Stage K over distinct blocks: item = (block k, block slot s, first member,
// member count) with the members the clusters sharing block k; the vectors of
// an item are its (member, right-hand side) pairs, nrl right-hand sides per
// launch, so that a block streamed once serves up to 8 vectors.
template <class TM_, class TIN, class TOUT>
struct PrecKP {
  using TM = TM_;
  using Acc = typename MT<TM>::Acc;
  struct Args {
    const TM* K;
    const float* kscale;  // FP16 blocks: row scales, index (kc_slot_begin[k] + s)*q2 + j
    const int4* items;
    const long long* kc_off;
    const int* kc_slot_begin;
    const int* members;
    const int* cl_slot_begin;
    const int* slot_lf;
    const long long* cl_tpos;
    int nb, q2, split;
    const TIN* t;
    TOUT* z;
    long long nf, tstride, tmul;  // t of (rhs, cluster) at rhs * tstride + cl_tpos * tmul
    int nrl;    // right-hand sides of an item: vector rr = member * nrl + rhs
    int nrhs;   // vectors of an item, member group width x nrl
    int total;  // right-hand sides of the launch: `groups` of nrl, item = entry of items * groups + group
    int groups;
    long long nitems;
  };
  // item (k, s * split + part, first member, members): rows
  // [part * hq, min(q^2, (part + 1) * hq)) of slot s, hq = ceil(q^2 / split)
  __device__ static bool decode(const Args& A, long long item, ItemInfo& it) {
    const int entry = (int)item / A.groups, grp = (int)item - entry * A.groups;
    const int4 e = A.items[entry];
    const int k = e.x, s = e.y / A.split, part = e.y % A.split;
    const int hq = (A.q2 + A.split - 1) / A.split;
    const int r0 = min(A.q2, part * hq);
    const int s0 = A.kc_slot_begin[k], ns = A.kc_slot_begin[k + 1] - s0;
    it.ncols = ns * A.q2;
    it.ld = (int)rup4(it.ncols);
    it.mat = A.K + A.kc_off[k] + ((long long)s * A.q2 + r0) * it.ld;
    it.nrows = min(A.q2, r0 + hq) - r0;
    it.face = s;
    it.nbr = r0;    // first row within the slot
    it.xoff = e.z;  // first member
    it.mask = e.w;  // members
    it.leaf = grp * A.nrl;  // first right-hand side
    it.aoff = (long long)(s0 + s) * A.q2 + r0;
    return it.nrows > 0;
  }
  __device__ static long long row_off(const Args&, const ItemInfo& it, int l) { return (long long)l * it.ld; }
  __device__ static Acc load_x(const Args& A, const ItemInfo& it, int rr, int c) {
    const int m = rr / A.nrl, rhs = it.leaf + rr - m * A.nrl;
    if (m >= it.mask || rhs >= A.total) return czero<Acc>();
    return cvt<Acc>(A.t[(long long)rhs * A.tstride + A.cl_tpos[A.members[it.xoff + m]] * A.tmul + c]);
  }
  __device__ static void store(const Args& A, const ItemInfo& it, const Acc* outs, int, int tid) {
    if (!outs) return;
    for (int idx = tid; idx < it.mask * A.nrl * it.nrows; idx += kThreads) {
      const int rr = idx / it.nrows, jj = idx % it.nrows, m = rr / A.nrl, rhs = it.leaf + rr - m * A.nrl;
      if (rhs >= A.total) continue;
      const int lf = A.slot_lf[A.cl_slot_begin[A.members[it.xoff + m]] + it.face];
      const long long o = (long long)(lf / 6) * A.nb + (long long)(lf % 6) * A.q2 + it.nbr + jj;
      A.z[(long long)rhs * A.nf + o] = cvt<TOUT>(rscale(outs[idx], A.kscale, it.aoff + jj));
    }
  }
};

// ---------------------------------------------------------------------------
// The kernel.
// ---------------------------------------------------------------------------
// gate: while a GMRES cycle is replayed from a graph, the word that says whether any
// right-hand side is still active (0: return at once); nullptr otherwise.
template <class P, int NR, int RPW>
__global__ void __launch_bounds__(kThreads) seg_gemv_kernel(const typename P::Args A, int xcap, int rowcap,
                                                            const int* gate) {
  if (gate && *gate == 0) return;
  using TM = typename P::TM;
  using Acc = typename P::Acc;
  using R_ = typename Real<Acc>::type;
  constexpr int VPL = MT<TM>::VPL;
  extern __shared__ __align__(16) unsigned char smraw[];
  Acc* xs = reinterpret_cast<Acc*>(smraw);
  Acc* outs = xs + NR * xcap;  // NR x rowcap
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nr = A.nrhs < NR ? A.nrhs : NR;
  for (long long item = blockIdx.x; item < A.nitems; item += gridDim.x) {
    ItemInfo it;
    if (!P::decode(A, item, it)) {
      P::store(A, it, nullptr, nr, tid);
      continue;
    }
    const int ncp = (it.ncols + VPL - 1) / VPL * VPL, ncs = VPL == 4 ? (ncp + 127) & ~127 : ncp;
    for (int idx = tid; idx < NR * ncp; idx += kThreads) {
      const int rr = idx / ncp, c = idx % ncp;
      xs[rr * ncs + staged<VPL>(c)] = (rr < nr && c < it.ncols) ? P::load_x(A, it, rr, c) : czero<Acc>();
    }
    __syncthreads();
    const TM* mat = reinterpret_cast<const TM*>(it.mat);
    const int nrows = it.nrows;
    for (int r0 = warp * RPW; r0 < nrows; r0 += kWarps * RPW) {
      constexpr int V = 2 * RPW * NR;
      R_ acc[V];  // (row, right-hand side, re/im)
#pragma unroll
      for (int i = 0; i < V; ++i) acc[i] = 0;
      const TM* row[RPW];
#pragma unroll
      for (int i = 0; i < RPW; ++i) row[i] = mat + P::row_off(A, it, min(r0 + i, nrows - 1));
#pragma unroll 2
      for (int c = lane * VPL; c < ncp; c += 32 * VPL) {
        Acc mv[RPW][VPL];
#pragma unroll
        for (int i = 0; i < RPW; ++i) MT<TM>::load(row[i] + c, mv[i]);
#pragma unroll
        for (int rr = 0; rr < NR; ++rr) {
          Acc xq[4];
          if constexpr (VPL == 4) load_staged(xs + rr * ncs, c, xq);
#pragma unroll
          for (int v = 0; v < VPL; ++v) {
            const Acc xv = VPL == 4 ? xq[v] : xs[rr * ncs + c + v];
#pragma unroll
            for (int i = 0; i < RPW; ++i) {
              Acc t;
              t.x = acc[2 * (i * NR + rr)];
              t.y = acc[2 * (i * NR + rr) + 1];
              cfma(t, mv[i][v], xv);
              acc[2 * (i * NR + rr)] = t.x;
              acc[2 * (i * NR + rr) + 1] = t.y;
            }
          }
        }
      }
      int first;
      warp_sums<R_, V>(acc, lane, first);
      constexpr int kHeld = V >= 32 ? V / 32 : 1, kSame = V >= 32 ? 1 : 32 / V;  // lanes with the same sums
      if (lane % kSame == 0) {
#pragma unroll
        for (int k = 0; k < kHeld; ++k) {
          const int s = first + k, i = s / (2 * NR), rr = (s / 2) % NR;
          if (r0 + i < nrows) reinterpret_cast<R_*>(outs)[2 * (rr * nrows + r0 + i) + (s & 1)] = acc[k];
        }
      }
    }
    __syncthreads();
    P::store(A, it, outs, nr, tid);
    __syncthreads();
  }
}

// Stage B: one CTA per leaf (persistent), one thread per row of the leaf's B
// block.  B is stored transposed (column c holds the nint q^2 rows), so a warp
// reads 32 consecutive rows of one column: coalesced loads and no cross-lane
// reductions.  The external-face values are staged in shared memory; t at the
// neighbours' internal slots gets r - B r_ext, z_ext = r_ext.  Several
// right-hand sides: NR of them per pass over the block, each B entry loaded
// once per pass and used NR times (rhs r of vector v at v + r * stride).
template <class TM, class TIN, class TOUT>
struct PrecBArgs {
  const TM* B;
  const float* bscale;  // FP16 blocks: row scales, index bsc[leaf*6 + k] + j
  const long long* b_off;
  const uint8_t* int_mask;
  const int* brd;  // per leaf, internal faces then external: input offsets
  const int* bto;  // per leaf, internal faces: t offsets
  const int* bsc;  // per leaf, internal faces: row-scale bases
  int nl, q2;
  const TIN* r;
  TOUT* z;
  TOUT* t;
  int nrhs;
  long long vstride, tstride;  // per right-hand side: r and z, t
  const int* gate;  // as in seg_gemv_kernel
  // work items: groups of leaves sharing one B block, as (first index into gleaves, count)
  const int2* groups;
  const int* gleaves;
  int ngroups;
  int parts;  // CTAs per item, each a part of the rows (the first one also writes z_ext)
};

template <class TM> __device__ __forceinline__ typename MT<TM>::Acc load_one(const TM* p);
template <> __device__ __forceinline__ float2 load_one<__half2>(const __half2* p) { return __half22float2(*p); }
template <> __device__ __forceinline__ float2 load_one<float2>(const float2* p) { return *p; }
template <> __device__ __forceinline__ double2 load_one<double2>(const double2* p) { return *p; }

template <class TM, class TIN, class TOUT, int NR>
__global__ void __launch_bounds__(kThreads) prec_b_kernel(const PrecBArgs<TM, TIN, TOUT> A) {
  if (A.gate && *A.gate == 0) return;
  using Acc = typename MT<TM>::Acc;
  extern __shared__ __align__(16) unsigned char smraw[];
  Acc* xs = reinterpret_cast<Acc*>(smraw);  // NR x (external columns)
  const int q2 = A.q2;
  // item: a group of leaves sharing one B block (same block, same internal-face mask); the
  // vectors of a pass are NR (leaf of the group, right-hand side) pairs, so every entry of B
  // loaded from L2 serves NR independent accumulations
  for (int idx_i = blockIdx.x; idx_i < A.ngroups * A.parts; idx_i += gridDim.x) {
    const int item = idx_i / A.parts, part = idx_i - item * A.parts;
    const int2 grp = A.groups[item];
    const int leaf0 = A.gleaves[grp.x];
    const int nint = __popc((unsigned)A.int_mask[leaf0]);
    const int ncols = (6 - nint) * q2, nrows = nint * q2;
    const TM* Bm = A.B + A.b_off[leaf0];
    const int ldr = (int)rup4(nrows);
    const int nvec = grp.y * A.nrhs;
    for (int v0 = 0; v0 < nvec; v0 += NR) {
      const int nr = min(NR, nvec - v0);
      __syncthreads();
      for (int idx = threadIdx.x; idx < NR * ncols; idx += blockDim.x) {
        const int rr = idx / ncols, c = idx - rr * ncols;
        if (rr >= nr) {  // summed all the same: a test per product costs more
          xs[idx] = czero<Acc>();
          continue;
        }
        const int vid = v0 + rr, leaf = A.gleaves[grp.x + vid / A.nrhs], rhs = vid % A.nrhs;
        const int k = c / q2;
        const long long o = (long long)rhs * A.vstride + A.brd[leaf * 6 + nint + k] + (c - k * q2);
        const Acc v = cvt<Acc>(A.r[o]);
        xs[rr * ncols + c] = v;
        if (part == 0) A.z[o] = cvt<TOUT>(v);
      }
      __syncthreads();
      if (nint == 0) continue;
      const int row_end = nrows * (part + 1) / A.parts;
      for (int row = nrows * part / A.parts + threadIdx.x; row < row_end; row += blockDim.x) {
        // few right-hand sides in complex double: four sums per row, since one sum is a chain of two
        // dependent FP64 operations per column (216 of them at p = 8)
        constexpr int kS = sizeof(TM) == sizeof(double2) && NR <= 2 ? 4 : 1;
        Acc acc[NR], sum[kS][NR];
#pragma unroll
        for (int i = 0; i < kS; ++i)
#pragma unroll
          for (int rr = 0; rr < NR; ++rr) sum[i][rr] = czero<Acc>();
        int c = 0;
#pragma unroll(kS == 4 ? 3 : 1)
        for (; c + 3 < ncols; c += 4) {
          Acc bv[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) bv[i] = load_one<TM>(Bm + (long long)(c + i) * ldr + row);
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int rr = 0; rr < NR; ++rr)
              cfma(sum[i % kS][rr], bv[i], xs[rr * ncols + c + i]);
        }
        for (; c < ncols; ++c) {
          const Acc bv = load_one<TM>(Bm + (long long)c * ldr + row);
#pragma unroll
          for (int rr = 0; rr < NR; ++rr)
            cfma(sum[0][rr], bv, xs[rr * ncols + c]);
        }
#pragma unroll
        for (int rr = 0; rr < NR; ++rr) {
          acc[rr] = sum[0][rr];
#pragma unroll
          for (int i = 1; i < kS; ++i) acc[rr] = cadd(acc[rr], sum[i][rr]);
        }
        const int k = row / q2, j = row - k * q2;
        // the loads of up to 8 vectors, then their stores (one after the other waited for each load:
        // 64 right-hand sides at 4^3 leaves, p = 8, both stages 114 us, so 102 us)
        constexpr int kIn = NR < 8 ? NR : 8;
#pragma unroll
        for (int r0 = 0; r0 < NR; r0 += kIn) {
          if (r0 >= nr) break;
          Acc rv[kIn];
          long long to[kIn];
#pragma unroll
          for (int i = 0; i < kIn; ++i) {
            const int vid = v0 + min(r0 + i, nr - 1), leaf = A.gleaves[grp.x + vid / A.nrhs], rhs = vid % A.nrhs;
            const int e = leaf * 6 + k;
            to[i] = (long long)rhs * A.tstride + A.bto[e] + j;
            rv[i] = csub(cvt<Acc>(A.r[(long long)rhs * A.vstride + A.brd[e] + j]),
                         rscale(acc[r0 + i], A.bscale, (long long)A.bsc[e] + j));
          }
#pragma unroll
          for (int i = 0; i < kIn; ++i)
            if (r0 + i < nr) A.t[to[i]] = cvt<TOUT>(rv[i]);
        }
      }
    }
  }
}

template <class P, int NR, int RPW>
cudaError_t launch_one(const typename P::Args& A, int xcap, int rowcap, int nsm, cudaStream_t st, long long* counter,
                       const int* gate, int bps = 0) {
  using Acc = typename P::Acc;
  const size_t smem = ((size_t)NR * xcap + (size_t)NR * rowcap) * sizeof(Acc);
  auto kern = seg_gemv_kernel<P, NR, RPW>;
  cudaError_t e = allow_dynamic_smem((const void*)kern, smem);
  if (e != cudaSuccess) return e;
  int occ = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kThreads, smem);
  if (e != cudaSuccess) return e;
  occ = std::max(occ, 1);
  if (bps > 0) occ = std::min(occ, bps);  // a tuned cap on resident CTAs per SM
  long long grid = std::min<long long>(A.nitems, (long long)nsm * occ);
  if (grid <= 0) return cudaSuccess;
  kern<<<(unsigned)grid, kThreads, smem, st>>>(A, xcap, rowcap, gate);
  ++*counter;
  return cudaGetLastError();
}

// launch_one with the rows per warp chosen at run time (1, 2, 4 or 8; at most kMaxAcc
// accumulators of RPW rows x NR right-hand sides per thread, fewer rows otherwise)
template <class P, int NR>
cudaError_t launch_shaped(const typename P::Args& A, int xcap, int rowcap, int nsm, cudaStream_t st,
                          long long* counter, const int* gate, LaunchShape sh) {
  constexpr int kMax = kMaxAcc<typename P::TM>;
  const int r = sh.rpw;
  if constexpr (NR * 8 <= kMax) {
    if (r >= 8) return launch_one<P, NR, 8>(A, xcap, rowcap, nsm, st, counter, gate, sh.bps);
  }
  if constexpr (NR * 4 <= kMax) {
    if (r >= 4) return launch_one<P, NR, 4>(A, xcap, rowcap, nsm, st, counter, gate, sh.bps);
  }
  if (r >= 2) return launch_one<P, NR, 2>(A, xcap, rowcap, nsm, st, counter, gate, sh.bps);
  return launch_one<P, NR, 1>(A, xcap, rowcap, nsm, st, counter, gate, sh.bps);
}

// group of nr right-hand sides -> index into the shape tables
inline int group_index(int nr) { return nr == 1 ? 0 : nr == 2 ? 1 : nr <= 4 ? 2 : 3; }

template <class P>
cudaError_t launch_group(const typename P::Args& B, int nr, int xcap, int rowcap, int nsm, cudaStream_t st,
                         long long* counter, const int* gate, LaunchShape sh) {
  if (nr == 1) return launch_shaped<P, 1>(B, xcap, rowcap, nsm, st, counter, gate, sh);
  if (nr == 2) return launch_shaped<P, 2>(B, xcap, rowcap, nsm, st, counter, gate, sh);
  if (nr <= 4) return launch_shaped<P, 4>(B, xcap, rowcap, nsm, st, counter, gate, sh);
  return launch_shaped<P, 8>(B, xcap, rowcap, nsm, st, counter, gate, sh);
}

// Right-hand sides (or vectors) of the next launch, at most `most` of `left`: in complex double
// whole powers of two, since the FP64 pipe is the bound and a group of 6 would compute 8 -- unless
// the whole product (entries of the matrices) takes no longer than the other launch does: 3 right-hand
// sides at 3^3 leaves, p = 5, 17.6 us as 2 + 1 and 12.5 us in one launch; 4^3 leaves, p = 10 (8.8
// million entries) 210 and 280 us.
constexpr long long kSplitEntries = 1000000;
template <class TM>
int next_group(int left, int most, long long entries) {
  int n = std::min(left, most);
  if (sizeof(TM) == sizeof(double2) && entries >= kSplitEntries)
    while (n & (n - 1)) n &= n - 1;
  return n;
}

// Launch over right-hand-side groups of at most `most` (each group re-reads the matrix);
// shapes[g]: the launch shape of group index g, tuned[g]: chosen by the tuner.  The defaults suit
// items of many rows; items of a face's few take no more rows per warp than give every warp some, and
// two with four right-hand sides in complex float where there are several per SM.  Measured: 3^3
// leaves, p = 5, complex double, 4 right-hand sides (9 rows): 25.4 us with 4 rows per warp, 12.9 us
// with 2; complex float, 4 right-hand sides: 6^3 leaves, p = 7 (25 rows) 23.1 us with 4, 18.9 us with
// 2; 3^3 leaves, p = 10 (one item per SM) 11.0 and 13.8 us.
template <class P, class Shift>
cudaError_t launch_groups(const hps_handle* h, typename P::Args A, int nrhs, int most, int xcap, int rowcap,
                          cudaStream_t st, Shift shift, const LaunchShape* shapes, const bool* tuned) {
  const int nsm = h->nsm;
  long long* counter = &h->prof.launches;
  for (int r0 = 0, nr; r0 < nrhs; r0 += nr) {
    typename P::Args B = A;
    nr = next_group<typename P::TM>(nrhs - r0, most, (long long)h->nl * h->nb * xcap);
    shift(B, r0);
    B.nrhs = nr;
    const int g = group_index(nr);
    LaunchShape sh = shapes[g];
    if (!tuned || !tuned[g]) {
      if (g == 2 && sizeof(typename P::Acc) == sizeof(float2) && rowcap < 128 && A.nitems >= 2LL * nsm) sh.rpw = std::min(sh.rpw, 2);
      while (sh.rpw > 1 && kWarps * (sh.rpw / 2) >= rowcap) sh.rpw >>= 1;
    }
    const cudaError_t e = launch_group<P>(B, nr, xcap, rowcap, nsm, st, counter, h->gate, sh);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Shared-memory columns staged per vector: the leaf's face data (apply), its interior source
// (right-hand side), or a cluster's internal right-hand side (stage K).
enum class XCap { Apply, Rhs, StageK };
int xcap_of(const hps_handle* h, XCap which) {
  int mx = which == XCap::Apply ? h->nb : which == XCap::Rhs ? h->ni : 0;
  if (which == XCap::StageK && h->has_precond)
    for (int c = 0; c < h->ct.ncl; ++c)
      mx = std::max(mx, (h->ct.cl_slot_begin[c + 1] - h->ct.cl_slot_begin[c]) * h->q * h->q);
  return (int)round_up(std::max(mx, 1), which == XCap::StageK ? 128 : 64);
}

// Accumulators of a launch of n right-hand sides: 1, 2, 4 or 8.
int round_up2(int n) { return n <= 2 ? n : n <= 4 ? 4 : 8; }

// Items per leaf of the applies: enough for several waves of the chip (24 per SM, about 6 for each
// resident CTA), as many as faces at most; whole leaves stage their vector once and divide evenly
// among the warps (216 rows at p = 8, a face's 36 do not).  In complex double, where the SM with the
// most rows sets the pace, finer ones down to 16 rows while there are fewer than 4 per SM: 3^3 leaves,
// p = 10, 40.2 us with 162 items, 33.6 us with 648.  More parts where the results of the
// right-hand sides of a launch would take more than 100 KB of shared memory beside their vectors,
// and fewer right-hand sides per launch (`most`) where the vectors themselves do not fit (body loads
// of 12^3 values and more in complex double).
struct LeafPlan {
  int parts, most;
};
LeafPlan leaf_plan(const hps_handle* h, int nrhs, size_t acc_bytes, int xcap) {
  LeafPlan l{1, 8};
  while (l.parts < 6 && (long long)h->nl * l.parts < 24LL * h->nsm) l.parts += l.parts < 3 ? 1 : 3;
  if (acc_bytes == sizeof(double2))
    while (l.parts < 24 && (long long)h->nl * l.parts < 4LL * h->nsm && h->nb >= 32 * l.parts) l.parts *= 2;
  auto smem = [&]() {
    return (size_t)std::min(round_up2(nrhs), l.most) * (xcap + (h->nb + l.parts - 1) / l.parts) * acc_bytes;
  };
  while (l.parts < 6 && smem() > (size_t)100 * 1024) l.parts += l.parts < 3 ? 1 : 3;
  while (l.most > 1 && smem() > (size_t)220 * 1024) l.most >>= 1;
  return l;
}

template <class TM, class TIN, class TOUT>
cudaError_t apply_t(const hps_handle* h, const TM* R, const TIN* f, TOUT* y, const double2* bvec, int nrhs,
                    cudaStream_t st) {
  using P = ApplyP<TM, TIN, TOUT>;
  typename P::Args A;
  A.R = R;
  A.ldR = h->ldR;
  A.nb = h->nb;
  A.q2 = h->q * h->q;
  A.g = GridDims{h->nx, h->ny, h->nz};
  A.f = f;
  A.y = y;
  A.bvec = bvec;
  A.nf = h->nf;
  A.nrhs = nrhs;
  const int xcap = xcap_of(h, XCap::Apply);
  const LeafPlan plan = leaf_plan(h, nrhs, sizeof(typename P::Acc), xcap);
  A.parts = plan.parts;
  A.inv = row_inv(A.q2);
  A.nitems = (long long)h->nl * A.parts;
  const LaunchShape* shapes = h->shapes.apply[std::is_same<TM, double2>::value ? 1 : 0];
  return launch_groups<P>(h, A, nrhs, plan.most, xcap, (h->nb + A.parts - 1) / A.parts, st, [&](typename P::Args& B, int r0) {
    B.f += (long long)r0 * h->nf;
    B.y += (long long)r0 * h->nf;
    if (B.bvec) B.bvec += (long long)r0 * h->nf;
  }, shapes, h->shapes.apply_tuned[std::is_same<TM, double2>::value ? 1 : 0]);
}

// Stage K of every block that the tensor cores do not take (use_tc: all but those of kc_tc), by the
// batched GEMV.  t of right-hand side r at t + r * rstride, cluster c's part at cl_tpos[c] * tmul.
template <class TM, class TT>
cudaError_t stage_k_simt(const hps_handle* h, const TM* K, const float* kscale, const TT* t, long long rstride,
                         long long tmul, TT* z, int nrhs, bool use_tc, cudaStream_t st) {
  const int q2 = h->q * h->q;
  using P = PrecKP<TM, TT, TT>;
  typename P::Args A;
  A.K = K;
  A.kscale = kscale;
  A.kc_off = h->dct.kc_off;
  A.kc_slot_begin = h->dct.kc_slot_begin;
  A.members = h->dct.kc_members;
  A.cl_slot_begin = h->dct.cl_slot_begin;
  A.slot_lf = h->dct.slot_lf;
  A.cl_tpos = h->dct.cl_tpos;
  A.split = h->ct.krow_split;
  A.nb = h->nb;
  A.q2 = q2;
  A.nf = h->nf;
  A.tstride = rstride;
  A.tmul = tmul;
  const int xcap = xcap_of(h, XCap::StageK);
  // An item of member groups of width w takes up to fit / w right-hand sides (fewer where the staged
  // vectors do not fit in shared memory), and a launch all of them, the groups of one block's rows one
  // after the other so that they find the rows in L2.  64 blocks of one cluster at p = 8 (8^3 leaves),
  // both stages: complex float with FP16 blocks, 12 right-hand sides, 454 us with 8 and 4 vectors in
  // two launches, 353 us with 4 at a time in one; complex double, 8 right-hand sides, 4.4 ms with 8
  // vectors (119 KB, one CTA per SM), 3.4 ms with 4 and two CTAs per SM.
  constexpr bool k64 = sizeof(TM) == sizeof(double2);
  int fit = k64 ? 8 : 4;
  while (fit > 1 && (size_t)fit * (xcap + q2) * sizeof(typename MT<TM>::Acc) > (size_t)(k64 ? 110 : 220) * 1024) fit >>= 1;
  for (int g = 0; g < 4; ++g) {
    const long long n = use_tc ? h->ct.kitems_ntc[g] : (long long)h->ct.kitems[g].size();
    if (n == 0) continue;
    A.items = h->dct.kitems[g];
    const int step = std::max(1, fit >> g);
    for (int r0 = 0; r0 < nrhs; r0 += A.total) {
      A.nrl = next_group<TM>(nrhs - r0, step, kSplitEntries);
      // all groups of one size in a launch; in complex float the last one may be smaller
      A.total = k64 ? (nrhs - r0) / A.nrl * A.nrl : nrhs - r0;
      A.groups = (A.total + A.nrl - 1) / A.nrl;
      A.nitems = n * A.groups;
      A.nrhs = A.nrl << g;
      A.t = t + (long long)r0 * rstride;
      A.z = z + (long long)r0 * h->nf;
      // shapes are tuned for single right-hand sides of the float kernels, on handles whose solves
      // run them; otherwise as many rows per warp as leave work for all 8 warps of an item, and with
      // several vectors no second turn for a few rows left (18 rows, p = 8, 12 right-hand sides at
      // 8^3 leaves: 418 us with 2 rows per warp, 353 us with 1)
      const bool tuned = h->shapes.k_tuned && A.nrl == 1 && !k64;
      const int rows = (q2 + A.split - 1) / A.split;
      const int half = A.nrhs == 1 || k64 ? 16 : 24, full = A.nrhs == 1 || k64 ? 32 : 40;
      const LaunchShape sh = tuned ? h->shapes.k[g] : LaunchShape{rows >= full ? 4 : rows >= half ? 2 : 1, 0};
      const cudaError_t e = launch_group<P>(A, A.nrhs, xcap, q2, h->nsm, st, &h->prof.launches, h->gate, sh);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

template <class TM, class TIN, class TOUT>
cudaError_t precond_t(const hps_handle* h, const TM* B, const TM* K, const TIN* r, TOUT* z, TOUT* t,
                      size_t scratch_bytes, int nrhs, cudaStream_t st, const float* bscale = nullptr, const float* kscale = nullptr,
                      bool use_tc = false) {
  const int q2 = h->q * h->q;
  const long long tstride = h->ct.tsize;
  // FP16 blocks with complex-float output on 2x2x2 clusters: stage B in tc_precond16.cu, and stage K
  // there too for one right-hand side and multiples of 64.  In between (and for ragged multiples)
  // the widely shared blocks take their complex-FP32 copies on the tensor cores and the others the
  // FP32 kernel: error against the exact product of the same blocks at p = 10 1.9e-7, on the FP16
  // tensor-core kernel 4.0e-7 (3.5e-6 with one sum per row), which is 103 instead of 514 us for 12
  // right-hand sides at 8^3 leaves, p = 8, but less than the FP32 that these calls have promised.
  if constexpr (std::is_same<TM, __half2>::value && std::is_same<TOUT, float2>::value) {
    const bool tc16 = precond_tc16_eligible(h, nrhs, scratch_bytes);
    if (precond_b16_eligible(h) && (tc16 || !precond_tc_multi_eligible(h, nrhs))) {
      constexpr VType kIn = std::is_same<TIN, float2>::value ? VType::C64
                            : std::is_same<TIN, float4>::value ? VType::DF : VType::C128;
      cudaEvent_t ev = h->prof.begin(st);
      cudaError_t e = launch_precond_b16(h, kIn, r, z, t, tc16, nrhs, st);
      h->prof.end(HPS_PHASE_PRECOND_B, ev, st);
      if (e != cudaSuccess) return e;
      ev = h->prof.begin(st);
      if (tc16) {
        e = launch_precond_tc16(h, t, z, nrhs, st);
      } else {
        // t as [position][right-hand side][nint0]; position p is cl_tpos / nint0
        if (use_tc) e = launch_precond_tc_vec(h, t, z, nrhs, h->tc_error, st);
        if (e == cudaSuccess) e = stage_k_simt(h, K, kscale, t, h->ct.nint0, nrhs, z, nrhs, use_tc, st);
      }
      h->prof.end(HPS_PHASE_PRECOND_K, ev, st);
      return e;
    }
  }
  {
    PrecBArgs<TM, TIN, TOUT> A;
    A.B = B;
    A.bscale = bscale;
    A.b_off = h->dct.b_off;
    A.int_mask = h->dct.int_mask;
    A.brd = h->dct.brd;
    A.bto = h->dct.bto;
    A.bsc = h->dct.bsc;
    A.nl = h->nl;
    A.q2 = q2;
    A.gate = h->gate;
    A.r = r;
    A.z = z;
    A.t = t;
    A.nrhs = nrhs;
    A.vstride = h->nf;
    A.tstride = tstride;
    A.groups = h->dct.bgroups;
    A.gleaves = h->dct.bgroup_leaves;
    A.ngroups = (int)h->ct.bgroups.size();
    using Acc = typename MT<TM>::Acc;
    cudaEvent_t ev = h->prof.begin(st);
    auto launch_b = [&](auto kern, int nr) -> cudaError_t {
      const size_t smem = (size_t)nr * h->ct.max_ext * q2 * sizeof(Acc) + 16;
      cudaError_t e2 = allow_dynamic_smem((const void*)kern, smem);
      int occ = 0;
      if (e2 == cudaSuccess) e2 = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kThreads, smem);
      if (e2 != cudaSuccess) return e2;
      // Where the items leave SMs idle, each is cut by rows into CTAs of a warp or more (64 leaves
      // at p = 8 in complex double: 32.5 us with one CTA and one sum per row, 28.5 us with 4 CTAs
      // and four sums; both with the timer's own ~8 us).  Not with many vectors per pass, which
      // every part would stage again: 64 right-hand sides, complex float, both stages at 4^3 leaves,
      // p = 8, 305 us in parts and 102 us whole; 2^3 leaves, p = 6, 86 and 52 us.
      PrecBArgs<TM, TIN, TOUT> C = A;
      const int rows = 3 * q2;
      C.parts = nr > 8 ? 1 : std::max(1, std::min((rows + 31) / 32, 2 * h->nsm / std::max(1, A.ngroups)));
      const int threads = C.parts > 1 ? std::min(kThreads, (int)round_up((rows + C.parts - 1) / C.parts, 32)) : kThreads;
      const int grid = (int)std::min<long long>((long long)A.ngroups * C.parts, (long long)h->nsm * std::max(occ, 1));
      kern<<<grid, threads, smem, st>>>(C);
      ++h->prof.launches;
      return cudaGetLastError();
    };
    // NR vectors (leaf of a group, right-hand side) per pass; shared memory for NR x (the most
    // external columns of any leaf: 3 q^2 when every cluster is 2x2x2, up to 6 q^2 for a leaf
    // alone in its cluster), halved while it does not fit
    const long long nvec = (long long)std::max(h->ct.max_group, 1) * nrhs;
    // (32 at a time with FP32 accumulators and many right-hand sides: each B entry read from L2
    // then feeds 32 accumulations)
    constexpr bool kWide = sizeof(Acc) == 8;
    int nr = nvec <= 1 ? 1 : nvec == 2 ? 2 : nvec <= 4 ? 4 : (kWide && nvec >= 32) ? 32 : 8;
    while (nr > 1 && (size_t)nr * h->ct.max_ext * q2 * sizeof(Acc) + 16 > (size_t)kMaxDynSmem) nr >>= 1;
    cudaError_t e;
    if (nr == 1) e = launch_b(prec_b_kernel<TM, TIN, TOUT, 1>, 1);
    else if (nr == 2) e = launch_b(prec_b_kernel<TM, TIN, TOUT, 2>, 2);
    else if (nr == 4) e = launch_b(prec_b_kernel<TM, TIN, TOUT, 4>, 4);
    else if (nr == 8) e = launch_b(prec_b_kernel<TM, TIN, TOUT, 8>, 8);
    else if constexpr (kWide) e = nr == 32 ? launch_b(prec_b_kernel<TM, TIN, TOUT, 32>, 32)
                                           : launch_b(prec_b_kernel<TM, TIN, TOUT, 16>, 16);
    else e = launch_b(prec_b_kernel<TM, TIN, TOUT, 8>, 8);
    h->prof.end(HPS_PHASE_PRECOND_B, ev, st);
    if (e != cudaSuccess) return e;
  }
  if (h->ct.nslots == 0) return cudaSuccess;
  cudaEvent_t ev = h->prof.begin(st);
  cudaError_t e = cudaSuccess;
  if constexpr (std::is_same<TOUT, float2>::value) {
    // many right-hand sides: every block once per 64 of them, on the tensor cores
    if (precond_tc_multi_eligible(h, nrhs)) {
      e = launch_precond_tc_multi(h, t, z, nrhs, h->tc_error, st);
      h->prof.end(HPS_PHASE_PRECOND_K, ev, st);
      return e;
    }
    for (int rhs = 0; use_tc && rhs < nrhs && e == cudaSuccess; ++rhs)
      e = launch_precond_tc(h, t + (long long)rhs * tstride, z + (long long)rhs * h->nf, h->tc_error, st);
  }
  if (e == cudaSuccess) e = stage_k_simt(h, K, kscale, t, tstride, 1, z, nrhs, use_tc, st);
  h->prof.end(HPS_PHASE_PRECOND_K, ev, st);
  return e;
}

}  // namespace

bool apply_tc_eligible(const hps_handle* h, int nrhs) {
  return h->opt.tc_apply && h->tc_error && h->R32 && nrhs >= 64 && nrhs % 64 == 0;
}

cudaError_t launch_apply(const hps_handle* h, bool fp32_matrix, VType tin, const void* f, VType tout, void* y,
                         const double2* bvec, int nrhs, bool residual, cudaStream_t st) {
  if (!residual) bvec = nullptr;
  if (!fp32_matrix) {
    if (tin == VType::C128 && tout == VType::C128)
      return apply_t(h, h->R64, (const double2*)f, (double2*)y, bvec, nrhs, st);
    return cudaErrorInvalidValue;
  }
  // the residual form b - (I + Pi R) f only exists for complex-double vectors
  if (bvec && !(tin == VType::C128 && tout == VType::C128)) return cudaErrorInvalidValue;
  // complex-double vectors on a lean handle: the compensated FP32 maps (FP64-accurate)
  if (tin == VType::C128 && tout == VType::C128 && compensated_maps(h)) return launch_apply_cf(h, (const double2*)f,
                                                                                               (double2*)y, bvec, nrhs, st);
  const bool tc = apply_tc_eligible(h, nrhs) && !bvec;
  if (tc && tin == VType::C64 && tout == VType::C64)
    return launch_apply_tc(h, (const float2*)f, y, false, nrhs, h->tc_error, st);
  if (tc && tin == VType::C64 && tout == VType::DF)
    return launch_apply_tc(h, (const float2*)f, y, true, nrhs, h->tc_error, st);
  if (tin == VType::C64 && (tout == VType::C64 || tout == VType::DF) && stream_apply_eligible(h, f, tout, nrhs))
    return launch_stream_apply(h, (const float2*)f, tout, y, nrhs, st);
  if (tin == VType::C64 && tout == VType::C64)
    return apply_t(h, h->R32, (const float2*)f, (float2*)y, nullptr, nrhs, st);
  if (tin == VType::C64 && tout == VType::C128)
    return apply_t(h, h->R32, (const float2*)f, (double2*)y, nullptr, nrhs, st);
  if (tin == VType::C128 && tout == VType::C128)
    return apply_t(h, h->R32, (const double2*)f, (double2*)y, bvec, nrhs, st);
  if (tin == VType::C64 && tout == VType::DF)
    return apply_t(h, h->R32, (const float2*)f, (float4*)y, nullptr, nrhs, st);
  if (tin == VType::DF && tout == VType::DF)
    return apply_t(h, h->R32, (const float4*)f, (float4*)y, nullptr, nrhs, st);
  return cudaErrorInvalidValue;
}

cudaError_t timed_apply(const hps_handle* h, int phase, bool fp32_matrix, VType tin, const void* f, VType tout,
                        void* y, const double2* bvec, int nrhs, bool residual, cudaStream_t st) {
  cudaEvent_t ev = h->prof.begin(st);
  cudaError_t e = launch_apply(h, fp32_matrix, tin, f, tout, y, bvec, nrhs, residual, st);
  h->prof.end(phase, ev, st);
  return e;
}

template <class TM>
cudaError_t rhs_t(const hps_handle* h, const TM* H, const double2* s, const double2* t, double2* b, int nrhs,
                  cudaStream_t st) {
  using P = RhsP<TM>;
  typename P::Args A;
  A.H = H;
  A.ldH = h->ldH;
  A.ni = h->ni;
  A.nb = h->nb;
  A.q2 = h->q * h->q;
  A.g = GridDims{h->nx, h->ny, h->nz};
  A.s = s;
  A.t = t;
  A.out = b;
  A.nf = h->nf;
  A.nint = h->nint;
  A.nrhs = nrhs;
  const int xcap = xcap_of(h, XCap::Rhs);
  const LeafPlan plan = leaf_plan(h, nrhs, sizeof(typename P::Acc), xcap);
  A.parts = plan.parts;
  A.inv = row_inv(A.q2);
  A.nitems = (long long)h->nl * A.parts;
  static const LaunchShape kDefault[4] = {{4, 0}, {4, 0}, {2, 0}, {2, 0}};
  return launch_groups<P>(h, A, nrhs, plan.most, xcap, (h->nb + A.parts - 1) / A.parts, st, [&](typename P::Args& B, int r0) {
    if (B.s) B.s += (long long)r0 * h->nint;
    if (B.t) B.t += (long long)r0 * h->nf;
    B.out += (long long)r0 * h->nf;
  }, kDefault, nullptr);
}

cudaError_t launch_rhs(const hps_handle* h, const double2* s, const double2* t, double2* b, int nrhs,
                       cudaStream_t st, bool compensated) {
  if (compensated && h->H16lo && h->H32) return launch_rhs_cf(h, s, t, b, nrhs, st);
  if (h->H64) return rhs_t(h, h->H64, s, t, b, nrhs, st);
  if (h->H16lo) return launch_rhs_cf(h, s, t, b, nrhs, st);
  return rhs_t(h, h->H32, s, t, b, nrhs, st);
}

cudaError_t launch_precond(const hps_handle* h, bool fp32_matrix, VType tin, const void* r, VType tout, void* z,
                           void* scratch, size_t scratch_bytes, int nrhs, cudaStream_t st, bool fp16_blocks) {
  if (!fp32_matrix) {
    if (tin == VType::C128 && tout == VType::C128)
      return precond_t(h, h->B64, h->Kc64, (const double2*)r, (double2*)z, (double2*)scratch, scratch_bytes, nrhs, st);
    return cudaErrorInvalidValue;
  }
  if (tout != VType::C64) return cudaErrorInvalidValue;
  // shared K blocks with many member clusters: complex-FP32 blocks on the tensor cores
  const bool tc = h->opt.tc_apply && h->Kc32 && h->tc_error && !h->ct.kc_tc.empty();
  if (fp16_blocks) {
    if (!h->Kc16 || !h->B16) return cudaErrorInvalidValue;
    auto run = [&](auto* in) {
      return precond_t(h, h->B16, h->Kc16, in, (float2*)z, (float2*)scratch, scratch_bytes, nrhs, st, h->B16s, h->Kc16s, tc);
    };
    if (tin == VType::C64) return run((const float2*)r);
    if (tin == VType::DF) return run((const float4*)r);
    return run((const double2*)r);
  }
  auto run = [&](auto* in) {
    return precond_t(h, h->B32, h->Kc32, in, (float2*)z, (float2*)scratch, scratch_bytes, nrhs, st, (const float*)nullptr,
                     (const float*)nullptr, tc);
  };
  if (tin == VType::C64) return run((const float2*)r);
  if (tin == VType::DF) return run((const float4*)r);
  return run((const double2*)r);
}

// ---------------------------------------------------------------------------
// Autotuner of the launch shapes (rows per warp, resident CTAs per SM) of the
// batched GEMV kernels, run once per shape at setup: every candidate is timed
// with CUDA events (one warm-up launch, then three) on the handle's own data,
// the fastest kept in a process-wide table keyed by (device, kernel, q,
// leaves, right-hand-side group, work items), so later handles of the same
// size reuse it.  The shapes do not change results (see LaunchShape).
// ---------------------------------------------------------------------------
namespace {

std::mutex g_tune_mu;
std::map<std::array<long long, 6>, LaunchShape> g_tuned;

template <class P>
LaunchShape tune_group(const hps_handle* h, const typename P::Args& A, int nr, int xcap, int rowcap,
                       const std::array<long long, 6>& key, LaunchShape dflt, cudaStream_t st) {
  {
    std::lock_guard<std::mutex> lock(g_tune_mu);
    auto it = g_tuned.find(key);
    if (it != g_tuned.end()) return it->second;
  }
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
    cudaGetLastError();
    if (e0) cudaEventDestroy(e0);
    return dflt;
  }
  long long dummy = 0;
  auto time_one = [&](LaunchShape sh) -> float {
    if (launch_group<P>(A, nr, xcap, rowcap, h->nsm, st, &dummy, nullptr, sh) != cudaSuccess) return 1e30f;
    cudaEventRecord(e0, st);
    for (int i = 0; i < 3; ++i)
      if (launch_group<P>(A, nr, xcap, rowcap, h->nsm, st, &dummy, nullptr, sh) != cudaSuccess) return 1e30f;
    cudaEventRecord(e1, st);
    if (cudaEventSynchronize(e1) != cudaSuccess) return 1e30f;
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    return ms / 3.f;
  };
  LaunchShape best = dflt;
  float tbest = time_one(dflt);
  const int nrp = nr <= 2 ? nr : nr <= 4 ? 4 : 8;
  const int rmax = std::min(8, kMaxAcc<typename P::TM> / nrp);
  for (int rpw = 1; rpw <= rmax; rpw *= 2)
    for (int bps = 0; bps <= 3; ++bps) {
      const LaunchShape sh{rpw, bps};
      if (sh.rpw == dflt.rpw && sh.bps == dflt.bps) continue;
      const float t = time_one(sh);
      if (t < 0.98f * tbest) {  // a clear win over the incumbent only
        tbest = t;
        best = sh;
      }
    }
  cudaGetLastError();
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  std::lock_guard<std::mutex> lock(g_tune_mu);
  g_tuned[key] = best;
  return best;
}

template <class TM, class TIN, class TOUT>
cudaError_t tune_apply(hps_handle* h, const TM* R, int kind, void* fbuf, void* ybuf, int nr, cudaStream_t st) {
  using P = ApplyP<TM, TIN, TOUT>;
  typename P::Args A;
  A.R = R;
  A.ldR = h->ldR;
  A.nb = h->nb;
  A.q2 = h->q * h->q;
  A.g = GridDims{h->nx, h->ny, h->nz};
  A.f = (const TIN*)fbuf;
  A.y = (TOUT*)ybuf;
  A.bvec = nullptr;
  A.nf = h->nf;
  A.nrhs = nr;
  const int xcap = xcap_of(h, XCap::Apply);
  const LeafPlan plan = leaf_plan(h, nr, sizeof(typename P::Acc), xcap);
  if (plan.most < nr) return cudaSuccess;  // such groups are not launched
  A.parts = plan.parts;
  A.inv = row_inv(A.q2);
  A.nitems = (long long)h->nl * A.parts;
  const int g = group_index(nr);
  const std::array<long long, 6> key{h->dev, kind, h->q, h->nl, nr, A.nitems};
  h->shapes.apply_tuned[kind][g] = true;
  h->shapes.apply[kind][g] = tune_group<P>(h, A, nr, xcap, (h->nb + A.parts - 1) / A.parts, key, h->shapes.apply[kind][g], st);
  return cudaSuccess;
}

template <class TM>
cudaError_t tune_stage_k(hps_handle* h, const TM* K, const float* kscale, void* t, void* z, bool tc, cudaStream_t st) {
  using P = PrecKP<TM, float2, float2>;
  typename P::Args A;
  A.K = K;
  A.kscale = kscale;
  A.kc_off = h->dct.kc_off;
  A.kc_slot_begin = h->dct.kc_slot_begin;
  A.members = h->dct.kc_members;
  A.cl_slot_begin = h->dct.cl_slot_begin;
  A.slot_lf = h->dct.slot_lf;
  A.cl_tpos = h->dct.cl_tpos;
  A.split = h->ct.krow_split;
  A.nb = h->nb;
  A.q2 = h->q * h->q;
  A.nf = h->nf;
  A.tstride = h->ct.tsize;
  A.tmul = 1;
  A.t = (const float2*)t;
  A.z = (float2*)z;
  for (int g = 0; g < 4; ++g) {
    const long long n = tc ? h->ct.kitems_ntc[g] : (long long)h->ct.kitems[g].size();
    if (n == 0) continue;
    A.items = h->dct.kitems[g];
    A.nitems = n;
    A.nrl = A.total = A.groups = 1;
    A.nrhs = 1 << g;
    const std::array<long long, 6> key{h->dev, 10 + (long long)sizeof(TM), h->q, h->nl, g, n};
    h->shapes.k[g] = tune_group<P>(h, A, 1 << g, xcap_of(h, XCap::StageK), A.q2, key, h->shapes.k[g], st);
  }
  return cudaSuccess;
}

}  // namespace

int autotune_shapes(hps_handle* h, cudaStream_t st) {
  const long long nf = h->nf;
  const int nr_max = std::min(8, std::max(1, h->opt.max_rhs));
  void *fbuf = nullptr, *ybuf = nullptr;
  const size_t bytes = (size_t)nr_max * nf * sizeof(double2);
  if (cudaMalloc(&fbuf, bytes) != cudaSuccess || cudaMalloc(&ybuf, bytes) != cudaSuccess) {
    cudaGetLastError();
    if (fbuf) cudaFree(fbuf);
    return HPS_OK;  // tuning is an optimization: keep the default shapes
  }
  cudaMemsetAsync(fbuf, 0, bytes, st);
  cudaMemsetAsync(ybuf, 0, bytes, st);
  std::vector<int> groups{1};
  if (nr_max > 1) groups.push_back(nr_max);
  for (int nr : groups) {
    // the inner apply of each form into the double-float basis, and FP64.  Where complex-FP32
    // operands take stream_apply.cu, the double-float ones (solves without the preconditioner) are
    // what is left for the FP32 maps.  A 16^3-leaf, p = 10 solve: 209.8 ms with the default
    // shapes, 202.1 ms with the tuned ones.
    if (h->R32) {
      if (stream_apply_eligible(h, fbuf, VType::DF, nr)) tune_apply<float2, float4, float4>(h, h->R32, 0, fbuf, ybuf, nr, st);
      else tune_apply<float2, float2, float4>(h, h->R32, 0, fbuf, ybuf, nr, st);
    }
    if (h->R64 && (h->opt.forms & HPS_FORM_FP64)) tune_apply<double2, double2, double2>(h, h->R64, 1, fbuf, ybuf, nr, st);
  }
  // SIMT stage K of the mixed solve (FP16 blocks when kept, else FP32)
  if (h->has_precond && h->ct.nslots > 0 && h->pc_scratch && !precond_b16_eligible(h)) {
    cudaMemsetAsync(h->pc_scratch, 0, (size_t)h->ct.tsize * sizeof(float2), st);
    const bool tc = h->opt.tc_apply && h->Kc32 && h->tc_error && !h->ct.kc_tc.empty();
    if (h->Kc16) tune_stage_k<__half2>(h, h->Kc16, h->Kc16s, h->pc_scratch, ybuf, tc, st);
    else if (h->Kc32) tune_stage_k<float2>(h, h->Kc32, nullptr, h->pc_scratch, ybuf, tc, st);
    h->shapes.k_tuned = true;
  }
  cudaStreamSynchronize(st);
  cudaGetLastError();
  cudaFree(fbuf);
  cudaFree(ybuf);
  h->shapes.tuned = true;
  return HPS_OK;
}

}  // namespace hps
