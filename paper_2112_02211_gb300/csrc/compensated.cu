// Compensated FP32 leaf maps for the memory-lean form: a map M (the ItI map R
// or the body-load map H, Sec. 2.2) is kept as its FP32 rounding M32 plus the
// rounding remainder M - M32 in FP16, scaled per row by sigma_i = max_j of the
// remainder's components, so that M32 + sigma_i lo_ij reproduces M to about
// 2^-24 * 2^-11 ~ 3e-11 relative, at 12 bytes per complex entry instead of 16
// (complex FP64).  Products with complex-double vectors x = x_hi + x_lo (two
// FP32 parts) are accumulated in double-float on the FP32 pipe:
//
//   M32 x_hi   exactly, each real product split by the FMA TwoProduct and
//              summed by Knuth's TwoSum into (sum, error) pairs;
//   M32 x_lo + sigma lo x_hi   in plain FP32 (terms 2^-24 smaller, so their
//              rounding is below the FP64-level target).
//
// This gives the lean form an FP64-accurate restart residual
// b - (I + Pi R) x, an FP64-accurate right-hand side b = tbar - Pi H s and
// complex-double applies, instead of FP32-accurate ones.  Item = (leaf, part): a
// part of the rows of the leaf's faces with a neighbour; the swap Pi is fused into the store as in
// the other applies (one writer per output slot).
//
// What bounds it: about 50 FP32 instructions per complex entry and right-hand side (12 bytes), on
// top of the warp reductions, which halve the sums in flight at every exchange, and the latency of
// the map entries, which are loaded one step ahead.  Measured, 8^3 leaves at p = 8:
// restart residual of 8 right-hand sides 2.23 -> 0.55 ms, of one 217 -> 103 us; right-hand side of 8
// sources 2.20 -> 0.54 ms (before: items of a face's 32 and 4 rows, one CTA per SM, full butterflies).
#include <algorithm>

#include "common.cuh"
#include "hps_internal.h"

namespace hps {

namespace {

constexpr int kT = 256;
constexpr int kW = kT / 32;
constexpr int kRPW = 2;  // rows per warp pass
constexpr int kNRMax = 4;  // most right-hand sides per pass over the block
constexpr int kCR = 48;    // rows per work item at most: a leaf is split so that the rows every
                           // pass over the right-hand sides re-reads stay in L2

// (sum, error) pair: value = s + c
struct cacc {
  float s, c;
};
__device__ __forceinline__ void cacc_prod(cacc& a, float x, float y) {
  const float p = __fmul_rn(x, y);
  const float e = __fmaf_rn(x, y, -p);
  const dfr t = df_two_sum(a.s, p);
  a.s = t.h;
  a.c = __fadd_rn(a.c, __fadd_rn(t.l, e));
}
__device__ __forceinline__ cacc cacc_merge(cacc a, cacc b) {
  const dfr t = df_two_sum(a.s, b.s);
  return {t.h, __fadd_rn(__fadd_rn(a.c, b.c), t.l)};
}
__device__ __forceinline__ cacc cacc_shfl(cacc a, int o) {
  return {__shfl_xor_sync(0xffffffffu, a.s, o), __shfl_xor_sync(0xffffffffu, a.c, o)};
}

struct CfArgs {
  const float2* M;     // FP32 rounding of the maps, per leaf nb x ld row-major
  const __half2* lo;   // remainder / row scale, same layout
  const float* scale;  // per row (leaf * nb + row)
  int ld, ncols, nb, q2;
  long long leaf_stride;  // elements per leaf of M / lo
  GridDims g;
  const double2* x;    // input [rhs][xstride]: face vectors (R) or interior vectors (H)
  long long xstride, xleaf;  // rhs stride, per-leaf offset unit
  double2* y;          // output [rhs][nf]
  const double2* b;    // R: residual mode y = b - (x + Pi R x), or nullptr (apply y = x + Pi R x)
  const double2* t;    // H: boundary data for the boundary-face slots, or nullptr
  long long nf;
  int nrhs, rhs_mode;  // rhs_mode: the map is H (b = tbar - Pi H s) instead of R
  int parts;           // items per leaf
  unsigned inv;        // row_inv(q2)
  long long nitems;
};

// One row's sums of one right-hand side.
struct CfSum {
  cacc re, im;
  float sre, sim;
};
__device__ __forceinline__ float pick(bool first, float a, float b) { return first ? a : b; }
__device__ __forceinline__ CfSum cf_pick(bool first, CfSum a, CfSum b) {
  return {{pick(first, a.re.s, b.re.s), pick(first, a.re.c, b.re.c)},
          {pick(first, a.im.s, b.im.s), pick(first, a.im.c, b.im.c)},
          pick(first, a.sre, b.sre),
          pick(first, a.sim, b.sim)};
}
__device__ __forceinline__ CfSum cf_exchange(CfSum keep, CfSum send, int o) {
  return {cacc_merge(keep.re, cacc_shfl(send.re, o)), cacc_merge(keep.im, cacc_shfl(send.im, o)),
          __fadd_rn(keep.sre, __shfl_xor_sync(0xffffffffu, send.sre, o)),
          __fadd_rn(keep.sim, __shfl_xor_sync(0xffffffffu, send.sim, o))};
}

// kNR right-hand sides per pass over the block (1, 2 or 4)
template <int kNR>
__global__ void __launch_bounds__(kT, kNR == 4 ? 2 : kNR == 2 ? 2 : 3) cf_gemv_kernel(const CfArgs A, int ncp) {
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* xh = reinterpret_cast<float2*>(smraw);  // kNR x ncp
  float2* xl = xh + kNR * ncp;                    // kNR x ncp
  double2* outs = reinterpret_cast<double2*>(xl + kNR * ncp);  // kNR x kCR
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int q2 = A.q2;
  for (long long item = blockIdx.x; item < A.nitems; item += gridDim.x) {
    const int leaf = (int)(item / A.parts), part = (int)(item % A.parts);
    unsigned mask = 0, flist = 0;
    int faces = 0;
#pragma unroll
    for (int f = 0; f < 6; ++f)
      if (A.g.neighbor(leaf, f) >= 0) {
        mask |= 1u << f;
        flist |= (unsigned)f << (4 * faces++);
      }
    const int row0 = faces * q2 * part / A.parts, nrow = faces * q2 * (part + 1) / A.parts - row0;
    auto place = [&](int l, int& face, int& j) {  // row l of the item
      const unsigned r = row0 + l, k = (r * A.inv) >> 20;
      j = (int)(r - k * q2);
      face = (flist >> (4 * k)) & 7u;
    };
    if (part == 0 && mask != 63u)
      // boundary faces: R rows unused (Pi is 0 there); H: the slot takes t (or 0)
      for (int idx = tid; idx < 6 * q2; idx += kT) {
        if ((mask >> (idx / q2)) & 1u) continue;
        for (int rr = 0; rr < A.nrhs; ++rr) {
          const long long o = (long long)rr * A.nf + (long long)leaf * A.nb + idx;
          if (A.rhs_mode) {
            A.y[o] = A.t ? A.t[o] : make_double2(0.0, 0.0);
          } else {
            const double2 xv = A.x[(long long)rr * A.xstride + (long long)leaf * A.nb + idx];
            A.y[o] = A.b ? csub(A.b[o], xv) : xv;
          }
        }
      }
    if (A.rhs_mode && !A.x) {  // no body load: h = 0
      for (int l = tid; l < nrow; l += kT) {
        int face, j;
        place(l, face, j);
        const long long o = (long long)A.g.neighbor(leaf, face) * A.nb + (long long)(face ^ 1) * q2 + j;
        for (int rr = 0; rr < A.nrhs; ++rr) A.y[(long long)rr * A.nf + o] = make_double2(0.0, 0.0);
      }
      continue;
    }
    const float2* Mb = A.M + (long long)leaf * A.leaf_stride;
    const __half2* Lb = A.lo + (long long)leaf * A.leaf_stride;
    const float* Sb = A.scale + (long long)leaf * A.nb;
    for (int r0 = 0; r0 < A.nrhs; r0 += kNR) {
      const int nr = min(kNR, A.nrhs - r0);
      __syncthreads();
#pragma unroll
      for (int rr = 0; rr < kNR; ++rr)
        for (int c = tid; c < ncp; c += kT) {
          double2 v = make_double2(0.0, 0.0);
          if (rr < nr && c < A.ncols) v = A.x[(long long)(r0 + rr) * A.xstride + (long long)leaf * A.xleaf + c];
          const float hr = __double2float_rn(v.x), hi = __double2float_rn(v.y);
          xh[rr * ncp + c] = make_float2(hr, hi);
          xl[rr * ncp + c] = make_float2(__double2float_rn(v.x - (double)hr), __double2float_rn(v.y - (double)hi));
        }
      __syncthreads();
      for (int rw = warp * kRPW; rw < nrow; rw += kW * kRPW) {
        constexpr int V = kRPW * kNR;
        CfSum acc[V];  // (row, right-hand side)
        float sig[kRPW];
        const float2* mrow[kRPW];
        const __half2* lrow[kRPW];
#pragma unroll
        for (int i = 0; i < kRPW; ++i) {
          int face, j;
          place(min(rw + i, nrow - 1), face, j);
          const int r = face * q2 + j;
          sig[i] = Sb[r];
          mrow[i] = Mb + (long long)r * A.ld;
          lrow[i] = Lb + (long long)r * A.ld;
        }
#pragma unroll
        for (int i = 0; i < V; ++i) acc[i] = {{0.f, 0.f}, {0.f, 0.f}, 0.f, 0.f};
        // entries one step ahead
        float4 m[kRPW];
        uint2 lraw[kRPW];
        int c = lane * 2;
        auto fetch = [&](int cc) {
          if (cc >= ncp) return;
#pragma unroll
          for (int i = 0; i < kRPW; ++i) {
            m[i] = __ldg(reinterpret_cast<const float4*>(mrow[i] + cc));
            lraw[i] = __ldg(reinterpret_cast<const uint2*>(lrow[i] + cc));
          }
        };
        fetch(c);
        for (; c < ncp; c += 64) {
          float4 mc[kRPW];
          uint2 lc[kRPW];
#pragma unroll
          for (int i = 0; i < kRPW; ++i) {
            mc[i] = m[i];
            lc[i] = lraw[i];
          }
          fetch(c + 64);
#pragma unroll
          for (int i = 0; i < kRPW; ++i) {
            const float2 l0 = __half22float2(*reinterpret_cast<const __half2*>(&lc[i].x));
            const float2 l1 = __half22float2(*reinterpret_cast<const __half2*>(&lc[i].y));
            const float2 mv[2] = {make_float2(mc[i].x, mc[i].y), make_float2(mc[i].z, mc[i].w)};
            const float2 lv[2] = {make_float2(l0.x * sig[i], l0.y * sig[i]), make_float2(l1.x * sig[i], l1.y * sig[i])};
#pragma unroll
            for (int v = 0; v < 2; ++v) {
#pragma unroll
              for (int rr = 0; rr < kNR; ++rr) {
                CfSum& a = acc[i * kNR + rr];
                const float2 h = xh[rr * ncp + c + v], l = xl[rr * ncp + c + v];
                // main part, exactly: (a + ib)(xr + i xi) with the high parts of x
                cacc_prod(a.re, mv[v].x, h.x);
                cacc_prod(a.re, -mv[v].y, h.y);
                cacc_prod(a.im, mv[v].x, h.y);
                cacc_prod(a.im, mv[v].y, h.x);
                // small part: M32 x_lo + sigma lo x_hi
                float tr = __fmaf_rn(mv[v].x, l.x, -__fmul_rn(mv[v].y, l.y));
                tr = __fmaf_rn(lv[v].x, h.x, tr);
                tr = __fmaf_rn(-lv[v].y, h.y, tr);
                float ti = __fmaf_rn(mv[v].x, l.y, __fmul_rn(mv[v].y, l.x));
                ti = __fmaf_rn(lv[v].x, h.y, ti);
                ti = __fmaf_rn(lv[v].y, h.x, ti);
                a.sre = __fadd_rn(a.sre, tr);
                a.sim = __fadd_rn(a.sim, ti);
              }
            }
          }
        }
        // warp sums: each step exchanges half of the sums still held (plain once one is left)
        int held = V, first = 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          if (held > 1) {
            held >>= 1;
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int k = 0; k < V / 2; ++k)
              if (k < held) acc[k] = cf_exchange(cf_pick(up, acc[k + held], acc[k]), cf_pick(up, acc[k], acc[k + held]), o);
            if (up) first += held;
          } else {
            acc[0] = cf_exchange(acc[0], acc[0], o);
          }
        }
        const int i = first / kNR, rr = first % kNR;
        if (lane % (32 / V) == 0 && rw + i < nrow)
          outs[rr * kCR + rw + i] = make_double2((double)acc[0].re.s + (double)acc[0].re.c + (double)acc[0].sre,
                                                 (double)acc[0].im.s + (double)acc[0].im.c + (double)acc[0].sim);
      }
      __syncthreads();
      for (int l = tid; l < nrow; l += kT) {
        int face, j;
        place(l, face, j);
        const long long dst = (long long)A.g.neighbor(leaf, face) * A.nb + (long long)(face ^ 1) * q2 + j;
        for (int rr = 0; rr < nr; ++rr) {
          const long long o = (long long)(r0 + rr) * A.nf + dst;
          const double2 gv = outs[rr * kCR + l];
          if (A.rhs_mode) {
            A.y[o] = make_double2(-gv.x, -gv.y);
          } else {
            const double2 xv = A.x[(long long)(r0 + rr) * A.xstride + dst];
            const double2 yv = cadd(xv, gv);
            A.y[o] = A.b ? csub(A.b[o], yv) : yv;
          }
        }
      }
    }
    __syncthreads();
  }
}

// Row-wise split of an FP64 map into its FP32 rounding (written elsewhere) and the
// remainder in FP16: lo = (M - fl32(M)) / sigma_row, sigma_row = max |remainder
// component| over the row (1 when the row is exactly representable).  One warp per row.
__global__ void split_lo_kernel(const double2* M, long long rows, int ld, __half2* lo, float* scale) {
  const int lane = threadIdx.x & 31;
  const long long row = (long long)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
  if (row >= rows) return;
  const double2* m = M + row * ld;
  float mx = 0.f;
  for (int c = lane; c < ld; c += 32) {
    const double2 v = m[c];
    mx = fmaxf(mx, fabsf((float)(v.x - (double)(float)v.x)));
    mx = fmaxf(mx, fabsf((float)(v.y - (double)(float)v.y)));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  const float sig = mx > 0.f ? mx : 1.f;
  if (lane == 0) scale[row] = sig;
  for (int c = lane; c < ld; c += 32) {
    const double2 v = m[c];
    const float rr = (float)((v.x - (double)(float)v.x) / (double)sig);
    const float ri = (float)((v.y - (double)(float)v.y) / (double)sig);
    lo[row * ld + c] = __floats2half2_rn(rr, ri);
  }
}

template <int kNR>
cudaError_t launch_cf_nr(const hps_handle* h, const CfArgs& A, int ncp, cudaStream_t st) {
  const size_t smem = (size_t)2 * kNR * ncp * sizeof(float2) + (size_t)kNR * kCR * sizeof(double2);
  auto kern = cf_gemv_kernel<kNR>;
  cudaError_t e = allow_dynamic_smem((const void*)kern, smem);
  if (e != cudaSuccess) return e;
  int occ = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kT, smem);
  if (e != cudaSuccess) return e;
  const long long grid = std::min<long long>(A.nitems, (long long)h->nsm * std::max(occ, 1));
  kern<<<(unsigned)grid, kT, smem, st>>>(A, ncp);
  ++h->prof.launches;
  return cudaGetLastError();
}

// one pass per group of up to 4 right-hand sides (a single right-hand side computes one)
cudaError_t launch_cf(const hps_handle* h, const CfArgs& A, int ncp, cudaStream_t st) {
  if (A.nrhs == 1) return launch_cf_nr<1>(h, A, ncp, st);
  if (A.nrhs == 2) return launch_cf_nr<2>(h, A, ncp, st);
  return launch_cf_nr<kNRMax>(h, A, ncp, st);
}

}  // namespace

cudaError_t launch_split_lo(const double2* M, long long rows, int ld, __half2* lo, float* scale, cudaStream_t st) {
  if (rows <= 0) return cudaSuccess;
  const int wpb = 8;
  split_lo_kernel<<<(unsigned)((rows + wpb - 1) / wpb), 32 * wpb, 0, st>>>(M, rows, ld, lo, scale);
  return cudaGetLastError();
}

bool compensated_maps(const hps_handle* h) { return h->R16lo != nullptr; }

// y = (I + Pi R) x (b == nullptr) or y = b - (I + Pi R) x with the compensated FP32 maps;
// x, y, b complex double [nrhs][nf].
cudaError_t launch_apply_cf(const hps_handle* h, const double2* x, double2* y, const double2* b, int nrhs,
                            cudaStream_t st) {
  if (!h->R32 || !h->R16lo) return cudaErrorInvalidValue;
  CfArgs A;
  A.M = h->R32;
  A.lo = h->R16lo;
  A.scale = h->R16ls;
  A.ld = h->ldR;
  A.ncols = h->nb;
  A.nb = h->nb;
  A.q2 = h->q * h->q;
  A.leaf_stride = (long long)h->nb * h->ldR;
  A.g = GridDims{h->nx, h->ny, h->nz};
  A.x = x;
  A.xstride = h->nf;
  A.xleaf = h->nb;
  A.y = y;
  A.b = b;
  A.t = nullptr;
  A.nf = h->nf;
  A.nrhs = nrhs;
  A.rhs_mode = 0;
  A.parts = (6 * A.q2 + kCR - 1) / kCR;
  A.inv = row_inv(A.q2);
  A.nitems = (long long)h->nl * A.parts;
  return launch_cf(h, A, (int)round_up(h->ldR, 2), st);
}

// b = tbar - Pi (H s) with the compensated FP32 maps H; s: [nrhs][nint] or nullptr.
cudaError_t launch_rhs_cf(const hps_handle* h, const double2* s, const double2* t, double2* b, int nrhs,
                          cudaStream_t st) {
  if (!h->H32 || !h->H16lo) return cudaErrorInvalidValue;
  CfArgs A;
  A.M = h->H32;
  A.lo = h->H16lo;
  A.scale = h->H16ls;
  A.ld = h->ldH;
  A.ncols = h->ni;
  A.nb = h->nb;
  A.q2 = h->q * h->q;
  A.leaf_stride = (long long)h->nb * h->ldH;
  A.g = GridDims{h->nx, h->ny, h->nz};
  A.x = s;
  A.xstride = h->nint;
  A.xleaf = h->ni;
  A.y = b;
  A.b = nullptr;
  A.t = t;
  A.nf = h->nf;
  A.nrhs = nrhs;
  A.rhs_mode = 1;
  A.parts = (6 * A.q2 + kCR - 1) / kCR;
  A.inv = row_inv(A.q2);
  A.nitems = (long long)h->nl * A.parts;
  return launch_cf(h, A, (int)round_up(h->ldH, 2), st);
}

}  // namespace hps
