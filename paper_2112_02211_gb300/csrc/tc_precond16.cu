// The cluster preconditioner with FP16 blocks where every cluster is 2x2x2 (z = J^{-1} r, Sec. 4,
// Algorithm 4 in face form):
//
// * stage B (prec_b16_kernel), any number of right-hand sides: a thread-block cluster of 4 CTAs per
//   up to 4 vectors that share their B blocks (right-hand sides, or members of one K block), two of
//   the 8 leaves a CTA, forms t = r_int - B r_ext (SIMT, two rows per thread, B stored transposed).
//   For the tensor-core stage K it finds the largest component t_max through distributed shared
//   memory and writes t / t_max as the tensor cores' operand: two FP16 terms hi + lo (~22 bits), each
//   as the rows conj(t) and the re/im swap of t.  Doing this here, once, replaces the conversion that
//   every 128-row tile of stage K would repeat (7 times at p = 8) on its way through shared memory.
//   Otherwise it writes t itself, for the SIMT stage K and the TF32 one of widely shared blocks.
// * stage K (tc_precond16_kernel), one right-hand side or a multiple of 64:
//   z_int = K_c t on the 5th-generation tensor cores
//   (tcgen05.mma.kind::f16, FP32 accumulation in TMEM).  A = K_c's FP16 copy (each row divided by
//   its FP32 scale s_row) as a real n x 2n matrix of interleaved (re, im) halves; B = the operand
//   rows; A B_hi + A B_lo = [Re | Im] of K_c t / (s_row t_max), multiplied back by s_row and t_max
//   in the epilogue.  K_c carries 2^-11 relative rounding (a fixed matrix); t is kept to ~2^-22,
//   so the result stays linear in t to FP32 level.  GMRES applies the preconditioner to V y in its
//   update and assumes that this equals sum_j y_j M^{-1} v_j; with one FP16 rounding of t (2^-11,
//   input-dependent) that would hold only to ~2e-4.  The tensor cores' sums truncate, so they are
//   kept short and added up in FP32 (kChunk); that is still 2e-7 to 4e-7 of the exact product of the
//   same blocks (p = 4 .. 12) where FP32 products and sums stay within 0.7e-7 to 2.4e-7, so other
//   numbers of right-hand sides take those (apply.cu).
//
// Vector v = position * nrhs + rhs (position: place of the member cluster in stage-K order), so
// the vectors of the clusters that share a block are consecutive.  A stage-K item is (block,
// 128-row tile, up to COLS vectors): as many members as COLS / nrhs holds, or COLS right-hand sides
// of one member.  The four operand planes of an item lie one after the other in shared memory, so
// one MMA of N = 4 COLS per K step of 16 makes all four products against one read of A (separate
// accumulators, added in the epilogue).  COLS = 16 keeps a stage at 24 KB and two CTAs per SM;
// COLS = 64 (48 KB stages, one CTA per SM, all of TMEM) reads a block fewer times where many
// vectors share it.  launch_precond_tc16 says where the line lies.
//
// Stage K's warp roles (192 threads, persistent, four stages): warp 0 TMA producer (A tile 128
// rows x 128 bytes, operand box 4 planes x COLS rows x 128 bytes), warp 1 TMEM allocation and the
// MMA issuer, warps 2..5 the epilogue.  Every wait is bounded; on a time-out the CTA sets the error
// word, waits (bounded) for its own copies and MMAs, frees TMEM and returns.
//
// Needs ClusterTables::tc16 (every cluster 2x2x2, 24 q^2 a multiple of 32).
#include <cooperative_groups.h>
#include <cuda.h>
#include <cuda_fp16.h>
#include <cudaTypedefs.h>

#include <algorithm>

#include "common.cuh"
#include "hps_internal.h"
#include "tc_common.cuh"

namespace hps {

namespace {

using namespace tc;

// ---------------------------------------------------------------------------
// Stage B
// ---------------------------------------------------------------------------
template <class TIN>
struct PrecB16Args {
  const __half2* B;       // FP16 blocks, transposed (column c holds the rows), rows divided by bscale
  const float* bscale;
  const long long* b_off;
  const int* brd;         // per leaf, internal faces then external: input offsets
  const int* bto;         // per leaf, internal faces: t offsets
  const int* bsc;         // per leaf, internal faces: row-scale bases
  const int* members;     // clusters in stage-K position order
  const int* leaves;      // 8 leaves of each cluster
  const int2* items;      // (first position, members), members of one K block
  const TIN* r;
  float2* z;
  float2* t32;            // [vector][n]: t itself; nullptr: op and tmax
  __half2* op;            // operand rows [4][ncl * nrhs][n]: conj hi, swap hi, conj lo, swap lo
  float* tmax;            // [ncl * nrhs]
  int q2, n, ncl, nrhs, rtiles;
  long long nf;
  const int* gate;
};

constexpr int kBCluster = 4;  // CTAs per leaf cluster: two of its 8 leaves each

// NR vectors per CTA, each entry of B loaded once for all of them; two rows per thread, so that
// each staged input value feeds two sums.  B comes from L2 (3 q^2 entries per row): the next
// entries of each row are in flight while the ones before them are used, the rows' offsets, scales and own inputs
// loaded before the sums.
template <class TIN, int NR>
__global__ void __cluster_dims__(kBCluster, 1, 1) __maxnreg__(80) prec_b16_kernel(const PrecB16Args<TIN> A) {
  namespace cg = cooperative_groups;
  if (A.gate && *A.gate == 0) return;  // the same for every CTA of the cluster
  extern __shared__ __align__(16) unsigned char b16_smem[];
  const int q2 = A.q2, n3 = 3 * q2, n = A.n;  // a leaf: n3 internal rows, n3 external columns
  const int nc = 2 * n3;                      // columns of the CTA's two leaves
  float2* xs = reinterpret_cast<float2*>(b16_smem);  // [NR][nc]
  __shared__ float red[20][NR], cmax[NR];
  __shared__ long long roff[NR];
  __shared__ int vpos[NR];
  const int item = blockIdx.x / kBCluster, l0 = (blockIdx.x % kBCluster) * 2;
  const int2 it = A.items[item / A.rtiles];
  const int first = (item % A.rtiles) * NR;
  const int nr = min(NR, it.y * A.nrhs - first), v0 = it.x * A.nrhs + first;
  const int tid = threadIdx.x, nt = blockDim.x;
  if (tid < NR) {
    const int v = v0 + min(tid, nr - 1), p = v / A.nrhs;
    vpos[tid] = p;
    roff[tid] = (long long)(v - p * A.nrhs) * A.nf;
  }
  __syncthreads();
  // the leaves of vector rr's cluster (vectors of an item share the B blocks, not the leaves)
  const int* leaves[NR];
  long long ro[NR];
#pragma unroll
  for (int rr = 0; rr < NR; ++rr) {
    leaves[rr] = A.leaves + 8 * A.members[vpos[rr]] + l0;
    ro[rr] = roff[rr];
  }
  for (int t = tid; t < nc; t += nt) {
    const int li = t >= n3, c = t - li * n3, k = c / q2;
#pragma unroll
    for (int rr = 0; rr < NR; ++rr) {
      if (rr < nr) {
        const long long o = ro[rr] + A.brd[leaves[rr][li] * 6 + 3 + k] + (c - k * q2);
        const float2 v = cvt<float2>(A.r[o]);
        xs[rr * nc + t] = v;
        A.z[o] = v;
      } else {
        xs[rr * nc + t] = make_float2(0.f, 0.f);
      }
    }
  }
  __syncthreads();
  constexpr int kRows = 2;
  constexpr int kU = NR == 4 ? 4 : 12;  // entries per row in flight (80 registers: 6 CTAs per SM at q = 6)
  const int hr = n3 / 2;  // rows of a thread: hr apart
  const bool on = tid < n3;
  float2 tv[kRows][NR];
  int to[kRows][NR];
  float mx[NR];
#pragma unroll
  for (int rr = 0; rr < NR; ++rr) mx[rr] = 0.f;
  if (on) {
    const int ldr = (int)rup4(n3);
    const int li = tid >= hr, row0 = tid - li * hr;
    const int leaf0 = leaves[0][li];
    const __half2* Bm = A.B + A.b_off[leaf0] + row0;
    const float2* x = xs + li * n3;
    __half2 b0[kRows][kU], b1[kRows][kU];
#pragma unroll
    for (int u = 0; u < kU; ++u)
#pragma unroll
      for (int i = 0; i < kRows; ++i) b0[i][u] = Bm[u * ldr + i * hr];
    float sc[kRows];
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      const int row = row0 + i * hr, k = row / q2, j = row - k * q2;
      sc[i] = A.bscale[A.bsc[leaf0 * 6 + k] + j];
#pragma unroll
      for (int rr = 0; rr < NR; ++rr) {
        const int e = leaves[rr][li] * 6 + k;
        to[i][rr] = A.bto[e] - vpos[rr] * n + j;
        tv[i][rr] = rr < nr ? cvt<float2>(A.r[ro[rr] + A.brd[e] + j]) : make_float2(0.f, 0.f);
      }
    }
    float2 acc[kRows][NR];
#pragma unroll
    for (int i = 0; i < kRows; ++i)
#pragma unroll
      for (int rr = 0; rr < NR; ++rr) acc[i][rr] = make_float2(0.f, 0.f);
    for (int c = 0; c < n3; c += kU) {  // n3 is a multiple of 12: q is even
      if (c + kU < n3) {
#pragma unroll
        for (int u = 0; u < kU; ++u)
#pragma unroll
          for (int i = 0; i < kRows; ++i) b1[i][u] = Bm[(c + kU + u) * ldr + i * hr];
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        float2 bv[kRows];
#pragma unroll
        for (int i = 0; i < kRows; ++i) {
          bv[i] = __half22float2(b0[i][u]);
          b0[i][u] = b1[i][u];
        }
#pragma unroll
        for (int rr = 0; rr < NR; ++rr) {
          const float2 xv = x[rr * nc + c + u];
#pragma unroll
          for (int i = 0; i < kRows; ++i) cfma(acc[i][rr], bv[i], xv);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < kRows; ++i)
#pragma unroll
      for (int rr = 0; rr < NR; ++rr) {
        tv[i][rr] = csub(tv[i][rr], make_float2(acc[i][rr].x * sc[i], acc[i][rr].y * sc[i]));
        if (A.t32 && rr < nr) A.t32[(long long)(v0 + rr) * n + to[i][rr]] = tv[i][rr];
        if (rr < nr) mx[rr] = fmaxf(mx[rr], fmaxf(fabsf(tv[i][rr].x), fabsf(tv[i][rr].y)));
      }
  }
  if (A.t32) return;  // the same for every CTA of the cluster
#pragma unroll
  for (int rr = 0; rr < NR; ++rr) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx[rr] = fmaxf(mx[rr], __shfl_xor_sync(0xffffffffu, mx[rr], o));
    if ((tid & 31) == 0) red[tid >> 5][rr] = mx[rr];
  }
  __syncthreads();
  if (tid < NR) {
    float m = 0.f;
    for (int w = 0; w < nt / 32; ++w) m = fmaxf(m, red[w][tid]);
    cmax[tid] = m;
  }
  cg::cluster_group cl = cg::this_cluster();
  cl.sync();
  const long long plane = (long long)A.ncl * A.nrhs * n;
#pragma unroll
  for (int rr = 0; rr < NR; ++rr) {
    if (rr >= nr) break;
    float m = 0.f;
#pragma unroll
    for (int w = 0; w < kBCluster; ++w) m = fmaxf(m, *cl.map_shared_rank(&cmax[rr], w));
    const long long v = v0 + rr;
    if (tid == 0 && l0 == 0) A.tmax[v] = m;
    // A maximum below the smallest normal float (a cluster far from every source, whose t holds
    // only subnormal values) would overflow the reciprocal: such a cluster's t is taken as 0, a
    // change below 2^-126 of the vector's scale.
    const float sc = m >= 0x1p-126f ? 1.f / m : 0.f;
    __half2* op = A.op + v * n;
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      if (!on) break;
      const float2 x = make_float2(tv[i][rr].x * sc, tv[i][rr].y * sc);
      const __half2 h = __floats2half2_rn(x.x, x.y);
      const __half2 l = __floats2half2_rn(x.x - __low2float(h), x.y - __high2float(h));
      __half2* d = op + to[i][rr];
      d[0] = __halves2half2(__low2half(h), __hneg(__high2half(h)));
      d[plane] = __halves2half2(__high2half(h), __low2half(h));
      d[2 * plane] = __halves2half2(__low2half(l), __hneg(__high2half(l)));
      d[3 * plane] = __halves2half2(__high2half(l), __low2half(l));
    }
  }
  cl.sync();  // no CTA leaves while another may read its maximum
}

// The operand rows [4][vector][nint0] lie at the start of the scratch, the maxima behind them.
float* operand_tmax(const ClusterTables& ct, const void* t, int nrhs) {
  return (float*)((__half2*)t + (size_t)4 * ct.ncl * nrhs * ct.nint0);
}

template <class TIN>
cudaError_t stage_b16(const hps_handle* h, const TIN* r, float2* z, float2* t, bool operand, int nrhs,
                      cudaStream_t st) {
  const ClusterTables& ct = h->ct;
  PrecB16Args<TIN> a;
  a.B = h->B16;
  a.bscale = h->B16s;
  a.b_off = h->dct.b_off;
  a.brd = h->dct.brd;
  a.bto = h->dct.bto;
  a.bsc = h->dct.bsc;
  a.members = h->dct.kc_members;
  a.leaves = h->dct.cl_leaves;
  a.r = r;
  a.z = z;
  a.t32 = operand ? nullptr : t;
  a.op = (__half2*)t;
  a.tmax = operand_tmax(ct, t, nrhs);
  a.q2 = h->q * h->q;
  a.n = ct.nint0;
  a.ncl = ct.ncl;
  a.nrhs = nrhs;
  a.nf = h->nf;
  a.gate = h->gate;
  // Vectors per item: the most (up to 4) that leave 4 CTAs per SM, and no more than any block has.
  // Measured at p = 8: 12^3 leaves of a bump medium, one right-hand side, 20.8 us with 1 vector
  // against 24.9 us with 4 (too few CTAs); 8^3 leaves, 12 right-hand sides, 45 us with 4.
  const int n3 = 3 * a.q2;
  auto ctas_of = [&](int k) {
    return (long long)ct.b16_count[tc16_members_per_item(k, nrhs)] * ((nrhs + k - 1) / k) * kBCluster;
  };
  int nr = 4;
  while (nr > 1 && (ctas_of(nr) < 4LL * h->nsm || (long long)ct.max_members * nrhs <= nr / 2)) nr >>= 1;
  const int P = tc16_members_per_item(nr, nrhs);
  a.items = h->dct.b16_items + ct.b16_begin[P];
  a.rtiles = (nrhs + nr - 1) / nr;
  const int threads = (int)round_up(n3, 32);
  const size_t smem = (size_t)nr * 2 * n3 * sizeof(float2);
  auto run = [&](auto kern) -> cudaError_t {
    const cudaError_t e = allow_dynamic_smem((const void*)kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)((long long)ct.b16_count[P] * a.rtiles * kBCluster), threads, smem, st>>>(a);
    ++h->prof.launches;
    return cudaGetLastError();
  };
  if (nr == 1) return run(prec_b16_kernel<TIN, 1>);
  if (nr == 2) return run(prec_b16_kernel<TIN, 2>);
  return run(prec_b16_kernel<TIN, 4>);
}

// ---------------------------------------------------------------------------
// Stage K
// ---------------------------------------------------------------------------
constexpr int kStages = 4;
constexpr int kTileM = 128;
constexpr int kKHalves = 64;            // K extent of a stage (128 bytes of FP16)
constexpr int kABytes = kTileM * 128;   // 16 KB
// Stages whose products the tensor cores add up before the sums move to FP32 registers.  The
// accumulation truncates, a loss of about one unit in the last place per step in one direction, so
// long sums drift.  Measured against the exact product of the same FP16 blocks, 2^3 leaves at p = 10
// (48 stages): 3.5e-6 with one sum, 4.0e-7 with 12 of 4 stages; 12^3 leaves at p = 8, both stages of
// one right-hand side: 39.7 us and 39.3 us.
constexpr int kChunk = 4;
constexpr int kThreads = 192;

template <int COLS> struct Shape {
  static constexpr int kBBytes = 4 * COLS * 128;           // operand planes conj hi, swap hi, conj lo, swap lo
  static constexpr int kStageBytes = kABytes + kBBytes;    // parts 1024-byte aligned
  static constexpr int kN = 4 * COLS;                      // accumulator columns
  static constexpr int kTmemCols = 2 * kN;                 // two accumulators
};

struct Pk16Args {
  int nint, kblocks, q2;
  long long nitems;
  const int4* items;       // (block, row tile, first position, members)
  int rtiles;              // COLS-RHS tiles of one member (nrhs > COLS), else 1
  int nrhs;
  const int* kc_slot_begin;
  const int* zoff;         // [position][24] output offset of each slot of the member's faces
  const float* kscale;     // FP16 row scales, index kc_slot_begin[k] q^2 + row
  const float* tmax;       // [vector]
  long long nf;
  float2* z;
  int* error;
  const int* gate;         // while a GMRES cycle is replayed: 0 = return at once
};

struct __align__(8) Bars {
  uint64_t full[kStages];
  uint64_t empty[kStages];
  uint64_t acc_full[2];
  uint64_t acc_empty[2];
  uint64_t drain;
  uint32_t tmem_base;
  int abort;
};

// block, row tile, first vector and vector count of an item
template <int COLS>
__device__ __forceinline__ void decode(const Pk16Args& a, long long item, int& blk, int& mt, int& v0, int& cnt) {
  const int4 e = a.items[item / a.rtiles];
  const int first = (int)(item % a.rtiles) * COLS;
  blk = e.x;
  mt = e.y;
  v0 = e.z * a.nrhs + first;
  cnt = min(COLS, e.w * a.nrhs - first);
}

template <int COLS>
__global__ void __launch_bounds__(kThreads, COLS == 16 ? 2 : 1)
    tc_precond16_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                        Pk16Args a) {
  using S = Shape<COLS>;
  constexpr int kStageBytes = S::kStageBytes, kTmemCols = S::kTmemCols;
  if (a.gate && *a.gate == 0) return;  // before any barrier or TMEM allocation
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* ring = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  Bars* bars = reinterpret_cast<Bars*>(ring + kStages * kStageBytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&bars->full[s], 1);
      mbar_init(&bars->empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&bars->acc_full[b], 1);
      mbar_init(&bars->acc_empty[b], 4);
    }
    mbar_init(&bars->drain, 1);
    bars->abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bars->tmem_base)),
                 "r"(kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = bars->tmem_base;

  auto fail = [&]() {
    atomicExch(a.error, 1);
    atomicExch(&bars->abort, 1);
  };

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      long long it = 0;
      bool ok = true;
      for (long long item = blockIdx.x; item < a.nitems && ok; item += gridDim.x) {
        int blk, mt, v0, cnt;
        decode<COLS>(a, item, blk, mt, v0, cnt);
        for (int kb = 0; kb < a.kblocks; ++kb, ++it) {
          const int s = (int)(it % kStages);
          const uint32_t ph = (uint32_t)((it / kStages) & 1);
          if (bars->abort || (it >= kStages && !mbar_wait(&bars->empty[s], ph ^ 1))) {
            fail();
            ok = false;
            break;
          }
          unsigned char* st = ring + s * kStageBytes;
          mbar_expect_tx(&bars->full[s], kStageBytes);
          tma_load_3d(st, &mapA, &bars->full[s], kb * kKHalves, mt * kTileM, blk);
          tma_load_3d(st + kABytes, &mapB, &bars->full[s], kb * kKHalves, v0, 0);
        }
      }
      for (long long j = (it > kStages ? it - kStages : 0); j < it; ++j)
        if (!mbar_wait(&bars->full[(int)(j % kStages)], (uint32_t)((j / kStages) & 1))) fail();
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    if (lane == 0) {
      const uint32_t idesc = instr_desc_f16(S::kN, kTileM);
      long long it = 0;
      long long local = 0;
      bool ok = true;
      for (long long item = blockIdx.x; item < a.nitems && ok; item += gridDim.x) {
        for (int kb = 0; kb < a.kblocks; ++kb, ++it) {
          const int b = (int)(local & 1);
          const uint32_t acc = tmem + (uint32_t)(b * S::kN);
          if (kb % kChunk == 0) {
            if (local >= 2 && !mbar_wait(&bars->acc_empty[b], (uint32_t)(((local >> 1) - 1) & 1))) {
              fail();
              ok = false;
              break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          }
          const int s = (int)(it % kStages);
          const uint32_t ph = (uint32_t)((it / kStages) & 1);
          if (bars->abort || !mbar_wait(&bars->full[s], ph)) {
            fail();
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t aa = smem_u32(ring + s * kStageBytes), bb = aa + kABytes;
#pragma unroll
          for (int kk = 0; kk < kKHalves / 16; ++kk) {
            const uint32_t off = kk * 32;  // 16 halves
            mma_f16(acc, smem_desc(aa + off), smem_desc(bb + off), idesc, (kb % kChunk == 0 && kk == 0) ? 0u : 1u);
          }
          mma_commit(&bars->empty[s]);
          if (kb % kChunk == kChunk - 1 || kb == a.kblocks - 1) {
            mma_commit(&bars->acc_full[b]);
            ++local;
          }
        }
      }
      mma_commit(&bars->drain);
      if (!mbar_wait(&bars->drain, 0)) fail();
    }
    __syncwarp();
  } else {
    // ---------------- epilogue: warps 2..5, each on the 32 TMEM lanes that it may read ----------------
    const int ew = warp & 3;
    const int chunks = (a.kblocks + kChunk - 1) / kChunk;
    long long local = 0;
    bool ok = true;
    for (long long item = blockIdx.x; item < a.nitems && ok; item += gridDim.x) {
      int blk, mt, v0, cnt;
      decode<COLS>(a, item, blk, mt, v0, cnt);
      const int row = mt * kTileM + ew * 32 + lane;
      const float ks = (row < a.nint) ? a.kscale[(long long)a.kc_slot_begin[blk] * a.q2 + row] : 0.f;
      const int sl = row / a.q2, j = row - sl * a.q2;
      const int* zo = a.zoff + sl;
      // offsets and scales of 16 vectors
      auto place = [&](int h0, int (&off)[16], float (&f)[16]) {
        int pos = (v0 + h0) / a.nrhs, rhs = v0 + h0 - pos * a.nrhs;
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          const bool on = h0 + c < cnt && row < a.nint;
          off[c] = on ? zo[pos * 24] : 0;
          f[c] = on ? a.tmax[v0 + h0 + c] : 0.f;
          if (++rhs == a.nrhs) {
            rhs = 0;
            ++pos;
          }
        }
      };
      int off[16];
      float f[16];
      if (COLS == 16) place(0, off, f);  // in flight during the sums
      float re[COLS], im[COLS];
#pragma unroll
      for (int c = 0; c < COLS; ++c) re[c] = im[c] = 0.f;
      for (int ch = 0; ch < chunks; ++ch, ++local) {
        const int b = (int)(local & 1);
        if (bars->abort || !mbar_wait(&bars->acc_full[b], (uint32_t)((local >> 1) & 1))) {
          fail();
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t taddr = tmem + ((uint32_t)(ew * 32) << 16) + (uint32_t)(b * S::kN);
#pragma unroll
        for (int h0 = 0; h0 < COLS; h0 += 16) {
          if (h0 >= cnt) break;
          uint32_t reh[16], imh[16], rel[16], iml[16];
          tmem_ld16(taddr + h0, reh);
          tmem_ld16(taddr + COLS + h0, imh);
          tmem_ld16(taddr + 2 * COLS + h0, rel);
          tmem_ld16(taddr + 3 * COLS + h0, iml);
          tmem_wait_ld();
#pragma unroll
          for (int c = 0; c < 16; ++c) {
            re[h0 + c] += __uint_as_float(reh[c]) + __uint_as_float(rel[c]);
            im[h0 + c] += __uint_as_float(imh[c]) + __uint_as_float(iml[c]);
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->acc_empty[b]);
      }
      if (!ok) break;
#pragma unroll
      for (int h0 = 0; h0 < COLS; h0 += 16) {
        if (h0 >= cnt) break;
        if (COLS > 16) place(h0, off, f);
        int rhs = (v0 + h0) % a.nrhs;
        if (row < a.nint) {
#pragma unroll
          for (int c = 0; c < 16; ++c) {
            if (h0 + c < cnt) {
              const float w = ks * f[c];
              a.z[(long long)rhs * a.nf + off[c] + j] = make_float2(re[h0 + c] * w, im[h0 + c] * w);
            }
            if (++rhs == a.nrhs) rhs = 0;
          }
        }
      }
    }
  }

  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
  }
}

}  // namespace

int tc16_members_per_item(int cols, int nrhs) { return nrhs >= cols ? 1 : cols / nrhs; }

bool precond_b16_eligible(const hps_handle* h) {
  return h->has_precond && h->opt.tc_apply && h->Kc16 && h->Kc16s && h->tc_error && h->ct.tc16;
}

bool precond_tc16_eligible(const hps_handle* h, int nrhs, size_t scratch_bytes) {
  return precond_b16_eligible(h) && (nrhs == 1 || nrhs % 64 == 0) && tc16_operand_bytes(h->ct, nrhs) <= scratch_bytes;
}

size_t tc16_operand_bytes(const ClusterTables& ct, int nrhs) {
  return (size_t)ct.ncl * nrhs * ((size_t)4 * ct.nint0 * sizeof(__half2) + sizeof(float));
}

size_t precond_scratch_bytes(const ClusterTables& ct, int nrhs) {
  const size_t t = (size_t)std::max<long long>(1, ct.tsize) * nrhs * sizeof(double2);
  return ct.tc16 ? std::max(t, tc16_operand_bytes(ct, nrhs)) : t;
}

cudaError_t launch_precond_b16(const hps_handle* h, VType tin, const void* r, float2* z, float2* t, bool operand,
                               int nrhs, cudaStream_t st) {
  if (!precond_b16_eligible(h)) return cudaErrorInvalidValue;
  if (tin == VType::C64) return stage_b16(h, (const float2*)r, z, t, operand, nrhs, st);
  if (tin == VType::DF) return stage_b16(h, (const float4*)r, z, t, operand, nrhs, st);
  return stage_b16(h, (const double2*)r, z, t, operand, nrhs, st);
}

cudaError_t launch_precond_tc16(const hps_handle* h, const void* t, float2* z, int nrhs, cudaStream_t st) {
  const ClusterTables& ct = h->ct;
  if (!precond_b16_eligible(h) || (nrhs != 1 && nrhs % 64 != 0)) return cudaErrorInvalidValue;
  auto encode = encoder();
  if (!encode) return cudaErrorNotSupported;
  const int nint = ct.nint0;
  // TMA: 16-byte aligned bases and strides (checked, not assumed)
  if ((reinterpret_cast<uintptr_t>(h->Kc16) | reinterpret_cast<uintptr_t>(t)) % 16 != 0 || (4LL * nint) % 16 != 0)
    return cudaErrorInvalidValue;
  // Items of 16 vectors unless that takes more than twice as many items as 64 would (blocks shared
  // by many vectors).  Measured per application of stage K at p = 8: 12^3 leaves of a bump medium,
  // one right-hand side (few blocks, up to ~190 members) 18.9 us at 16 against 51 us at 64 columns.
  auto count_of = [&](int cols) {
    return (long long)ct.tc16_count[tc16_members_per_item(cols, nrhs)] * ((nrhs + cols - 1) / cols);
  };
  const int cols = count_of(16) <= 2 * count_of(64) ? 16 : 64;
  const int P = tc16_members_per_item(cols, nrhs);
  CUtensorMap mapA, mapB;
  // three-dimensional FP16 arrays [d2][d1][2 nint halves] in boxes of 64 halves x b1 rows x b2
  auto map3 = [&](CUtensorMap* m, void* base, cuuint64_t d1, cuuint64_t d2, cuuint32_t b1, cuuint32_t b2) {
    cuuint64_t dims[3] = {(cuuint64_t)(2 * nint), d1, d2};
    cuuint64_t strides[2] = {(cuuint64_t)nint * 4, (cuuint64_t)nint * 4 * d1};
    cuuint32_t box[3] = {kKHalves, b1, b2};
    cuuint32_t es[3] = {1, 1, 1};
    return encode(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
  };
  if (!map3(&mapA, (void*)h->Kc16, (cuuint64_t)nint, (cuuint64_t)ct.nkc, kTileM, 1) ||
      !map3(&mapB, const_cast<void*>(t), (cuuint64_t)ct.ncl * nrhs, 4, (cuuint32_t)cols, 4))
    return cudaErrorInvalidValue;
  Pk16Args a;
  a.nint = nint;
  a.kblocks = 2 * nint / kKHalves;
  a.q2 = h->q * h->q;
  a.items = h->dct.tc16_items + ct.tc16_begin[P];
  a.rtiles = (nrhs + cols - 1) / cols;
  a.nrhs = nrhs;
  a.kc_slot_begin = h->dct.kc_slot_begin;
  a.zoff = h->dct.zoff;
  a.kscale = h->Kc16s;
  a.tmax = operand_tmax(ct, t, nrhs);
  a.nf = h->nf;
  a.z = z;
  a.error = h->tc_error;
  a.gate = h->gate;
  a.nitems = count_of(cols);
  auto run = [&](auto kern, int stage_bytes, int per_sm) -> cudaError_t {
    const int smem = kStages * stage_bytes + (int)sizeof(Bars) + 1024;
    const cudaError_t e = allow_dynamic_smem((const void*)kern, smem);
    if (e != cudaSuccess) return e;
    const int grid = (int)std::min<long long>(a.nitems, (long long)per_sm * h->nsm);
    kern<<<grid, kThreads, smem, st>>>(mapA, mapB, a);
    ++h->prof.launches;
    return cudaGetLastError();
  };
  return cols == 16 ? run(tc_precond16_kernel<16>, Shape<16>::kStageBytes, 2)
                    : run(tc_precond16_kernel<64>, Shape<64>::kStageBytes, 1);
}

}  // namespace hps
