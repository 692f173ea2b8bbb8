// y = (I + Pi R) f with the rows of the leaf maps streamed through shared memory by bulk copies
// (Sec. 2.2, Sec. 3.1), in complex float for any number of right-hand sides that the tensor-core
// apply does not take (tc_apply.cu: multiples of 64).
//
// One CTA per SM, persistent over an equal share of all matrix rows that are read (rows of faces
// with a neighbour, leaf after leaf): a producer thread keeps a ring of row chunks (4 warps x RPW
// rows) and the leaves' input vectors in flight with cp.async.bulk; groups of four warps take the
// chunks in turn, RPW rows a warp, 16 bytes per lane and load, and reduce them with halving
// exchanges (warp_sums).  A
// chunk in shared memory serves all right-hand sides, NR at a time, so the maps are read from HBM
// once whatever their number, and the staged input values are shared by RPW rows.  Each lane then
// holds one (row, right-hand side): y = f + g goes straight to the neighbour's slot (the swap Pi
// fused into the store, one writer per slot); f at that slot was loaded before the sums.
//
// What bounds it: HBM for one right-hand side, shared-memory reads of the staged values and the
// FP32 pipe for several.  The kernel that this replaces here (seg_gemv_kernel) read the maps once
// per 8 right-hand sides and lost time to the gaps between a CTA's items (stage, sync, sum, sync,
// store).  Measured: 7x6x5 leaves, p = 9, 16 right-hand sides 152 -> 86 us (132 with seg_gemv_kernel's
// new reductions); 8^3, p = 8, 8 right-hand sides 125 -> 88 us, one 48 -> 43 us; 12^3, p = 8, one
// 122 -> 114 us (5.2 TB/s).  In complex double the FP64 pipe is the bound and seg_gemv_kernel, with
// more warps resident, is the faster one (9^3, p = 8: 268 against 277 us).
//
// Every wait is bounded: on a time-out the CTA sets the error word, its producer stops, waits
// (bounded) for the copies in flight and returns, and its consumers go through their remaining chunks
// without waiting, on whatever the ring holds (hps_status and the solves report it).
#include <algorithm>

#include "common.cuh"
#include "hps_internal.h"
#include "tc_common.cuh"

namespace hps {

namespace {

using namespace tc;

constexpr int kGroup = 4;  // warps that share a chunk
constexpr int kMaxStages = 8;
// Groups of warps: registers allow fewer with more accumulators per thread.  The number of stages
// is a multiple of it, so that a stage's chunks all belong to one group, which waits for each of
// its phases.
template <int NR> constexpr int kGroups = NR <= 2 ? 4 : NR == 4 ? 3 : 2;
constexpr size_t kSmem = 220 * 1024;

template <class T>
struct StreamArgs {
  const T* R;
  int ld, nb, q2;
  unsigned inv;        // row_inv(q2)
  GridDims g;
  int nl;
  const T* f;
  void* y;
  long long nf, rows;   // values per right-hand side; matrix rows that are read
  int nrhs, stages;
  long long spin;    // tries per bounded wait
  int skip_arrival;  // test hook: CTA 0's first warp does not give back the first chunk
  int* error;
  const int* gate;
};

struct __align__(8) StreamBars {
  uint64_t full[kMaxStages], empty[kMaxStages];
  uint64_t xfull[2], xempty[2];
  int abort;
};

__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// Faces with a neighbour of the leaves before leaf l (closed form: six per leaf less the faces on
// the six sides of the grid).
__device__ __forceinline__ long long faces_before(const GridDims& g, long long l) {
  const long long nxy = (long long)g.nx * g.ny, iz = l / nxy, rem = l - iz * nxy, iy = rem / g.nx, ix = rem - iy * g.nx;
  const long long lines = iz * g.ny + iy;
  return 6 * l - (lines + (ix > 0)) - lines - (iz * g.nx + min(rem, (long long)g.nx)) -
         (iz * g.nx + max(0LL, rem - (long long)(g.ny - 1) * g.nx)) - min(l, nxy) -
         max(0LL, l - (long long)(g.nz - 1) * nxy);
}

// Walk over the CTA's rows [row, end) in chunks that stay inside one leaf.
struct Walk {
  long long row, end;  // rows still to do
  int leaf, lrow, lrows;
  int ix, iy, iz;
  unsigned mask, flist;
  __device__ void enter(const GridDims& g, int q2) {  // faces of the current leaf
    mask = (ix > 0 ? 1u : 0u) | (ix + 1 < g.nx ? 2u : 0u) | (iy > 0 ? 4u : 0u) | (iy + 1 < g.ny ? 8u : 0u) |
           (iz > 0 ? 16u : 0u) | (iz + 1 < g.nz ? 32u : 0u);
    flist = 0;
    int n = 0;
#pragma unroll
    for (int f = 0; f < 6; ++f)
      if ((mask >> f) & 1u) flist |= (unsigned)f << (4 * n++);
    lrows = n * q2;
  }
  template <class A>
  __device__ void start(const A& a) {
    // equal shares in whole groups of 4 rows
    const long long quads = (a.rows + 3) / 4;
    row = min(a.rows, 4 * (quads * blockIdx.x / gridDim.x));
    end = min(a.rows, 4 * (quads * (blockIdx.x + 1) / gridDim.x));
    const long long face = row / a.q2;
    long long lo = 0, hi = a.nl - 1;  // the last leaf with faces_before <= face
    while (lo < hi) {
      const long long mid = (lo + hi + 1) / 2;
      if (faces_before(a.g, mid) <= face) lo = mid;
      else hi = mid - 1;
    }
    leaf = (int)lo;
    ix = leaf % a.g.nx;
    iy = leaf / a.g.nx % a.g.ny;
    iz = leaf / (a.g.nx * a.g.ny);
    enter(a.g, a.q2);
    lrow = (int)(row - faces_before(a.g, lo) * a.q2);
  }
  __device__ bool more() const { return row < end; }
  __device__ int count(int chunk) const { return (int)min((long long)min(chunk, lrows - lrow), end - row); }
  // past a chunk of n rows; true when the next one is in another leaf
  __device__ bool advance(const GridDims& g, int q2, int n) {
    row += n;
    lrow += n;
    if (lrow < lrows || row >= end) return false;
    ++leaf;  // every leaf of a grid with rows has a neighbour
    if (++ix == g.nx) {
      ix = 0;
      if (++iy == g.ny) {
        iy = 0;
        ++iz;
      }
    }
    lrow = 0;
    enter(g, q2);
    return true;
  }
};

template <class T> struct Lane;
template <> struct Lane<float2> {
  static constexpr int VPL = 2;
  __device__ static __forceinline__ void load(const float2* p, float2 (&v)[2]) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = make_float2(t.x, t.y);
    v[1] = make_float2(t.z, t.w);
  }
};
__device__ __forceinline__ float2 add_out(float2 f, float2 g, float2*) { return cadd(f, g); }
__device__ __forceinline__ float4 add_out(float2 f, float2 g, float4*) {
  const dfr re = df_two_sum(f.x, g.x), im = df_two_sum(f.y, g.y);
  return make_float4(re.h, im.h, re.l, im.l);
}

template <class T, class TOUT, int NR, int RPW>
__global__ void __launch_bounds__(32 * (kGroups<NR> * kGroup + 1), 1) stream_apply_kernel(const StreamArgs<T> a) {
  if (a.gate && *a.gate == 0) return;
  using R_ = typename Real<T>::type;
  constexpr int VPL = Lane<T>::VPL, kChunk = kGroup * RPW, kG = kGroups<NR>, kWarps = kG * kGroup;
  extern __shared__ __align__(128) unsigned char sa_smem[];
  const int nb = a.nb, ld = a.ld, q2 = a.q2, nrhs = a.nrhs;
  T* ring = reinterpret_cast<T*>(sa_smem);
  T* xs = ring + (size_t)a.stages * kChunk * ld;  // [2][nrhs][nb]
  StreamBars* bars = reinterpret_cast<StreamBars*>(xs + (size_t)2 * nrhs * nb);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < a.stages; ++s) {
      mbar_init(&bars->full[s], 1);
      mbar_init(&bars->empty[s], kGroup);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&bars->xfull[b], 1);
      mbar_init(&bars->xempty[b], kWarps);
    }
    bars->abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  volatile int* abort = &bars->abort;
  auto fail = [&]() {
    atomicExch(a.error, 1);
    *abort = 1;
  };
  Walk w;
  w.start(a);
  if (warp == kWarps) {
    // ---------------- producer ----------------
    if (lane != 0 || !w.more()) return;
    long long it = 0;
    int nx = 0;
    bool fresh = true;
    for (bool ok = true; w.more() && ok; ++it) {
      if (fresh) {  // the leaf's vectors
        const int b = nx & 1;
        if (nx >= 2 && !mbar_wait(&bars->xempty[b], (uint32_t)(((nx >> 1) - 1) & 1), a.spin)) {
          fail();
          break;
        }
        mbar_expect_tx(&bars->xfull[b], (uint32_t)(nrhs * nb * sizeof(T)));
        for (int r = 0; r < nrhs; ++r)
          bulk_load(xs + ((size_t)b * nrhs + r) * nb, a.f + r * a.nf + (long long)w.leaf * nb, nb * sizeof(T),
                    &bars->xfull[b]);
        ++nx;
      }
      const int s = (int)(it % a.stages), n = w.count(kChunk);
      if (*abort || (it >= a.stages && !mbar_wait(&bars->empty[s], (uint32_t)((it / a.stages - 1) & 1), a.spin))) {
        fail();
        break;
      }
      mbar_expect_tx(&bars->full[s], (uint32_t)(n * ld * sizeof(T)));
      T* dst = ring + (size_t)s * kChunk * ld;
      const T* M = a.R + (long long)w.leaf * nb * ld;
      for (int d = 0; d < n;) {  // runs of rows that are consecutive in memory
        const unsigned r = w.lrow + d, k = (r * a.inv) >> 20;
        const int j = (int)(r - k * q2), face = (w.flist >> (4 * k)) & 7;
        const int run = w.mask == 63u ? n : min(n - d, q2 - j);
        bulk_load(dst + (size_t)d * ld, M + (long long)(face * q2 + j) * ld, (uint32_t)(run * ld * sizeof(T)),
                  &bars->full[s]);
        d += run;
      }
      fresh = w.advance(a.g, q2, n);
    }
    // copies in flight land before the CTA leaves (bounded)
    for (long long j = it > a.stages ? it - a.stages : 0; j < it; ++j)
      if (!mbar_wait(&bars->full[(int)(j % a.stages)], (uint32_t)((j / a.stages) & 1), a.spin)) fail();
    for (int j = nx > 2 ? nx - 2 : 0; j < nx; ++j)
      if (!mbar_wait(&bars->xfull[j & 1], (uint32_t)((j >> 1) & 1), a.spin)) fail();
    return;
  }
  // ---------------- consumers ----------------
  // After a time-out no branch depends on it: the lanes of a warp may leave a wait differently, and
  // they meet again in warp_sums.
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    if (mbar_wait(bar, parity, 1)) return;
    for (long long i = 1; i < a.spin; ++i)
      if (*abort || mbar_wait(bar, parity, 1)) return;
    fail();
  };
  constexpr int V = 2 * RPW * NR;
  constexpr int kHeld = V >= 32 ? V / 32 : 1, kSame = V >= 32 ? 1 : 32 / V;
  constexpr int kMine = kHeld >= 2 ? kHeld / 2 : 1;  // complex results per lane
  TOUT* y = reinterpret_cast<TOUT*>(a.y);
  int nx = 0;
  bool fresh = true;
  for (long long it = 0; w.more(); ++it) {
    const int s = (int)(it % a.stages), n = w.count(kChunk), leaf = w.leaf;
    if (fresh) {
      wait(&bars->xfull[nx & 1], (uint32_t)((nx >> 1) & 1));
      ++nx;
      // the leaf's first rows are this CTA's: its faces on the boundary of the cube only copy
      if (w.lrow == 0 && w.mask != 63u)
        for (int idx = threadIdx.x; idx < 6 * q2; idx += 32 * kWarps)
          if (!((w.mask >> (idx / q2)) & 1u))
            for (int r = 0; r < nrhs; ++r) {
              const long long o = r * a.nf + (long long)leaf * nb + idx;
              y[o] = add_out(a.f[o], czero<T>(), (TOUT*)nullptr);
            }
    }
    if (it % kG != warp / kGroup) {  // another group's chunk
      fresh = w.advance(a.g, q2, n);
      if (fresh && lane == 0) mbar_arrive(&bars->xempty[(nx - 1) & 1]);
      continue;
    }
    const T* x = xs + (size_t)((nx - 1) & 1) * nrhs * nb;
    wait(&bars->full[s], (uint32_t)((it / a.stages) & 1));
    const int l0 = warp % kGroup * RPW;
    if (l0 < n) {
      const T* row[RPW];
#pragma unroll
      for (int i = 0; i < RPW; ++i) row[i] = ring + ((size_t)s * kChunk + min(l0 + i, n - 1)) * ld;
      for (int r0 = 0; r0 < nrhs; r0 += NR) {
        // this lane's results: sums number first + k are (row, right-hand side, re/im)
        int first = 0, held = V;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
          if (held > 1) {
            held >>= 1;
            if (lane & o) first += held;
          }
        long long out[kMine];
        T fv[kMine];
#pragma unroll
        for (int m = 0; m < kMine; ++m) {
          const int c = first / 2 + m, i = c / NR, rr = r0 + c % NR;
          const unsigned lr = w.lrow + l0 + i, k = (lr * a.inv) >> 20;
          const int j = (int)(lr - k * q2), face = (w.flist >> (4 * k)) & 7;
          const int step = face >> 1 == 0 ? 1 : face >> 1 == 1 ? a.g.nx : a.g.nx * a.g.ny;
          const int nbr = leaf + (face & 1 ? step : -step);
          const bool on = l0 + i < n && rr < nrhs && (kHeld > 1 || (lane % kSame == 0 && !(first & 1)));
          out[m] = on ? rr * a.nf + (long long)nbr * nb + (long long)(face ^ 1) * q2 + j : -1;
          fv[m] = on ? a.f[out[m]] : czero<T>();
        }
        R_ acc[V];
#pragma unroll
        for (int i = 0; i < V; ++i) acc[i] = 0;
        const T* xr[NR];
#pragma unroll
        for (int rr = 0; rr < NR; ++rr) xr[rr] = x + (size_t)min(r0 + rr, nrhs - 1) * nb;
#pragma unroll 2
        for (int c = lane * VPL; c < nb; c += 32 * VPL) {
          T mv[RPW][VPL];
#pragma unroll
          for (int i = 0; i < RPW; ++i) Lane<T>::load(row[i] + c, mv[i]);
#pragma unroll
          for (int rr = 0; rr < NR; ++rr) {
            T xv[VPL];
            Lane<T>::load(xr[rr] + c, xv);
#pragma unroll
            for (int v = 0; v < VPL; ++v) {
#pragma unroll
              for (int i = 0; i < RPW; ++i) {
                T t;
                t.x = acc[2 * (i * NR + rr)];
                t.y = acc[2 * (i * NR + rr) + 1];
                cfma(t, mv[i][v], xv[v]);
                acc[2 * (i * NR + rr)] = t.x;
                acc[2 * (i * NR + rr) + 1] = t.y;
              }
            }
          }
        }
        int dummy;
        warp_sums<R_, V>(acc, lane, dummy);
#pragma unroll
        for (int m = 0; m < kMine; ++m) {
          T g;
          if constexpr (kHeld > 1) {
            g.x = acc[2 * m];
            g.y = acc[2 * m + 1];
          } else {  // re and im ended in lanes kSame apart
            g.x = acc[0];
            g.y = __shfl_xor_sync(0xffffffffu, acc[0], kSame);
          }
          if (out[m] >= 0) y[out[m]] = add_out(fv[m], g, (TOUT*)nullptr);
        }
      }
    }
    __syncwarp();
    if (lane == 0 && !(a.skip_arrival && blockIdx.x == 0 && warp == 0 && it == 0)) mbar_arrive(&bars->empty[s]);
    fresh = w.advance(a.g, q2, n);
    if (fresh && lane == 0) mbar_arrive(&bars->xempty[(nx - 1) & 1]);
  }
}

template <class T, class TOUT, int NR, int RPW>
cudaError_t launch(const hps_handle* h, const StreamArgs<T>& a, size_t smem, cudaStream_t st) {
  auto kern = stream_apply_kernel<T, TOUT, NR, RPW>;
  const cudaError_t e = allow_dynamic_smem((const void*)kern, smem);
  if (e != cudaSuccess) return e;
  const int grid = (int)std::min<long long>(h->nsm, (a.rows + kGroup * RPW - 1) / (kGroup * RPW));
  kern<<<grid, 32 * (kGroups<NR> * kGroup + 1), smem, st>>>(a);
  ++h->prof.launches;
  return cudaGetLastError();
}

template <class T, class TOUT, int NR>
cudaError_t launch_rpw(const hps_handle* h, const StreamArgs<T>& a, int rpw, size_t smem, cudaStream_t st) {
  if (rpw == 4) return launch<T, TOUT, NR, 4>(h, a, smem, st);
  if (rpw == 2) return launch<T, TOUT, NR, 2>(h, a, smem, st);
  return launch<T, TOUT, NR, 1>(h, a, smem, st);
}

// Rows per warp and ring stages for nrhs right-hand sides; false when the ring does not fit.  As
// many rows per warp as leave one stage per group of warps (two stages with half the rows were no
// faster: 94 against 86 us in the 16-RHS case above).
bool plan(const hps_handle* h, int nrhs, int& rpw, int& stages, size_t& smem) {
  const size_t fixed = (size_t)2 * nrhs * h->nb * sizeof(float2) + sizeof(StreamBars) + 128;
  if (fixed >= kSmem) return false;
  const int groups = nrhs <= 2 ? kGroups<1> : nrhs <= 4 ? kGroups<4> : kGroups<8>;
  for (rpw = 4; rpw >= 1; rpw /= 2) {
    const size_t stage = (size_t)kGroup * rpw * h->ldR * sizeof(float2);
    stages = (int)std::min<size_t>(kMaxStages, (kSmem - fixed) / stage) / groups * groups;
    smem = fixed + stages * stage;
    if (stages >= groups) return true;
  }
  return false;
}

template <class T, class TOUT>
cudaError_t run(const hps_handle* h, const T* R, const T* f, TOUT* y, int nrhs, cudaStream_t st) {
  StreamArgs<T> a;
  a.R = R;
  a.ld = h->ldR;
  a.nb = h->nb;
  a.q2 = h->q * h->q;
  a.inv = row_inv(a.q2);
  a.g = GridDims{h->nx, h->ny, h->nz};
  a.nl = h->nl;
  a.nf = h->nf;
  const long long nx = h->nx, ny = h->ny, nz = h->nz;
  a.rows = (6 * nx * ny * nz - 2 * (nx * ny + nx * nz + ny * nz)) * a.q2;
  a.spin = h->test_spin > 0 ? h->test_spin : kSpinLimit;
  a.skip_arrival = h->test_skip_arrival;
  a.error = h->tc_error;
  a.gate = h->gate;
  // as many right-hand sides per launch as fit beside the ring
  int per = nrhs, rpw = 1;
  size_t smem = 0;
  while (per > 1 && !plan(h, per, rpw, a.stages, smem)) per = (per + 1) / 2;
  for (int r0 = 0; r0 < nrhs; r0 += per) {
    a.nrhs = std::min(per, nrhs - r0);
    if (!plan(h, a.nrhs, rpw, a.stages, smem)) return cudaErrorInvalidValue;
    a.f = f + (long long)r0 * h->nf;
    a.y = y + (long long)r0 * h->nf;
    cudaError_t e;
    if (a.nrhs == 1) e = launch_rpw<T, TOUT, 1>(h, a, rpw, smem, st);
    else if (a.nrhs == 2) e = launch_rpw<T, TOUT, 2>(h, a, rpw, smem, st);
    else if (a.nrhs <= 4) e = launch_rpw<T, TOUT, 4>(h, a, rpw, smem, st);
    else e = launch_rpw<T, TOUT, 8>(h, a, rpw, smem, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// The batched GEMV (apply.cu) is the faster one for up to 8 right-hand sides where the maps come from
// L2 and its items fill the chip: maps of at most half of L2 inside a solve (double-float results),
// which applies them at every step, and of a third in single calls, whose maps may have left it; faces
// of at most 256 KB, so that few CTAs do not work long at one item; and leaves for an item per SM,
// unless their rows are short.  Measured, us, GEMV and streamed, maps in L2: 4^3 leaves, p = 8, one
// right-hand side 9.2 and 12.9; 6^3, p = 7, one 12.4 and 18.9; 8^3, p = 6, one 17.1 and 23.1, eight
// 39.8 and 37.4; 6^3, p = 8 (67 MB), one 15.0 and 22.9, after an L2 flush 35.5 and 27.3.  On the other
// side: 7^3, p = 8 (110 MB), two 49 and 34; 2^3, p = 12 (faces of 480 KB), one 10.7 and 8.8; 4^3,
// p = 8, 16 right-hand sides 35 and 25.
bool stream_apply_better(const hps_handle* h, VType tout, int nrhs) {
  if (nrhs > 8) return true;
  const double row = h->ldR * sizeof(float2);
  const double bytes = (6.0 * h->nl - 2.0 * (h->nx * h->ny + h->nx * h->nz + h->ny * h->nz)) * h->q * h->q * row;
  const bool in_l2 = bytes <= (tout == VType::DF ? 64.0 : 40.0) * (1 << 20);
  const bool short_items = h->q * h->q * row <= 256.0 * 1024 && (6LL * h->nl >= h->nsm || h->nb <= 96);
  return !(in_l2 && short_items);
}

}  // namespace

bool stream_apply_eligible(const hps_handle* h, const void* f, VType tout, int nrhs) {
  int rpw, stages;
  size_t smem;
  return h->tc_error && h->nl > 1 && reinterpret_cast<uintptr_t>(f) % 16 == 0 && plan(h, 1, rpw, stages, smem) &&
         stream_apply_better(h, tout, nrhs);
}

cudaError_t launch_stream_apply(const hps_handle* h, const float2* f, VType tout, void* y, int nrhs, cudaStream_t st) {
  if (tout == VType::C64) return run<float2, float2>(h, h->R32, f, (float2*)y, nrhs, st);
  if (tout == VType::DF) return run<float2, float4>(h, h->R32, f, (float4*)y, nrhs, st);
  return cudaErrorInvalidValue;
}

}  // namespace hps
