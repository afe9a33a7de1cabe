// Persistent FP32 V_loc plane kernel for N x N planes whose occupied columns are the full disk
// |n1|, |n2| <= XM (cubic and other cells whose sphere projection is a full disk), a whole line in
// one thread's registers.
//
// The work per (pair, z plane) unit: the inverse n2 transform of the occupied x columns, the inverse
// n1 transform of every row, the product with V_loc(r), the forward n1 transform and the forward n2
// transform of the occupied columns back to the column buffer.
//  * Persistent blocks with a static round-robin over the units; each unit's slice of the column
//    buffer (ldcb contiguous complex values) moves into and out of shared memory with bulk
//    asynchronous copies (cp.async.bulk, completion on an mbarrier for loads and bulk groups for
//    stores), three slices in flight, so the column gathers and scatters are shared-memory accesses
//    and the global latency hides behind the transforms of the previous unit.
//  * The column phases of consecutive units overlap: the first CW warps run the forward n2 transforms
//    of unit k while the next CW run the inverse n2 transforms of unit k + 1, two tiles in shared
//    memory; per unit the block spends one column-transform time instead of two.
//  * The tile keeps only the 2 XM + 1 occupied columns (odd pitch: conflict-free column and row
//    access), and the disk bound is a compile-time constant, so the zero inputs of the inverse
//    transforms and the unused outputs of the forward transforms drop out of the arithmetic.
//  * Packed arithmetic and prime-factor transforms (line_dft.cuh) without a twiddle table, V_loc in
//    the order that the lanes' rows read together (plane_lines.cuh), and one copy of each transform.
// What bounds it: 8 warps per SM (the registers of a line) with the FP32 pipe half busy (53% at 64 x 64,
// 49% at 96 x 96), the rest dependent-issue waits and, where 3 of 4 warps have rows, barriers.
//
// 128 pairs on one GB300, ms, against the best kernel before (64: this kernel with scalar four-step
// transforms and a copy of them per use; 96: two threads per line; others: line-resident):
//   N        48    50    54    60    64    72    75    80    96
//   before  .048  .056  .077  .087  .100  .173  .267  .287  .402
//   here    .039  .055  .060  .065  .075  .167  .223  .215  .326
// Every wait is bounded: a block whose copy does not complete sets the error flag, waits (again
// bounded) for the copies it has in flight and leaves.
#include <cstdlib>

#include "fft.cuh"
#include "kernels.cuh"
#include "plane_lines.cuh"
#include "tc.cuh"

namespace wdf {
namespace {

using namespace tc;

constexpr long kCopyWaitLimit = 1L << 24;

__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void bulk_store(void *dst, const void *src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)), "r"(bytes) : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// all but the newest bulk store have finished reading shared memory
__device__ __forceinline__ void bulk_wait_read_but_one() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

template <int N, int XM> __device__ __forceinline__ constexpr bool on_disk(int i) { return i <= XM || i >= N - XM; }
// compact column of natural index x on the disk
template <int N, int XM> __device__ __forceinline__ constexpr int compact(int x) { return x <= XM ? x : x - (N - (2 * XM + 1)); }

typedef ld::CA<float> O;  // packed complex arithmetic
typedef O::C C;

// warps of the row phase (one row per thread) and of one direction of the column phases
template <int N, int XM> struct PipeShape {
  static constexpr int CW = (2 * XM + 1 + 31) / 32, RW = (N + 31) / 32, W = RW > 2 * CW ? RW : 2 * CW, threads = 32 * W;
  static constexpr int blocks = 8 / W > 0 ? 8 / W : 1;  // 8 warps of up to 255 registers per SM
};

template <int N, int XM>
__global__ void __launch_bounds__(PipeShape<N, XM>::threads, PipeShape<N, XM>::blocks) k_plane_pipe(Geo g, const int *__restrict__ jidx,
                                                      PlaneArgs<float> pa, long nunits, int *err) {
  constexpr int NX = 2 * XM + 1;
  constexpr int CT = 32 * PipeShape<N, XM>::CW;  // threads of one column direction
  extern __shared__ __align__(128) unsigned char smraw[];
  const int ldcb = g.ldcb;
  float2 *slices = reinterpret_cast<float2 *>(smraw);  // 3 x ldcb
  C *tiles = reinterpret_cast<C *>(slices + 3 * ldcb);   // 2 x N x NX
  uint64_t *bar = reinterpret_cast<uint64_t *>(tiles + 2 * N * NX);  // 3 (8-byte aligned as the tiles are)
  const int t = threadIdx.x, half = t < CT ? 0 : t < 2 * CT ? 1 : 2, l = t - half * CT;
  const long G = gridDim.x, u0 = blockIdx.x;
  pdl_begin();
  pdl_wait();
  if (u0 >= nunits) return;
  const int cnt = (int)((nunits - 1 - u0) / G) + 1;
  const uint32_t bytes = (uint32_t)ldcb * (uint32_t)sizeof(float2);
  float2 *cb = pa.cb;
  int issued[3] = {0, 0, 0};  // loads issued into each slice (thread 0)
  if (t == 0) {
#pragma unroll
    for (int i = 0; i < 3; ++i) mbar_init(&bar[i], 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (t == 0) {
    bulk_load(slices, cb + u0 * ldcb, bytes, &bar[0]);
    issued[0] = 1;
    if (cnt > 1) {
      bulk_load(slices + ldcb, cb + (u0 + G) * ldcb, bytes, &bar[1]);
      issued[1] = 1;
    }
  }
  // Phases: 0 the inverse columns of unit 0; 2 k + 1 the rows of unit k; 2 k + 2 the forward columns of unit k
  // (first half of the threads) and the inverse columns of unit k + 1 (second half). One copy of the
  // inverse and one of the forward transform serve rows and columns: with a copy for each use (four) the
  // kernel waited for instruction fetch (1.4 to 2.2 "no instruction" stalls per issue).
  const int x = l <= XM ? l : l + (N - NX);  // natural n1 of this thread's column
  bool stop = false;
#pragma unroll 1
  for (int ph = 0; ph <= 2 * cnt && !stop; ++ph) {
    const bool rows = ph & 1;
    const int kf = rows ? ph >> 1 : (ph >> 1) - 1, ki = ph >> 1;  // unit of the rows or forward columns; of the inverse columns
    bool inv = rows ? t < N : half == 1 && l < NX && ki < cnt;
    const bool fwd = rows ? t < N : half == 0 && l < NX && kf >= 0;
    bool fail = false;
    const int mine = rows || half == 0 ? max(kf, 0) : ki;  // the unit whose tile and slice this thread uses
    C *tcur = tiles + (mine & 1) * N * NX;
    float2 *sl = slices + (mine % 3) * ldcb;
    if (inv && !rows && !mbar_wait(&bar[ki % 3], (uint32_t)((ki / 3) & 1), kCopyWaitLimit)) {
      inv = false;
      fail = true;
    }
    C v[N];
    if (inv) {
      if (rows) {
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] = on_disk<N, XM>(i) ? tcur[t * NX + compact<N, XM>(i)] : O::zero();
      } else {
#pragma unroll
        for (int y = 0; y < N; ++y) {
          v[y] = O::zero();
          if (on_disk<N, XM>(y)) {
            const int jj = __ldg(jidx + y * N + x);
            if (jj >= 0) v[y] = O::get(sl[jj]);
          }
        }
      }
      ld::Dft<float, N, 1, ld::Band<N, XM, 1, 0>>::run(v);
      if (rows) {
        const float *plane = pa.field + (size_t)((u0 + (long)kf * G) % g.n3) * N * N;
        constexpr int GR = lines_group(N);
#pragma unroll
        for (int c = 0; c < N / GR; ++c) {
          float f[GR];
          load_run<float, GR, N>(f, plane, t, c * GR);
#pragma unroll
          for (int e = 0; e < GR; ++e) v[c * GR + e] = O::scale(v[c * GR + e], f[e]);
        }
      } else {
#pragma unroll
        for (int y = 0; y < N; ++y) tcur[y * NX + l] = v[y];
      }
    }
    if (fwd) {
      if (!rows) {
#pragma unroll
        for (int y = 0; y < N; ++y) v[y] = tcur[y * NX + l];
      }
      ld::Dft<float, N, -1>::run(v);
      if (rows) {
#pragma unroll
        for (int i = 0; i < N; ++i)
          if (on_disk<N, XM>(i)) tcur[t * NX + compact<N, XM>(i)] = v[i];
      } else {
#pragma unroll
        for (int y = 0; y < N; ++y)
          if (on_disk<N, XM>(y)) {
            const int jj = __ldg(jidx + y * N + x);
            if (jj >= 0) sl[jj] = O::put(v[y]);
          }
        fence_proxy_async();
      }
    }
    stop = __syncthreads_or(fail);
    if (!stop && !rows && kf >= 0 && t == 0) {
      bulk_store(cb + (u0 + (long)kf * G) * ldcb, slices + (kf % 3) * ldcb, bytes);
      if (kf + 2 < cnt) {
        const int b = (kf + 2) % 3;
        bulk_wait_read_but_one();  // the store of unit kf - 1 from this slice has read it
        bulk_load(slices + b * ldcb, cb + (u0 + (long)(kf + 2) * G) * ldcb, bytes, &bar[b]);
        ++issued[b];
      }
    }
  }
  if (t == 0) {
    if (stop) {  // let every load this block issued land before the block's shared memory goes away
      bool ok = true;
#pragma unroll
      for (int b = 0; b < 3; ++b)
        if (issued[b] > 0) ok &= mbar_wait(&bar[b], (uint32_t)((issued[b] - 1) & 1), kCopyWaitLimit);
      (void)ok;
      atomicExch(err, 1);
    }
    bulk_wait_all();
  }
}

template <int N, int XM> size_t pipe_smem(const Geo &g) {
  return sizeof(float2) * (3 * (size_t)g.ldcb + 2 * (size_t)N * (2 * XM + 1)) + 3 * sizeof(uint64_t);
}

template <int N, int XM> void pipe_launch(const FftCtx<float> &f, int npair, const PlaneArgs<float> &pa, cudaStream_t st) {
  static int nsm = 0;
  if (nsm == 0) {
    int dev = 0;
    WDF_CUDA_TRY(cudaGetDevice(&dev));
    WDF_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  }
  constexpr int TH = PipeShape<N, XM>::threads;
  const size_t sm = pipe_smem<N, XM>(f.g);
  int per_sm = 0;
  WDF_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_plane_pipe<N, XM>, TH, sm));
  if (per_sm < 1) per_sm = 1;
  const long nunits = (long)npair * f.g.n3;
  const long grid = std::min<long>(nunits, (long)nsm * per_sm);
  PlaneArgs<float> a = pa;
  a.field = f.vgroup;
  launch_pdl("plane_vloc", 32, nunits, k_plane_pipe<N, XM>, dim3((unsigned)grid), dim3(TH), sm, st, f.g, f.jidx, a, nunits, f.err);
  WDF_CUDA_TRY(cudaGetLastError());
}

bool pipe_enabled() {
  static const bool on = std::getenv("WDF_NO_PIPE_PLANE") == nullptr;
  return on;
}

}  // namespace

// the (N, disk bound) pairs this kernel is compiled for
#define WDF_PIPE_SIZES(X) X(48, 11) X(50, 11) X(54, 12) X(60, 13) X(64, 14) X(64, 15) X(72, 16) X(75, 17) X(80, 18) X(96, 22)

bool plane_pipe_available(const Geo &g, const int *err) {
  if (!pipe_enabled() || err == nullptr || g.n1 != g.n2) return false;
  if (g.ymax > g.xmax || g.nxact != 2 * g.xmax + 1 || g.ldcb % 2 != 0) return false;
#define X(N, XM) \
  if (g.n1 == N && g.xmax == XM) return true;
  WDF_PIPE_SIZES(X)
#undef X
  return false;
}

void set_plane_pipe_limits(const Geo &g) {
#define X(N, XM) \
  if (g.n1 == N && g.n2 == N && pipe_smem<N, XM>(g) <= 227 * 1024) raise_smem_limit(k_plane_pipe<N, XM>, pipe_smem<N, XM>(g));
  WDF_PIPE_SIZES(X)
#undef X
}

bool launch_plane_pipe(const FftCtx<float> &f, int npair, const PlaneArgs<float> &pa, cudaStream_t st) {
  if (npair <= 0 || !plane_pipe_available(f.g, f.err)) return false;
#define X(N, XM)                          \
  if (f.g.n1 == N && f.g.xmax == XM) {    \
    pipe_launch<N, XM>(f, npair, pa, st); \
    return true;                          \
  }
  WDF_PIPE_SIZES(X)
#undef X
  return false;
}

}  // namespace wdf
