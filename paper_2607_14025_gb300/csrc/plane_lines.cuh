// Plane kernels with whole lines in the registers of a few lanes, for N x N planes whose occupied
// columns lie in |n1|, |n2| <= N / 4 (every alias-free grid: twice the orbitals' band fits).
//
// Work of a block: P consecutive (pair, z) units. Per unit the inverse n2 transforms of the nx
// occupied columns, the inverse n1 transforms of the N rows, the pointwise product, and the way
// back (OP_VLOC; OP_G2R stops on the grid, OP_PROD_R2G starts there).
//
// A line of N = L M points belongs to L lanes (LW = 32 / L lines a warp). Lane h holds the samples
// x[L m + h], does an M-point DFT in registers (line_dft.cuh: prime-factor maps, zero inputs
// pruned), and after an exchange through a small buffer of its own warp owns k = h KI + i
// (i < KI = M / L) of all L sub-transforms: one twiddle product and an L-point DFT give
// X[k + M j]. The forward transform runs the same steps backwards from that layout, so a row's two
// transforms and the product between them stay in registers. With L = 1 (FP32 up to N = 80) a lane
// has the whole line and there is neither exchange nor twiddle table.
//
// Shared memory holds only the occupied columns (pitch 2 (N / 4) + 1, odd), so several blocks share
// an SM and one block's barriers (two per plane group) hide behind the others' arithmetic. P and
// the W warps of a block are chosen so that the 32-lane tasks of the column phases and of the row
// phase both come out even (Lines<T, N>). The three phases share one copy of the inverse and one of the
// forward code, which keeps the double-float kernels (about 3,500 FP32 instructions a transform)
// inside the instruction cache.
#pragma once

#include <cstdlib>

#include "kernels.cuh"
#include "line_dft.cuh"

namespace wdf {

// lanes per line, planes and warps per block, blocks per SM the registers are bounded for, chunks
// of the exchange. Registers: 2 N (FP32) or 4 M (double-float) hold the line. Shared memory: one
// plane's tile is N (2 (N / 4) + 1) values. L is the fewest lanes that divide their own share of the
// line (L | N / L) with at most 80 points a lane in FP32 and 30 in double-float and FP64; C keeps the
// exchange at 10 values or fewer per lane and chunk (12 in FP32); B is what the registers and
// the tiles leave.
template <typename T, int N> struct Lines {
  static constexpr int L = 0, P = 1, W = 1, B = 1, C = 1;  // L = 0: no instance
};
#define WDF_LINES(T, N, L_, P_, W_, B_, C_) \
  template <> struct Lines<T, N> {          \
    static constexpr int L = L_, P = P_, W = W_, B = B_, C = C_; \
  };
WDF_LINES(float, 24, 1, 8, 3, 5, 1)
WDF_LINES(float, 30, 1, 6, 3, 5, 1)
WDF_LINES(float, 32, 1, 6, 3, 4, 1)
WDF_LINES(float, 36, 1, 5, 3, 4, 1)
WDF_LINES(float, 40, 1, 8, 5, 3, 1)
WDF_LINES(float, 45, 1, 4, 3, 4, 1)
WDF_LINES(float, 48, 1, 4, 3, 4, 1)
WDF_LINES(float, 50, 1, 5, 4, 3, 1)
WDF_LINES(float, 54, 1, 7, 6, 2, 1)
WDF_LINES(float, 60, 1, 1, 1, 12, 1)
WDF_LINES(float, 64, 1, 1, 1, 9, 1)
WDF_LINES(float, 72, 1, 3, 4, 2, 1)
WDF_LINES(float, 75, 1, 2, 4, 2, 1)
WDF_LINES(float, 80, 1, 2, 4, 2, 1)
WDF_LINES(float, 96, 2, 1, 3, 3, 4)
WDF_LINES(df64, 24, 1, 8, 3, 4, 1)
WDF_LINES(df64, 30, 1, 6, 3, 3, 1)
WDF_LINES(df64, 32, 2, 3, 3, 5, 2)
WDF_LINES(df64, 36, 2, 4, 5, 3, 3)
WDF_LINES(df64, 40, 2, 4, 5, 2, 2)
WDF_LINES(df64, 45, 3, 2, 5, 3, 5)
WDF_LINES(df64, 48, 2, 2, 3, 4, 4)
WDF_LINES(df64, 50, 5, 2, 9, 2, 2)
WDF_LINES(df64, 54, 3, 1, 3, 5, 3)
WDF_LINES(df64, 60, 2, 1, 2, 4, 3)
WDF_LINES(df64, 64, 4, 1, 4, 4, 2)
WDF_LINES(df64, 72, 3, 1, 4, 3, 4)
WDF_LINES(df64, 75, 5, 1, 7, 2, 3)
WDF_LINES(df64, 80, 4, 1, 5, 2, 5)
WDF_LINES(df64, 96, 4, 1, 6, 2, 3)
WDF_LINES(double, 24, 1, 8, 3, 4, 1)
WDF_LINES(double, 30, 1, 6, 3, 3, 1)
WDF_LINES(double, 32, 2, 3, 3, 5, 2)
WDF_LINES(double, 36, 2, 4, 5, 3, 3)
WDF_LINES(double, 40, 2, 4, 5, 2, 2)
WDF_LINES(double, 45, 3, 2, 5, 3, 5)
WDF_LINES(double, 48, 2, 2, 3, 4, 4)
WDF_LINES(double, 50, 5, 2, 9, 2, 2)
WDF_LINES(double, 54, 3, 1, 3, 4, 3)
WDF_LINES(double, 60, 2, 1, 2, 4, 3)
WDF_LINES(double, 64, 4, 1, 4, 4, 2)
WDF_LINES(double, 72, 3, 1, 4, 2, 4)
WDF_LINES(double, 75, 5, 1, 7, 2, 3)
WDF_LINES(double, 80, 4, 1, 5, 2, 5)
WDF_LINES(double, 96, 4, 1, 6, 2, 3)
#undef WDF_LINES

// Padding of the exchange buffer: line l, source s, slot a of a chunk sits at l PL + s QS + a. A
// warp stores for one register with (l, s) = (lane / L, lane % L) and loads with (l, a) =
// (lane / L, KC (lane % L) + const); PL and QS are the smallest for which neither meets a bank twice
// within the lanes that one pass serves (16 lanes of 8 bytes, 8 of 16), or with the fewest meetings.
template <int L, int KC, int EB> struct ExPad {
  static constexpr int G = 128 / EB, LW = 32 / L, MC = KC * L;
  static constexpr int meetings(int pl, int q) {
    int bad = 0;
    for (int g0 = 0; g0 < LW * L; g0 += G) {
      for (int a = g0; a < g0 + G && a < LW * L; ++a)
        for (int b = a + 1; b < g0 + G && b < LW * L; ++b) {
          if (((a / L) * pl + (a % L) * q - (b / L) * pl - (b % L) * q) % G == 0) ++bad;
          if (((a / L) * pl + (a % L) * KC - (b / L) * pl - (b % L) * KC) % G == 0) ++bad;
        }
    }
    return bad;
  }
  static constexpr int best() {  // pl * 64 + q
    int b = 0, bm = 1 << 30;
    for (int q = MC; q < MC + 4; ++q)
      for (int pl = (L - 1) * q + MC; pl < (L - 1) * q + MC + 8; ++pl) {
        const int m = meetings(pl, q) * 16 + (pl - L * MC);
        if (m < bm) {
          bm = m;
          b = pl * 64 + q;
        }
      }
    return b;
  }
  static constexpr int PL = best() / 64, QS = best() % 64, size = LW * PL;
};

template <typename T, int N> struct LineXf {
  typedef ld::CA<T> O;
  typedef typename O::C Cx;
  static constexpr int L = Lines<T, N>::L, M = N / L, KI = M / L, C = Lines<T, N>::C, KC = KI / C, LW = 32 / L, XB = N / 4;
  static_assert(L == 1 || (M % L == 0 && KI % C == 0), "lines split evenly over their lanes");
  typedef ExPad<L, KC, (int)sizeof(Cx)> Pad;

  // in: v[m] = x[L m + h]; out: v[j KI + i] = X[h KI + i + M j]. ex: the warp's buffer at this line
  // (every lane of the warp calls; `on` false: the lane stores nothing)
  static __device__ __forceinline__ void inverse(Cx (&v)[M], int h, bool on, Cx *ex, const Cx *tw) {
    ld::Dft<T, M, 1, ld::Band<N, XB, L, 0, L>>::run(v);
    if constexpr (L > 1) {
#pragma unroll
      for (int c = 0; c < C; ++c) {
        if (on)
#pragma unroll
          for (int a = 0; a < L; ++a)
#pragma unroll
            for (int i = 0; i < KC; ++i) ex[h * Pad::QS + a * KC + i] = v[a * KI + c * KC + i];
        __syncwarp();
#pragma unroll
        for (int s = 0; s < L; ++s)
#pragma unroll
          for (int i = 0; i < KC; ++i) v[s * KI + c * KC + i] = ex[s * Pad::QS + h * KC + i];
        __syncwarp();
      }
#pragma unroll
      for (int s = 1; s < L; ++s) {
        const Cx *w = tw + s * h * KI;
#pragma unroll
        for (int i = 0; i < KI; ++i) v[s * KI + i] = O::twiddle(v[s * KI + i], w[s * i], false);
      }
#pragma unroll
      for (int i = 0; i < KI; ++i) {
        Cx b[L];
#pragma unroll
        for (int s = 0; s < L; ++s) b[s] = v[s * KI + i];
        ld::Dft<T, L, 1>::run(b);
#pragma unroll
        for (int j = 0; j < L; ++j) v[j * KI + i] = b[j];
      }
    }
  }

  // the inverse's steps backwards: in v[j KI + i] = x[h KI + i + M j], out v[m] = Y[L m + h]
  static __device__ __forceinline__ void forward(Cx (&v)[M], int h, bool on, Cx *ex, const Cx *tw) {
    if constexpr (L > 1) {
#pragma unroll
      for (int i = 0; i < KI; ++i) {
        Cx b[L];
#pragma unroll
        for (int j = 0; j < L; ++j) b[j] = v[j * KI + i];
        ld::Dft<T, L, -1>::run(b);
#pragma unroll
        for (int s = 0; s < L; ++s) v[s * KI + i] = b[s];
      }
#pragma unroll
      for (int s = 1; s < L; ++s) {
        const Cx *w = tw + s * h * KI;
#pragma unroll
        for (int i = 0; i < KI; ++i) v[s * KI + i] = O::twiddle(v[s * KI + i], w[s * i], true);
      }
#pragma unroll
      for (int c = 0; c < C; ++c) {
        if (on)
#pragma unroll
          for (int s = 0; s < L; ++s)
#pragma unroll
            for (int i = 0; i < KC; ++i) ex[s * Pad::QS + h * KC + i] = v[s * KI + c * KC + i];
        __syncwarp();
#pragma unroll
        for (int a = 0; a < L; ++a)
#pragma unroll
          for (int i = 0; i < KC; ++i) v[a * KI + c * KC + i] = ex[h * Pad::QS + a * KC + i];
        __syncwarp();
      }
    }
    ld::Dft<T, M, -1>::run(v);
  }
};

// largest power of two (at most 4) that divides a
__host__ __device__ constexpr int align_of(int a) { return a % 4 == 0 ? 4 : a % 2 == 0 ? 2 : 1; }
// V_loc for the FP32 kernels: x in groups of G = lines_group(N), [z][x / G][y][G], so that the lanes
// of a warp (consecutive rows y) read consecutive 4 G-byte words. In natural order every lane's
// 16-byte read is in a cache line of its own, and those lookups took 42% of the L1 throughput at
// 48 x 48.
__host__ __device__ constexpr int lines_group(int n) { return align_of(n); }

// E consecutive reals of row l from x0 on: FP32 from the grouped layout, FP64-class from natural order
template <typename T, int E, int N> __device__ __forceinline__ void load_run(T (&f)[E], const T *__restrict__ plane, int l, int x0) {
  if constexpr (std::is_same<T, float>::value) {
    constexpr int G = lines_group(N);
    static_assert(E % G == 0, "whole groups");
    const float *p = plane + (size_t)x0 * N + l * G;
#pragma unroll
    for (int c = 0; c < E / G; ++c) {
      const float *q = p + c * G * N;
      if constexpr (G == 4) {
        const float4 w = __ldg(reinterpret_cast<const float4 *>(q));
        f[4 * c] = w.x;
        f[4 * c + 1] = w.y;
        f[4 * c + 2] = w.z;
        f[4 * c + 3] = w.w;
      } else if constexpr (G == 2) {
        const float2 w = __ldg(reinterpret_cast<const float2 *>(q));
        f[2 * c] = w.x;
        f[2 * c + 1] = w.y;
      } else {
        f[c] = __ldg(q);
      }
    }
  } else {
    const T *p = plane + (size_t)l * N + x0;
    if constexpr (std::is_same<T, df64>::value && E % 2 == 0 && N % 2 == 0) {  // 16 bytes at a time
#pragma unroll
      for (int c = 0; c < E / 2; ++c) {
        const float4 w = __ldg(reinterpret_cast<const float4 *>(p + 2 * c));
        f[2 * c] = df64(w.x, w.y);
        f[2 * c + 1] = df64(w.z, w.w);
      }
    } else {
#pragma unroll
      for (int c = 0; c < E; ++c) f[c] = p[c];
    }
  }
}

template <typename T, int N, int OP>
__global__ void __launch_bounds__(32 * Lines<T, N>::W, Lines<T, N>::B)
    k_plane_lines(Geo g, const cplx<T> *__restrict__ twg, const int *__restrict__ jidx, PlaneArgs<T> pa, int nunits, int ppb) {
  typedef LineXf<T, N> X;
  typedef ld::CA<T> O;
  typedef typename O::C Cx;
  typedef cplx<T> Gx;  // in global memory
  constexpr int L = X::L, M = X::M, KI = X::KI, LW = X::LW, XB = X::XB;
  constexpr int W = Lines<T, N>::W, PITCH = 2 * XB + 1, TH = 32 * W;
  constexpr bool STAGE = std::is_same<T, float>::value;  // column-buffer slices through shared memory
  extern __shared__ __align__(16) unsigned char smraw[];
  Cx *tw = reinterpret_cast<Cx *>(smraw);
  Cx *exb = tw + (L > 1 ? N : 0);
  Cx *tile = exb + (L > 1 ? W * X::Pad::size : 0);
  Gx *slice = reinterpret_cast<Gx *>((reinterpret_cast<uintptr_t>(tile + ppb * N * PITCH) + 15) & ~(uintptr_t)15);
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int nx = g.nxact, xmax = g.xmax, ldcb = g.ldcb;
  const int u0 = blockIdx.x * ppb, np = min(ppb, nunits - u0);
  Gx *cb = pa.cb + (size_t)u0 * ldcb;
  pdl_begin();
  if constexpr (L > 1)
    for (int i = t; i < N; i += TH) tw[i] = O::get(twg[i]);
  // the tile's columns between the occupied ones and the compile-time band read as zero
  if (OP != OP_PROD_R2G && nx < PITCH) {
    const int gap = PITCH - nx;
    for (int i = t; i < np * N * gap; i += TH) tile[(i / gap) * PITCH + xmax + 1 + i % gap] = O::zero();
  }
  pdl_wait();
  if constexpr (STAGE) {
    if (OP != OP_PROD_R2G) {
      const float4 *s = reinterpret_cast<const float4 *>(cb);
      float4 *d = reinterpret_cast<float4 *>(slice);
      for (int i = t; i < np * ldcb / 2; i += TH) d[i] = s[i];
    }
  }
  __syncthreads();
  const bool lane_on = L == 1 || lane < LW * L;
  const int sub = lane_on ? lane / L : 0, h = lane_on ? lane % L : 0;
  Cx *ex = exb + (L > 1 ? warp * X::Pad::size + sub * X::Pad::PL : 0);
  const T *field = pa.field;
  Cx v[M];
  // phases: 0 columns inverse, 1 rows, 2 columns forward
#pragma unroll 1
  for (int ph = (OP == OP_PROD_R2G ? 1 : 0); ph < (OP == OP_G2R ? 2 : 3); ++ph) {
    const int per = ph == 1 ? N : nx, count = np * per;
#pragma unroll 1
    for (int task = warp; task * LW < count; task += W) {
      const int line = task * LW + sub;
      const bool live = lane_on && line < count;
      const int p = live ? line / per : 0, l = live ? line - p * per : 0;
      Cx *tl = tile + p * N * PITCH;
      const Gx *sl = STAGE ? slice + p * ldcb : cb + (size_t)p * ldcb;
      const int x = l <= xmax ? l : l + (N - nx);         // natural n1 of column l
      const int cl = l <= xmax ? l : l + (PITCH - nx);    // its place in the tile
      Cx *trow = tl + l * PITCH;
      const int u = u0 + p, q = u / g.n3, z = u - q * g.n3;
      if (ph < 2) {
        if (OP != OP_PROD_R2G) {
          if (ph == 0) {
#pragma unroll
            for (int m = 0; m < M; ++m) {
              v[m] = O::zero();
              if (ld::Band<N, XB, L, 0, L>::at(m)) {
                const int jj = live ? __ldg(jidx + (L * m + h) * N + x) : -1;
                if (jj >= 0) v[m] = O::get(sl[jj]);
              }
            }
          } else {
#pragma unroll
            for (int m = 0; m < M; ++m) {
              v[m] = O::zero();
              if (ld::Band<N, XB, L, 0, L>::at(m)) {
                const int n = L * m + h;
                if (L == 1 || n <= XB || n >= N - XB) v[m] = trow[n <= XB ? n : n - (N - PITCH)];
              }
            }
          }
          X::inverse(v, h, lane_on, ex, tw);
        }
        if (ph == 0) {
          if (live)
#pragma unroll
            for (int j = 0; j < L; ++j)
#pragma unroll
              for (int i = 0; i < KI; ++i) tl[(h * KI + i + M * j) * PITCH + cl] = O::norm(v[j * KI + i]);
          continue;
        }
        const size_t row = (size_t)z * N * N + (size_t)l * N + h * KI;  // real-space point i of run j: row + M j + i
        if (OP == OP_G2R) {
          Gx *out = pa.grid + (size_t)q * g.n3 * N * N + row;
          if (live)
#pragma unroll
            for (int j = 0; j < L; ++j)
#pragma unroll
              for (int i = 0; i < KI; ++i) out[M * j + i] = O::put(O::norm(v[j * KI + i]));
          continue;
        }
        const T *f = field + (size_t)(z + (OP == OP_PROD_R2G ? q % pa.nocc * g.n3 : 0)) * N * N;
        const Gx *dv = OP == OP_PROD_R2G ? pa.grid + (size_t)(q / pa.nocc) * g.n3 * N * N + row : nullptr;
#pragma unroll
        for (int j = 0; j < L; ++j) {
          T fv[KI];
          load_run<T, KI, N>(fv, f, l, h * KI + M * j);
#pragma unroll
          for (int i = 0; i < KI; ++i)
            v[j * KI + i] = O::scale(OP == OP_PROD_R2G ? O::get(dv[M * j + i]) : v[j * KI + i], fv[i]);
        }
      } else {
#pragma unroll
        for (int j = 0; j < L; ++j)
#pragma unroll
          for (int i = 0; i < KI; ++i) v[j * KI + i] = tl[(h * KI + i + M * j) * PITCH + cl];
      }
      if (OP != OP_G2R) {
        X::forward(v, h, lane_on, ex, tw);
        if (live) {
          if (ph == 1) {
#pragma unroll
            for (int m = 0; m < M; ++m)
              if (ld::Band<N, XB, L, 0, L>::at(m)) {
                const int n = L * m + h;
                if (L == 1 || n <= XB || n >= N - XB) trow[n <= XB ? n : n - (N - PITCH)] = O::norm(v[m]);
              }
          } else {
            Gx *so = STAGE ? slice + p * ldcb : cb + (size_t)p * ldcb;
#pragma unroll
            for (int m = 0; m < M; ++m)
              if (ld::Band<N, XB, L, 0, L>::at(m)) {
                const int jj = __ldg(jidx + (L * m + h) * N + x);
                if (jj >= 0) so[jj] = O::put(O::norm(v[m]));
              }
          }
        }
      }
    }
    __syncthreads();
  }
  if constexpr (STAGE) {
    if (OP != OP_G2R) {
      float4 *s = reinterpret_cast<float4 *>(cb);
      const float4 *d = reinterpret_cast<const float4 *>(slice);
      for (int i = t; i < np * ldcb / 2; i += TH) s[i] = d[i];
    }
  }
}

template <typename T, int N> size_t lines_smem(const Geo &g, int ppb) {
  typedef LineXf<T, N> X;
  typedef Lines<T, N> D;
  size_t n = (size_t)ppb * N * (2 * (N / 4) + 1);
  if (D::L > 1) n += N + (size_t)D::W * X::Pad::size;
  if (std::is_same<T, float>::value) n += (size_t)ppb * g.ldcb;
  return n * sizeof(cplx<T>) + 16;  // 16: the slices of an odd tile start on the next 16 bytes
}

template <typename T, int N> void lines_limits_n(const Geo &g) {
  if (g.n1 != N || g.n2 != N) return;
  const size_t sm = lines_smem<T, N>(g, Lines<T, N>::P);
  if (sm > 227 * 1024) return;
  raise_smem_limit(k_plane_lines<T, N, OP_VLOC>, sm);
  if constexpr (!std::is_same<T, float>::value) {
    raise_smem_limit(k_plane_lines<T, N, OP_G2R>, sm);
    raise_smem_limit(k_plane_lines<T, N, OP_PROD_R2G>, sm);
  }
}

template <typename T, int N, int OP>
void lines_launch_op(const char *cls, const FftCtx<T> &f, int npair, const PlaneArgs<T> &pa, cudaStream_t st) {
  typedef Lines<T, N> D;
  const int nunits = npair * f.g.n3;
  PlaneArgs<T> a = pa;
  if (std::is_same<T, float>::value) a.field = f.vgroup;
  // few units: fewer planes per block, so that every SM has its blocks before a block has a second
  // plane (8 solves on 24 x 24: 96 units, 12 blocks of 8 planes against 96 of one)
  const int ppb = std::max(1, std::min(D::P, (nunits + 152 * D::B - 1) / (152 * D::B)));
  const dim3 grid((unsigned)((nunits + ppb - 1) / ppb));
  launch_pdl(cls, bits_of<T>(), nunits, k_plane_lines<T, N, OP>, grid, dim3(32 * D::W), lines_smem<T, N>(f.g, ppb), st, f.g, f.tw1, f.jidx,
               a, nunits, ppb);
  WDF_CUDA_TRY(cudaGetLastError());
}

template <typename T, int N> bool lines_launch_n(const FftCtx<T> &f, int op, int npair, const PlaneArgs<T> &pa, cudaStream_t st) {
  if (f.g.n1 != N) return false;
  if (op == OP_VLOC) lines_launch_op<T, N, OP_VLOC>("plane_vloc", f, npair, pa, st);
  if constexpr (!std::is_same<T, float>::value) {
    if (op == OP_G2R) lines_launch_op<T, N, OP_G2R>("plane_g2r", f, npair, pa, st);
    if (op == OP_PROD_R2G) lines_launch_op<T, N, OP_PROD_R2G>("plane_prod", f, npair, pa, st);
  }
  return true;
}

}  // namespace wdf

// the entry points of one translation unit: launch_NAME and set_NAME_limits over its sizes
#define WDF_LINES_UNIT(NAME, T, ...)                                                                               \
  namespace wdf {                                                                                                  \
  template <int... Ns> static bool NAME##_go(const FftCtx<T> &f, int op, int n, const PlaneArgs<T> &pa, cudaStream_t st) { \
    return (lines_launch_n<T, Ns>(f, op, n, pa, st) || ...);                                                       \
  }                                                                                                                \
  template <int... Ns> static void NAME##_lim(const Geo &g) { (lines_limits_n<T, Ns>(g), ...); }                   \
  bool launch_##NAME(const FftCtx<T> &f, int op, int n, const PlaneArgs<T> &pa, cudaStream_t st) {                 \
    return NAME##_go<__VA_ARGS__>(f, op, n, pa, st);                                                               \
  }                                                                                                                \
  void set_##NAME##_limits(const Geo &g) { NAME##_lim<__VA_ARGS__>(g); }                                           \
  }
