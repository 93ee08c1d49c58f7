// Batched Cholesky factorisations of the RPA tail on GB300 (sm_103a): V = L L^H,
// 1 - Pi' and V^-1 - chi0 with their log-determinants and traces, and the
// inverse of the V factors.
//
// What bounds it.  An SM's FP64 pipe takes 64 clocks per warp instruction on
// each of its four sub-partitions (two DFMA lanes per clock and SM), so one
// complex N = 768 factorisation is 151e6 clocks (73 ms) of one SM's pipe but
// 0.5 ms of all 152: a matrix that stays on one SM, or on a cluster of eight,
// is bound by that pipe and by its own serial phases, whatever else is idle.
// Every panel step is therefore spread over the whole GPU: a launch covers
// the panel rows or the trailing tiles of every matrix, and the kernel boundary is
// the only synchronisation.  The tile that holds the next diagonal block factors it at
// once, so a panel costs two launches.  Matrices up to 64 stay in one CTA's
// shared memory, one launch in all.
//
// Panel width.  Few matrices are bound by the chain of a panel: diagonal
// block, rows, update of the next diagonal block.  Its FP64 instructions per
// column grow with the panel width (every warp instruction is 64 clocks however
// few lanes it has), so panels of 16 columns, 16 lanes per row and 16 x 16
// tiles are about 22 us, two of them 44 where one of 32 columns took 95.  The FP64 modes
// always take 16 columns (with many matrices the FP64 pipe bounds either
// width); per matrix the arithmetic and its order do not depend on the batch,
// the lanes per row or the tile, so a matrix gives the same bits alone, in a
// batch or in a ragged launch.  The inverse form takes 32 columns when its
// trailing tiles fill the GPU, since each panel converts and adds the whole
// trailing matrix in FP64.
//
// Measured on GB300, panel launches (and one CTA or an 8-CTA cluster per matrix
// instead): one complex N = 768 factor of V 1.5 ms (19.9); 16 matrices of
// N = 768 in FP64 9.7 ms (30.1); 32 in the inverse form 8.8 ms (17.6); 320 of
// N = 512 in the inverse form 19.4 ms (34.7); 64 of N = 300 1.6 ms (18.6); 16
// real ones of N = 64 0.065 ms (0.285).  The 16 FP64 matrices need 7.6 ms of
// the FP64 pipe, so larger batches (chol_g64_use) leave all but 1/(N /
// 128) of the trailing updates to the tensor cores, one block column of 128
// columns at a time: 16 of N = 768 4.4 ms (9.9 without), 320 of N = 512 in the inverse
// form 14.4 (19.3).  What is left is the FP64 work inside the block columns and, for few
// matrices, two launches of some 20 us each per panel.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "fp64_elem.cuh"
#include "g64.h"
#include "rpa_internal.h"

namespace rpa {
namespace {

constexpr int CB = 32;                   // block edge of the triangular inverse
constexpr int SMALL_N = 64;              // largest matrix of the one-launch kernel
constexpr int INIT_BLOCKS = 32;          // CTAs per matrix that form V^-1 - chi (<= SMALL_N)

// Lower-triangular index -> (i, j), j <= i.
__device__ __forceinline__ void tri_ij(int t, int& i, int& j) {
  int k = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while ((k + 1) * (k + 2) / 2 <= t) ++k;
  while (k * (k + 1) / 2 > t) --k;
  i = k;
  j = t - k * (k + 1) / 2;
}

// The matrices of one launch: n_mat equal ones at a stride, or a task table.
struct CholBatch {
  const CholTask* tasks;  // null: the uniform form below
  double* mats;
  long bstride;
  double* out;
  int* status;
  const double *Wn, *Vc, *ldV;
  int N, mode, status_base, n_w;
};

template <bool C>
__device__ __forceinline__ CholTask task_of(const CholBatch& B, int b) {
  if (B.tasks) return B.tasks[b];
  CholTask t;
  const long q = B.mode == 2 ? b / B.n_w : 0;
  const long NN = (long)B.N * B.N * (C ? 2 : 1);
  t.A = B.mats + (long)b * B.bstride;
  t.out = B.out ? B.out + (B.mode == 1 ? b : 2 * b) : nullptr;
  t.W = B.Wn + q * NN;
  t.Vc = B.Vc + q * NN;
  t.ldv = B.ldV + q;
  t.status = B.status;
  t.N = B.N;
  t.mode = B.mode;
  t.code = 1 + B.status_base + b;
  return t;
}

// x -= a * conj(b)
template <bool C>
__device__ __forceinline__ void msub_conj(Elem<C>& x, Elem<C> a, Elem<C> b) {
  x.re = fma(-a.re, b.re, x.re);
  if constexpr (C) {
    x.re = fma(-a.im, b.im, x.re);
    x.im = fma(-a.im, b.re, x.im);
    x.im = fma(a.re, b.im, x.im);
  }
}
template <bool C>
__device__ __forceinline__ Elem<C> scale(Elem<C> a, double s) {
  a.re *= s;
  if constexpr (C) a.im *= s;
  return a;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// Sum over the CTA's 256 threads in a fixed order, valid in thread 0.
__device__ __forceinline__ double block_sum(double v, double* red) {
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < 8; ++w) s += red[w];
  __syncthreads();
  return s;
}

// 1 / x, correctly rounded: for a normal positive x the hardware approximation and
// two Newton-Raphson steps r += r (1 - x r), four FP64 instructions on the serial
// chain of a panel.  The last step rounds r (1 + e) with e exact up to its own rounding, which is
// the nearest value but for the significand 2 - 2^-52, whose reciprocal lies next to a
// midpoint (Markstein, 1990); it and the values outside the range go through the division.
__device__ __forceinline__ double fast_rcp(double x) {
  const int hi = __double2hiint(x);
  if (hi < (2 << 20) || hi >= (2044 << 20) || ((hi | 0xFFF00000) & __double2loint(x)) == -1) return 1.0 / x;
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  r = fma(r, fma(-x, r, 1.0), r);
  return fma(r, fma(-x, r, 1.0), r);
}

template <bool C, int NB>
struct DiagShared {
  Elem<C> col[2][NB];  // the current column (unscaled), double-buffered
  double rd[2];        // reciprocal of the current pivot
  double piv[NB];      // pivots (mode 0: pivot - 1)
  double l[NB], rs[NB];
  int bad;
};

// Factor of the diagonal block D (lower triangle, nb x nb, shared memory) by
// the CTA's 256 threads; L goes to Lout (leading dimension ld).  The first
// column needs no update; the others' elements stay in registers, in column
// order, so that whole warps retire as the columns do (NB = 16: one element
// per thread of four warps, one per sub-partition).  A column costs one
// barrier: the columns stay unscaled (x_rc -= x_rk conj(x_ck) / d_k), which leaves one
// reciprocal on the serial chain; all square roots, logarithms and scalings
// follow at the end, one per thread.  Returns (thread 0) the block's share of
// the log-determinant, NaN and S.bad on a non-positive pivot.
template <bool C, int NB>
__device__ double diag_factor(Elem<C> (*D)[CB + 1], DiagShared<C, NB>& S, int nb, int mode, double* Lout, long ld) {
  constexpr int UPD = NB * (NB - 1) / 2;  // elements of columns 1 ..
  constexpr int E = (UPD + 255) / 256;
  const int tid = threadIdx.x;
  Elem<C> x[E];
  int er[E], ec[E];
  if (tid == 0) S.bad = 0;
  auto publish = [&](int r, int c, const Elem<C>& v, int buf) {
    S.col[buf][r] = v;
    if (r == c) {
      const double u = v.re;
      S.piv[r] = u;
      S.rd[buf] = fast_rcp(mode == 0 ? 1.0 + u : u);
    }
  };
#pragma unroll
  for (int k = 0; k < E; ++k) {
    const int e = tid + 256 * k;
    er[k] = ec[k] = -1;
    x[k] = zero_elem<C>();
    if (e < UPD) {
      int i, j;
      tri_ij(UPD - 1 - e, i, j);
      const int r = NB - 1 - j, c = NB - 1 - i;
      if (r < nb) {
        er[k] = r;
        ec[k] = c;
        x[k] = D[r][c];
      }
    }
  }
  Elem<C> x0 = zero_elem<C>();  // column 0, one element per thread
  if (tid < nb) {
    x0 = D[tid][0];
    publish(tid, 0, x0, 0);
  }
  __syncthreads();
  for (int c = 0; c + 1 < nb; ++c) {
    const int buf = c & 1;
    const double rd = S.rd[buf];
#pragma unroll
    for (int k = 0; k < E; ++k)
      if (ec[k] > c) {
        msub_conj<C>(x[k], scale<C>(S.col[buf][er[k]], rd), S.col[buf][ec[k]]);
        if (ec[k] == c + 1) publish(er[k], c + 1, x[k], buf ^ 1);
      }
    __syncthreads();
  }
  double lg = 0.0;
  if (tid < nb) {
    const double u = S.piv[tid];
    const double p = mode == 0 ? 1.0 + u : u;
    const bool ok = p > 0.0;
    const double l = sqrt(p);
    S.l[tid] = l;
    S.rs[tid] = fast_rcp(l);
    lg = !ok ? nan("") : mode == 0 ? log1p(u) : log(p);
    if (!ok) S.bad = 1;
  }
  __syncthreads();
  auto put = [&](int r, int c, const Elem<C>& v) {
    Elem<C> w = scale<C>(v, S.rs[c]);
    if (r == c) {
      w = zero_elem<C>();
      w.re = S.l[r];
    }
    st_elem<C>(Lout, r * ld + c, w);
  };
  if (tid < nb) put(tid, 0, x0);
#pragma unroll
  for (int k = 0; k < E; ++k)
    if (ec[k] >= 0) put(er[k], ec[k], x[k]);
  return tid < 32 ? warp_sum(lg) : 0.0;
}

// Log-determinant bookkeeping of one diagonal block (thread 0): out[0] grows
// panel by panel, the last panel of mode 2 adds ln det V.
__device__ __forceinline__ void diag_report(const CholTask& t, double lg, int bad, bool first, bool last) {
  if (bad && t.status) atomicCAS(t.status, 0, t.code);
  if (!t.out) return;
  double v = first ? lg : t.out[0] + lg;
  if (last && t.mode == 2) v += *t.ldv;
  t.out[0] = v;
}

// Rows of a panel: X L_kk^H = A_panel, LPR lanes per row (lane g of a row
// owns columns c = LPR j + g).  16 lanes keep a row's serial chain short (a
// column is six FP64 instructions of its warp), 4 lanes use fewer instructions
// per row.  Ls[c][c'] holds L_kk[c'][c], rs the reciprocal diagonal.  `A` is
// this row's panel (invalid rows take part in the shuffles).
template <bool C, int NB, int LPR, class ST>
__device__ __forceinline__ void panel_row(const double* A, bool valid, const Elem<C> (*Ls)[CB + 1],
                                          const double* rs, const ST& store) {
  constexpr int J = NB / LPR;
  const int lane = threadIdx.x & 31, g = lane & (LPR - 1), q0 = lane & ~(LPR - 1);
  Elem<C> x[J];
#pragma unroll
  for (int j = 0; j < J; ++j) x[j] = valid ? ld_elem<C>(A, LPR * j + g) : zero_elem<C>();
#pragma unroll
  for (int c = 0; c < NB; ++c) {
    Elem<C> v = scale<C>(x[c / LPR], rs[c]);
    v.re = __shfl_sync(0xffffffffu, v.re, q0 | (c & (LPR - 1)));
    if constexpr (C) v.im = __shfl_sync(0xffffffffu, v.im, q0 | (c & (LPR - 1)));
    if (g == (c & (LPR - 1))) x[c / LPR] = v;
#pragma unroll
    for (int j = c / LPR; j < J; ++j)
      if (j > c / LPR || g > (c & (LPR - 1))) msub_conj<C>(x[j], v, Ls[c][LPR * j + g]);
  }
  if (valid)
#pragma unroll
    for (int j = 0; j < J; ++j) store(LPR * j + g, x[j]);
}

// --------------------------------------------------- per-panel kernels ----

// First launch of modes 1 and 2, nblk CTAs per matrix.  Mode 1: the strict
// upper triangle becomes zero.  Mode 2: M = V^-1 - chi over the lower
// triangle and the trace Tr(chi V), as one partial sum per CTA in the first
// row's strict upper triangle (columns 1 .. nblk, free until the first panel).
template <bool C>
__global__ void __launch_bounds__(256) chol_init_kernel(const __grid_constant__ CholBatch B, int nblk) {
  __shared__ double red[8];
  const int b = blockIdx.x / nblk, blk = blockIdx.x % nblk;
  const CholTask t = task_of<C>(B, b);
  const int N = t.N;
  if (t.mode == 1) {
    for (int r = blk; r < N; r += nblk)
      for (int c = r + 1 + threadIdx.x; c < N; c += 256) st_elem<C>(t.A, (long)r * N + c, zero_elem<C>());
    return;
  }
  double s = 0.0;
  for (int r = blk; r < N; r += nblk) {
    const long r0 = (long)r * N;
    for (int c = threadIdx.x; c <= r; c += 256) {
      const Elem<C> x = ld_elem<C>(t.A, r0 + c), v = ld_elem<C>(t.Vc, r0 + c), w = ld_elem<C>(t.W, r0 + c);
      double p = x.re * v.re;
      if constexpr (C) p = fma(x.im, v.im, p);
      s += r == c ? p : 2.0 * p;
      Elem<C> m;
      m.re = -w.re - x.re;
      if constexpr (C) m.im = -w.im - x.im;
      st_elem<C>(t.A, r0 + c, m);
    }
  }
  s = block_sum(s, red);
  if (threadIdx.x == 0) {
    Elem<C> e = zero_elem<C>();
    e.re = s;
    st_elem<C>(t.A, 1 + blk, e);
  }
}

// The diagonal block at kb of every matrix, and with the first (kb = 0) the
// traces (mode 0: Tr Pi = -sum Y_jj; mode 2: the partial sums of chol_init_kernel).
template <bool C, int NB>
__global__ void __launch_bounds__(256) chol_first_kernel(const __grid_constant__ CholBatch B, int nblk, int kb) {
  __shared__ Elem<C> D[NB][CB + 1];
  __shared__ DiagShared<C, NB> S;
  __shared__ double red[8];
  const CholTask t = task_of<C>(B, blockIdx.x);
  const int N = t.N, tid = threadIdx.x, nb = min(NB, N - kb);
  if (t.mode != 1 && kb == 0) {
    double s = 0.0;
    if (t.mode == 0) {
      for (int j = tid; j < N; j += 256) s -= ld_elem<C>(t.A, (long)j * N + j).re;
    } else if (tid < nblk) {
      s = ld_elem<C>(t.A, 1 + tid).re;
    }
    s = block_sum(s, red);
    if (tid == 0) t.out[1] = s;
  }
  for (int i = tid; i < NB * NB; i += 256) {
    const int r = i / NB, c = i % NB;
    if (r < nb && c <= r) D[r][c] = ld_elem<C>(t.A, (long)(kb + r) * N + kb + c);
  }
  __syncthreads();
  const double lg = diag_factor<C, NB>(D, S, nb, t.mode, t.A + ((long)kb * N + kb) * (C ? 2 : 1), N);
  if (tid == 0) diag_report(t, lg, S.bad, kb == 0, N - kb <= NB);
}

// Block columns (chol_outer below) of matrices out of the digit split's range:
// A[r][c] -= sum_{k < J0} L[r][k] conj(L[c][k]), J0 <= c < cend, in FP64.
template <bool C>
__global__ void __launch_bounds__(256) chol_outer_kernel(int N, double* __restrict__ mats, long bstride, int J0,
                                                         int cend, int per, const int* __restrict__ only) {
  constexpr int T = 32, KS = 16;
  __shared__ Elem<C> S1[T][KS + 1], S2[T][KS + 1];
  const int b = blockIdx.x / per, tile = blockIdx.x % per;
  if (!(only[b] & 1)) return;
  const int nc = (cend - J0 + T - 1) / T, TI = tile / nc, TJ = tile % nc;
  if (TI < TJ) return;
  double* A = mats + (long)b * bstride;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  Elem<C> o[2][2];
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int r = J0 + TI * T + ty + 16 * u, c = J0 + TJ * T + tx + 16 * v;
      o[u][v] = r < N && c < N ? ld_elem<C>(A, (long)r * N + c) : zero_elem<C>();
    }
  for (int k0 = 0; k0 < J0; k0 += KS) {
    for (int i = tid; i < T * KS; i += 256) {
      const int r = i / KS, k = k0 + i % KS;
      const int ri = J0 + TI * T + r, rj = J0 + TJ * T + r;
      S1[r][i % KS] = ri < N && k < J0 ? ld_elem<C>(A, (long)ri * N + k) : zero_elem<C>();
      S2[r][i % KS] = rj < N && k < J0 ? ld_elem<C>(A, (long)rj * N + k) : zero_elem<C>();
    }
    __syncthreads();
#pragma unroll 4
    for (int k = 0; k < KS; ++k)
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int v = 0; v < 2; ++v) msub_conj<C>(o[u][v], S1[ty + 16 * u][k], S2[tx + 16 * v][k]);
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int r = J0 + TI * T + ty + 16 * u, c = J0 + TJ * T + tx + 16 * v;
      if (r < N && c < cend && c <= r) st_elem<C>(A, (long)r * N + c, o[u][v]);
    }
}

// Panel rows below the diagonal block at kb (full panels only: kb + NB < N).
// Mode 2 also stores the float-float copy of L_{i,kb+c} at (row kb + c, column
// i) of the free strict upper triangle, where a trailing tile's operand rows
// are contiguous.
template <bool C, int NB, int LPR, int WARPS>
__global__ void __launch_bounds__(32 * WARPS) chol_panel_kernel(const __grid_constant__ CholBatch B, int kb, int per) {
  __shared__ Elem<C> Ls[NB][CB + 1];
  __shared__ double rs[NB];
  const int b = blockIdx.x / per, blk = blockIdx.x % per;
  const CholTask t = task_of<C>(B, b);
  const int N = t.N, tid = threadIdx.x;
  const int r0 = kb + NB + blk * (32 / LPR) * WARPS;
  if (r0 >= N) return;
  for (int i = tid; i < NB * NB; i += 32 * WARPS) {
    const int r = i / NB, c = i % NB;
    if (c <= r) {
      const Elem<C> e = ld_elem<C>(t.A, (long)(kb + r) * N + kb + c);
      Ls[c][r] = e;
      if (c == r) rs[r] = fast_rcp(e.re);
    }
  }
  __syncthreads();
  const int i = r0 + tid / LPR;
  const bool valid = i < N;
  double* row = t.A + ((long)i * N + kb) * (C ? 2 : 1);
  double* A = t.A;
  const bool ff = t.mode == 2;
  panel_row<C, NB, LPR>(row, valid, Ls, rs, [&](int c, const Elem<C>& v) {
    st_elem<C>(row, c, v);
    if (ff) st_ff<C>(A, (long)(kb + c) * N + i, to_ff<C>(v));
  });
}

// Trailing update with the panel at kb: tiles of edge 16 U of the lower
// triangle beyond it, U x U outputs per thread; FP64 (FF = false) or, on the
// split-precision path, float-float on the FP32 pipe (about 2^-45 of the
// update, five times the FP64 pipe's rate).  Tile (0, 0) goes on to factor
// the next diagonal block.  Only columns below cend (a multiple of the panel
// width, or at least N).
template <bool C, bool FF, int NB, int U>
__global__ void __launch_bounds__(256, FF ? 3 : 2)
    chol_update_kernel(const __grid_constant__ CholBatch B, int kb, int per, int cend) {
  static_assert(NB <= 16 * U, "the first tile holds the next diagonal block");
  constexpr int T = 16 * U, SR = NB > T ? NB : T;
  __shared__ Elem<C> S1[SR][CB + 1];
  __shared__ Elem<C> S2[NB][CB + 1];
  __shared__ DiagShared<C, NB> S;
  const int b = blockIdx.x / per, tile = blockIdx.x % per;
  const CholTask t = task_of<C>(B, b);
  const int N = t.N, m0 = kb + NB, m = N - m0;
  if (m <= 0) return;
  const int nt = (m + T - 1) / T;
  int TI, TJ;
  if (cend < N) {
    const int nc = (cend - m0 + T - 1) / T;
    TI = tile / nc;
    TJ = tile % nc;
    if (TI >= nt || TI < TJ) return;
  } else {
    if (tile >= nt * (nt + 1) / 2) return;
    tri_ij(tile, TI, TJ);
  }
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  double* A = t.A;
  Elem<C> o[U][U];  // the tile's own values, in flight during the product
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < U; ++v) {
      const int r = m0 + TI * T + ty + 16 * u, c = m0 + TJ * T + tx + 16 * v;
      o[u][v] = (r < N && c <= r) ? ld_elem<C>(A, (long)r * N + c) : zero_elem<C>();
    }
  if constexpr (FF) {
    FFE<C>(*F1)[CB + 1] = reinterpret_cast<FFE<C>(*)[CB + 1]>(S1);
    FFE<C>(*F2)[CB + 1] = reinterpret_cast<FFE<C>(*)[CB + 1]>(S2);
    for (int i = tid; i < NB * T; i += 256) {
      const int r = i % T, c = i / T;
      const int ri = m0 + TI * T + r, rj = m0 + TJ * T + r;
      const long up = (long)(kb + c) * N;
      F1[c][r] = ri < N ? ld_ff<C>(A, up + ri) : FFE<C>{};
      F2[c][r] = rj < N ? conj_ff<C>(ld_ff<C>(A, up + rj)) : FFE<C>{};
    }
    __syncthreads();
    FFE<C> acc[U][U] = {};
#pragma unroll 2
    for (int c = 0; c < NB; ++c) {
      FFE<C> fa[U], fb[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        fa[u] = F1[c][ty + 16 * u];
        fb[u] = F2[c][tx + 16 * u];
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = 0; v < U; ++v) ff_mac_e<C>(acc[u][v], fa[u], fb[v]);
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int v = 0; v < U; ++v) {
        o[u][v].re -= (double)acc[u][v].rh + (double)acc[u][v].rl;
        if constexpr (C) o[u][v].im -= (double)acc[u][v].ih + (double)acc[u][v].il;
      }
  } else {
    for (int i = tid; i < NB * T; i += 256) {
      const int r = i / NB, c = i % NB;
      const int ri = m0 + TI * T + r, rj = m0 + TJ * T + r;
      S1[c][r] = ri < N ? ld_elem<C>(A, (long)ri * N + kb + c) : zero_elem<C>();
      S2[c][r] = rj < N ? ld_elem<C>(A, (long)rj * N + kb + c) : zero_elem<C>();
    }
    __syncthreads();
#pragma unroll 4
    for (int c = 0; c < NB; ++c) {
      Elem<C> a[U], bv[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        a[u] = S1[c][ty + 16 * u];
        bv[u] = S2[c][tx + 16 * u];
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = 0; v < U; ++v) msub_conj<C>(o[u][v], a[u], bv[v]);
    }
  }
  const bool diag = tile == 0;
  if (diag) __syncthreads();  // S1 is read no more
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < U; ++v) {
      const int lr = ty + 16 * u, lc = tx + 16 * v;
      const int r = m0 + TI * T + lr, c = m0 + TJ * T + lc;
      if (diag && lr < NB && lc < NB)
        S1[lr][lc] = o[u][v];
      else if (r < N && c <= r && c < cend)
        st_elem<C>(A, (long)r * N + c, o[u][v]);
    }
  if (!diag) return;
  __syncthreads();
  const int nb = min(NB, m);
  const double lg = diag_factor<C, NB>(S1, S, nb, t.mode, A + ((long)m0 * N + m0) * (C ? 2 : 1), N);
  if (tid == 0) diag_report(t, lg, S.bad, false, m <= NB);
}

// N <= 64: the whole matrix in one CTA's shared memory, all modes, one launch
// (up to four panels of 16 columns: diagonal block, rows, trailing elements).
template <bool C>
__global__ void __launch_bounds__(256) chol_small_kernel(const __grid_constant__ CholBatch B) {
  extern __shared__ __align__(16) double m_raw[];  // SMALL_N x (SMALL_N + 1) elements
  constexpr int NB = 16;
  __shared__ Elem<C> D[NB][CB + 1];
  __shared__ DiagShared<C, NB> S;
  __shared__ double red[8];
  constexpr long LD = SMALL_N + 1;
  const CholTask t = task_of<C>(B, blockIdx.x);
  const int N = t.N, tid = threadIdx.x;
  double s = 0.0;
  for (int i = tid; i < N * N; i += 256) {
    const int r = i / N, c = i % N;
    if (c > r) continue;
    Elem<C> x = ld_elem<C>(t.A, i);
    if (t.mode == 2) {
      const Elem<C> v = ld_elem<C>(t.Vc, i), w = ld_elem<C>(t.W, i);
      double p = x.re * v.re;
      if constexpr (C) p = fma(x.im, v.im, p);
      s += r == c ? p : 2.0 * p;
      x.re = -w.re - x.re;
      if constexpr (C) x.im = -w.im - x.im;
    } else if (t.mode == 0 && r == c) {
      s -= x.re;
    }
    st_elem<C>(m_raw, r * LD + c, x);
  }
  s = block_sum(s, red);  // its barriers also order the loads before the factor
  if (tid == 0 && t.mode != 1) t.out[1] = s;
  for (int kb = 0; kb < N; kb += NB) {
    const int nb = min(NB, N - kb), m0 = kb + nb, m = N - m0;
    for (int i = tid; i < NB * NB; i += 256) {
      const int r = i / NB, c = i % NB;
      if (r < nb && c <= r) D[r][c] = ld_elem<C>(m_raw, (kb + r) * LD + kb + c);
    }
    __syncthreads();
    const double lg = diag_factor<C, NB>(D, S, nb, t.mode, m_raw + (kb * LD + kb) * (C ? 2 : 1), LD);
    if (tid == 0) diag_report(t, lg, S.bad, kb == 0, m <= 0);
    __syncthreads();
    if (m <= 0) break;
    for (int i = tid; i < NB * NB; i += 256) {
      const int r = i / NB, c = i % NB;
      if (c <= r) D[c][r] = ld_elem<C>(m_raw, (kb + r) * LD + kb + c);
    }
    __syncthreads();
    // at most 48 rows, four lanes each
    if (tid < 192) {
      const int i = m0 + (tid >> 2);
      double* row = m_raw + ((long)min(i, N - 1) * LD + kb) * (C ? 2 : 1);
      panel_row<C, NB, 4>(row, i < N, D, S.rs, [&](int c, const Elem<C>& v) { st_elem<C>(row, c, v); });
    }
    __syncthreads();
    for (int e = tid; e < m * (m + 1) / 2; e += 256) {
      int r, c;
      tri_ij(e, r, c);
      const long ro = (m0 + r) * LD, co = (m0 + c) * LD;
      Elem<C> x = ld_elem<C>(m_raw, ro + m0 + c);
#pragma unroll 4
      for (int k = 0; k < NB; ++k) msub_conj<C>(x, ld_elem<C>(m_raw, ro + kb + k), ld_elem<C>(m_raw, co + kb + k));
      st_elem<C>(m_raw, ro + m0 + c, x);
    }
    __syncthreads();
  }
  if (t.mode != 1) return;
  for (int i = tid; i < N * N; i += 256) {
    const int r = i / N, c = i % N;
    st_elem<C>(t.A, i, c <= r ? ld_elem<C>(m_raw, r * LD + c) : zero_elem<C>());
  }
}

// ------------------------------------------------ triangular inverse ------
// X = L^-1 by doubling: the 32 x 32 diagonal blocks are inverted on their own,
// then for s = 32, 64, ... every aligned pair of inverted blocks of size s
// joins into one of size 2 s, X21 = -X22 (L21 X11), as two tiled products
// over all pairs and matrices: log2(N/32) levels of two launches whose tiles
// fill the GPU, instead of one CTA per column block that walks down all rows
// (N^2/2 tile products one after another for the first block).

template <bool C>
__global__ void __launch_bounds__(128) trinv_diag_kernel(int N, const double* __restrict__ Lb, double* __restrict__ Xb) {
  __shared__ Elem<C> Ls[CB][CB + 1];
  __shared__ double rs[CB];
  const int nt = (N + CB - 1) / CB;
  const int b = blockIdx.x / nt, k0 = (blockIdx.x % nt) * CB, tid = threadIdx.x;
  const long NN = (long)N * N * (C ? 2 : 1);
  const double* L = Lb + b * NN;
  double* X = Xb + b * NN;
  // padding rows and columns of a short block act as the identity
  for (int i = tid; i < CB * CB; i += 128) {
    const int r = i / CB, c = i % CB;
    Elem<C> e = zero_elem<C>();
    if (r == c) e.re = 1.0;
    if (k0 + r < N && c <= r) e = ld_elem<C>(L, (long)(k0 + r) * N + k0 + c);
    Ls[c][r] = conj_e<C>(e);  // [column][row]
  }
  __syncthreads();
  if (tid < CB) rs[tid] = 1.0 / Ls[tid][tid].re;
  __syncthreads();
  // column j of X solves L x = e_j, four lanes per column (lane g owns rows
  // 4 k + g): the same walk as a panel row, on L itself
  const int lane = tid & 31, g = lane & 3, q0 = lane & ~3, j = tid >> 2;
  Elem<C> x[CB / 4];
#pragma unroll
  for (int k = 0; k < CB / 4; ++k) {
    x[k] = zero_elem<C>();
    if (4 * k + g == j) x[k].re = 1.0;
  }
#pragma unroll
  for (int c = 0; c < CB; ++c) {
    Elem<C> v = scale<C>(x[c / 4], rs[c]);
    v.re = __shfl_sync(0xffffffffu, v.re, q0 | (c & 3));
    if constexpr (C) v.im = __shfl_sync(0xffffffffu, v.im, q0 | (c & 3));
    if (g == (c & 3)) x[c / 4] = v;
#pragma unroll
    for (int k = c / 4; k < CB / 4; ++k)
      if (k > c / 4 || g > (c & 3)) msub_conj<C>(x[k], v, Ls[c][4 * k + g]);
  }
#pragma unroll
  for (int k = 0; k < CB / 4; ++k) {
    const int r = 4 * k + g;
    if (k0 + r < N && k0 + j < N) st_elem<C>(X, (long)(k0 + r) * N + k0 + j, r >= j ? x[k] : zero_elem<C>());
  }
}

// One level of the doubling: PASS 0: T21 = L21 X11 into X's own storage of
// the mirrored block (rows of block 1, columns of block 2: the strict upper
// triangle, free until the end), transposed; PASS 1: X21 = -X22 T21.
// K ranges skip the operands' zero triangles.
template <bool C, int PASS, int U>
__global__ void __launch_bounds__(256) trinv_join_kernel(int N, int s, const double* __restrict__ Lb,
                                                         double* __restrict__ Xb, int tiles, int n_pairs) {
  constexpr int T = 16 * U;  // tile edge
  __shared__ Elem<C> S1[CB][T + 1];
  __shared__ Elem<C> S2[CB][T + 1];
  const int nt = s / T;
  int bid = blockIdx.x;
  const int tile = bid % tiles;
  bid /= tiles;
  const int p = bid % n_pairs, b = bid / n_pairs;
  const int TI = tile / nt, TJ = tile % nt;
  const int c0 = 2 * s * p, r0 = c0 + s;  // block 1 (columns), block 2 (rows)
  const int row0 = r0 + TI * T, col0 = c0 + TJ * T;
  if (row0 >= N) return;
  const long NN = (long)N * N * (C ? 2 : 1);
  const double* L = Lb + b * NN;
  double* X = Xb + b * NN;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  Elem<C> o[U][U];
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < U; ++v) o[u][v] = zero_elem<C>();
  // PASS 0: sum over k of L[row][k] X[k][col], k in block 1 from the column's tile on
  // PASS 1: sum over k of X[row][k] T[k][col], k in block 2 up to the row's tile
  const int ka = PASS == 0 ? col0 / CB * CB : r0, kz = PASS == 0 ? r0 : min(row0 + T, N);
  for (int k0 = ka; k0 < kz; k0 += CB) {
    for (int i = tid; i < CB * T; i += 256) {
      const int r = i / CB, c = i % CB;
      if (PASS == 0) {
        const int kr = i / T, kc = i % T;
        S1[c][r] = row0 + r < N ? ld_elem<C>(L, (long)(row0 + r) * N + k0 + c) : zero_elem<C>();
        S2[kr][kc] = ld_elem<C>(X, (long)(k0 + kr) * N + col0 + kc);
      } else {
        S1[c][r] = (row0 + r < N && k0 + c < N) ? ld_elem<C>(X, (long)(row0 + r) * N + k0 + c) : zero_elem<C>();
        // T[k][col] is stored at X[col][k]
        S2[c][r] = k0 + c < N ? ld_elem<C>(X, (long)(col0 + r) * N + k0 + c) : zero_elem<C>();
      }
    }
    __syncthreads();
#pragma unroll 4
    for (int c = 0; c < CB; ++c) {
      Elem<C> a[U], bv[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        a[u] = S1[c][ty + 16 * u];
        bv[u] = S2[c][tx + 16 * u];
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = 0; v < U; ++v) mac<C>(o[u][v], a[u], bv[v]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < U; ++v) {
      const int r = row0 + ty + 16 * u, c = col0 + tx + 16 * v;
      if (r >= N) continue;
      Elem<C> e = o[u][v];
      if (PASS == 1) {
        e.re = -e.re;
        if constexpr (C) e.im = -e.im;
      }
      st_elem<C>(X, PASS == 0 ? (long)c * N + r : (long)r * N + c, e);
    }
}

// Clears the strict upper triangle that held the doubling's intermediates.
template <bool C>
__global__ void __launch_bounds__(256) clear_upper_kernel(int N, double* __restrict__ Xb) {
  const int b = blockIdx.x / N, r = blockIdx.x % N;
  double* X = Xb + (long)b * N * N * (C ? 2 : 1);
  for (int c = r + 1 + threadIdx.x; c < N; c += 256) st_elem<C>(X, (long)r * N + c, zero_elem<C>());
}

// ------------------------------------------------------------ host side ---

template <bool C>
cudaError_t small_attr() {
  // per device, set once (the attribute belongs to the device's context)
  static std::mutex mu;
  static bool done[MAX_DEVICES] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= MAX_DEVICES) dev = 0;
  std::lock_guard<std::mutex> lk(mu);
  if (done[dev]) return cudaSuccess;
  const cudaError_t e =
      cudaFuncSetAttribute(chol_small_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)(SMALL_N * (SMALL_N + 1) * sizeof(Elem<C>)));
  done[dev] = e == cudaSuccess;
  return e;
}

// Inverse form: panels of 32 columns once the trailing tiles of half the
// matrix's panels fill the GPU several times over.
bool panel32(int N, long n_mat) {
  const long h = (N / 2 + 31) / 32;
  return n_mat * h * (h + 1) / 2 >= 8L * device_sm_count();
}

// Block columns of OUTER columns (modes 0 and 2 with planes): the panels update
// only inside their block column, and each block column takes everything to its
// left at once as a digit product on the tensor cores (g64.cu),
// A[J0.., J] -= L[J0.., < J0] L[J, < J0]^H, whose planes are made of the finished columns.
constexpr int OUTER = 128;

struct OuterBytes {
  size_t a, b, ea, eb, one;  // planes and exponents of one matrix, the largest block column
};
OuterBytes outer_bytes(int cplx, int N) {
  OuterBytes o{};
  for (int J0 = OUTER; J0 < N; J0 += OUTER) {
    o.a = std::max(o.a, g64_plane_bytes(cplx, 0, N - J0, J0, 1));
    o.b = std::max(o.b, g64_plane_bytes(cplx, 1, std::min(OUTER, N - J0), J0, 1));
  }
  o.ea = sizeof(int) * (size_t)g64_rpad(cplx, 0, N);
  o.eb = sizeof(int) * (size_t)g64_rpad(cplx, 1, OUTER);
  o.one = o.a + o.b + o.ea + o.eb;
  return o;
}

cudaError_t chol_outer(int cplx, int N, int n_mat, double* mats, long bstride, int J0, const CholOuter& x, int* status,
                       cudaStream_t s) {
  const OuterBytes t = outer_bytes(cplx, N);
  const long cs = cplx ? 2 : 1;
  const int C = std::min(OUTER, N - J0), R = N - J0;
  const size_t fb = ((sizeof(int) * (size_t)n_mat + 1023) / 1024) * 1024;
  int* flag = (int*)x.work;
  if (x.bytes < fb + t.one) return cudaErrorInvalidValue;
  const int room = (int)std::min<size_t>((size_t)n_mat, (x.bytes - fb) / t.one);
  if (cudaError_t e = cudaMemsetAsync(flag, 0, sizeof(int) * (size_t)n_mat, s)) return e;
  for (int b0 = 0; b0 < n_mat; b0 += room) {
    const int nb = std::min(room, n_mat - b0);
    char* p = (char*)x.work + fb;
    double* Ab = mats + b0 * bstride;
    // conj(L) by rows, its rows J0.. and J0 .. J0 + C - 1
    auto src = [&](int rows) {
      G64Src g{};
      g.base = Ab + (long)J0 * N * cs;
      g.stride = bstride / cs;
      g.ld = N;
      g.by_rows = 1;
      g.conj = 1;
      g.nb = nb;
      g.R = rows;
      g.K = J0;
      return g;
    };
    G64Op oa{}, ob{};
    oa.planes = (uint16_t*)p;
    ob.planes = (uint16_t*)(p + t.a * (size_t)nb);
    oa.e = (int*)(p + (t.a + t.b) * (size_t)nb);
    ob.e = (int*)(p + (t.a + t.b + t.ea) * (size_t)nb);
    oa.stride = (long)(g64_plane_bytes(cplx, 0, R, J0, 1) / 2);
    ob.stride = (long)(g64_plane_bytes(cplx, 1, C, J0, 1) / 2);
    oa.Rpad = g64_rpad(cplx, 0, R);
    ob.Rpad = g64_rpad(cplx, 1, C);
    oa.n_kb = ob.n_kb = g64_nkb(cplx, J0);
    if (cudaError_t e = g64_slice(cplx, 0, src(R), oa, flag + b0, 1, s)) return e;
    if (cudaError_t e = g64_slice(cplx, 1, src(C), ob, flag + b0, 1, s)) return e;
    G64Out o{};
    o.base = Ab + ((long)J0 * N + J0) * cs;
    o.stride = bstride / cs;
    o.s0 = N;
    o.t0 = 1;
    o.rd = o.cd = 1 << 30;
    o.R = R;
    o.C = C;
    o.add = o.neg = 1;
    o.tri = 2;
    if (cudaError_t e = g64_product(cplx, oa, ob, G64Index{nullptr, nullptr, 1, 1}, o, nb, 0, nullptr, 0, flag + b0, 1,
                                    status, nullptr, s))
      return e;
    const int per = ((R + 31) / 32) * ((C + 31) / 32);
    if (cplx)
      chol_outer_kernel<true><<<(unsigned)(nb * per), 256, 0, s>>>(N, Ab, bstride, J0, J0 + C, per, flag + b0);
    else
      chol_outer_kernel<false><<<(unsigned)(nb * per), 256, 0, s>>>(N, Ab, bstride, J0, J0 + C, per, flag + b0);
  }
  return cudaGetLastError();
}
int outer_launches(int cplx, int N, int n_mat, size_t bytes) {
  const OuterBytes t = outer_bytes(cplx, N);
  const size_t fb = ((sizeof(int) * (size_t)n_mat + 1023) / 1024) * 1024;
  const int room = (int)std::min<size_t>((size_t)n_mat, (bytes - fb) / t.one);
  return (n_mat + room - 1) / room * 6;
}

// Launches of one batch whose largest matrix is N (tasks sorted by size,
// largest first, when ragged: Ns[b] is task b's size, so that each panel
// covers only the prefix that still has one).
template <bool C>
cudaError_t chol_run(const CholBatch& B, int N, int n_mat, const int* Ns, int mode, cudaStream_t s, int* n_launch,
                     const CholOuter* outer) {
  int nl = 0;
  if (N <= SMALL_N) {
    if (cudaError_t e = small_attr<C>()) return e;
    chol_small_kernel<C><<<n_mat, 256, SMALL_N * (SMALL_N + 1) * sizeof(Elem<C>), s>>>(B);
    if (n_launch) *n_launch = 1;
    return cudaGetLastError();
  }
  if (mode != 0) {
    chol_init_kernel<C><<<n_mat * INIT_BLOCKS, 256, 0, s>>>(B, INIT_BLOCKS);
    ++nl;
  }
  const bool wide = mode == 2 && panel32(N, n_mat);
  if (wide)
    chol_first_kernel<C, 32><<<n_mat, 256, 0, s>>>(B, INIT_BLOCKS, 0);
  else
    chol_first_kernel<C, 16><<<n_mat, 256, 0, s>>>(B, INIT_BLOCKS, 0);
  ++nl;
  const long sms = device_sm_count();
  const int NB = wide ? 32 : 16;
  int live = n_mat;
  for (int kb = 0; kb + NB < N; kb += NB) {
    while (Ns && live > 0 && Ns[live - 1] <= kb + NB) --live;
    const int m = N - kb - NB;
    // rows: 8 per CTA with 16 lanes each while that leaves SMs free, else 64
    // with four lanes each (80 instead of 128 FP64 instructions per row)
    const int per64 = (m + 63) / 64, per8 = (m + 7) / 8;
    const bool few = (long)live * per8 <= 4 * sms;
    if (wide) {
      if (few)
        chol_panel_kernel<C, 32, 16, 4><<<(unsigned)(live * per8), 128, 0, s>>>(B, kb, per8);
      else
        chol_panel_kernel<C, 32, 4, 8><<<(unsigned)(live * per64), 256, 0, s>>>(B, kb, per64);
    } else {
      if (few)
        chol_panel_kernel<C, 16, 16, 4><<<(unsigned)(live * per8), 128, 0, s>>>(B, kb, per8);
      else
        chol_panel_kernel<C, 16, 4, 8><<<(unsigned)(live * per64), 256, 0, s>>>(B, kb, per64);
    }
    ++nl;
    const long n32 = (m + 31) / 32, n16 = (m + 15) / 16;
    int per32 = (int)(n32 * (n32 + 1) / 2), per16 = (int)(n16 * (n16 + 1) / 2), cend = N;
    if (outer) {
      cend = std::min(N, (kb / OUTER + 1) * OUTER);
      if (kb + NB == cend) {  // the next block column
        if (cudaError_t e = chol_outer(C ? 1 : 0, N, n_mat, B.mats, B.bstride, cend, *outer, B.status, s)) return e;
        if (wide)
          chol_first_kernel<C, 32><<<n_mat, 256, 0, s>>>(B, INIT_BLOCKS, cend);
        else
          chol_first_kernel<C, 16><<<n_mat, 256, 0, s>>>(B, INIT_BLOCKS, cend);
        nl += 1 + outer_launches(C ? 1 : 0, N, n_mat, outer->bytes);
        continue;
      }
      if (cend < N) {
        const int w = cend - kb - NB;
        per32 = (int)(n32 * ((w + 31) / 32));
        per16 = (int)(n16 * ((w + 15) / 16));
      }
    }
    // 16 x 16 tiles until 32 x 32 ones give every SM two (they read less)
    const bool t32 = live * (long)per32 >= 2 * sms;
    if (mode == 2) {
      if (wide)
        chol_update_kernel<C, true, 32, 2><<<(unsigned)(live * per32), 256, 0, s>>>(B, kb, per32, cend);
      else if (t32)
        chol_update_kernel<C, true, 16, 2><<<(unsigned)(live * per32), 256, 0, s>>>(B, kb, per32, cend);
      else
        chol_update_kernel<C, true, 16, 1><<<(unsigned)(live * per16), 256, 0, s>>>(B, kb, per16, cend);
    } else if (t32) {
      chol_update_kernel<C, false, 16, 2><<<(unsigned)(live * per32), 256, 0, s>>>(B, kb, per32, cend);
    } else {
      chol_update_kernel<C, false, 16, 1><<<(unsigned)(live * per16), 256, 0, s>>>(B, kb, per16, cend);
    }
    ++nl;
  }
  if (n_launch) *n_launch = nl;
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_cholesky(int cplx, int N, int n_mat, double* mats, long bstride, int mode, double* out,
                            int* status, int status_base, cudaStream_t s, const double* Wn, const double* Vc,
                            const double* ldV, int n_w, const CholOuter* outer, int* n_launch) {
  if (n_mat == 0) return cudaSuccess;
  if (mode == 2 && (!Wn || !Vc || !ldV || n_w <= 0)) return cudaErrorInvalidValue;
  if (mode != 1 && !out) return cudaErrorInvalidValue;
  const long nt = (N + 15) / 16;
  if ((long)n_mat * std::max<long>(nt * (nt + 1) / 2, INIT_BLOCKS) > 0x7fffffffL) return cudaErrorInvalidValue;
  const CholBatch B{nullptr, mats, bstride, out, status, Wn, Vc, ldV, N, mode, status_base, std::max(n_w, 1)};
  if (outer && (N <= OUTER || mode == 1 || !outer->work)) outer = nullptr;
  return cplx ? chol_run<true>(B, N, n_mat, nullptr, mode, s, n_launch, outer)
              : chol_run<false>(B, N, n_mat, nullptr, mode, s, n_launch, outer);
}

// The digit products save FP64 work (mode 0) or a fifth of it on the FP32 pipe (mode
// 2) and add some 60 us of launches per block column.  Measured, log-det step of
// one q with and without: complex N = 384, 8 frequencies 2.07 and 2.25 ms, N = 512,
// 16 4.07 and 5.39, N = 768, 8 5.71 and 8.29; real N = 384, 16 equal, N = 512, 16
// 2.36 and 2.54, N = 768, 16 4.15 and 5.15.  Inverse form: 16 real of N = 733 2.12 and
// 1.65 (not taken), 32 complex of N = 768 7.4 and 9.2, 320 of N = 512 14.4 and 19.3.
bool chol_g64_use(int cplx, int N, int n, int mode) {
  const double macs = (cplx ? 4.0 : 1.0) * N * (double)N * N * n;
  return N >= 384 && n >= 8 && macs >= (mode == 2 ? 2.5e10 : 1.5e9);
}

int cholesky_launches(int N, int n_mat, int mode) {
  if (n_mat <= 0) return 0;
  if (N <= SMALL_N) return 1;
  return (mode != 0 ? 2 : 1) + 2 * ((N - 1) / (mode == 2 && panel32(N, n_mat) ? 32 : 16));
}

cudaError_t launch_cholesky_ragged(int cplx, const CholTask* tasks, const CholTask* host, int n_tasks, cudaStream_t s,
                                   int* n_launch) {
  if (n_launch) *n_launch = 0;
  if (n_tasks <= 0) return cudaSuccess;
  std::vector<int> Ns(n_tasks);
  int big = 0;
  for (int i = 0; i < n_tasks; ++i) {
    if (host[i].mode != host[0].mode || (i && host[i].N > host[i - 1].N)) return cudaErrorInvalidValue;
    Ns[i] = host[i].N;
    if (host[i].N > SMALL_N) big = i + 1;
  }
  const int mode = host[0].mode;
  int total = 0;
  for (int part = 0; part < 2; ++part) {
    const int lo = part ? big : 0, n = part ? n_tasks - big : big;
    if (n == 0) continue;
    CholBatch B{};
    B.tasks = tasks + lo;
    int nl = 0;
    const cudaError_t e = cplx ? chol_run<true>(B, Ns[lo], n, Ns.data() + lo, mode, s, &nl, nullptr)
                               : chol_run<false>(B, Ns[lo], n, Ns.data() + lo, mode, s, &nl, nullptr);
    if (e != cudaSuccess) return e;
    total += nl;
  }
  if (n_launch) *n_launch = total;
  return cudaSuccess;
}

namespace {
template <bool C>
cudaError_t trinv_run(int N, int n_q, const double* L, double* X, cudaStream_t s) {
  const int nt = (N + CB - 1) / CB;
  const long sms = device_sm_count();
  trinv_diag_kernel<C><<<n_q * nt, 128, 0, s>>>(N, L, X);
  for (int sz = CB; sz < N; sz *= 2) {
    const int pairs = (N - sz + 2 * sz - 1) / (2 * sz);
    // 16 x 16 tiles (a quarter of the FP64 work each, the same sums) while 32 x 32 ones leave SMs idle
    if ((long)n_q * pairs * (sz / 32) * (sz / 32) >= 2 * sms) {
      const int tiles = (sz / 32) * (sz / 32);
      trinv_join_kernel<C, 0, 2><<<n_q * pairs * tiles, 256, 0, s>>>(N, sz, L, X, tiles, pairs);
      trinv_join_kernel<C, 1, 2><<<n_q * pairs * tiles, 256, 0, s>>>(N, sz, L, X, tiles, pairs);
    } else {
      const int tiles = (sz / 16) * (sz / 16);
      trinv_join_kernel<C, 0, 1><<<n_q * pairs * tiles, 256, 0, s>>>(N, sz, L, X, tiles, pairs);
      trinv_join_kernel<C, 1, 1><<<n_q * pairs * tiles, 256, 0, s>>>(N, sz, L, X, tiles, pairs);
    }
  }
  if (N > CB) clear_upper_kernel<C><<<n_q * N, 256, 0, s>>>(N, X);
  return cudaGetLastError();
}
}  // namespace

int trinv_launches(int N) {
  int n = N > CB ? 2 : 1;
  for (int sz = CB; sz < N; sz *= 2) n += 2;
  return n;
}

cudaError_t launch_trinv(int cplx, int N, int n_q, const double* L, double* X, cudaStream_t s) {
  if (n_q == 0) return cudaSuccess;
  return cplx ? trinv_run<true>(N, n_q, L, X, s) : trinv_run<false>(N, n_q, L, X, s);
}

}  // namespace rpa
