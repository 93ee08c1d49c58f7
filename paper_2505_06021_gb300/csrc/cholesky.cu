// Batched Cholesky factorisations of the RPA tail on GB300 (sm_103a): V = L L^H,
// 1 - Pi' and V^-1 - chi0 with their log-determinants and traces, and the
// inverse of the V factors.
//
// What bounds it.  An SM issues two DFMA lanes per clock, so one complex
// N = 768 factorisation is 151e6 clocks (73 ms) of one SM's FP64 pipe but
// 0.5 ms of all 152: a matrix that stays on one SM, or on a cluster of eight,
// is bound by that pipe and by its own serial phases, whatever else is idle.
// Every panel step is therefore spread over the whole GPU: a launch covers
// the panel rows (16 or 64 per CTA) or the trailing 32 x 32 tiles of every
// matrix, and the kernel boundary is the only synchronisation.  The tile that
// holds the next diagonal block factors it at once, so a panel costs two
// launches.  Per matrix the arithmetic and its order do not depend on the
// batch, so a matrix gives the same bits alone, in a batch or in a ragged
// launch.  Matrices up to 64 stay in one CTA's shared memory, one launch in all.
//
// Measured on GB300, one CTA or an 8-CTA cluster per matrix before, panel
// launches now: one complex N = 768 factor of V 19.9 -> 2.4 ms; 16 matrices of
// N = 768 in FP64 30.1 -> 9.7 ms; 32 in the inverse form 17.6 -> 8.8 ms; 320 of
// N = 512 in the inverse form 34.7 -> 19.4 ms; 64 of N = 300 18.6 -> 1.6 ms; 16
// real ones of N = 64 0.285 -> 0.065 ms.  What is left is the FP64 pipe (the 16
// FP64 matrices need 7.6 ms of it) and, for few matrices, two launches of some
// 20 us each per panel.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "fp64_elem.cuh"
#include "rpa_internal.h"

namespace rpa {
namespace {

constexpr int CB = 32;                   // panel width and trailing tile edge
constexpr int SMALL_N = 64;              // largest matrix of the one-launch kernel
constexpr int TRI = CB * (CB + 1) / 2;   // elements of a diagonal block's lower triangle
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

template <bool C>
struct DiagShared {
  Elem<C> col[2][CB];  // the current column (unscaled), double-buffered
  double rd[2];        // reciprocal of the current pivot
  double piv[CB];      // pivots (mode 0: pivot - 1)
  double l[CB], rs[CB];
  int bad;
};

// Factor of the diagonal block D (lower triangle, nb x nb, shared memory) by
// the CTA's 256 threads; L goes to Lout (leading dimension ld).  Each thread
// keeps two or three elements of the triangle in registers, in column order,
// so that whole warps retire as the columns do.  A column costs one barrier:
// the columns stay unscaled (x_rc -= x_rk conj(x_ck) / d_k), which leaves one
// reciprocal on the serial chain; all square roots, logarithms and scalings
// follow at the end, one per thread.  Returns (thread 0) the block's share of
// the log-determinant, NaN and *S.bad on a non-positive pivot.
template <bool C>
__device__ double diag_factor(Elem<C> (*D)[CB + 1], DiagShared<C>& S, int nb, int mode, double* Lout, long ld) {
  const int tid = threadIdx.x;
  Elem<C> x[3];
  int er[3], ec[3];
  if (tid == 0) S.bad = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int e = tid + 256 * k;
    er[k] = ec[k] = -1;
    x[k] = zero_elem<C>();
    if (e < TRI) {
      int i, j;
      tri_ij(TRI - 1 - e, i, j);
      const int r = CB - 1 - j, c = CB - 1 - i;
      if (r < nb) {
        er[k] = r;
        ec[k] = c;
        x[k] = D[r][c];
      }
    }
  }
  auto publish = [&](int k, int buf) {
    S.col[buf][er[k]] = x[k];
    if (er[k] == ec[k]) {
      const double u = x[k].re;
      S.piv[er[k]] = u;
      S.rd[buf] = 1.0 / (mode == 0 ? 1.0 + u : u);
    }
  };
  if (ec[0] == 0) publish(0, 0);
  __syncthreads();
  for (int c = 0; c < nb; ++c) {
    const int buf = c & 1;
    const double rd = S.rd[buf];
#pragma unroll
    for (int k = 0; k < 3; ++k)
      if (ec[k] > c) {
        msub_conj<C>(x[k], scale<C>(S.col[buf][er[k]], rd), S.col[buf][ec[k]]);
        if (ec[k] == c + 1) publish(k, buf ^ 1);
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
    S.rs[tid] = 1.0 / l;
    lg = !ok ? nan("") : mode == 0 ? log1p(u) : log(p);
    if (!ok) S.bad = 1;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 3; ++k)
    if (ec[k] >= 0) {
      Elem<C> v = scale<C>(x[k], S.rs[ec[k]]);
      if (er[k] == ec[k]) {
        v = zero_elem<C>();
        v.re = S.l[er[k]];
      }
      st_elem<C>(Lout, er[k] * ld + ec[k], v);
    }
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

// Rows of a panel: X L_kk^H = A_panel, four lanes per row (lane g of a row
// owns columns c = 4 j + g), so that the serial chain of a row is 32 short
// steps and a warp's FP64 instructions carry eight rows.  Ls[c][c'] holds
// L_kk[c'][c], rs the reciprocal diagonal.  `row` is this quad's row (invalid
// rows take part in the shuffles).
template <bool C, class ST>
__device__ __forceinline__ void panel_row(const double* A, long ld, bool valid, const Elem<C> (*Ls)[CB + 1],
                                          const double* rs, const ST& store) {
  const int lane = threadIdx.x & 31, g = lane & 3, q0 = lane & ~3;
  Elem<C> x[CB / 4];
#pragma unroll
  for (int j = 0; j < CB / 4; ++j) x[j] = valid ? ld_elem<C>(A, 4 * j + g) : zero_elem<C>();
#pragma unroll
  for (int c = 0; c < CB; ++c) {
    Elem<C> v = scale<C>(x[c / 4], rs[c]);
    v.re = __shfl_sync(0xffffffffu, v.re, q0 | (c & 3));
    if constexpr (C) v.im = __shfl_sync(0xffffffffu, v.im, q0 | (c & 3));
    if (g == (c & 3)) x[c / 4] = v;
#pragma unroll
    for (int j = c / 4; j < CB / 4; ++j)
      if (j > c / 4 || g > (c & 3)) msub_conj<C>(x[j], v, Ls[c][4 * j + g]);
  }
  if (valid)
#pragma unroll
    for (int j = 0; j < CB / 4; ++j) store(4 * j + g, x[j]);
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

// The first diagonal block of every matrix, and the traces (mode 0: Tr Pi =
// -sum Y_jj; mode 2: the partial sums of chol_init_kernel).
template <bool C>
__global__ void __launch_bounds__(256) chol_first_kernel(const __grid_constant__ CholBatch B, int nblk) {
  __shared__ Elem<C> D[CB][CB + 1];
  __shared__ DiagShared<C> S;
  __shared__ double red[8];
  const CholTask t = task_of<C>(B, blockIdx.x);
  const int N = t.N, tid = threadIdx.x, nb = min(CB, N);
  if (t.mode != 1) {
    double s = 0.0;
    if (t.mode == 0) {
      for (int j = tid; j < N; j += 256) s -= ld_elem<C>(t.A, (long)j * N + j).re;
    } else if (tid < nblk) {
      s = ld_elem<C>(t.A, 1 + tid).re;
    }
    s = block_sum(s, red);
    if (tid == 0) t.out[1] = s;
  }
  for (int i = tid; i < CB * CB; i += 256) {
    const int r = i / CB, c = i % CB;
    if (r < nb && c <= r) D[r][c] = ld_elem<C>(t.A, (long)r * N + c);
  }
  __syncthreads();
  const double lg = diag_factor<C>(D, S, nb, t.mode, t.A, N);
  if (tid == 0) diag_report(t, lg, S.bad, true, N <= CB);
}

// Panel rows below the diagonal block at kb (full panels only: kb + CB < N).
// Mode 2 also stores the float-float copy of L_{i,kb+c} at (row kb + c, column
// i) of the free strict upper triangle, where a trailing tile's operand rows
// are contiguous.
template <bool C, int WARPS>
__global__ void __launch_bounds__(32 * WARPS) chol_panel_kernel(const __grid_constant__ CholBatch B, int kb, int per) {
  __shared__ Elem<C> Ls[CB][CB + 1];
  __shared__ double rs[CB];
  const int b = blockIdx.x / per, blk = blockIdx.x % per;
  const CholTask t = task_of<C>(B, b);
  const int N = t.N, tid = threadIdx.x;
  const int r0 = kb + CB + blk * 8 * WARPS;
  if (r0 >= N) return;
  for (int i = tid; i < CB * CB; i += 32 * WARPS) {
    const int r = i / CB, c = i % CB;
    if (c <= r) Ls[c][r] = ld_elem<C>(t.A, (long)(kb + r) * N + kb + c);
  }
  __syncthreads();
  if (tid < CB) rs[tid] = 1.0 / Ls[tid][tid].re;
  __syncthreads();
  const int i = r0 + (tid >> 2);
  const bool valid = i < N;
  double* row = t.A + ((long)i * N + kb) * (C ? 2 : 1);
  double* A = t.A;
  const bool ff = t.mode == 2;
  panel_row<C>(row, N, valid, Ls, rs, [&](int c, const Elem<C>& v) {
    st_elem<C>(row, c, v);
    if (ff) st_ff<C>(A, (long)(kb + c) * N + i, to_ff<C>(v));
  });
}

// Trailing update with the panel at kb: 32 x 32 tiles of the lower triangle
// beyond it, 2 x 2 outputs per thread; FP64 (FF = false) or, on the
// split-precision path, float-float on the FP32 pipe (about 2^-45 of the
// update, five times the FP64 pipe's rate).  Tile (0, 0) goes on to factor
// the next diagonal block.
template <bool C, bool FF>
__global__ void __launch_bounds__(256, FF ? 3 : 2)
    chol_update_kernel(const __grid_constant__ CholBatch B, int kb, int per) {
  __shared__ Elem<C> S1[CB][CB + 1];
  __shared__ Elem<C> S2[CB][CB + 1];
  __shared__ DiagShared<C> S;
  const int b = blockIdx.x / per, tile = blockIdx.x % per;
  const CholTask t = task_of<C>(B, b);
  const int N = t.N, m0 = kb + CB, m = N - m0;
  if (m <= 0) return;
  const int nt = (m + CB - 1) / CB;
  if (tile >= nt * (nt + 1) / 2) return;
  int TI, TJ;
  tri_ij(tile, TI, TJ);
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  double* A = t.A;
  Elem<C> o[2][2];  // the tile's own values, in flight during the product
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int r = m0 + TI * CB + ty + 16 * u, c = m0 + TJ * CB + tx + 16 * v;
      o[u][v] = (r < N && c <= r) ? ld_elem<C>(A, (long)r * N + c) : zero_elem<C>();
    }
  if constexpr (FF) {
    FFE<C>(*F1)[CB + 1] = reinterpret_cast<FFE<C>(*)[CB + 1]>(S1);
    FFE<C>(*F2)[CB + 1] = reinterpret_cast<FFE<C>(*)[CB + 1]>(S2);
    for (int i = tid; i < CB * CB; i += 256) {
      const int r = i % CB, c = i / CB;
      const int ri = m0 + TI * CB + r, rj = m0 + TJ * CB + r;
      const long up = (long)(kb + c) * N;
      F1[c][r] = ri < N ? ld_ff<C>(A, up + ri) : FFE<C>{};
      F2[c][r] = rj < N ? conj_ff<C>(ld_ff<C>(A, up + rj)) : FFE<C>{};
    }
    __syncthreads();
    FFE<C> acc[2][2] = {};
#pragma unroll 2
    for (int c = 0; c < CB; ++c) {
      const FFE<C> a0 = F1[c][ty], a1 = F1[c][ty + 16];
      const FFE<C> b0 = F2[c][tx], b1 = F2[c][tx + 16];
      ff_mac_e<C>(acc[0][0], a0, b0);
      ff_mac_e<C>(acc[0][1], a0, b1);
      ff_mac_e<C>(acc[1][0], a1, b0);
      ff_mac_e<C>(acc[1][1], a1, b1);
    }
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        o[u][v].re -= (double)acc[u][v].rh + (double)acc[u][v].rl;
        if constexpr (C) o[u][v].im -= (double)acc[u][v].ih + (double)acc[u][v].il;
      }
  } else {
    for (int i = tid; i < CB * CB; i += 256) {
      const int r = i / CB, c = i % CB;
      const int ri = m0 + TI * CB + r, rj = m0 + TJ * CB + r;
      S1[c][r] = ri < N ? ld_elem<C>(A, (long)ri * N + kb + c) : zero_elem<C>();
      S2[c][r] = rj < N ? ld_elem<C>(A, (long)rj * N + kb + c) : zero_elem<C>();
    }
    __syncthreads();
#pragma unroll 4
    for (int c = 0; c < CB; ++c) {
      const Elem<C> a0 = S1[c][ty], a1 = S1[c][ty + 16];
      const Elem<C> b0 = S2[c][tx], b1 = S2[c][tx + 16];
      msub_conj<C>(o[0][0], a0, b0);
      msub_conj<C>(o[0][1], a0, b1);
      msub_conj<C>(o[1][0], a1, b0);
      msub_conj<C>(o[1][1], a1, b1);
    }
  }
  if (tile == 0) {
    __syncthreads();  // S1 is read no more
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int v = 0; v < 2; ++v) S1[ty + 16 * u][tx + 16 * v] = o[u][v];
    __syncthreads();
    const int nb = min(CB, m);
    const double lg = diag_factor<C>(S1, S, nb, t.mode, A + ((long)m0 * N + m0) * (C ? 2 : 1), N);
    if (tid == 0) diag_report(t, lg, S.bad, false, m <= CB);
    return;
  }
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int r = m0 + TI * CB + ty + 16 * u, c = m0 + TJ * CB + tx + 16 * v;
      if (r < N && c <= r) st_elem<C>(A, (long)r * N + c, o[u][v]);
    }
}

// N <= 64: the whole matrix in one CTA's shared memory, all modes, one launch
// (two panels: diagonal block, rows, trailing block, diagonal block).
template <bool C>
__global__ void __launch_bounds__(256) chol_small_kernel(const __grid_constant__ CholBatch B) {
  extern __shared__ __align__(16) double m_raw[];  // SMALL_N x (SMALL_N + 1) elements
  __shared__ Elem<C> D[CB][CB + 1];
  __shared__ DiagShared<C> S;
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
  for (int kb = 0; kb < N; kb += CB) {
    const int nb = min(CB, N - kb), m0 = kb + nb;
    for (int i = tid; i < CB * CB; i += 256) {
      const int r = i / CB, c = i % CB;
      if (r < nb && c <= r) D[r][c] = ld_elem<C>(m_raw, (kb + r) * LD + kb + c);
    }
    __syncthreads();
    const double lg = diag_factor<C>(D, S, nb, t.mode, m_raw + (kb * LD + kb) * (C ? 2 : 1), LD);
    if (tid == 0) diag_report(t, lg, S.bad, kb == 0, m0 >= N);
    __syncthreads();
    if (m0 >= N) break;
    for (int i = tid; i < CB * CB; i += 256) {
      const int r = i / CB, c = i % CB;
      if (c <= r) D[c][r] = ld_elem<C>(m_raw, r * LD + c);
    }
    __syncthreads();
    // at most 32 rows: the first four warps
    if (tid < 128) {
      const int i = m0 + (tid >> 2);
      double* row = m_raw + (long)min(i, N - 1) * LD * (C ? 2 : 1);
      panel_row<C>(row, LD, i < N, D, S.rs, [&](int c, const Elem<C>& v) { st_elem<C>(row, c, v); });
    }
    __syncthreads();
    const int m = N - m0;
    for (int e = tid; e < TRI; e += 256) {
      int r, c;
      tri_ij(e, r, c);
      if (r >= m) continue;
      const long ro = (m0 + r) * LD, co = (m0 + c) * LD;
      Elem<C> x = ld_elem<C>(m_raw, ro + m0 + c);
#pragma unroll 4
      for (int k = 0; k < CB; ++k) msub_conj<C>(x, ld_elem<C>(m_raw, ro + k), ld_elem<C>(m_raw, co + k));
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
template <bool C, int PASS>
__global__ void __launch_bounds__(256) trinv_join_kernel(int N, int s, const double* __restrict__ Lb,
                                                         double* __restrict__ Xb, int tiles, int n_pairs) {
  __shared__ Elem<C> S1[CB][CB + 1];
  __shared__ Elem<C> S2[CB][CB + 1];
  const int nt = s / CB;
  int bid = blockIdx.x;
  const int tile = bid % tiles;
  bid /= tiles;
  const int p = bid % n_pairs, b = bid / n_pairs;
  const int TI = tile / nt, TJ = tile % nt;
  const int c0 = 2 * s * p, r0 = c0 + s;  // block 1 (columns), block 2 (rows)
  const int row0 = r0 + TI * CB, col0 = c0 + TJ * CB;
  if (row0 >= N) return;
  const long NN = (long)N * N * (C ? 2 : 1);
  const double* L = Lb + b * NN;
  double* X = Xb + b * NN;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  Elem<C> o[2][2];
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) o[u][v] = zero_elem<C>();
  // PASS 0: sum over k of L[row][k] X[k][col], k in block 1 from the column's tile on
  // PASS 1: sum over k of X[row][k] T[k][col], k in block 2 up to the row's tile
  const int ka = PASS == 0 ? col0 : r0, kz = PASS == 0 ? r0 : min(row0 + CB, N);
  for (int k0 = ka; k0 < kz; k0 += CB) {
    for (int i = tid; i < CB * CB; i += 256) {
      const int r = i / CB, c = i % CB;
      if (PASS == 0) {
        S1[c][r] = row0 + r < N ? ld_elem<C>(L, (long)(row0 + r) * N + k0 + c) : zero_elem<C>();
        S2[r][c] = ld_elem<C>(X, (long)(k0 + r) * N + col0 + c);
      } else {
        S1[c][r] = (row0 + r < N && k0 + c < N) ? ld_elem<C>(X, (long)(row0 + r) * N + k0 + c) : zero_elem<C>();
        // T[k][col] is stored at X[col][k]
        S2[c][r] = k0 + c < N ? ld_elem<C>(X, (long)(col0 + r) * N + k0 + c) : zero_elem<C>();
      }
    }
    __syncthreads();
#pragma unroll 4
    for (int c = 0; c < CB; ++c) {
      const Elem<C> a0 = S1[c][ty], a1 = S1[c][ty + 16];
      const Elem<C> b0 = S2[c][tx], b1 = S2[c][tx + 16];
      mac<C>(o[0][0], a0, b0);
      mac<C>(o[0][1], a0, b1);
      mac<C>(o[1][0], a1, b0);
      mac<C>(o[1][1], a1, b1);
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
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

// Launches of one batch whose largest matrix is N (tasks sorted by size,
// largest first, when ragged: Ns[b] is task b's size, so that each panel
// covers only the prefix that still has one).
template <bool C>
cudaError_t chol_run(const CholBatch& B, int N, int n_mat, const int* Ns, int mode, cudaStream_t s, int* n_launch) {
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
  chol_first_kernel<C><<<n_mat, 256, 0, s>>>(B, INIT_BLOCKS);
  ++nl;
  const int sms = device_sm_count();
  int live = n_mat;
  for (int kb = 0; kb + CB < N; kb += CB) {
    while (Ns && live > 0 && Ns[live - 1] <= kb + CB) --live;
    const int m = N - kb - CB;
    // 16 rows per CTA while 64 would leave SMs idle (a CTA's rows queue on
    // its SM's FP64 pipe: 64 rows are 34 us, 16 are 9)
    const int per64 = (m + 63) / 64, per16 = (m + 15) / 16;
    if ((long)live * per64 >= 2L * sms)
      chol_panel_kernel<C, 8><<<(unsigned)(live * per64), 256, 0, s>>>(B, kb, per64);
    else
      chol_panel_kernel<C, 2><<<(unsigned)(live * per16), 64, 0, s>>>(B, kb, per16);
    const int nt = (m + CB - 1) / CB, per = nt * (nt + 1) / 2;
    if (mode == 2)
      chol_update_kernel<C, true><<<(unsigned)(live * per), 256, 0, s>>>(B, kb, per);
    else
      chol_update_kernel<C, false><<<(unsigned)(live * per), 256, 0, s>>>(B, kb, per);
    nl += 2;
  }
  if (n_launch) *n_launch = nl;
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_cholesky(int cplx, int N, int n_mat, double* mats, long bstride, int mode, double* out,
                            int* status, int status_base, cudaStream_t s, const double* Wn, const double* Vc,
                            const double* ldV, int n_w) {
  if (n_mat == 0) return cudaSuccess;
  if (mode == 2 && (!Wn || !Vc || !ldV || n_w <= 0)) return cudaErrorInvalidValue;
  if (mode != 1 && !out) return cudaErrorInvalidValue;
  const long nt = (N + CB - 1) / CB;
  if ((long)n_mat * std::max<long>(nt * (nt + 1) / 2, INIT_BLOCKS) > 0x7fffffffL) return cudaErrorInvalidValue;
  const CholBatch B{nullptr, mats, bstride, out, status, Wn, Vc, ldV, N, mode, status_base, std::max(n_w, 1)};
  return cplx ? chol_run<true>(B, N, n_mat, nullptr, mode, s, nullptr)
              : chol_run<false>(B, N, n_mat, nullptr, mode, s, nullptr);
}

int cholesky_launches(int N, int n_mat, int mode) {
  if (n_mat <= 0) return 0;
  if (N <= SMALL_N) return 1;
  return (mode != 0 ? 2 : 1) + 2 * ((N - 1) / CB);
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
    const cudaError_t e = cplx ? chol_run<true>(B, Ns[lo], n, Ns.data() + lo, mode, s, &nl)
                               : chol_run<false>(B, Ns[lo], n, Ns.data() + lo, mode, s, &nl);
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
  trinv_diag_kernel<C><<<n_q * nt, 128, 0, s>>>(N, L, X);
  for (int sz = CB; sz < N; sz *= 2) {
    const int tiles = (sz / CB) * (sz / CB), pairs = (N - sz + 2 * sz - 1) / (2 * sz);
    trinv_join_kernel<C, 0><<<n_q * pairs * tiles, 256, 0, s>>>(N, sz, L, X, tiles, pairs);
    trinv_join_kernel<C, 1><<<n_q * pairs * tiles, 256, 0, s>>>(N, sz, L, X, tiles, pairs);
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
