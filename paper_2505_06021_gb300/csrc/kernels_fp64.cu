// FP64 kernels of the RPA hot path on GB300 (sm_103a).
//
// GB300 executes FP64 at about 1/58 of its FP32 rate (1.2 TFLOP/s measured
// for DFMA and DGEMM), so every kernel here is bound by the FP64 pipe and is
// organised to issue as few FP64 instructions per useful result as possible.
// Larger chi0 and sandwich calls run as digit products on the tensor cores
// (g64.cu) and come here only for matrices those cannot hold (`only` flags).
//   * chi0: the product conj(C_P,t) C_Q,t is formed once per t and reused for
//     a group of G frequencies (2 DFMA per frequency instead of 4), and only
//     the lower triangle of tiles is computed (chi0 is Hermitian);
//   * the sandwich uses the Cholesky factor L of V (triangular operands, lower
//     output only) instead of the dense V^(1/2);
//   * the factorisation of 1 - Pi (cholesky.cu) keeps the diagonal in "pivot minus one"
//     form so that ln det = sum log1p(u) keeps its digits as Pi -> 0;
//   * the inverse form used with the split-precision chi0 needs no sandwich at
//     all: det(1 - V^(1/2) chi V^(1/2)) = det(V^-1 - chi) det V and
//     Tr(V^(1/2) chi V^(1/2)) = Tr(chi V), with V^-1 = X^H X, X = L^-1, formed
//     once per q.
// All reductions run in a fixed order, so results are bit-reproducible.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>

#include "fp64_elem.cuh"
#include "rpa_internal.h"

namespace rpa {
namespace {

// ---------------------------------------------------------------- helpers --

int num_sms_fp64() { return device_sm_count(); }

// Lower-triangular tile index -> (I, J), J <= I.
__device__ __forceinline__ void tri_index(int t, int& I, int& J) {
  int i = (int)((sqrt(8.0 * (double)t + 1.0) - 1.0) * 0.5);
  while ((i + 1) * (i + 2) / 2 <= t) ++i;
  while (i * (i + 1) / 2 > t) --i;
  I = i;
  J = t - i * (i + 1) / 2;
}

// ------------------------------------------------------------ d table -----

__global__ void dtab_kernel(BatchGeom g, const double* __restrict__ eps_occ, const double* __restrict__ eps_virt,
                            const int* __restrict__ kidx, const int* __restrict__ kqidx,
                            const double* __restrict__ omega, double zeta_k, double* __restrict__ dtab) {
  const long total = (long)g.n_qb * g.n_k * g.n_w * g.n_ov;
  for (long idx = blockIdx.x * (long)blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
    long r = idx;
    const int t = (int)(r % g.n_ov);
    r /= g.n_ov;
    const int w = (int)(r % g.n_w);
    r /= g.n_w;
    const int pair = (int)r;  // qb * n_k + j
    const int i = t / g.n_virt, a = t - i * g.n_virt;
    const double delta = eps_virt[(long)kqidx[pair] * g.n_virt + a] - eps_occ[(long)kidx[pair] * g.n_occ + i];
    const double om = omega[w];
    dtab[idx] = zeta_k * (-4.0 * delta / (delta * delta + om * om));
  }
}

// --------------------------------------------------------------- chi0 -----
// Grid: one CTA per (q in batch, lower tile pair (I, J), frequency group).
// Tile 16 U x 16 U outputs, 256 threads, each thread U x U outputs (rows
// ty + 16 u, columns tx + 16 v) for G frequencies.  An output's sum does not
// depend on U or G.

constexpr int TK = 16;  // t-chunk

template <bool C, int G, int U>
__global__ void __launch_bounds__(256, 1)
    chi0_fp64_kernel(BatchGeom g, const double* const* __restrict__ Cptrs, const double* __restrict__ dtab,
                     double* __restrict__ chi, int n_tiles, int n_wg, const int* __restrict__ only) {
  constexpr int CT = 16 * U;  // output tile edge
  __shared__ Elem<C> As[TK][CT];
  __shared__ Elem<C> Bs[TK][CT];
  __shared__ double Ds[G][TK];

  int bid = blockIdx.x;
  const int wg = bid % n_wg;
  bid /= n_wg;
  const int tile = bid % n_tiles;
  const int qb = bid / n_tiles;
  if (only && !(only[qb] & 1)) return;
  int I, J;
  tri_index(tile, I, J);
  const int w0 = wg * G;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int N = g.n_aux, n_ov = g.n_ov;

  Elem<C> acc[G][U * U];
#pragma unroll
  for (int k = 0; k < G; ++k)
#pragma unroll
    for (int m = 0; m < U * U; ++m) acc[k][m] = zero_elem<C>();

  for (int j = 0; j < g.n_k; ++j) {
    const double* Cj = Cptrs[qb * g.n_k + j];
    const double* dj = dtab + ((long)(qb * g.n_k + j) * g.n_w) * n_ov;
    for (int t0 = 0; t0 < n_ov; t0 += TK) {
      for (int idx = tid; idx < CT * TK; idx += 256) {
        const int r = idx / TK, tt = idx % TK, t = t0 + tt;
        const int P = I * CT + r, Q = J * CT + r;
        As[tt][r] = (P < N && t < n_ov) ? ld_elem<C>(Cj, (long)P * n_ov + t) : zero_elem<C>();
        Bs[tt][r] = (Q < N && t < n_ov) ? ld_elem<C>(Cj, (long)Q * n_ov + t) : zero_elem<C>();
      }
      for (int idx = tid; idx < G * TK; idx += 256) {
        const int k = idx / TK, tt = idx % TK, t = t0 + tt, w = w0 + k;
        Ds[k][tt] = (t < n_ov && w < g.n_w) ? dj[(long)w * n_ov + t] : 0.0;
      }
      __syncthreads();
#pragma unroll 4
      for (int tt = 0; tt < TK; ++tt) {
        // p = conj(a) * b
        Elem<C> p[U * U], aa[U], bb[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          aa[u] = As[tt][ty + 16 * u];
          bb[u] = Bs[tt][tx + 16 * u];
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int v = 0; v < U; ++v) {
            if constexpr (C) {
              p[U * u + v].re = fma(aa[u].re, bb[v].re, aa[u].im * bb[v].im);
              p[U * u + v].im = fma(aa[u].re, bb[v].im, -aa[u].im * bb[v].re);
            } else {
              p[U * u + v].re = aa[u].re * bb[v].re;
            }
          }
#pragma unroll
        for (int k = 0; k < G; ++k) {
          const double d = Ds[k][tt];
#pragma unroll
          for (int m = 0; m < U * U; ++m) {
            acc[k][m].re = fma(d, p[m].re, acc[k][m].re);
            if constexpr (C) acc[k][m].im = fma(d, p[m].im, acc[k][m].im);
          }
        }
      }
      __syncthreads();
    }
  }
  // write the lower triangle and its Hermitian mirror
  const long NN = (long)N * N;
#pragma unroll
  for (int k = 0; k < G; ++k) {
    const int w = w0 + k;
    if (w >= g.n_w) break;
    double* out = chi + ((long)qb * g.n_w + w) * NN * (C ? 2 : 1);
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int v = 0; v < U; ++v) {
        const int P = I * CT + ty + 16 * u, Q = J * CT + tx + 16 * v;
        if (P >= N || Q >= N || Q > P) continue;
        Elem<C> e = acc[k][U * u + v];
        if (P == Q) {
          if constexpr (C) e.im = 0.0;
          st_elem<C>(out, (long)P * N + Q, e);
        } else {
          st_elem<C>(out, (long)P * N + Q, e);
          st_elem<C>(out, (long)Q * N + P, conj_e<C>(e));
        }
      }
  }
}

template <bool C, int G, int U>
cudaError_t chi0_launch_g(const BatchGeom& g, const double* const* Cptrs, const double* dtab, double* chi,
                          cudaStream_t s, const int* only) {
  const int nt = (g.n_aux + 16 * U - 1) / (16 * U);
  const int n_tiles = nt * (nt + 1) / 2;
  const int n_wg = (g.n_w + G - 1) / G;
  const long blocks = (long)n_tiles * n_wg * g.n_qb;
  if (blocks > 0x7fffffffL) return cudaErrorInvalidConfiguration;
  chi0_fp64_kernel<C, G, U><<<(unsigned)blocks, 256, 0, s>>>(g, Cptrs, dtab, chi, n_tiles, n_wg, only);
  return cudaGetLastError();
}

// Tile edge and frequency group.  A CTA issues (4 + 2 G) FP64 instructions
// per complex (P, Q, t) (1 + G real) for G frequencies, and its SM's FP64
// pipe serves all CTAs that sit there, so the choice minimises the number of
// CTAs the fullest SM gets times a CTA's work: large groups share the product
// conj(C_P) C_Q when there is work for every SM, small tiles and groups spread
// a small response (a 32 x 32 tile of 8 frequencies holds the pipe for 4.6k
// clocks per 1000 real t).  Measured at N_aux 64, 112 t, 16 frequencies, real:
// 272 us with 32 x 32 tiles of 8 frequencies (6 CTAs), see the table in the
// design notes for the present time.
template <bool C>
cudaError_t chi0_dispatch(const BatchGeom& g, const double* const* Cptrs, const double* dtab, double* chi,
                          cudaStream_t s, const int* only) {
  const int Gs[6] = {10, 8, 5, 4, 2, 1};
  const long sms = num_sms_fp64();
  int bG = 8, bU = 2;
  double best = 1e300;
  for (int U = 2; U >= 1; --U)
    for (int G : Gs) {
      const long nt = (g.n_aux + 16 * U - 1) / (16 * U);
      const long blocks = nt * (nt + 1) / 2 * ((g.n_w + G - 1) / G) * g.n_qb;
      const double work = (C ? 4.0 + 2.0 * G : 1.0 + G) * U * U;
      // the last wave counts as a whole one while there are few
      const double waves = blocks >= 16 * sms ? (double)blocks / sms : (double)((blocks + sms - 1) / sms);
      const double cost = waves * work * (U == 1 ? 1.05 : 1.0);  // smaller tiles read the operands more often
      if (cost < best) {
        best = cost;
        bG = G;
        bU = U;
      }
    }
#define RPA_CHI0_G(G)                                                   \
  case G:                                                               \
    return bU == 2 ? chi0_launch_g<C, G, 2>(g, Cptrs, dtab, chi, s, only)     \
                   : chi0_launch_g<C, G, 1>(g, Cptrs, dtab, chi, s, only)
  switch (bG) {
    RPA_CHI0_G(10);
    RPA_CHI0_G(5);
    RPA_CHI0_G(4);
    RPA_CHI0_G(2);
    RPA_CHI0_G(1);
    default:
      return bU == 2 ? chi0_launch_g<C, 8, 2>(g, Cptrs, dtab, chi, s, only) : chi0_launch_g<C, 8, 1>(g, Cptrs, dtab, chi, s, only);
  }
#undef RPA_CHI0_G
}

// ----------------------------------------------------------- sandwich -----
// MODE 0: T = X L      (L lower triangular; K-range of output column tile J
//                       starts at J*64)
// MODE 1: Y = -L^H T   (lower output tiles only; K-range of row tile I starts
//                       at I*64)
// GT x GT output tile (64, 32 or 16), 256 threads, U x U outputs per thread,
// U = GT / 16.

constexpr int GK = 16;

template <bool C, int MODE, int U>
__global__ void __launch_bounds__(256)
    sandwich_kernel(int N, int n_w, const double* __restrict__ Xb, const double* __restrict__ Lb,
                    double* __restrict__ Ob, int n_tiles_row, int tiles_per_mat, const int* __restrict__ only) {
  constexpr int GT = 16 * U;
  __shared__ Elem<C> As[GK][GT];
  __shared__ Elem<C> Bs[GK][GT];
  const int b = blockIdx.x / tiles_per_mat;
  if (only && !(only[b] & 1)) return;
  const int tile = blockIdx.x % tiles_per_mat;
  int I, J;
  if (MODE == 0) {
    I = tile / n_tiles_row;
    J = tile % n_tiles_row;
  } else {
    tri_index(tile, I, J);
  }
  const long NN = (long)N * N;
  const int cs = C ? 2 : 1;
  const double* X = Xb + (long)b * NN * cs;
  const double* L = Lb + (long)(b / n_w) * NN * cs;
  double* O = Ob + (long)b * NN * cs;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;

  Elem<C> acc[U][U];
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < U; ++v) acc[u][v] = zero_elem<C>();

  const int k_begin = (MODE == 0 ? J : I) * GT;
  for (int k0 = k_begin; k0 < N; k0 += GK) {
    for (int idx = tid; idx < GK * GT; idx += 256) {
      if (MODE == 0) {
        // A = X[P][R] (row-major, R contiguous): idx -> (p, kk) with kk fastest
        const int p = idx / GK, kk = idx % GK, P = I * GT + p, R = k0 + kk;
        As[kk][p] = (P < N && R < N) ? ld_elem<C>(X, (long)P * N + R) : zero_elem<C>();
        // B = L[R][Q], zero above the diagonal (R < Q)
        const int q = idx % GT, kb = idx / GT, Q = J * GT + q, R2 = k0 + kb;
        Bs[kb][q] = (Q < N && R2 < N && R2 >= Q) ? ld_elem<C>(L, (long)R2 * N + Q) : zero_elem<C>();
      } else {
        // A[P][R] = conj(L[R][P]), zero for R < P; read L rows R, P contiguous
        const int p = idx % GT, kk = idx / GT, P = I * GT + p, R = k0 + kk;
        As[kk][p] = (P < N && R < N && R >= P) ? conj_e<C>(ld_elem<C>(L, (long)R * N + P)) : zero_elem<C>();
        const int q = idx % GT, Q = J * GT + q;
        Bs[kk][q] = (Q < N && R < N) ? ld_elem<C>(X, (long)R * N + Q) : zero_elem<C>();
      }
    }
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < GK; ++kk) {
      Elem<C> a[U], bv[U];
#pragma unroll
      for (int u = 0; u < U; ++u) a[u] = As[kk][ty + 16 * u];
#pragma unroll
      for (int v = 0; v < U; ++v) bv[v] = Bs[kk][tx + 16 * v];
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = 0; v < U; ++v) mac<C>(acc[u][v], a[u], bv[v]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < U; ++v) {
      const int P = I * GT + ty + 16 * u, Q = J * GT + tx + 16 * v;
      if (P >= N || Q >= N) continue;
      Elem<C> e = acc[u][v];
      if (MODE == 1) {
        e.re = -e.re;
        if constexpr (C) e.im = -e.im;
      }
      st_elem<C>(O, (long)P * N + Q, e);
    }
}

// ------------------------------------------------------------- energy -----

__global__ void energy_kernel(int n_q, int n_w, const double* __restrict__ parts, const double* __restrict__ w_q,
                              const double* __restrict__ zeta_w, double* __restrict__ eps, double* __restrict__ Ec) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  // Neumaier-compensated sums in a fixed order: q inside, frequency outside.
  double E = 0.0, Ec_c = 0.0;
  for (int w = 0; w < n_w; ++w) {
    double e = 0.0, c = 0.0;
    for (int q = 0; q < n_q; ++q) {
      const double v = parts[2 * ((long)q * n_w + w)] + parts[2 * ((long)q * n_w + w) + 1];
      eps[(long)q * n_w + w] = v;
      const double x = w_q[q] * v;
      const double t = e + x;
      c += (fabs(e) >= fabs(x)) ? (e - t) + x : (x - t) + e;
      e = t;
    }
    const double x = zeta_w[w] * (e + c);
    const double t = E + x;
    Ec_c += (fabs(E) >= fabs(x)) ? (E - t) + x : (x - t) + E;
    E = t;
  }
  *Ec = (E + Ec_c) / (2.0 * M_PI);
}

}  // namespace

// ------------------------------------------------------------ launchers ----

cudaError_t launch_dtab(const BatchGeom& g, const double* eps_occ, const double* eps_virt, const int* kidx,
                        const int* kqidx, const double* omega, double zeta_k, double* dtab, cudaStream_t s) {
  const long total = (long)g.n_qb * g.n_k * g.n_w * g.n_ov;
  if (total == 0) return cudaSuccess;
  const long blocks = std::min<long>((total + 255) / 256, 152L * 16);
  dtab_kernel<<<(unsigned)blocks, 256, 0, s>>>(g, eps_occ, eps_virt, kidx, kqidx, omega, zeta_k, dtab);
  return cudaGetLastError();
}

cudaError_t launch_chi0_fp64(const BatchGeom& g, const double* const* Cptrs, const double* dtab, double* chi,
                             cudaStream_t s, const int* only) {
  return g.cplx ? chi0_dispatch<true>(g, Cptrs, dtab, chi, s, only) : chi0_dispatch<false>(g, Cptrs, dtab, chi, s, only);
}

namespace {
template <bool C, int MODE, int U>
cudaError_t sandwich_pass_u(int N, int n_batch, int n_w, const double* X, const double* L, double* O, cudaStream_t s,
                            const int* only) {
  const int nt = (N + 16 * U - 1) / (16 * U);
  const int per = MODE == 0 ? nt * nt : nt * (nt + 1) / 2;
  if ((long)n_batch * per > 0x7fffffffL) return cudaErrorInvalidValue;
  sandwich_kernel<C, MODE, U><<<(unsigned)(n_batch * per), 256, 0, s>>>(N, n_w, X, L, O, nt, per, only);
  return cudaGetLastError();
}

// One triangular product.  Every tile size issues the same FP64 instructions,
// and one 64 x 64 tile of N = 768 keeps an SM's FP64 pipe busy for 3 ms, so the
// largest tile (fewest operand reads) is taken that still gives every SM two
// CTAs to balance.
template <bool C, int MODE>
cudaError_t sandwich_pass(int N, int n_batch, int n_w, const double* X, const double* L, double* O, cudaStream_t s,
                            const int* only) {
  const long sms = num_sms_fp64();
  auto blocks = [&](int gt) {
    const long nt = (N + gt - 1) / gt;
    return n_batch * (MODE == 0 ? nt * nt : nt * (nt + 1) / 2);
  };
  if (blocks(64) >= 4 * sms) return sandwich_pass_u<C, MODE, 4>(N, n_batch, n_w, X, L, O, s, only);
  if (blocks(32) >= 2 * sms) return sandwich_pass_u<C, MODE, 2>(N, n_batch, n_w, X, L, O, s, only);
  return sandwich_pass_u<C, MODE, 1>(N, n_batch, n_w, X, L, O, s, only);
}
}  // namespace

cudaError_t launch_sandwich(int cplx, int N, int n_batch, int n_w, const double* chi, const double* L, double* T,
                            double* Y, cudaStream_t s, const int* only) {
  if (n_batch == 0) return cudaSuccess;
  if (cplx) {
    if (cudaError_t e = sandwich_pass<true, 0>(N, n_batch, n_w, chi, L, T, s, only)) return e;
    return sandwich_pass<true, 1>(N, n_batch, n_w, T, L, Y, s, only);
  }
  if (cudaError_t e = sandwich_pass<false, 0>(N, n_batch, n_w, chi, L, T, s, only)) return e;
  return sandwich_pass<false, 1>(N, n_batch, n_w, T, L, Y, s, only);
}

cudaError_t launch_gram(int cplx, int N, int n_q, const double* X, double* Wn, cudaStream_t s, const int* only) {
  return cplx ? sandwich_pass<true, 1>(N, n_q, 1, X, X, Wn, s, only)
              : sandwich_pass<false, 1>(N, n_q, 1, X, X, Wn, s, only);
}

cudaError_t launch_energy_reduce(int n_q, int n_w, const double* parts, const double* w_q, const double* zeta_w,
                                 double* eps, double* Ec, cudaStream_t s) {
  energy_kernel<<<1, 32, 0, s>>>(n_q, n_w, parts, w_q, zeta_w, eps, Ec);
  return cudaGetLastError();
}

__global__ void __launch_bounds__(256) copy16_kernel(uint4* __restrict__ dst, const uint4* __restrict__ src, long n) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) dst[i] = src[i];
}

cudaError_t launch_copy_d2d(void* dst, const void* src, size_t bytes, cudaStream_t s, uint64_t* n_launch) {
  if (bytes == 0) return cudaSuccess;
  if (bytes % 16 || (uintptr_t)dst % 16 || (uintptr_t)src % 16)
    return cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToDevice, s);
  const long n = (long)(bytes / 16);
  const unsigned blocks = (unsigned)std::min<long>((n + 255) / 256, (long)num_sms_fp64() * 8);
  copy16_kernel<<<blocks, 256, 0, s>>>((uint4*)dst, (const uint4*)src, n);
  if (n_launch) ++*n_launch;
  return cudaGetLastError();
}

}  // namespace rpa
