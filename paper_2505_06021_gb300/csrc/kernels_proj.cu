// Periodic projector (Sec. 2.3) on GB300: S(k) = U D U^H, R(k) = Theta(D(k) -
// eps_d), R~ = prod_k R(k), T(k) = U(k) R~ U(k)^H, c~(k) = T(k) c(k).
//
// Eigendecomposition: one-sided (Hestenes) Jacobi on the columns of W = S(k),
// all k-points of the job in every launch.  Orthogonalising the columns of
// a Hermitian positive definite S by rotations V gives S V = W = U D: the
// eigenvalues are the column norms of W, the eigenvectors the columns of V
// (accumulated alongside, orthonormal to rounding and accurate to
// eps/gap even for the tiny eigenvalues the projector removes).  A sweep is
// Np - 1 rounds of the round-robin (circle) ordering of Np columns (Np = N
// rounded up to even, a zero padding column); a round rotates Np/2 disjoint
// column pairs, a CTA or a warp per (k-point, pair), so a launch has no
// inter-CTA dependency and a round is one kernel launch.  Per pair: alpha =
// |w_p|^2, beta = |w_q|^2, gamma = w_p^H w_q; with
// e = conj(gamma)/|gamma|, zeta = (beta - alpha)/(2|gamma|),
// t = sign(zeta)/(|zeta| + sqrt(1 + zeta^2)), c = 1/sqrt(1 + t^2), s = c t:
//   w_p <- c w_p - s e w_q,   w_q <- s w_p + c e w_q,
// which makes the pair orthogonal (the 2 x 2 Hermitian Jacobi rotation).  The
// largest |gamma|/sqrt(alpha beta) of a sweep decides convergence on the host.
//
// Start of the iteration (proj.cu, bases of some size): the sweeps above begin
// from eigenvectors of nearly full accuracy instead of I.  One-sided Jacobi in FP32
// (its pipe is 64 times the FP64 one; in shared memory, 32 columns at a time)
// gives them to about 1e-6; they are
// refined by matrix products on the tensor cores (g64.cu): Newton-Schulz steps
// V <- V - V (V^H V - I) / 2 for orthonormality, and first-order corrections
// V <- V + V E, E_ij = (V^H S V)_ij / (lambda_j - lambda_i) where that is small (the
// quadratically convergent refinement of Ogita and Aishima, 2018, without its
// cluster step).  Then the columns of W = S V are made orthogonal to rounding by
// the same first-order rotations from G = W^H W (whose entries are accurate
// relative to both columns, so this holds for the tiny eigenvalues too), and the
// few pairs that need large rotations are rotated one by one; where G still
// shows a cosine above 1e-14, the FP64 sweeps finish.  Measured, 16 overlaps of 256
// functions: 0.7 ms of products stand for three FP64 sweeps of 255 rounds (23 us each,
// 17.8 ms), 13.1 ms in all instead of 29.9; the most of it is the FP32 sweeps
// (7 ms) and the refinement's products.
//
// Since the eigenvalues are taken in ascending order and R~ is a product over
// k, R~ removes the m lowest positions at every k-point, m the largest count
// of eigenvalues below eps_d; T(k) c = c - U_m (U_m^H c), U_m the m lowest
// eigenvectors of S(k).
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <mutex>

#include "fp64_elem.cuh"
#include "rpa_internal.h"

namespace rpa {
namespace {

__device__ __forceinline__ void round_pair(int n, int r, int i, int& p, int& q) {
  if (i == 0) {
    p = 0;
    q = 1 + (r % (n - 1));
  } else {
    p = 1 + ((r + i) % (n - 1));
    q = 1 + ((r + n - 1 - i) % (n - 1));
  }
}

// W[k][j][mu] = S(k)[mu][j] = conj(S(k)[j][mu]) (S Hermitian), V[k] = I;
// padding columns j >= N are zero in both.
template <bool C>
__global__ void __launch_bounds__(256) proj_load_kernel(ProjPtrs P, int N, int Np, double* __restrict__ W,
                                                        double* __restrict__ V) {
  const int k = blockIdx.y, j = blockIdx.x;
  const double* S = P.S[k];
  double* w = W + ((size_t)k * Np + j) * N * (C ? 2 : 1);
  double* v = V + ((size_t)k * Np + j) * N * (C ? 2 : 1);
  for (int mu = threadIdx.x; mu < N; mu += blockDim.x) {
    Elem<C> e = j < N ? conj_e<C>(ld_elem<C>(S, (long)j * N + mu)) : zero_elem<C>();
    st_elem<C>(w, mu, e);
    Elem<C> one = zero_elem<C>();
    one.re = (mu == j) ? 1.0 : 0.0;
    st_elem<C>(v, mu, one);
  }
}

// x <- c x - s e y, y <- s x + c e y for element mu of columns x, y.
template <bool C>
__device__ __forceinline__ void rotate_pair(double* xc, double* yc, int mu, double c, double s, double er, double ei) {
  const Elem<C> x = ld_elem<C>(xc, mu), y = ld_elem<C>(yc, mu);
  Elem<C> xn, yn;
  if constexpr (C) {
    const double eyr = er * y.re - ei * y.im, eyi = er * y.im + ei * y.re;
    xn.re = c * x.re - s * eyr;
    xn.im = c * x.im - s * eyi;
    yn.re = s * x.re + c * eyr;
    yn.im = s * x.im + c * eyi;
  } else {
    xn.re = c * x.re - s * er * y.re;
    yn.re = s * x.re + c * er * y.re;
  }
  st_elem<C>(xc, mu, xn);
  st_elem<C>(yc, mu, yn);
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The 2 x 2 rotation that makes columns with norms^2 a, b and inner product g
// orthogonal: c, s, e = conj(g)/|g|.
__device__ __forceinline__ void pair_rotation(double a, double b, double gr, double gi, double g, double& c, double& s,
                                              double& er, double& ei) {
  const double zeta = (b - a) / (2.0 * g);
  const double t = (zeta >= 0.0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
  c = 1.0 / sqrt(1.0 + t * t);
  s = c * t;
  er = gr / g;
  ei = -gi / g;
}

// |x|^2, |y|^2, conj(x) y over this thread's share of two columns.
template <bool C>
__device__ __forceinline__ void pair_dots(const double* xc, const double* yc, int N, int first, int step, double& a,
                                          double& b, double& gr, double& gi) {
  a = b = gr = gi = 0.0;
  for (int mu = first; mu < N; mu += step) {
    const Elem<C> x = ld_elem<C>(xc, mu), y = ld_elem<C>(yc, mu);
    if constexpr (C) {
      a = fma(x.re, x.re, fma(x.im, x.im, a));
      b = fma(y.re, y.re, fma(y.im, y.im, b));
      gr = fma(x.re, y.re, fma(x.im, y.im, gr));  // conj(x) y
      gi = fma(x.re, y.im, fma(-x.im, y.re, gi));
    } else {
      a = fma(x.re, x.re, a);
      b = fma(y.re, y.re, b);
      gr = fma(x.re, y.re, gr);
    }
  }
  a = warp_sum(a);
  b = warp_sum(b);
  gr = warp_sum(gr);
  if constexpr (C) gi = warp_sum(gi);
}

// The rotation of a CTA's column pair from its warps' sums, by thread 0 alone: its
// roots, divisions and sums are FP64 instructions of one warp (64 clocks of a
// sub-partition each, however few lanes take part), and seven more warps that
// repeat them would share the same four pipes.  rot: c, s, e (re, im), 1 if the
// cosine is above thresh; returns the cosine (thread 0), 0 elsewhere.  off_max (or null)
// takes the cosine before the rotation is computed.
__device__ __forceinline__ double cta_rotation(double (*red)[4], double* rot, double a, double b, double gr, double gi,
                                               double thresh, unsigned long long* off_max) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double off = 0.0;
  if (lane == 0) {
    red[wid][0] = a;
    red[wid][1] = b;
    red[wid][2] = gr;
    red[wid][3] = gi;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    a = b = gr = gi = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      a += red[w][0];
      b += red[w][1];
      gr += red[w][2];
      gi += red[w][3];
    }
    const double g = sqrt(gr * gr + gi * gi);
    off = (a > 0.0 && b > 0.0) ? g / sqrt(a * b) : 0.0;
    if (off_max) atomicMax(off_max, (unsigned long long)__double_as_longlong(off));
    if (off > thresh) {
      double c, s, er, ei;
      pair_rotation(a, b, gr, gi, g, c, s, er, ei);
      rot[0] = c;
      rot[1] = s;
      rot[2] = er;
      rot[3] = ei;
      rot[4] = 1.0;
    } else {
      rot[4] = 0.0;
    }
  }
  __syncthreads();
  return off;
}

// One round r: columns (p, q) of pair i of W[k] are rotated, by a CTA each
// (WARP = false) or, when the pairs of all k-points fill the GPU, by a warp each,
// four to a CTA: no barriers, and once most pairs are orthogonal a round is
// the FP64 pipe's time for the inner products.  Calls on 63 functions and 1, 9 and
// 16 k-points: 7.1, 8.6 and 12 ms (9.7, 17.2 and 29.8 with the rotation in all eight
// warps of the CTA).
template <bool C, bool WARP>
__global__ void __launch_bounds__(WARP ? 128 : 256) jacobi_round_kernel(int N, int Np, int r, double* __restrict__ W,
                                                                        double* __restrict__ V, double thresh,
                                                                        unsigned long long* __restrict__ off_max) {
  __shared__ double red[8][4], rot[5];
  const int lane = threadIdx.x & 31, k = blockIdx.y;
  const int i = WARP ? blockIdx.x * 4 + (threadIdx.x >> 5) : blockIdx.x;
  if (i >= Np / 2) return;
  int p, q;
  round_pair(Np, r, i, p, q);
  double* wp = W + ((size_t)k * Np + p) * N * (C ? 2 : 1);
  double* wq = W + ((size_t)k * Np + q) * N * (C ? 2 : 1);
  const int first = WARP ? lane : threadIdx.x, step = WARP ? 32 : 256;
  double a, b, gr, gi, c, s, er, ei;
  pair_dots<C>(wp, wq, N, first, step, a, b, gr, gi);
  if constexpr (WARP) {
    const double g = sqrt(gr * gr + gi * gi);
    const double off = (a > 0.0 && b > 0.0) ? g / sqrt(a * b) : 0.0;
    if (first == 0) atomicMax(off_max, (unsigned long long)__double_as_longlong(off));
    if (!(off > thresh)) return;
    pair_rotation(a, b, gr, gi, g, c, s, er, ei);
  } else {
    cta_rotation(red, rot, a, b, gr, gi, thresh, off_max);
    if (rot[4] == 0.0) return;
    c = rot[0];
    s = rot[1];
    er = rot[2];
    ei = rot[3];
  }
  double* vp = V + ((size_t)k * Np + p) * N * (C ? 2 : 1);
  double* vq = V + ((size_t)k * Np + q) * N * (C ? 2 : 1);
  for (int mu = first; mu < N; mu += step) {
    rotate_pair<C>(wp, wq, mu, c, s, er, ei);
    rotate_pair<C>(vp, vq, mu, c, s, er, ei);
  }
}

// The few columns that the refinement could not tell apart (the eigenvalues
// far below FP32's resolution, near-degenerate ones): those with a cosine
// above 1e-14 in G = W^H W (above 1e-3 where they are too many), swept among
// themselves, one CTA per k-point.  More than CLUSTER_MAX are left to the sweeps
// over all columns.
constexpr int CLUSTER_MAX = 24;
template <bool C>
__global__ void __launch_bounds__(256) proj_cluster_kernel(int N, int Np, const double* __restrict__ G,
                                                           double* __restrict__ W, double* __restrict__ V,
                                                           double thresh) {
  __shared__ double red[8][4], rot[5], offs;
  __shared__ int list[CLUSTER_MAX], cnt;
  extern __shared__ unsigned char mark[];
  const int k = blockIdx.x, tid = threadIdx.x;
  const double* g = G + (size_t)k * N * N * (C ? 2 : 1);
  for (int j = tid; j < N; j += 256) mark[j] = 0;
  __syncthreads();
  for (int j = 0; j < N; ++j) {
    const double gj = ld_elem<C>(g, (long)j * N + j).re;
    for (int i = tid; i < N; i += 256) {
      if (i == j) continue;
      const Elem<C> x = ld_elem<C>(g, (long)j * N + i);
      double v = x.re * x.re;
      if constexpr (C) v += x.im * x.im;
      const double gg = gj * ld_elem<C>(g, (long)i * N + i).re;
      if (v > 1e-28 * gg) mark[i] |= v > 1e-6 * gg ? 3 : 1;  // (j is marked as i's partner)
    }
  }
  __syncthreads();
  if (tid == 0) {
    int n = 0;
    for (int bits = 1; bits <= 3; bits += 2) {
      n = 0;
      for (int j = 0; j < N; ++j)
        if ((mark[j] & bits) == bits) {
          if (n < CLUSTER_MAX) list[n] = j;
          ++n;
        }
      if (n <= CLUSTER_MAX) break;
    }
    cnt = n;
  }
  __syncthreads();
  if (cnt < 2 || cnt > CLUSTER_MAX) return;
  double* wk = W + (size_t)k * Np * N * (C ? 2 : 1);
  double* vk = V + (size_t)k * Np * N * (C ? 2 : 1);
  for (int sweep = 0; sweep < 12; ++sweep) {
    double worst = 0.0;
    for (int u = 0; u < cnt; ++u)
      for (int v = u + 1; v < cnt; ++v) {
        const long op = (long)list[u] * N * (C ? 2 : 1), oq = (long)list[v] * N * (C ? 2 : 1);
        double a, b, gr, gi;
        pair_dots<C>(wk + op, wk + oq, N, tid, 256, a, b, gr, gi);
        worst = fmax(worst, cta_rotation(red, rot, a, b, gr, gi, thresh, nullptr));
        const double c = rot[0], s = rot[1], er = rot[2], ei = rot[3];
        const bool turn = rot[4] != 0.0;
        __syncthreads();  // rot and red are free again
        if (!turn) continue;
        for (int mu = tid; mu < N; mu += 256) {  // a thread's own elements: no barrier between pairs
          rotate_pair<C>(wk + op, wk + oq, mu, c, s, er, ei);
          rotate_pair<C>(vk + op, vk + oq, mu, c, s, er, ei);
        }
      }
    if (tid == 0) offs = worst;
    __syncthreads();
    if (offs <= 1e-14) break;
  }
}

// ---- FP32 start ----

template <bool C>
struct Flt;
template <>
struct Flt<true> {
  float re, im;
};
template <>
struct Flt<false> {
  float re;
};

// Sum of squares of S(k) (W, N columns of N), one CTA per k-point, fixed order, and
// from it the scale of the FP32 start.  Columns of a root mean square norm outside
// [2^-50, 2^60] get a NaN, which rejects the start: beyond it the FP32 sum or the digit
// products' range may not hold S.
template <bool C>
__global__ void __launch_bounds__(256) proj_norm_kernel(int N, int Np, const double* __restrict__ W,
                                                        float* __restrict__ scale) {
  __shared__ double red[8];
  const double* w = W + (size_t)blockIdx.x * Np * N * (C ? 2 : 1);
  const long n = (long)N * N * (C ? 2 : 1);
  float s = 0.f;
  for (long i = threadIdx.x; i < n; i += 256) {
    const float x = (float)w[i];
    s = fmaf(x, x, s);
  }
  const double t = warp_sum((double)s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
  __syncthreads();
  if (threadIdx.x == 0) {
    double u = 0.0;
    for (int i = 0; i < 8; ++i) u += red[i];
    const double norm = sqrt(u / N);
    scale[blockIdx.x] = norm >= 0x1p-50 && norm <= 0x1p60 ? (float)(1.0 / norm) : __int_as_float(0x7fffffff);
  }
}

// W32 = scale S, V32 = I (Np columns of N each, as in FP64).
template <bool C>
__global__ void __launch_bounds__(256) proj_load32_kernel(int N, int Np, const double* __restrict__ W,
                                                          const float* __restrict__ scale, float* __restrict__ W32,
                                                          float* __restrict__ V32) {
  const int k = blockIdx.y, j = blockIdx.x;
  const size_t c0 = ((size_t)k * Np + j) * N * (C ? 2 : 1);
  const float sc = scale[k];
  for (int i = threadIdx.x; i < N * (C ? 2 : 1); i += blockDim.x) {
    W32[c0 + i] = (float)W[c0 + i] * sc;
    V32[c0 + i] = i == (C ? 2 : 1) * j ? 1.f : 0.f;
  }
}

// Rotates columns p, q of W and V (N elements each), by one warp, where their
// cosine is above thresh; returns the cosine.  Columns below 1e-6 of the typical
// norm (FP32 noise) count as that long.
template <bool C>
__device__ __forceinline__ float rotate32(Flt<C>* wp, Flt<C>* wq, Flt<C>* vp, Flt<C>* vq, int N, float thresh) {
  const int lane = threadIdx.x & 31;
  float a = 0.f, b = 0.f, gr = 0.f, gi = 0.f;
#pragma unroll 4
  for (int mu = lane; mu < N; mu += 32) {
    const Flt<C> x = wp[mu], y = wq[mu];
    a = fmaf(x.re, x.re, a);
    b = fmaf(y.re, y.re, b);
    gr = fmaf(x.re, y.re, gr);
    if constexpr (C) {
      a = fmaf(x.im, x.im, a);
      b = fmaf(y.im, y.im, b);
      gr = fmaf(x.im, y.im, gr);
      gi = fmaf(x.re, y.im, fmaf(-x.im, y.re, gi));
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
    gr += __shfl_xor_sync(0xffffffffu, gr, o);
    if constexpr (C) gi += __shfl_xor_sync(0xffffffffu, gi, o);
  }
  const float g = sqrtf(gr * gr + gi * gi);
  const float off = g / sqrtf(fmaxf(a, 1e-12f) * fmaxf(b, 1e-12f));
  if (!(off > thresh)) return off;  // (a NaN ends here too: the start is then rejected)
  const float zeta = (b - a) / (2.f * g);
  const float t = (zeta >= 0.f ? 1.f : -1.f) / (fabsf(zeta) + sqrtf(1.f + zeta * zeta));
  const float c = rsqrtf(1.f + t * t), s = c * t, er = gr / g, ei = -gi / g;
  auto rot = [&](Flt<C>* xc, Flt<C>* yc) {
#pragma unroll 4
    for (int mu = lane; mu < N; mu += 32) {
      const Flt<C> x = xc[mu], y = yc[mu];
      Flt<C> xn, yn;
      if constexpr (C) {
        const float eyr = er * y.re - ei * y.im, eyi = er * y.im + ei * y.re;
        xn.re = c * x.re - s * eyr;
        xn.im = c * x.im - s * eyi;
        yn.re = s * x.re + c * eyr;
        yn.im = s * x.im + c * eyi;
      } else {
        xn.re = c * x.re - s * er * y.re;
        yn.re = s * x.re + c * er * y.re;
      }
      xc[mu] = xn;
      yc[mu] = yn;
    }
  };
  rot(wp, wq);
  rot(vp, vq);
  return off;
}

// A block round of the FP32 sweeps: a CTA takes two blocks of B columns of W
// and V of one k-point into shared memory, rotates every pair across them (B
// rounds of B disjoint pairs, a warp each) and writes them back; the first block
// round of a sweep also rotates the pairs within the blocks (2 B - 1 rounds).  A
// sweep then reads and writes the columns nb - 1 times, not Np - 1, and has as
// many launches (nb blocks).  What bounds a round inside the CTA is each warp's
// chain of loads, sums and rotation (2.8 us; shared memory 44 % and issue 47 %
// busy).  Sweeps of 16 overlaps of 256 functions: 21 ms less than with a launch per
// round in global memory.
template <bool C, int B>
__global__ void __launch_bounds__(32 * B) jacobi32_block_kernel(int N, int Np, int nb, int br, float* __restrict__ W32,
                                                                float* __restrict__ V32, float thresh,
                                                                unsigned* __restrict__ off_max) {
  extern __shared__ __align__(16) float cols32[];
  __shared__ unsigned worst;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const size_t m0 = (size_t)blockIdx.y * Np * N;
  Flt<C>* w = reinterpret_cast<Flt<C>*>(cols32);  // 2 B columns of W, then of V
  Flt<C>* v = w + (size_t)2 * B * N;
  Flt<C>* wg = reinterpret_cast<Flt<C>*>(W32) + m0;
  Flt<C>* vg = reinterpret_cast<Flt<C>*>(V32) + m0;
  int bp, bq;
  round_pair(nb, br, blockIdx.x, bp, bq);
  const Flt<C> zero{};
  if (threadIdx.x == 0) worst = 0;
#pragma unroll
  for (int h = 0; h < 2; ++h) {  // (columns past Np count as zero: never rotated)
    const int col = (h ? bq : bp) * B + wid, lc = h * B + wid;
#pragma unroll 4
    for (int mu = lane; mu < N; mu += 32) {
      w[(size_t)lc * N + mu] = col < Np ? wg[(size_t)col * N + mu] : zero;
      v[(size_t)lc * N + mu] = col < Np ? vg[(size_t)col * N + mu] : zero;
    }
  }
  __syncthreads();
  const int rounds = br == 0 ? 2 * B - 1 : B;
  unsigned mine = 0;
  for (int r = 0; r < rounds; ++r) {
    int p = wid, q = B + (wid + r) % B;
    if (br == 0) round_pair(2 * B, r, wid, p, q);
    const float off = rotate32<C>(w + (size_t)p * N, w + (size_t)q * N, v + (size_t)p * N, v + (size_t)q * N, N, thresh);
    mine = max(mine, __float_as_uint(off));
    __syncthreads();
  }
  if (lane == 0) atomicMax(&worst, mine);
  __syncthreads();
  if (threadIdx.x == 0) atomicMax(off_max, worst);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int col = (h ? bq : bp) * B + wid, lc = h * B + wid;
    if (col < Np)
#pragma unroll 4
      for (int mu = lane; mu < N; mu += 32) {
        wg[(size_t)col * N + mu] = w[(size_t)lc * N + mu];
        vg[(size_t)col * N + mu] = v[(size_t)lc * N + mu];
      }
  }
}

// One round of the FP32 sweeps on columns too long for that: a warp per column
// pair and k-point, in global memory.
template <bool C>
__global__ void __launch_bounds__(128) jacobi32_round_kernel(int N, int Np, int r, float* __restrict__ W32,
                                                             float* __restrict__ V32, float thresh,
                                                             unsigned* __restrict__ off_max) {
  const int i = blockIdx.x * 4 + (threadIdx.x >> 5);
  if (i >= Np / 2) return;
  int p, q;
  round_pair(Np, r, i, p, q);
  const size_t m0 = (size_t)blockIdx.y * Np * N;
  Flt<C>* w = reinterpret_cast<Flt<C>*>(W32) + m0;
  Flt<C>* v = reinterpret_cast<Flt<C>*>(V32) + m0;
  const float off = rotate32<C>(w + (size_t)p * N, w + (size_t)q * N, v + (size_t)p * N, v + (size_t)q * N, N, thresh);
  if ((threadIdx.x & 31) == 0) atomicMax(off_max, __float_as_uint(off));
}

__global__ void __launch_bounds__(256) proj_widen_kernel(long n, const float* __restrict__ x, double* __restrict__ y) {
  for (long i = blockIdx.x * 256L + threadIdx.x; i < n; i += gridDim.x * 256L) y[i] = (double)x[i];
}

// In place over column j of M(k) (N x N at a stride N^2): ORTHO: -(M - I) / 2,
// the largest |M - I| into *dev; else the correction
// E_ij = M_ij / (M_jj - M_ii) where it is below lim, zero elsewhere (diag: the
// M_ii, saved before the launch), and the largest |M_ij| / sqrt(M_ii M_jj)
// into *dev.
template <bool C, bool ORTHO>
__global__ void __launch_bounds__(256) proj_corr_kernel(int N, double* __restrict__ M, const double* __restrict__ diag,
                                                        float lim, unsigned* __restrict__ dev) {
  const int k = blockIdx.y, j = blockIdx.x;
  double* col = M + ((size_t)k * N + j) * N * (C ? 2 : 1);
  const double lj = ORTHO ? 0.0 : diag[(size_t)k * N + j], inv = ORTHO ? 0.0 : 1.0 / lj;
  float dm = 0.f;
  bool bad = false;
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    Elem<C> e = ld_elem<C>(col, i);
    double f;
    if constexpr (ORTHO) {
      if (i == j) e.re -= 1.0;
      f = -0.5;
      float v = fabsf((float)e.re);
      if constexpr (C) v = fmaxf(v, fabsf((float)e.im));
      dm = fmaxf(dm, v);
      bad |= !(v < 1e30f);
    } else {
      // (relative to M_jj, so that the FP32 range holds any scale of M)
      const double li = diag[(size_t)k * N + i], gap = lj - li;
      float v = fabsf((float)(e.re * inv));
      if constexpr (C) v = fmaxf(v, fabsf((float)(e.im * inv)));
      f = i != j && v < lim * fabsf((float)(gap * inv)) ? 1.0 / gap : 0.0;
      if (i != j) {
        const float c = v * rsqrtf((float)(li * inv));
        dm = fmaxf(dm, c);
        bad |= !(c < 1e30f);
      }
    }
    e.re *= f;
    if constexpr (C) e.im *= f;
    st_elem<C>(col, i, e);
  }
  if (bad) dm = __int_as_float(0x7f800000);
  dm = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(dm)));
  if ((threadIdx.x & 31) == 0) atomicMax(dev, __float_as_uint(dm));
}

template <bool C>
__global__ void __launch_bounds__(256) proj_diag_kernel(int N, const double* __restrict__ M, double* __restrict__ diag) {
  const int k = blockIdx.y, i = blockIdx.x * 256 + threadIdx.x;
  if (i < N) diag[(size_t)k * N + i] = ld_elem<C>(M + (size_t)k * N * N * (C ? 2 : 1), (long)i * N + i).re;
}

// Per k-point: eigenvalue of column j = |w_j|, ascending rank (ties by index),
// count below eps_d (into m by atomicMax); lam_sorted[k][rank] and
// by_rank[k][rank] = j for the N real columns.
template <bool C>
__global__ void __launch_bounds__(256) proj_rank_kernel(int N, int Np, const double* __restrict__ W, double eps_d,
                                                        double* __restrict__ lam_sorted, int* __restrict__ by_rank,
                                                        int* __restrict__ m) {
  extern __shared__ double lam[];
  const int k = blockIdx.x;
  for (int j = threadIdx.x; j < Np; j += blockDim.x) {
    const double* w = W + ((size_t)k * Np + j) * N * (C ? 2 : 1);
    double s = 0.0;
    for (int mu = 0; mu < N; ++mu) {
      const Elem<C> x = ld_elem<C>(w, mu);
      s = fma(x.re, x.re, s);
      if constexpr (C) s = fma(x.im, x.im, s);
    }
    lam[j] = sqrt(s);
  }
  __syncthreads();
  int below = 0;
  for (int j = threadIdx.x; j < Np; j += blockDim.x) {
    // the padding column (zero) is not an eigenvector of S
    if (j >= N) continue;
    int rank = 0;
    for (int l = 0; l < N; ++l) rank += (lam[l] < lam[j]) || (lam[l] == lam[j] && l < j);
    lam_sorted[(size_t)k * N + rank] = lam[j];
    by_rank[(size_t)k * N + rank] = j;
    below += lam[j] - eps_d < 0.0;
  }
  below = __reduce_add_sync(0xffffffffu, below);
  __shared__ int wsum[8];
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = below;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += wsum[w];
    atomicMax(m, t);
  }
}

// X[k][r][n] = sum_mu conj(u_r[mu]) c[mu][n] for the r < m lowest
// eigenvectors u_r = V[k][by_rank[r]].
template <bool C>
__global__ void __launch_bounds__(256) proj_x_kernel(ProjPtrs P, int N, int Np, int n_mo, const double* __restrict__ V,
                                                     const int* __restrict__ by_rank, const int* __restrict__ m,
                                                     double* __restrict__ X) {
  const int r = blockIdx.x, k = blockIdx.y;
  if (r >= *m) return;
  const int j = by_rank[(size_t)k * N + r];
  if (j < 0 || j >= N) return;  // ranks are a permutation unless an eigenvalue is NaN
  const double* u = V + ((size_t)k * Np + j) * N * (C ? 2 : 1);
  const double* c = P.c[k];
  double* x = X + ((size_t)k * N + r) * n_mo * (C ? 2 : 1);
  for (int n = threadIdx.x; n < n_mo; n += blockDim.x) {
    Elem<C> acc = zero_elem<C>();
    for (int mu = 0; mu < N; ++mu) mac<C>(acc, conj_e<C>(ld_elem<C>(u, mu)), ld_elem<C>(c, (long)mu * n_mo + n));
    st_elem<C>(x, n, acc);
  }
}

// c~[mu][n] = c[mu][n] - sum_{r < m} u_r[mu] X[r][n]  (may run in place: X
// was formed from c before).
template <bool C>
__global__ void __launch_bounds__(256) proj_apply_kernel(ProjPtrs P, int N, int Np, int n_mo,
                                                         const double* __restrict__ V, const int* __restrict__ by_rank,
                                                         const int* __restrict__ m, const double* __restrict__ X) {
  const int mu = blockIdx.x, k = blockIdx.y;
  const int mm = *m;
  const double* c = P.c[k];
  double* out = P.out[k];
  for (int n = threadIdx.x; n < n_mo; n += blockDim.x) {
    Elem<C> v = ld_elem<C>(c, (long)mu * n_mo + n);
    for (int r = 0; r < mm; ++r) {
      const int j = by_rank[(size_t)k * N + r];
      if (j < 0 || j >= N) continue;
      Elem<C> u = ld_elem<C>(V + ((size_t)k * Np + j) * N * (C ? 2 : 1), mu);
      u.re = -u.re;
      if constexpr (C) u.im = -u.im;
      mac<C>(v, u, ld_elem<C>(X + ((size_t)k * N + r) * n_mo * (C ? 2 : 1), n));
    }
    st_elem<C>(out, (long)mu * n_mo + n, v);
  }
}

}  // namespace

cudaError_t launch_proj_load(int cplx, const ProjPtrs& P, int n_mat, int N, int Np, double* W, double* V,
                             cudaStream_t s) {
  const dim3 grid(Np, n_mat);
  if (cplx)
    proj_load_kernel<true><<<grid, 256, 0, s>>>(P, N, Np, W, V);
  else
    proj_load_kernel<false><<<grid, 256, 0, s>>>(P, N, Np, W, V);
  return cudaGetLastError();
}

cudaError_t launch_proj_load32(int cplx, int n_mat, int N, int Np, const double* W, float* scale, float* W32, float* V32,
                               cudaStream_t s) {
  const dim3 grid(Np, n_mat);
  if (cplx) {
    proj_norm_kernel<true><<<n_mat, 256, 0, s>>>(N, Np, W, scale);
    proj_load32_kernel<true><<<grid, 256, 0, s>>>(N, Np, W, scale, W32, V32);
  } else {
    proj_norm_kernel<false><<<n_mat, 256, 0, s>>>(N, Np, W, scale);
    proj_load32_kernel<false><<<grid, 256, 0, s>>>(N, Np, W, scale, W32, V32);
  }
  return cudaGetLastError();
}

// Shared memory of a block round at most (2 B columns of W and V).
constexpr size_t J32_SMEM = 225 * 1024;

// The launch limit of a block kernel, per device and set once to the most any
// basis takes: it belongs to the function, which the contexts of all threads share.
template <bool C, int B>
static cudaError_t jacobi32_attr() {
  static std::mutex mu;
  static bool done[MAX_DEVICES] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= MAX_DEVICES) dev = 0;
  std::lock_guard<std::mutex> lk(mu);
  if (done[dev]) return cudaSuccess;
  const cudaError_t e =
      cudaFuncSetAttribute(jacobi32_block_kernel<C, B>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)J32_SMEM);
  done[dev] = e == cudaSuccess;
  return e;
}

// One sweep of the FP32 iteration; returns the launches made, or a negative
// CUDA error.
template <bool C, int B>
static int jacobi32_blocks(int n_mat, int N, int Np, float* W32, float* V32, float thresh, unsigned* off_max,
                           cudaStream_t s) {
  const size_t sh = sizeof(Flt<C>) * 4 * B * (size_t)N;
  cudaError_t e = jacobi32_attr<C, B>();
  const int nb = 2 * ((Np + 2 * B - 1) / (2 * B));
  for (int br = 0; br < nb - 1 && e == cudaSuccess; ++br) {
    jacobi32_block_kernel<C, B><<<dim3(nb / 2, n_mat), 32 * B, sh, s>>>(N, Np, nb, br, W32, V32, thresh, off_max);
    e = cudaGetLastError();
  }
  return e == cudaSuccess ? nb - 1 : -(int)e;
}
template <bool C>
static int jacobi32_sweep(int n_mat, int N, int Np, float* W32, float* V32, float thresh, unsigned* off_max,
                          cudaStream_t s) {
  // blocks of 16 columns while 32 columns of W and V fit in shared memory
  // (complex N <= 450), of 8 up to twice that
  const size_t col = sizeof(Flt<C>) * 4 * (size_t)N, room = J32_SMEM;
  if (16 * col <= room) return jacobi32_blocks<C, 16>(n_mat, N, Np, W32, V32, thresh, off_max, s);
  if (8 * col <= room) return jacobi32_blocks<C, 8>(n_mat, N, Np, W32, V32, thresh, off_max, s);
  for (int r = 0; r < Np - 1; ++r)
    jacobi32_round_kernel<C><<<dim3((Np / 2 + 3) / 4, n_mat), 128, 0, s>>>(N, Np, r, W32, V32, thresh, off_max);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? Np - 1 : -(int)e;
}

int launch_jacobi32_sweep(int cplx, int n_mat, int N, int Np, float* W32, float* V32, float thresh, unsigned* off_max,
                          cudaStream_t s) {
  return cplx ? jacobi32_sweep<true>(n_mat, N, Np, W32, V32, thresh, off_max, s)
              : jacobi32_sweep<false>(n_mat, N, Np, W32, V32, thresh, off_max, s);
}

cudaError_t launch_proj_widen(long n, const float* x, double* y, cudaStream_t s) {
  proj_widen_kernel<<<(unsigned)std::min<long>((n + 255) / 256, (long)device_sm_count() * 8), 256, 0, s>>>(n, x, y);
  return cudaGetLastError();
}

cudaError_t launch_proj_corr(int cplx, int n_mat, int N, bool ortho, double* M, double* diag, float lim,
                             unsigned* dev, cudaStream_t s) {
  const dim3 grid(N, n_mat), gd((N + 255) / 256, n_mat);
  if (!ortho) {
    if (cplx)
      proj_diag_kernel<true><<<gd, 256, 0, s>>>(N, M, diag);
    else
      proj_diag_kernel<false><<<gd, 256, 0, s>>>(N, M, diag);
  }
  if (cplx) {
    if (ortho)
      proj_corr_kernel<true, true><<<grid, 256, 0, s>>>(N, M, diag, lim, dev);
    else
      proj_corr_kernel<true, false><<<grid, 256, 0, s>>>(N, M, diag, lim, dev);
  } else {
    if (ortho)
      proj_corr_kernel<false, true><<<grid, 256, 0, s>>>(N, M, diag, lim, dev);
    else
      proj_corr_kernel<false, false><<<grid, 256, 0, s>>>(N, M, diag, lim, dev);
  }
  return cudaGetLastError();
}

cudaError_t launch_jacobi_round(int cplx, int n_mat, int N, int Np, int r, double* W, double* V, double thresh,
                                unsigned long long* off_max, cudaStream_t s) {
  // a warp per pair from eight pairs per SM on
  if ((long)Np / 2 * n_mat >= 8L * device_sm_count()) {
    const dim3 grid((Np / 2 + 3) / 4, n_mat);
    if (cplx)
      jacobi_round_kernel<true, true><<<grid, 128, 0, s>>>(N, Np, r, W, V, thresh, off_max);
    else
      jacobi_round_kernel<false, true><<<grid, 128, 0, s>>>(N, Np, r, W, V, thresh, off_max);
  } else {
    const dim3 grid(Np / 2, n_mat);
    if (cplx)
      jacobi_round_kernel<true, false><<<grid, 256, 0, s>>>(N, Np, r, W, V, thresh, off_max);
    else
      jacobi_round_kernel<false, false><<<grid, 256, 0, s>>>(N, Np, r, W, V, thresh, off_max);
  }
  return cudaGetLastError();
}

cudaError_t launch_proj_cluster(int cplx, int n_mat, int N, int Np, const double* G, double* W, double* V, double thresh,
                                cudaStream_t s) {
  if (cplx)
    proj_cluster_kernel<true><<<n_mat, 256, N, s>>>(N, Np, G, W, V, thresh);
  else
    proj_cluster_kernel<false><<<n_mat, 256, N, s>>>(N, Np, G, W, V, thresh);
  return cudaGetLastError();
}

cudaError_t launch_proj_finish(int cplx, const ProjPtrs& P, int n_mat, int N, int Np, int n_mo, const double* W,
                               const double* V, double eps_d, double* lam_sorted, int* by_rank, int* m, double* X,
                               cudaStream_t s) {
  const size_t sh = sizeof(double) * Np;
  if (sh > 48 * 1024) return cudaErrorInvalidValue;
  if (cplx) {
    proj_rank_kernel<true><<<n_mat, 256, sh, s>>>(N, Np, W, eps_d, lam_sorted, by_rank, m);
    proj_x_kernel<true><<<dim3(N, n_mat), 256, 0, s>>>(P, N, Np, n_mo, V, by_rank, m, X);
    proj_apply_kernel<true><<<dim3(N, n_mat), 256, 0, s>>>(P, N, Np, n_mo, V, by_rank, m, X);
  } else {
    proj_rank_kernel<false><<<n_mat, 256, sh, s>>>(N, Np, W, eps_d, lam_sorted, by_rank, m);
    proj_x_kernel<false><<<dim3(N, n_mat), 256, 0, s>>>(P, N, Np, n_mo, V, by_rank, m, X);
    proj_apply_kernel<false><<<dim3(N, n_mat), 256, 0, s>>>(P, N, Np, n_mo, V, by_rank, m, X);
  }
  return cudaGetLastError();
}

}  // namespace rpa
