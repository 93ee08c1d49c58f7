// Products of FP64 matrices on the tensor cores (g64.cu): operands in eight
// 7-bit digit planes, integer accumulation, FP64 results.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "rpa_internal.h"

namespace rpa {

constexpr int G64_TAB = 48;  // matrices a pointer table of one launch names

// Batched operand: element (b, r, k), r < R, k < K, of matrix b at
//   p + r ld + k (by rows) or p + k ld + r (by columns), p = tab[b] or base + b stride
// (elements of 16 bytes complex, 8 real), optionally conjugated.
struct G64Src {
  const double* tab[G64_TAB];
  const double* base;
  long stride, ld;
  int use_tab, by_rows, conj, nb, R, K;
  int no_diag;  // element (r, r) counts as zero (g64_product adds its terms, see G64Diag)
  int by_element;  // the rows' spread is bounded so that single elements keep their accuracy (g64.cu)
};

// A sliced operand in device memory: planes, one exponent per row (|x| < 2^e).
struct G64Op {
  uint16_t* planes;
  int* e;
  long stride;   // uint16 units per matrix
  int Rpad, n_kb;
};

// Where a product goes: element (b, r, c) of output b at
//   p + (r / rd) s1 + (r % rd) s0 + (c / cd) t1 + (c % cd) t0.
struct G64Out {
  double* tab[G64_TAB];
  double* base;
  long stride, s0, s1, t0, t1;
  int use_tab, rd, cd, R, C;
  int add;    // add to what is there
  int neg;    // negate
  int tri;    // 0: all, 1: c <= r and the conjugate mirrored, 2: c <= r only
};

// Row counts and bytes of an operand's planes: `role` 0 = left (blocks of 128
// rows), 1 = right (blocks of 32 complex or 64 real rows).
int g64_rpad(int cplx, int role, int R);
inline int g64_nkb(int cplx, int K) { return ((cplx ? 2 * K : K) + 15) / 16; }
size_t g64_plane_bytes(int cplx, int role, int R, int K, int nb);

// Exponents and digit planes of an operand.  A row that holds an infinity or
// NaN, leaves the range 2^+-60 or spreads too far raises bit 0 of a flag (the
// caller then keeps the FP64 kernels' result), a row whose largest entry stands
// out of its root mean square bit 1 (the product then takes the digit pairs of
// one more level).
// frep = 0: one word *flag for all matrices; else matrix b raises flag[b frep
// .. b frep + frep - 1].  Two launches.
cudaError_t g64_slice(int cplx, int role, const G64Src& src, const G64Op& op, int* flag, int frep, cudaStream_t s);

// out[b](r, c) = sum_k conj(A[ia](r, k)) B[ib](c, k), ia = ta ? ta[b] : b / diva
// (ib alike), b < nb.  kmode: 0 every k, 1 only k >= the column tile's first
// column, 2 only k >= the row tile's first row (for triangular operands whose
// other half is zero).  A time-out sets *status.  With part (g64_part_bytes)
// the K range may be split over CTAs.  flag: the operands'
// flags, one word (per_b = 0) or one per matrix b (per_b = 1; where its bit 0 is
// set, nothing is stored).  Launches: 1 or 2 (*n_launch += them).
// Matrices with a dominant diagonal (V, chi0 and their factors) would lose the
// digits of their other entries to it, so both operands are sliced without
// their diagonals, and the product adds the two terms k = r and k = c in FP64
// from the operands themselves (untabled, square).
struct G64Diag {
  int on;
  G64Src A, B;
};
struct G64Index {
  const short* ta;  // host tables of nb entries (nb <= G64_TAB), or null
  const short* tb;
  int diva, divb;
};
cudaError_t g64_product(int cplx, const G64Op& A, const G64Op& B, const G64Index& ix, const G64Out& out, int nb,
                        int kmode, void* part, size_t part_bytes, const int* flag, int per_b, int* status,
                        uint64_t* n_launch, cudaStream_t s, const G64Diag* diag = nullptr);

// Triangular products of the tail (A4-A5) as digit products: Y[b] = -(L^H chi[b]
// L), lower triangle, L of matrix b / n_w, with T as scratch (chi and Y may be
// the same); Wn[q] = -(X[q]^H X[q]), lower triangle.  `work` holds the planes of some
// matrices at a time (at least two; tail_g64_bytes of n are enough for n at
// once); a matrix out of the split's range goes through the FP64
// kernels.  n in tail_g64_use: matrices per q (its answer decides the bits of
// an FP64 job, so it may not depend on how many q share the call).
bool tail_g64_use(int cplx, int N, int n);
size_t tail_g64_bytes(int cplx, int N, int n_mat, size_t most = (size_t)1 << 30);
cudaError_t launch_sandwich_g64(int cplx, int N, int n_batch, int n_w, const double* chi, const double* L, double* T,
                                double* Y, void* work, size_t work_bytes, int* status, uint64_t* n_launch,
                                cudaStream_t s);
cudaError_t launch_gram_g64(int cplx, int N, int n_q, const double* X, double* Wn, void* work, size_t work_bytes,
                            int* status, uint64_t* n_launch, cudaStream_t s);

// FP64 chi0 on this product: whether the size takes it, its workspace, and
// the launch for all q of g (q out of the split's range are redone by the FP64 kernel).
// The workspace holds the planes of some frequencies at a time (chi0_g64_freqs at
// most, one at least); the result does not depend on how many.
bool chi0_g64_use(const BatchGeom& g);
int chi0_g64_freqs(const BatchGeom& g);
size_t chi0_g64_bytes(const BatchGeom& g, int n_freq);
cudaError_t launch_chi0_g64(const BatchGeom& g, const double* const* Cptrs, const double* dtab, double* chi,
                            void* work, size_t work_bytes, int* status, uint64_t* n_launch, cudaStream_t s);

}  // namespace rpa
