// FP64 products on the tcgen05 tensor cores of GB300 (sm_103a).
//
// An SM's FP64 pipe issues two DFMA lanes per clock (1.2 TFLOP/s for the whole
// GPU), its tensor pipe 8192 BF16 flops.  A product of FP64 matrices is
// therefore cut into exact pieces (an error-free split in the manner of
// Ozaki, Ogita, Oishi and Rump): row r of an operand is scaled by one exponent
// e_r (|x| < 2^e_r) to integers F = round(x 2^(55 - e_r)), whose eight balanced
// base-128 digits (|d| <= 64) are exact in BF16.  Digit pairs (i, j) of level
// l = i + j <= 7 are multiplied, 36 of 64; levels l >= 8 lie 2^-56 below the
// leading one.  Every level has its own FP32 accumulator in TMEM, whose
// integer sums stay below 2^24 for 768 real k up to level 4 whatever the data
// (level l adds l + 1 products of at most 2^12 each); levels 5 to 7, 2^-35
// and less, could round only for data whose digits all agree.  Every 768 k the
// accumulators are added into two 64-bit integers per output, so splitting K
// over CTAs, or batching, changes no bit of the result.
//
// Error: the dropped levels and the rounding of F, about 2^-56 max|a| max|b|
// sqrt(K) per output, against 2^-53 sqrt(K) (partial sums) for a chain of
// DFMA.  Emulated on Gaussian rows: 1.3e-16 against 3.2e-16 (norm, relative)
// for K = 128, 1.1e-16 against 2.0e-15 for K = 4096.  The dropped levels scale
// with the rows' largest entries, so where one stands far out of its row's root
// mean square (row_flags), the seven pairs of level 8 are multiplied too; the
// error left is the rounding of F, 2^-56 (max|a| |b| + |a| max|b|).  Rows whose
// typical entry lies so far below the largest that even this could exceed the
// DFMA chain's error, and rows with an infinity or NaN or outside 2^+-60, are
// flagged, and the callers keep the FP64 kernels' result.
//
// Tile: 128 rows x 64 real columns.  Complex data is embedded as real rows
// X = (re_0, im_0, ...) on the left and X over Y = (im_0, -re_0, ...) on the
// right, 32 complex columns, so that the 64 columns are [Re | Im] of
// sum conj(a) b.  Eight levels of 64 columns fill the 512 TMEM columns.
// Digit planes j, j+1, ... of the right operand are adjacent in a stage, so
// one MMA of N = 64 n multiplies one left plane with n right planes into n
// adjacent accumulators: 12 MMAs per 16 k, 1152 tensor-pipe clocks.  Operands
// are stored pre-blocked in the order the MMAs read them (32 KB + 16 KB per 16
// k) and arrive by two bulk copies per stage.
#include "g64.h"

#include <math.h>
#include <string.h>

#include <algorithm>
#include <mutex>

#include "fp64_elem.cuh"
#include "tc_ptx.cuh"

namespace rpa {
namespace {

constexpr int NP = 8;                        // digit planes
constexpr int KBLK = 16;                     // real k per K-block
constexpr int KBC = 48;                      // K-blocks per exact accumulation (768 real k)
constexpr int A_BLOCK = NP * 128 * KBLK * 2; // bytes per left row block and K-block (32 KB)
constexpr int B_BLOCK = NP * 64 * KBLK * 2;  // right (16 KB)
constexpr int G_STAGES = 4;
constexpr int G_STAGE = A_BLOCK + B_BLOCK;
constexpr int G_EPI = 8;                     // epilogue warps
constexpr int G_THREADS = 64 + 32 * G_EPI;
constexpr size_t G_SMEM = (size_t)G_STAGES * G_STAGE + 1024 + 256;
constexpr size_t PART_ITEM = 32ull * 256 * sizeof(longlong2);  // split-K partial of one tile
constexpr int E_ZERO = -4000;                // exponent of a zero row

// ------------------------------------------------------------- slicing ----

// F = round(x 2^(55 - e)) for |x| < 2^e.
__device__ __forceinline__ long long fix55(double x, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int E = (int)((b >> 52) & 0x7ff);
  if (E == 0 || e == E_ZERO) return 0;
  const int sh = min(max(1029 + e - E, 1), 63);
  const unsigned long long h = ((b & 0xFFFFFFFFFFFFFull) | (1ull << 52)) << 9;
  const long long f = (long long)((h + (1ull << (sh - 1))) >> sh);
  return (long long)b < 0 ? -f : f;
}
// F = round(c d 2^(55 - e)) for |c d| < 2^e: the 106-bit product of the two
// significands, its top 64 bits kept.
__device__ __forceinline__ long long fix55_mul(unsigned long long cb, unsigned long long db, int e) {
  const int Ec = (int)((cb >> 52) & 0x7ff), Ed = (int)((db >> 52) & 0x7ff);
  if (Ec == 0 || Ed == 0 || e == E_ZERO) return 0;
  const unsigned long long mc = (cb << 11) | (1ull << 63), md = (db << 11) | (1ull << 63);
  const unsigned long long hi = __umul64hi(mc, md) >> 1;  // |c d| = hi 2^(Ec + Ed - 2107)
  const int sh = min(max(2052 + e - Ec - Ed, 1), 63);
  const long long f = (long long)((hi + (1ull << (sh - 1))) >> sh);
  return (long long)(cb ^ db) < 0 ? -f : f;
}

constexpr unsigned long long DIGIT_BIAS = 64ull | 64ull << 7 | 64ull << 14 | 64ull << 21 | 64ull << 28 | 64ull << 35 |
                                          64ull << 42 | 64ull << 49;

// Digit d of plane P of G = F + DIGIT_BIAS as the FP32 bits of d 2^(-7 P) (exact,
// |d| <= 64).
template <int P>
__device__ __forceinline__ uint32_t digit_bits(unsigned long long G) {
  constexpr int s = 7 * (7 - P);
  const uint32_t v = (uint32_t)(G >> s);
  const uint32_t f = (P == 0 ? v : (v & 127u)) | 0x4B000000u;
  constexpr float sc = 1.0f / (float)(1ull << (7 * P));
  return __float_as_uint(fmaf(__uint_as_float(f), sc, -8388672.0f * sc));
}

// Digit planes of 16 consecutive real k of one row: G in order.  Left: row
// of the 128-row block; right: X in row `row`, Y in row 32 + row (complex).
template <int ROLE, bool C, int P = 0>
__device__ __forceinline__ void store_digits(const unsigned long long (&G)[16], uint16_t* blk, int row) {
  if constexpr (P < NP) {
    uint32_t x[8], y[8];
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      const uint32_t a = digit_bits<P>(G[2 * v]), b = digit_bits<P>(G[2 * v + 1]);
      x[v] = __byte_perm(a, b, 0x7632);
      if (ROLE == 1 && C) y[v] = __byte_perm(b, a ^ 0x80000000u, 0x7632);
    }
    uint16_t* d = blk + P * ((ROLE == 0 ? 128 : 64) * KBLK);
    auto put = [&](int r, const uint32_t(&w)[8]) {
      uint4* q = reinterpret_cast<uint4*>(d + ((r >> 3) * 16 + (r & 7)) * 8);
      q[0] = make_uint4(w[0], w[1], w[2], w[3]);
      q[8] = make_uint4(w[4], w[5], w[6], w[7]);
    };
    put(row, x);
    if constexpr (ROLE == 1 && C) put(32 + row, y);
    store_digits<ROLE, C, P + 1>(G, blk, row);
  }
}

template <bool C>
__device__ __forceinline__ const double* src_ptr(const G64Src& s, int b) {
  return s.use_tab ? s.tab[b] : s.base + b * s.stride * (C ? 2 : 1);
}

// |x| as FP32 bits (truncated; 0 only for zero, 1 below 2^-126, all ones at or
// above 2^127).
__device__ __forceinline__ uint32_t abs_bits32(unsigned long long b) {
  const uint32_t hi = (uint32_t)(b >> 32) & 0x7fffffffu, lo = (uint32_t)b;
  if (hi < (897u << 20)) return (hi | lo) ? 1u : 0u;
  if (hi >= (1150u << 20)) return 0xffffffffu;
  return __funnelshift_l(lo, hi, 3) - (896u << 23);
}

// What decides a row's exponent and its flags: largest |x| (FP32 bits, truncated),
// sum of squares, sum of the FP32 exponents and count of the nonzero entries.
struct RowStat {
  uint32_t m = 0;
  float ss = 0.f;
  int es = 0, nz = 0;
  __device__ __forceinline__ void add(uint32_t v) {
    m = max(m, v);
    ss = fmaf(__uint_as_float(v), __uint_as_float(v), ss);
    es += (int)(v >> 23);
    nz += v != 0;
  }
  __device__ __forceinline__ void join(const RowStat& o) {
    m = max(m, o.m);
    ss += o.ss;
    es += o.es;
    nz += o.nz;
  }
  __device__ __forceinline__ void warp_join() {
    m = __reduce_max_sync(0xffffffffu, m);
    es = __reduce_add_sync(0xffffffffu, es);
    nz = __reduce_add_sync(0xffffffffu, nz);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  }
};

// Bit 0 (FP64 kernels): an infinity, a NaN, values outside 2^+-60, or a mean
// binary exponent more than 1.5 + log2(K) / 2 below the largest entry's: then
// 2^-56 max|a| |b| can exceed the DFMA chain's error, about 2^-53 sqrt(K) / 5
// of |a| |b| for typical entries.  (Gaussian rows: 2.4 at K = 128, 2.8 at 8192.
// Sums of less than 64 terms, the short ends of triangular operands: 8, as
// their few exponents scatter.)
// Bit 1 (level 8 too): (max / rms)^2 above `spread` sqrt(K / 128), where the
// dropped levels could exceed it.
//
// These bounds are for the norm of an output row.  A single element sum_k a_k b_k can
// be far smaller than |a| |b| where the large entries of one row meet the small ones
// of the other (halves scaled by 2^-g in turn: mean gap 2.5 + g / 2), and the split's
// error is not.  Operands whose products are results of their own (`by_element`: the
// unweighted rows of chi0, AO -> MO) are held to the gap up to which the error per element,
// over sum_k |a_k b_k|, stays within about twice a DFMA chain's.  Emulated, split over
// chain at g = 0, 2, 4, 6, 8, levels to 7: K = 128 0.57, 1.9, 7, 31, 130, K = 2048 0.19, 0.6, 2.6,
// 9, 39; with level 8 0.09, 0.34, 1.4, 5.5, 23 and 0.03, 0.1, 0.3, 1.6, 5.3.  So level 8
// from a gap of 4.25 (one Gaussian row in 10^6 has one), the FP64 kernels
// from 4.6 at K = 128, a quarter more per factor of two.
constexpr float SPREAD = 40.f;            // as given: Gaussian rows reach 20
constexpr float SPREAD_WEIGHTED = 100.f;  // times the smooth frequency weights (a factor 2 of spread of their own)
constexpr float TINY = 8.7e-19f;          // 2^-60
__device__ __forceinline__ int row_flags(const RowStat& r, float spread, bool by_element) {
  const float m = __uint_as_float(r.m), n = (float)max(r.nz, 1);
  if (r.m >= 0x7f800000u || !(m < 1.1e18f) || !(m > TINY)) return 1;
  const float gap = (float)(r.m >> 23) - (float)r.es / n, lg = log2f(n);
  if (by_element) {
    if (gap > (n < 16.f ? 8.f : n < 64.f ? 5.2f : 4.6f + 0.25f * fmaxf(lg - 7.f, 0.f))) return 1;
    if (gap > 4.25f) return 2;
  } else if (gap > (n < 64.f ? 8.f : 1.5f + 0.5f * lg)) {
    return 1;
  }
  return m * m <= spread * sqrtf(n * (1.0f / 128.0f)) * r.ss / n ? 0 : 2;
}
// The row's exponent; raises its flags.
__device__ __forceinline__ int row_exponent(const RowStat& r, float spread, bool by_element, int* flag,
                                            int nflag = 1) {
  if (r.m == 0) return E_ZERO;
  if (const int bits = row_flags(r, spread, by_element))
    for (int i = 0; i < nflag; ++i) atomicOr(flag + i, bits);
  if (r.m >= 0x7f800000u) return 1100;
  return (int)(__float_as_uint(__uint_as_float(r.m) * 1.000001f) >> 23) - 126;
}

// Exponent and flags of every row of every matrix: one warp per
// row (by rows), or 32 rows per CTA with eight warps along k (by columns).
template <bool C>
__global__ void __launch_bounds__(256) g64_exp_kernel(const __grid_constant__ G64Src src, int Rpad, int* __restrict__ e,
                                                      int* __restrict__ flag, int frep) {
  __shared__ RowStat sr[8][32];
  const int rows = src.by_rows ? 8 : 32, nblk = (Rpad + rows - 1) / rows;
  const int b = blockIdx.x / nblk, r0 = (blockIdx.x % nblk) * rows;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double* p = src_ptr<C>(src, b);
  const int r = r0 + (src.by_rows ? warp : lane);
  RowStat st;
  if (r < src.R) {
    const int k0 = src.by_rows ? lane : warp, dk = src.by_rows ? 32 : 8;
    for (int k = k0; k < src.K; k += dk) {
      if (src.no_diag && k == r) continue;
      const Elem<C> x = ld_elem<C>(p, src.by_rows ? (long)r * src.ld + k : (long)k * src.ld + r);
      st.add(abs_bits32((unsigned long long)__double_as_longlong(x.re)));
      if constexpr (C) st.add(abs_bits32((unsigned long long)__double_as_longlong(x.im)));
    }
  }
  if (src.by_rows) {
    st.warp_join();
    if (lane != 0) return;
  } else {
    sr[warp][lane] = st;
    __syncthreads();
    if (warp != 0) return;
    for (int w = 1; w < 8; ++w) st.join(sr[w][lane]);
  }
  if (r < Rpad)
    e[(long)b * Rpad + r] = r < src.R ? row_exponent(st, SPREAD, src.by_element, flag + (long)b * frep, max(frep, 1))
                                         : E_ZERO;
}

// One thread per (matrix, row, K-block); consecutive threads take consecutive
// rows, so the blocked stores coalesce.
template <bool C, int ROLE>
__global__ void __launch_bounds__(256) g64_slice_kernel(const __grid_constant__ G64Src src, const __grid_constant__ G64Op op) {
  constexpr int kpb = C ? 8 : 16;                             // k per K-block
  constexpr int RB = ROLE == 0 ? 128 : (C ? 32 : 64);         // rows per block
  const long per = (long)op.Rpad * op.n_kb, total = per * src.nb;
  for (long idx = blockIdx.x * 256L + threadIdx.x; idx < total; idx += gridDim.x * 256L) {
    const int b = (int)(idx / per);
    const long rem = idx - b * per;
    const int r = (int)(rem % op.Rpad), kb = (int)(rem / op.Rpad);
    const double* p = src_ptr<C>(src, b);
    const int e = op.e[(long)b * op.Rpad + r];
    unsigned long long G[16];
#pragma unroll
    for (int v = 0; v < kpb; ++v) {
      const int k = kb * kpb + v;
      Elem<C> x = zero_elem<C>();
      if (r < src.R && k < src.K && !(src.no_diag && k == r)) x = ld_elem<C>(p, src.by_rows ? (long)r * src.ld + k : (long)k * src.ld + r);
      if constexpr (C) {
        if (src.conj) x.im = -x.im;
        G[2 * v] = (unsigned long long)fix55(x.re, e) + DIGIT_BIAS;
        G[2 * v + 1] = (unsigned long long)fix55(x.im, e) + DIGIT_BIAS;
      } else {
        G[v] = (unsigned long long)fix55(x.re, e) + DIGIT_BIAS;
      }
    }
    uint16_t* blk = op.planes + b * op.stride + ((long)(r / RB) * op.n_kb + kb) * ((ROLE == 0 ? A_BLOCK : B_BLOCK) / 2);
    store_digits<ROLE, C>(G, blk, r % RB);
  }
}

// --------------------------------------------------------------- product --

struct G64Params {
  const uint16_t *A, *B;
  const int *eA, *eB;
  long sA, sB;
  int RpA, RpB, n_kb, diva, divb, use_ta, use_tb;
  short ta[G64_TAB], tb[G64_TAB];
  int nb, nI, nJ, tri, n_tiles, n_split, cps;  // cps: chunks per split
  int kmode, n_items;
  longlong2* part;
  const int* flag;  // null, the operands' one flag word, or (per_b) a word per matrix
  int per_b;
  int* status;
  G64Out out;
  G64Diag diag;
};

// One MMA: left plane i, right planes j .. j + n - 1, accumulators g .. g + n - 1.
struct GMma {
  int i, j, n, g;
};
// Levels 0-3 first, then 4-7; the first entry of each half starts its four
// accumulators at the first K-block of a chunk.
__device__ constexpr GMma kG[12] = {{0, 0, 4, 0}, {1, 0, 3, 1}, {2, 0, 2, 2}, {3, 0, 1, 3}, {0, 4, 4, 4}, {1, 3, 4, 4},
                                    {2, 2, 4, 4}, {3, 1, 4, 4}, {4, 0, 4, 4}, {5, 0, 3, 5}, {6, 0, 2, 6}, {7, 0, 1, 7}};
constexpr bool g_table_ok() {
  constexpr GMma t[12] = {{0, 0, 4, 0}, {1, 0, 3, 1}, {2, 0, 2, 2}, {3, 0, 1, 3}, {0, 4, 4, 4}, {1, 3, 4, 4},
                          {2, 2, 4, 4}, {3, 1, 4, 4}, {4, 0, 4, 4}, {5, 0, 3, 5}, {6, 0, 2, 6}, {7, 0, 1, 7}};
  for (int a = 0; a < NP; ++a)
    for (int b = 0; b < NP; ++b) {
      int c = 0;
      for (const GMma& m : t)
        if (m.i == a && b >= m.j && b < m.j + m.n) {
          ++c;
          if (m.g + b - m.j != a + b) return false;
        }
      if (c != (a + b < NP ? 1 : 0)) return false;
    }
  return true;
}
static_assert(g_table_ok(), "digit-pair table is inconsistent");

struct GItem {
  int b, I, J, ia, ib, kb0, kb1, local;  // local: tile index within (split, b)
};
template <bool C>
__device__ __forceinline__ GItem g_item(const G64Params& p, int item) {
  GItem r;
  const int tile = item % p.n_tiles;
  int q = item / p.n_tiles;
  r.b = q % p.nb;
  const int ks = q / p.nb;
  if (p.tri) {
    // row block I holds min(nJ, (C ? 4 : 2)(I + 1)) column tiles
    int t = tile, I = 0;
    while (true) {
      const int c = min(p.nJ, (C ? 4 : 2) * (I + 1));
      if (t < c) break;
      t -= c;
      ++I;
    }
    r.I = I;
    r.J = t;
  } else {
    r.I = tile / p.nJ;
    r.J = tile % p.nJ;
  }
  r.ia = p.use_ta ? p.ta[r.b] : r.b / p.diva;
  r.ib = p.use_tb ? p.tb[r.b] : r.b / p.divb;
  const int lo = min(p.n_kb, p.kmode == 1 ? r.J * 4 : p.kmode == 2 ? r.I * (C ? 16 : 8) : 0);
  r.kb0 = min(p.n_kb, lo + ks * p.cps * KBC);
  r.kb1 = min(p.n_kb, r.kb0 + p.cps * KBC);
  if (ks == p.n_split - 1) r.kb1 = p.n_kb;
  r.local = r.b * p.n_tiles + tile;
  return r;
}

// (hi 2^28 + lo) 2^ex rounded to FP64, integer arithmetic only.
__device__ __forceinline__ double to_f64(long long hi, long long lo, int ex) {
  // 128-bit T = hi 2^28 + lo
  long long h = hi >> 36;
  unsigned long long l = (unsigned long long)hi << 28;
  const unsigned long long l2 = l + (unsigned long long)lo;
  h += (lo >> 63) + (l2 < l ? 1 : 0);
  l = l2;
  if (h == 0 && l == 0) return 0.0;
  const bool neg = h < 0;
  if (neg) {
    l = ~l + 1ull;
    h = ~h + (l == 0 ? 1 : 0);
  }
  // normalise to a 64-bit significand with its top bit set
  int msb;
  unsigned long long m;
  bool sticky = false;
  if (h) {
    const int z = __clzll(h);
    msb = 127 - z;
    m = z ? ((unsigned long long)h << z) | (l >> (64 - z)) : (unsigned long long)h;
    sticky = z ? (l << z) != 0 : l != 0;
  } else {
    const int z = __clzll((long long)l);
    msb = 63 - z;
    m = l << z;
  }
  // round to 53 bits, ties to even
  unsigned long long r = m >> 11;
  const unsigned long long rest = m & 2047ull;
  if (rest > 1024 || (rest == 1024 && (sticky || (r & 1)))) ++r;  // r = 2^53 carries into the exponent below
  const int E = msb + ex + 1023;
  if (E <= 1 || E >= 2046) return scalbn(neg ? -(double)r : (double)r, msb + ex - 52);
  const unsigned long long bits = ((unsigned long long)E << 52) + (r - (1ull << 52));
  return __longlong_as_double((long long)(bits | (neg ? 1ull << 63 : 0ull)));
}

template <bool C>
__device__ __forceinline__ Elem<C> src_at(const G64Src& s, int b, int r, int k) {
  Elem<C> x = ld_elem<C>(s.base + b * s.stride * (C ? 2 : 1), s.by_rows ? (long)r * s.ld + k : (long)k * s.ld + r);
  if (s.conj) x = conj_e<C>(x);
  return x;
}
// v += conj(A(r, k)) B(c, k) for k = r and k = c.
template <bool C>
__device__ __forceinline__ void add_diag(const G64Diag& d, int ia, int ib, int r, int c, Elem<C>& v) {
  mac<C>(v, conj_e<C>(src_at<C>(d.A, ia, r, r)), src_at<C>(d.B, ib, c, r));
  if (r != c) mac<C>(v, conj_e<C>(src_at<C>(d.A, ia, r, c)), src_at<C>(d.B, ib, c, c));
}

// Writes one thread's 16 complex (32 real) outputs of row r: columns c0 + u.
template <bool C, bool DIAG>
__device__ __forceinline__ void g_store(const G64Params& p, const GItem& it, int row, int half, const long long (&hi)[32],
                                        const long long (&lo)[32]) {
  const G64Out& o = p.out;
  const int r = it.I * 128 + row;
  if (r >= o.R || (p.per_b && (p.flag[it.b] & 1))) return;
  double* out = o.use_tab ? o.tab[it.b] : o.base + it.b * o.stride * (C ? 2 : 1);
  const int eA = p.eA[(long)it.ia * p.RpA + r];
  const int* eB = p.eB + (long)it.ib * p.RpB;
  const long ro = (long)(r / o.rd) * o.s1 + (long)(r % o.rd) * o.s0;
  constexpr int NC = C ? 16 : 32;
  const int c0 = it.J * (C ? 32 : 64) + half * NC;
#pragma unroll
  for (int u = 0; u < NC; ++u) {
    const int c = c0 + u;
    if (c >= o.C || (o.tri && c > r)) continue;
    const int ex = eA + eB[c] - 61;
    Elem<C> v;
    v.re = to_f64(hi[u], lo[u], ex);
    if constexpr (C) v.im = to_f64(hi[16 + u], lo[16 + u], ex);
    if constexpr (DIAG) add_diag<C>(p.diag, it.ia, it.ib, r, c, v);
    if (o.neg) {
      v.re = -v.re;
      if constexpr (C) v.im = -v.im;
    }
    const long at = ro + (long)(c / o.cd) * o.t1 + (long)(c % o.cd) * o.t0;
    if (o.add) {
      const Elem<C> w = ld_elem<C>(out, at);
      v.re += w.re;
      if constexpr (C) v.im += w.im;
    }
    if constexpr (C)
      if (o.tri == 1 && c == r) v.im = 0.0;
    st_elem<C>(out, at, v);
    if (o.tri == 1 && c != r) st_elem<C>(out, (long)c * o.s0 + (long)r * o.t0, conj_e<C>(v));
  }
}

// One producer thread (bulk copies), one MMA thread, eight epilogue warps; a
// persistent CTA per SM.  Epilogue warp w: rows 32 (w & 3) .., column half.
template <bool C, bool DIAG>
__global__ void __launch_bounds__(G_THREADS, 1) g64_kernel(const __grid_constant__ G64Params p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + G_STAGES * G_STAGE);
  uint64_t* empty = full + G_STAGES;
  uint64_t* acc_full = empty + G_STAGES;
  uint64_t* acc_empty = acc_full + 1;
  uint64_t* drain = acc_empty + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int ERR = 1 + (1 << 30);
  if (threadIdx.x == 0) {
    for (int i = 0; i < G_STAGES; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    mbar_init(acc_full, 1);
    mbar_init(acc_empty, 32 * G_EPI);
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      int armed[G_STAGES];
      for (int i = 0; i < G_STAGES; ++i) armed[i] = -1;
      bool ok = true;
      for (int item = blockIdx.x; item < p.n_items && ok; item += gridDim.x) {
        const GItem it = g_item<C>(p, item);
        const uint16_t* a = p.A + it.ia * p.sA + (long)it.I * p.n_kb * (A_BLOCK / 2);
        const uint16_t* b = p.B + it.ib * p.sB + (long)it.J * p.n_kb * (B_BLOCK / 2);
        for (int kb = it.kb0; kb < it.kb1; ++kb) {
          ok = mbar_wait(&empty[stage], phase ^ 1u, abort_flag, p.status, ERR + 21, 2000);
          if (!ok) break;
          uint8_t* sa = smem + stage * G_STAGE;
          mbar_expect_tx(&full[stage], G_STAGE);
          bulk_load(sa, a + (long)kb * (A_BLOCK / 2), A_BLOCK, &full[stage]);
          bulk_load(sa + A_BLOCK, b + (long)kb * (B_BLOCK / 2), B_BLOCK, &full[stage]);
          armed[stage] = (int)phase;
          if (++stage == G_STAGES) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
      // every armed stage's copy must have landed before the CTA exits
      for (int i = 0; i < G_STAGES; ++i) {
        if (armed[i] < 0) continue;
        const unsigned long long t0 = gtime();
        while (!mbar_try(&full[i], (uint32_t)armed[i]) && gtime() - t0 < WAIT_NS) {
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0, acc_phase = 0;
      bool ok = true;
      const uint64_t d0 = sdesc(smem_u32(smem));
      for (int item = blockIdx.x; item < p.n_items && ok; item += gridDim.x) {
        const GItem it = g_item<C>(p, item);
        const bool more = p.flag && (p.flag[p.per_b ? it.b : 0] & 2);
        for (int c0 = it.kb0; c0 < it.kb1 && ok; c0 += KBC) {
          const int c1 = min(it.kb1, c0 + KBC);
          ok = mbar_wait(acc_empty, acc_phase ^ 1u, abort_flag, p.status, ERR + 22);
          if (!ok) break;
          fence_after();
          for (int kb = c0; kb < c1; ++kb) {
            ok = mbar_wait(&full[stage], phase, abort_flag, p.status, ERR + 23);
            if (!ok) break;
            fence_after();
            const uint64_t da = d0 + (uint64_t)((stage * G_STAGE) >> 4);
            const uint64_t db = da + (uint64_t)(A_BLOCK >> 4);
#pragma unroll
            for (int m = 0; m < 12; ++m)
              mma(tmem + 64u * (uint32_t)kG[m].g, da + (uint64_t)((kG[m].i * 128 * KBLK * 2) >> 4),
                  db + (uint64_t)((kG[m].j * 64 * KBLK * 2) >> 4), idesc(64u * (uint32_t)kG[m].n),
                  !(kb == c0 && (m == 0 || m == 4)));
            if (more) {  // level 8, into level 7's accumulator
#pragma unroll
              for (int i = 1; i < NP; ++i)
                mma(tmem + 64u * 7u, da + (uint64_t)((i * 128 * KBLK * 2) >> 4),
                    db + (uint64_t)(((8 - i) * 64 * KBLK * 2) >> 4), idesc(64u), true);
            }
            mma_commit(&empty[stage]);
            if (++stage == G_STAGES) {
              stage = 0;
              phase ^= 1u;
            }
          }
          if (ok) mma_commit(acc_full);
          acc_phase ^= 1u;
        }
      }
      // all MMAs issued by this thread must be complete before TMEM is freed
      mma_commit(drain);
      const unsigned long long t0 = gtime();
      while (!mbar_try(drain, 0) && gtime() - t0 < WAIT_NS) {
      }
    }
  } else {
    const int quad = warp & 3, half = (warp - 2) >> 2;
    const int row = quad * 32 + lane;
    constexpr int NC = C ? 16 : 32;
    const uint32_t tl = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(half * NC);
    uint32_t acc_phase = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < p.n_items && ok; item += gridDim.x) {
      const GItem it = g_item<C>(p, item);
      long long hi[32], lo[32];
#pragma unroll
      for (int u = 0; u < 32; ++u) hi[u] = lo[u] = 0;
      for (int c0 = it.kb0; c0 < it.kb1; c0 += KBC) {
        ok = mbar_wait(acc_full, acc_phase, abort_flag, p.status, ERR + 24, 20000);
        if (!ok) break;
        fence_after();
#pragma unroll
        for (int u = 0; u < 32; u += 4) {
          // complex: accumulators 0-15 are Re columns, 16-31 the Im columns 32 further
          const uint32_t col = C && u >= 16 ? 32u + (uint32_t)(u - 16) : (uint32_t)u;
          float v[NP][4];
#pragma unroll
          for (int l = 0; l < NP; ++l) tmem_ld4(tl + 64u * l + col, v[l]);
          tmem_wait_ld();
#pragma unroll
          for (int w = 0; w < 4; ++w) {
            // level l holds its integer sum times 2^(-7 l)
            long long h = 0, q = 0;
#pragma unroll
            for (int l = 0; l < 4; ++l) {
              h += (long long)__float2int_rn(v[l][w] * (float)(1ull << (7 * l))) * (long long)(1 << (7 * (3 - l)));
              q += (long long)__float2int_rn(v[4 + l][w] * (float)(1ull << (7 * (4 + l)))) *
                   (long long)(1 << (7 * (3 - l)));
            }
            hi[u + w] += h;
            lo[u + w] += q;
          }
        }
        fence_before();
        mbar_arrive(acc_empty);
        acc_phase ^= 1u;
      }
      if (!ok) break;
      if (p.n_split == 1) {
        g_store<C, DIAG>(p, it, row, half, hi, lo);
      } else {
        longlong2* d = p.part + (long)item * (32 * 256) + (threadIdx.x - 64);
#pragma unroll
        for (int u = 0; u < 32; ++u) d[u * 256] = make_longlong2(hi[u], lo[u]);
      }
    }
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
}

// Sum of the split-K partials (exact) and the store, one CTA per tile.
template <bool C>
__global__ void __launch_bounds__(256) g64_reduce_kernel(const __grid_constant__ G64Params p) {
  const int per = p.nb * p.n_tiles;
  const GItem it = g_item<C>(p, blockIdx.x);
  long long hi[32], lo[32];
#pragma unroll
  for (int u = 0; u < 32; ++u) hi[u] = lo[u] = 0;
  for (int ks = 0; ks < p.n_split; ++ks) {
    const longlong2* d = p.part + ((long)ks * per + blockIdx.x) * (32 * 256) + threadIdx.x;
#pragma unroll
    for (int u = 0; u < 32; ++u) {
      const longlong2 v = d[u * 256];
      hi[u] += v.x;
      lo[u] += v.y;
    }
  }
  const int warp = (threadIdx.x >> 5) + 2;
  g_store<C, false>(p, it, (warp & 3) * 32 + (threadIdx.x & 31), (warp - 2) >> 2, hi, lo);
}

cudaError_t g64_attr() {
  static std::mutex mu;
  static bool done[MAX_DEVICES] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= MAX_DEVICES) dev = 0;
  std::lock_guard<std::mutex> lk(mu);
  if (done[dev]) return cudaSuccess;
  cudaError_t e = cudaSuccess;
  for (auto* k : {g64_kernel<true, false>, g64_kernel<false, false>, g64_kernel<true, true>, g64_kernel<false, true>})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G_SMEM);
  done[dev] = e == cudaSuccess;
  return e;
}

unsigned grid_for(long n, long per_sm) {
  return (unsigned)std::max<long>(1, std::min<long>((n + 255) / 256, (long)device_sm_count() * per_sm));
}

}  // namespace

int g64_rpad(int cplx, int role, int R) {
  const int rb = role == 0 ? 128 : (cplx ? 32 : 64);
  return (R + rb - 1) / rb * rb;
}

size_t g64_plane_bytes(int cplx, int role, int R, int K, int nb) {
  const size_t blocks = (size_t)g64_rpad(cplx, role, R) / (role == 0 ? 128 : (cplx ? 32 : 64));
  return blocks * g64_nkb(cplx, K) * (role == 0 ? A_BLOCK : B_BLOCK) * nb;
}

cudaError_t g64_slice(int cplx, int role, const G64Src& src, const G64Op& op, int* flag, int frep, cudaStream_t s) {
  const int rows = src.by_rows ? 8 : 32;
  const unsigned gb = (unsigned)((long)src.nb * ((op.Rpad + rows - 1) / rows));
  const unsigned gs = grid_for((long)op.Rpad * op.n_kb * src.nb, 16);
  if (cplx) {
    g64_exp_kernel<true><<<gb, 256, 0, s>>>(src, op.Rpad, op.e, flag, frep);
    if (role == 0)
      g64_slice_kernel<true, 0><<<gs, 256, 0, s>>>(src, op);
    else
      g64_slice_kernel<true, 1><<<gs, 256, 0, s>>>(src, op);
  } else {
    g64_exp_kernel<false><<<gb, 256, 0, s>>>(src, op.Rpad, op.e, flag, frep);
    if (role == 0)
      g64_slice_kernel<false, 0><<<gs, 256, 0, s>>>(src, op);
    else
      g64_slice_kernel<false, 1><<<gs, 256, 0, s>>>(src, op);
  }
  return cudaGetLastError();
}

cudaError_t g64_product(int cplx, const G64Op& A, const G64Op& B, const G64Index& ix, const G64Out& out, int nb,
                        int kmode, void* part, size_t part_bytes, const int* flag, int per_b, int* status,
                        uint64_t* n_launch, cudaStream_t s, const G64Diag* diag) {
  if (nb <= 0) return cudaSuccess;
  if (A.n_kb != B.n_kb || ((ix.ta || ix.tb || out.use_tab) && nb > G64_TAB)) return cudaErrorInvalidValue;
  if (cudaError_t e = g64_attr()) return e;
  G64Params p;
  memset(&p, 0, sizeof p);
  p.A = A.planes;
  p.B = B.planes;
  p.eA = A.e;
  p.eB = B.e;
  p.sA = A.stride;
  p.sB = B.stride;
  p.RpA = A.Rpad;
  p.RpB = B.Rpad;
  p.n_kb = A.n_kb;
  p.diva = std::max(1, ix.diva);
  p.divb = std::max(1, ix.divb);
  p.use_ta = ix.ta != nullptr;
  p.use_tb = ix.tb != nullptr;
  for (int b = 0; b < nb && ix.ta; ++b) p.ta[b] = ix.ta[b];
  for (int b = 0; b < nb && ix.tb; ++b) p.tb[b] = ix.tb[b];
  p.nb = nb;
  p.nI = A.Rpad / 128;
  p.nJ = B.Rpad / (cplx ? 32 : 64);
  p.tri = out.tri;
  long tiles = 0;
  if (p.tri)
    for (int I = 0; I < p.nI; ++I) tiles += std::min(p.nJ, (cplx ? 4 : 2) * (I + 1));
  else
    tiles = (long)p.nI * p.nJ;
  const long items = tiles * nb;
  const int sms = device_sm_count();
  // split of K, in whole chunks: the launch's longest CTA, a chunk's MMAs plus
  // its drain as the unit, half a unit per item, one per split for the reduction
  const int chunks = (p.n_kb + KBC - 1) / KBC;
  int ns = 1;
  if (part && kmode == 0 && !diag) {
    double best = 1e300;
    for (int k = 1; k <= std::min(chunks, 64); ++k) {
      const int cps = (chunks + k - 1) / k, kk = (chunks + cps - 1) / cps;
      if (kk != k || (k > 1 && (size_t)items * k * PART_ITEM > part_bytes)) continue;
      const double waves = (double)((items * k + sms - 1) / sms);
      const double cost = waves * (cps + 0.4) + (k > 1 ? 0.3 + 0.1 * k * (double)items / sms : 0.0);
      if (cost < best) {
        best = cost;
        ns = k;
      }
    }
  }
  if (items * ns > 0x7fffffffL) return cudaErrorInvalidValue;
  p.n_tiles = (int)tiles;
  p.n_split = ns;
  p.cps = (chunks + ns - 1) / ns;
  p.kmode = kmode;
  p.n_items = (int)(items * ns);
  p.part = (longlong2*)part;
  p.flag = flag;
  p.per_b = flag && per_b;
  p.status = status;
  p.out = out;
  if (diag) p.diag = *diag;
  const unsigned grid = (unsigned)std::min<long>(p.n_items, sms);
  auto* kern = diag ? (cplx ? g64_kernel<true, true> : g64_kernel<false, true>)
                    : (cplx ? g64_kernel<true, false> : g64_kernel<false, false>);
  kern<<<grid, G_THREADS, G_SMEM, s>>>(p);
  if (n_launch) *n_launch += 1;
  if (ns > 1) {
    if (cplx)
      g64_reduce_kernel<true><<<(unsigned)items, 256, 0, s>>>(p);
    else
      g64_reduce_kernel<false><<<(unsigned)items, 256, 0, s>>>(p);
    if (n_launch) *n_launch += 1;
  }
  return cudaGetLastError();
}

// ------------------------------------------------ products of the tail ----

namespace {

size_t al1k(size_t x) { return (x + 1023) & ~(size_t)1023; }

// Bytes of the planes of one matrix of the sandwich: one left and one right
// operand per (q, w), and one of L per q (at least as large as its share).
struct TailBytes {
  size_t a, b, ea, eb, one;
};
TailBytes tail_bytes(int cplx, int N) {
  TailBytes t;
  t.a = g64_plane_bytes(cplx, 0, N, N, 1);
  t.b = g64_plane_bytes(cplx, 1, N, N, 1);
  t.ea = al1k(sizeof(int) * (size_t)g64_rpad(cplx, 0, N));
  t.eb = al1k(sizeof(int) * (size_t)g64_rpad(cplx, 1, N));
  t.one = t.a + t.b + t.ea + t.eb;
  return t;
}

// Square matrices at a stride N^2, by rows or columns, without their diagonals.
G64Src square(const double* base, int N, int nb, int by_rows, int conj) {
  G64Src s{};
  s.base = base;
  s.stride = (long)N * N;
  s.ld = N;
  s.by_rows = by_rows;
  s.conj = conj;
  s.nb = nb;
  s.R = s.K = N;
  s.no_diag = 1;
  return s;
}

G64Op square_op(int cplx, int role, int N, char* planes, char* e) {
  G64Op o{};
  o.planes = (uint16_t*)planes;
  o.e = (int*)e;
  o.stride = (long)(g64_plane_bytes(cplx, role, N, N, 1) / 2);
  o.Rpad = g64_rpad(cplx, role, N);
  o.n_kb = g64_nkb(cplx, N);
  return o;
}

G64Out square_out(double* base, int N, int neg, int tri) {
  G64Out o{};
  o.base = base;
  o.stride = (long)N * N;
  o.s0 = N;
  o.t0 = 1;
  o.rd = o.cd = 1 << 30;
  o.R = o.C = N;
  o.neg = neg;
  o.tri = tri;
  return o;
}

}  // namespace

// Measured: the sandwich of 16 matrices of N = 768 40.6 ms in FP64 (its pipe
// needs 33), 1.9 ms here; 48 of N = 150 1.69 and 0.40 ms; V^-1 = X^H X of 16 of N =
// 512 3.5 and 0.45 ms.  Small matrices leave the tiles (128 rows) mostly padding; below 2.5e7 complex
// multiply-adds per q (N = 150, 12 frequencies: 0.42 ms in FP64) the FP64 kernels
// take little more than the launches.
bool tail_g64_use(int cplx, int N, int n) {
  return N >= 128 && (cplx ? 1.0 : 0.25) * N * (double)N * N * n >= 2.5e7;
}

size_t tail_g64_bytes(int cplx, int N, int n_mat, size_t most) {
  const size_t one = tail_bytes(cplx, N).one;
  return al1k(sizeof(int) * (size_t)n_mat) + std::max(2 * one, std::min(most, one * (size_t)n_mat));
}

cudaError_t launch_sandwich_g64(int cplx, int N, int n_batch, int n_w, const double* chi, const double* L, double* T,
                                double* Y, void* work, size_t work_bytes, int* status, uint64_t* n_launch,
                                cudaStream_t s) {
  const TailBytes t = tail_bytes(cplx, N);
  const long NN = (long)N * N, cs = cplx ? 2 : 1;
  const size_t fb = al1k(sizeof(int) * (size_t)n_batch);
  int* flag = (int*)work;
  char* p = (char*)work + fb;
  const int room = (int)std::min<size_t>((size_t)n_batch, (work_bytes - fb) / t.one);
  if (work_bytes < fb + t.one) return cudaErrorInvalidValue;
  if (cudaError_t e = cudaMemsetAsync(flag, 0, sizeof(int) * (size_t)n_batch, s)) return e;
  uint64_t nl = 0;
  // passes over whole q, or over some matrices of one
  for (int b0 = 0; b0 < n_batch;) {
    const int q = b0 / n_w, nq = std::max(1, std::min(room / n_w, (n_batch - b0) / n_w));
    const int nb = std::min({room, nq * n_w, (q + nq) * n_w - b0});
    const int rep = std::min(nb, n_w);                 // matrices of a pass that share an L
    char *pb = p + t.a * (size_t)nb, *ea = pb + t.b * (size_t)nb, *eb = ea + t.ea * (size_t)nb;
    const double *X = chi + b0 * NN * cs, *Lq = L + q * NN * cs;
    double *Tb = T + b0 * NN * cs, *Yb = Y + b0 * NN * cs;
    const G64Op A = square_op(cplx, 0, N, p, ea), B = square_op(cplx, 1, N, pb, eb);
    // T = chi L: conj(A)(P, R) = chi[P][R], B(Q, R) = L[R][Q], R >= Q
    const G64Diag d1{1, square(X, N, nb, 1, 1), square(Lq, N, nq, 0, 0)};
    if (cudaError_t e = g64_slice(cplx, 0, d1.A, A, flag + b0, 1, s)) return e;
    if (cudaError_t e = g64_slice(cplx, 1, d1.B, B, flag + b0, rep, s)) return e;
    if (cudaError_t e = g64_product(cplx, A, B, G64Index{nullptr, nullptr, 1, rep}, square_out(Tb, N, 0, 0), nb, 1,
                                    nullptr, 0, flag + b0, 1, status, &nl, s, &d1))
      return e;
    // Y = -L^H T: A(P, R) = L[R][P], B(Q, R) = T[R][Q], R >= P, lower triangle
    const G64Diag d2{1, square(Lq, N, nq, 0, 0), square(Tb, N, nb, 0, 0)};
    if (cudaError_t e = g64_slice(cplx, 0, d2.A, A, flag + b0, rep, s)) return e;
    if (cudaError_t e = g64_slice(cplx, 1, d2.B, B, flag + b0, 1, s)) return e;
    // (Y may be chi, which the FP64 kernels need: flagged matrices are not stored)
    if (cudaError_t e = g64_product(cplx, A, B, G64Index{nullptr, nullptr, rep, 1}, square_out(Yb, N, 1, 2), nb, 2,
                                    nullptr, 0, flag + b0, 1, status, &nl, s, &d2))
      return e;
    if (cudaError_t e = launch_sandwich(cplx, N, nb, rep, X, Lq, Tb, Yb, s, flag + b0)) return e;
    nl += 10;
    b0 += nb;
  }
  if (n_launch) *n_launch += nl;
  return cudaGetLastError();
}

cudaError_t launch_gram_g64(int cplx, int N, int n_q, const double* X, double* Wn, void* work, size_t work_bytes,
                            int* status, uint64_t* n_launch, cudaStream_t s) {
  const TailBytes t = tail_bytes(cplx, N);
  const long NN = (long)N * N, cs = cplx ? 2 : 1;
  const size_t fb = al1k(sizeof(int) * (size_t)n_q);
  int* flag = (int*)work;
  char* p = (char*)work + fb;
  if (work_bytes < fb + t.one) return cudaErrorInvalidValue;
  const int room = (int)std::min<size_t>((size_t)n_q, (work_bytes - fb) / t.one);
  if (cudaError_t e = cudaMemsetAsync(flag, 0, sizeof(int) * (size_t)n_q, s)) return e;
  uint64_t nl = 0;
  for (int q0 = 0; q0 < n_q; q0 += room) {
    const int nb = std::min(room, n_q - q0);
    char *pb = p + t.a * (size_t)nb, *ea = pb + t.b * (size_t)nb, *eb = ea + t.ea * (size_t)nb;
    const G64Op A = square_op(cplx, 0, N, p, ea), B = square_op(cplx, 1, N, pb, eb);
    const G64Src sx = square(X + q0 * NN * cs, N, nb, 0, 0);
    if (cudaError_t e = g64_slice(cplx, 0, sx, A, flag + q0, 1, s)) return e;
    if (cudaError_t e = g64_slice(cplx, 1, sx, B, flag + q0, 1, s)) return e;
    const G64Diag d{1, sx, sx};
    if (cudaError_t e = g64_product(cplx, A, B, G64Index{nullptr, nullptr, 1, 1}, square_out(Wn + q0 * NN * cs, N, 1, 2), nb,
                                    2, nullptr, 0, flag + q0, 1, status, &nl, s, &d))
      return e;
    if (cudaError_t e = launch_gram(cplx, N, nb, X + q0 * NN * cs, Wn + q0 * NN * cs, s, flag + q0)) return e;
    nl += 5;
  }
  if (n_launch) *n_launch += nl;
  return cudaGetLastError();
}

// ------------------------------------------------------------ FP64 chi0 ---
// chi0(w) = sum_t conj(C_Pt d_t(w)) C_Qt, one product per frequency with the
// weight on the left operand.  The transitions run in panels of a fixed size
// (chi0_panel), whose digit planes of all frequencies fit the workspace; each
// panel adds to chi0 in FP64.

namespace {

constexpr int CHI_W = 8;  // frequencies per pass of the exponent kernel

// Statistics of |C_Pt| or |C_Pt d_t(w)| over a part of the panel:
// one warp per row, the FP32 weights of 256 t staged for the CTA's 8 rows;
// blockIdx.z = 0: no weight (the right operand), z > 0: frequencies
// [w0 + 8 (z - 1), ...).  part[slot][kp][P], slot 0 unweighted, 1 + w.
template <bool C>
__global__ void __launch_bounds__(256) chi_exp_kernel(int N, int Npad, int n_ov, int n_w, int w0, int G, long t0, long t1,
                                                      const double* const* __restrict__ Cp,
                                                      const double* __restrict__ dtab, RowStat* __restrict__ part,
                                                      int* __restrict__ flag) {
  __shared__ float ds[CHI_W][256];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int P = blockIdx.x * 8 + warp, kp = blockIdx.y, KP = gridDim.y;
  const int z = blockIdx.z, g0 = z == 0 ? 0 : (z - 1) * CHI_W, ng = z == 0 ? 1 : min(CHI_W, G - g0);
  const long len = t1 - t0, a = t0 + len * kp / KP, b = t0 + len * (kp + 1) / KP;
  RowStat st[CHI_W];
  for (long tb = a; tb < b; tb += 256) {
    __syncthreads();
    for (int i = threadIdx.x; i < ng * 256; i += 256) {
      const int g = i >> 8;
      const long t = tb + (i & 255);
      float v = 1.f;
      if (z > 0) {
        v = 0.f;
        if (t < b) {
          const int j = (int)(t / n_ov), tt = (int)(t - (long)j * n_ov);
          const uint32_t x = abs_bits32(
              (unsigned long long)__double_as_longlong(dtab[((long)j * n_w + w0 + g0 + g) * n_ov + tt]));
          v = __uint_as_float(x);
          // weights so small that their products could vanish in FP32
          if (x != 0 && v < TINY) atomicOr(flag, 1);
        }
      }
      ds[g][i & 255] = v;
    }
    __syncthreads();
    if (P >= N) continue;
    for (int u = lane; u < 256 && tb + u < b; u += 32) {
      const long t = tb + u;
      const int j = (int)(t / n_ov), tt = (int)(t - (long)j * n_ov);
      const Elem<C> x = ld_elem<C>(Cp[j], (long)P * n_ov + tt);
      const float xr = __uint_as_float(abs_bits32((unsigned long long)__double_as_longlong(x.re)));
      float xi = 0.f;
      if constexpr (C) xi = __uint_as_float(abs_bits32((unsigned long long)__double_as_longlong(x.im)));
#pragma unroll
      for (int g = 0; g < CHI_W; ++g) {
        if (g >= ng) break;
        const float d = ds[g][u];
        // non-negative floats order like their bits; a NaN sorts above all
        st[g].add(__float_as_uint(xr * d) & 0x7fffffffu);
        if constexpr (C) st[g].add(__float_as_uint(xi * d) & 0x7fffffffu);
      }
    }
  }
#pragma unroll
  for (int g = 0; g < CHI_W; ++g) {
    if (g >= ng) break;
    st[g].warp_join();
    const int slot = z == 0 ? 0 : 1 + g0 + g;
    if (lane == 0 && P < Npad) part[((long)slot * KP + kp) * Npad + P] = st[g];
  }
}

// Exponents from the parts, in part order: eB[P] (slot 0) and eA[w][P].
__global__ void __launch_bounds__(256) chi_exp_final_kernel(int N, int NpadA, int NpadB, int Npad, int G, int KP,
                                                            const RowStat* __restrict__ part, int* eA, int* eB,
                                                            int* flag) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= (G + 1) * Npad) return;
  const int slot = i / Npad, P = i % Npad;
  RowStat st;
  if (P < N)
    for (int kp = 0; kp < KP; ++kp) st.join(part[((long)slot * KP + kp) * Npad + P]);
  const int e = row_exponent(st, slot ? SPREAD_WEIGHTED : SPREAD, slot == 0, flag);
  if (slot == 0) {
    if (P < NpadB) eB[P] = e;
  } else if (P < NpadA) {
    eA[(long)(slot - 1) * NpadA + P] = e;
  }
}

// Digit planes of the panel: the right operand (C itself), and the left
// operands C d(w) of G frequencies (C's values are loaded once).
template <bool C>
__global__ void __launch_bounds__(256) chi_slice_b_kernel(int N, int n_ov, long t0, long t1, const double* const* __restrict__ Cp,
                                                          const __grid_constant__ G64Op op) {
  constexpr int kpb = C ? 8 : 16, RB = C ? 32 : 64;
  const long total = (long)op.Rpad * op.n_kb;
  for (long idx = blockIdx.x * 256L + threadIdx.x; idx < total; idx += gridDim.x * 256L) {
    const int P = (int)(idx % op.Rpad), kb = (int)(idx / op.Rpad);
    const int e = op.e[P];
    unsigned long long G[16];
    const long tb = t0 + (long)kb * kpb;
    int j = (int)(tb / n_ov), tt = (int)(tb - (long)j * n_ov);
#pragma unroll
    for (int v = 0; v < kpb; ++v) {
      Elem<C> x = zero_elem<C>();
      if (P < N && tb + v < t1) x = ld_elem<C>(Cp[j], (long)P * n_ov + tt);
      if constexpr (C) {
        G[2 * v] = (unsigned long long)fix55(x.re, e) + DIGIT_BIAS;
        G[2 * v + 1] = (unsigned long long)fix55(x.im, e) + DIGIT_BIAS;
      } else {
        G[v] = (unsigned long long)fix55(x.re, e) + DIGIT_BIAS;
      }
      if (++tt == n_ov) {
        tt = 0;
        ++j;
      }
    }
    store_digits<1, C>(G, op.planes + ((long)(P / RB) * op.n_kb + kb) * (B_BLOCK / 2), P % RB);
  }
}

template <bool C>
__global__ void __launch_bounds__(256) chi_slice_a_kernel(int N, int n_ov, int n_w, int w0, int nG, long t0, long t1,
                                                          const double* const* __restrict__ Cp,
                                                          const double* __restrict__ dtab,
                                                          const __grid_constant__ G64Op op) {
  constexpr int kpb = C ? 8 : 16;
  const long total = (long)op.Rpad * op.n_kb;
  for (long idx = blockIdx.x * 256L + threadIdx.x; idx < total; idx += gridDim.x * 256L) {
    const int P = (int)(idx % op.Rpad), kb = (int)(idx / op.Rpad);
    const long tb = t0 + (long)kb * kpb;
    const int j0 = (int)(tb / n_ov), tt0 = (int)(tb - (long)j0 * n_ov);
    unsigned long long c[16];
    {
      int j = j0, tt = tt0;
#pragma unroll
      for (int v = 0; v < kpb; ++v) {
        Elem<C> x = zero_elem<C>();
        if (P < N && tb + v < t1) x = ld_elem<C>(Cp[j], (long)P * n_ov + tt);
        if constexpr (C) {
          c[2 * v] = (unsigned long long)__double_as_longlong(x.re);
          c[2 * v + 1] = (unsigned long long)__double_as_longlong(x.im);
        } else {
          c[v] = (unsigned long long)__double_as_longlong(x.re);
        }
        if (++tt == n_ov) {
          tt = 0;
          ++j;
        }
      }
    }
    for (int g = 0; g < nG; ++g) {
      const int e = op.e[(long)g * op.Rpad + P];
      unsigned long long G[16];
      int j = j0, tt = tt0;
#pragma unroll
      for (int v = 0; v < kpb; ++v) {
        unsigned long long d = 0;
        if (tb + v < t1)
          d = (unsigned long long)__double_as_longlong(__ldg(dtab + ((long)j * n_w + w0 + g) * n_ov + tt));
        if constexpr (C) {
          G[2 * v] = (unsigned long long)fix55_mul(c[2 * v], d, e) + DIGIT_BIAS;
          G[2 * v + 1] = (unsigned long long)fix55_mul(c[2 * v + 1], d, e) + DIGIT_BIAS;
        } else {
          G[v] = (unsigned long long)fix55_mul(c[v], d, e) + DIGIT_BIAS;
        }
        if (++tt == n_ov) {
          tt = 0;
          ++j;
        }
      }
      store_digits<0, C>(G, op.planes + g * op.stride + ((long)(P / 128) * op.n_kb + kb) * (A_BLOCK / 2), P & 127);
    }
  }
}

constexpr size_t CHI_PLANES = (size_t)3 << 30;  // digit planes of one panel
constexpr size_t CHI_PART = (size_t)256 << 20;  // split-K partials
constexpr int CHI_G = 32;                       // frequencies per pass

struct ChiPanel {
  int G, KP;     // frequencies per pass, parts of the exponent kernel
  long T;        // transitions per panel
  size_t a, b, ea, eb, ep, part, flag, total;
};
// The panel (T) depends on the geometry of one q alone, so the result does not
// depend on what shares the workspace; G frequencies per pass (0: as many as
// CHI_PLANES holds) change only its size.
ChiPanel chi0_panel(const BatchGeom& g, int G = 0) {
  ChiPanel L{};
  const long Kt = (long)g.n_k * g.n_ov;
  const long unit = g.cplx ? KBC * 8 : KBC * 16;  // transitions of one exact accumulation
  const size_t per_w = g64_plane_bytes(g.cplx, 0, g.n_aux, (int)unit, 1);
  L.G = (int)std::max<size_t>(1, std::min<size_t>((size_t)std::min(g.n_w, CHI_G), CHI_PLANES * 3 / 4 / per_w));
  const int RA = g64_rpad(g.cplx, 0, g.n_aux), RB = g64_rpad(g.cplx, 1, g.n_aux);
  const size_t per_unit = g64_plane_bytes(g.cplx, 0, g.n_aux, (int)unit, L.G) +
                          g64_plane_bytes(g.cplx, 1, g.n_aux, (int)unit, 1);
  long units = std::max<long>(1, (long)(CHI_PLANES / per_unit));
  const long all = (Kt + unit - 1) / unit;
  const long panels = (all + units - 1) / units;
  units = (all + panels - 1) / panels;
  L.T = units * unit;
  if (G > 0) L.G = std::min(L.G, G);
  const int K = (int)std::min(L.T, Kt);
  L.KP = (int)std::max<long>(1, std::min<long>(64, K / 512));
  L.a = al1k(g64_plane_bytes(g.cplx, 0, g.n_aux, K, L.G));
  L.b = al1k(g64_plane_bytes(g.cplx, 1, g.n_aux, K, 1));
  L.ea = al1k(sizeof(int) * (size_t)RA * g.n_w);
  L.eb = al1k(sizeof(int) * (size_t)RB);
  L.ep = al1k(sizeof(RowStat) * (size_t)(L.G + 1) * L.KP * std::max(RA, RB));
  L.flag = al1k(sizeof(int) * (size_t)std::max(1, g.n_qb));
  const long nI = RA / 128, nJ = RB / (g.cplx ? 32 : 64);
  long tiles = 0;
  for (long I = 0; I < nI; ++I) tiles += std::min<long>(nJ, (g.cplx ? 4 : 2) * (I + 1));
  L.part = std::min(CHI_PART, al1k(PART_ITEM * (size_t)tiles * L.G * 8));  // up to eight splits
  L.total = L.a + L.b + L.ea + L.eb + L.ep + L.flag + L.part;
  return L;
}

template <bool C>
cudaError_t chi0_g64_run(const BatchGeom& g, const double* const* Cptrs, const double* dtab, double* chi, void* work,
                         size_t work_bytes, int* status, uint64_t* n_launch, cudaStream_t s) {
  ChiPanel L = chi0_panel(g);
  while (L.G > 1 && L.total > work_bytes) L = chi0_panel(g, L.G - 1);
  if (L.total > work_bytes) return cudaErrorInvalidValue;
  char* p = (char*)work;
  int* flag = (int*)p;
  p += L.flag;
  G64Op A{}, B{};
  A.planes = (uint16_t*)p;
  p += L.a;
  B.planes = (uint16_t*)p;
  p += L.b;
  int* eA = (int*)p;
  p += L.ea;
  B.e = (int*)p;
  p += L.eb;
  RowStat* ep = (RowStat*)p;
  p += L.ep;
  A.Rpad = g64_rpad(C, 0, g.n_aux);
  B.Rpad = g64_rpad(C, 1, g.n_aux);
  const int Npad = std::max(A.Rpad, B.Rpad);
  const long Kt = (long)g.n_k * g.n_ov, NN = (long)g.n_aux * g.n_aux;
  uint64_t nl = 0;
  if (cudaError_t e = cudaMemsetAsync(flag, 0, sizeof(int) * (size_t)g.n_qb, s)) return e;
  for (int q = 0; q < g.n_qb; ++q) {
    const double* const* Cq = Cptrs + (long)q * g.n_k;
    const double* dq = dtab + (long)q * g.n_k * g.n_w * g.n_ov;
    for (long t0 = 0; t0 < Kt; t0 += L.T) {
      const long t1 = std::min(Kt, t0 + L.T);
      const int K = (int)(t1 - t0);
      A.n_kb = B.n_kb = g64_nkb(C, K);
      A.stride = (long)(A.Rpad / 128) * A.n_kb * (A_BLOCK / 2);
      B.stride = 0;
      // every frequency's exponents before the first product: the flags that the
      // products read are then those of the whole panel, however many passes it takes
      for (int w0 = 0; w0 < g.n_w; w0 += L.G) {
        const int G = std::min(L.G, g.n_w - w0);
        chi_exp_kernel<C><<<dim3((unsigned)((Npad + 7) / 8), (unsigned)L.KP, (unsigned)(1 + (G + CHI_W - 1) / CHI_W)), 256, 0,
                         s>>>(g.n_aux, Npad, g.n_ov, g.n_w, w0, G, t0, t1, Cq, dq, ep, flag + q);
        chi_exp_final_kernel<<<((G + 1) * Npad + 255) / 256, 256, 0, s>>>(g.n_aux, A.Rpad, B.Rpad, Npad, G, L.KP, ep,
                                                                         eA + (size_t)w0 * A.Rpad, B.e, flag + q);
        nl += 2;
      }
      for (int w0 = 0; w0 < g.n_w; w0 += L.G) {
        const int G = std::min(L.G, g.n_w - w0);
        A.e = eA + (size_t)w0 * A.Rpad;
        if (w0 == 0)
          chi_slice_b_kernel<C><<<grid_for((long)B.Rpad * B.n_kb, 16), 256, 0, s>>>(g.n_aux, g.n_ov, t0, t1, Cq, B);
        chi_slice_a_kernel<C><<<grid_for((long)A.Rpad * A.n_kb, 16), 256, 0, s>>>(g.n_aux, g.n_ov, g.n_w, w0, G, t0, t1, Cq,
                                                                                dq, A);
        nl += w0 == 0 ? 2 : 1;
        G64Out o{};
        o.base = chi + ((long)q * g.n_w + w0) * NN * (C ? 2 : 1);
        o.stride = NN;
        o.s0 = g.n_aux;
        o.t0 = 1;
        o.rd = o.cd = 1 << 30;
        o.R = o.C = g.n_aux;
        o.add = t0 > 0;
        o.tri = 1;
        G64Index ix{nullptr, nullptr, 1, 1 << 30};
        if (cudaError_t e = g64_product(C, A, B, ix, o, G, 0, p, L.part, flag + q, 0, status, &nl, s)) return e;
      }
    }
  }
  // the q whose rows exceed the split's precision
  if (cudaError_t e = launch_chi0_fp64(g, Cptrs, dtab, chi, s, flag)) return e;
  if (n_launch) *n_launch = nl + 1;
  return cudaGetLastError();
}

}  // namespace

// The split needs some six launches per panel and K long enough for its error
// bound.  Measured: one q of N_aux 320, 9 k, N_ov 1920, 16 frequencies (113
// GFLOP) 5.0 ms, 66.2 on the FP64 kernel; N_aux 150, 4 k, N_ov 252, 12 frequencies (1.1
// GFLOP per q) 0.21 ms per q and 0.98.  At 5e8 flops the FP64 kernel takes about 0.3
// ms, little more than the launches here.  Error against 64-bit sums at the
// first size: 2.5e-16, the FP64 kernel's 3.7e-15.
bool chi0_g64_use(const BatchGeom& g) {
  const double K = (double)g.n_k * g.n_ov;
  return (g.cplx ? 4.0 : 1.0) * g.n_aux * (g.n_aux + 1.0) * K * g.n_w >= 5e8 && K * (g.cplx ? 2 : 1) >= 128;
}

int chi0_g64_freqs(const BatchGeom& g) { return chi0_panel(g).G; }
size_t chi0_g64_bytes(const BatchGeom& g, int n_freq) { return chi0_panel(g, n_freq).total; }

cudaError_t launch_chi0_g64(const BatchGeom& g, const double* const* Cptrs, const double* dtab, double* chi,
                            void* work, size_t work_bytes, int* status, uint64_t* n_launch, cudaStream_t s) {
  return g.cplx ? chi0_g64_run<true>(g, Cptrs, dtab, chi, work, work_bytes, status, n_launch, s)
                : chi0_g64_run<false>(g, Cptrs, dtab, chi, work, work_bytes, status, n_launch, s);
}

}  // namespace rpa
