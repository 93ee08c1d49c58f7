// Float-float sums (h, l), |l| at most half a unit in the last place of h: Knuth's
// TwoSum, Dekker's TwoProd (by fma), a renormalisation per call.  Plain C++ on the
// host (compiled without contraction), round-to-nearest intrinsics on the device.
#pragma once
#include <math.h>

#ifdef __CUDACC__
#define RPA_FF __host__ __device__ __forceinline__
#else
#define RPA_FF inline
#endif

namespace rpa {

#ifdef __CUDA_ARCH__
RPA_FF float ff_add(float a, float b) { return __fadd_rn(a, b); }
RPA_FF float ff_sub(float a, float b) { return __fsub_rn(a, b); }
RPA_FF float ff_mul(float a, float b) { return __fmul_rn(a, b); }
#else
RPA_FF float ff_add(float a, float b) { return a + b; }
RPA_FF float ff_sub(float a, float b) { return a - b; }
RPA_FF float ff_mul(float a, float b) { return a * b; }
#endif

// h + l as a pair, |l| well below |h|.
RPA_FF void ff_norm(float& h, float& l) {
  const float s = h;
  h = ff_add(s, l);
  l = ff_sub(l, ff_sub(h, s));
}

// a + b = s + e exactly.
RPA_FF void ff_two_sum(float a, float b, float& s, float& e) {
  s = ff_add(a, b);
  const float v = ff_sub(s, a);
  e = ff_add(ff_sub(a, ff_sub(s, v)), ff_sub(b, v));
}

// (kx + ky)(x0 + x1) as p + t, ky x1 left out: the product's error and the cross terms in t.
RPA_FF void ff_prod(float kx, float ky, float x0, float x1, float& p, float& t) {
  p = ff_mul(kx, x0);
  t = fmaf(kx, x0, -p);
  t = fmaf(kx, x1, t);
  t = fmaf(ky, x0, t);
}

// (h, l) += p + t, t far below p.
RPA_FF void ff_acc(float& h, float& l, float p, float t) {
  float e;
  ff_two_sum(h, p, h, e);
  l = ff_add(l, ff_add(e, t));
  ff_norm(h, l);
}

// (h, l) += (kx + ky)(x0 + x1), 15 instructions.
RPA_FF void ff_fma(float& h, float& l, float kx, float ky, float x0, float x1) {
  float p, t;
  ff_prod(kx, ky, x0, x1, p, t);
  ff_acc(h, l, p, t);
}

// Two such terms, 27 instructions: the products are added first, all four error terms
// before they meet l.  Closer than two single steps (tests: 0.8 of their error).
RPA_FF void ff_fma2(float& h, float& l, float kx, float ky, float x0, float x1, float mx, float my, float y0, float y1) {
  float p, t, q, v, e, d;
  ff_prod(kx, ky, x0, x1, p, t);
  ff_prod(mx, my, y0, y1, q, v);
  ff_two_sum(p, q, p, e);
  ff_two_sum(h, p, h, d);
  l = ff_add(l, ff_add(ff_add(d, e), ff_add(t, v)));
  ff_norm(h, l);
}

}  // namespace rpa
