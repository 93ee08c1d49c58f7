// Host side of the periodic projector (Sec. 2.3): the Jacobi sweep loop with
// its convergence test, the rpa_projector entry point, and the regularised MO
// coefficients of AO-form jobs that carry overlap matrices.
#include <cuda_runtime.h>
#include <float.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "g64.h"
#include "proj_internal.h"
#include "rpa_internal.h"
#include "rpa_runtime.h"

namespace rpa {

namespace {
size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }
constexpr int kMaxSweeps = 60;
}  // namespace

ProjLayout proj_layout(int cplx, int n_mat, int N, int n_mo) {
  ProjLayout L;
  const size_t es = cplx ? 16 : 8;
  L.Np = N + (N & 1);
  L.W = 0;
  L.V = L.W + al256(es * (size_t)n_mat * L.Np * N);
  L.lam = L.V + al256(es * (size_t)n_mat * L.Np * N);
  L.rank = L.lam + al256(sizeof(double) * (size_t)n_mat * N);
  L.X = L.rank + al256(sizeof(int) * (size_t)n_mat * N);
  L.flags = L.X + al256(es * (size_t)n_mat * N * n_mo);
  L.bytes = L.flags + 256;
  return L;
}

// ------------------------------------------------------- fast start -------

namespace {

// S, one N x N product per k-point, the FP32 columns (W32, V32), diagonals,
// flags, and the digit planes of a group of k-points.
struct FastLayout {
  size_t S, M, f32, diag, flags, ea, eb, pa, pb, bytes;
  int group;
};
FastLayout fast_layout(int cplx, int n_mat, int N) {
  FastLayout L{};
  const size_t es = cplx ? 16 : 8, Np = N + (N & 1);
  L.S = 0;
  L.M = L.S + al256(es * n_mat * Np * N);
  L.f32 = L.M + al256(es * n_mat * N * N);
  L.diag = L.f32 + 2 * al256(es / 2 * n_mat * Np * N);
  L.flags = L.diag + al256(sizeof(double) * n_mat * N);
  const size_t a = g64_plane_bytes(cplx, 0, N, N, 1), b = g64_plane_bytes(cplx, 1, N, N, 1);
  L.group = (int)std::max<size_t>(1, std::min<size_t>((size_t)n_mat, ((size_t)512 << 20) / (a + b)));
  L.ea = L.flags + 256 + al256(sizeof(float) * n_mat);
  L.eb = L.ea + al256(sizeof(int) * (size_t)L.group * g64_rpad(cplx, 0, N));
  L.pa = (L.eb + al256(sizeof(int) * (size_t)L.group * g64_rpad(cplx, 1, N)) + 1023) & ~(size_t)1023;
  L.pb = L.pa + a * L.group;
  L.bytes = L.pb + b * L.group;
  return L;
}

constexpr int kSweeps32 = 14;
constexpr int kPolish = 4;
// largest cosine at which the columns count as orthogonal without an FP64 sweep
// that finds them so (the sweeps' own bar is this or wider)
constexpr float kOrthogonal = 1e-14f;

}  // namespace

// Bases below 64 functions keep the FP64 sweeps from V = I (7.1 ms for 63 functions
// at one k-point, 12 at 16); 64 functions take 2.5 and 2.8 ms with the start, 7.1
// and 12.3 without.
size_t proj_fast_bytes(int cplx, int n_mat, int N) {
  if (N < 64) return 0;
  const size_t b = fast_layout(cplx, n_mat, N).bytes;
  return b <= ((size_t)4 << 30) ? b : 0;
}

// out (columns of N at so per k-point) = or += conj(A) B over rows of A and B,
// as digit products (A rows or columns of matrices at sa, B columns at sb).
static cudaError_t fast_product(int cplx, int n_mat, int N, char* ws, const double* A, long sa, int a_rows, int a_conj,
                                const double* B, long sb, double* out, long so, int add, uint64_t* nl, cudaStream_t s) {
  const FastLayout L = fast_layout(cplx, n_mat, N);
  const size_t cs = cplx ? 2 : 1;
  int* flag = (int*)(ws + L.flags + 64);  // digit-plane flags (only bit 1 matters here)
  int* status = (int*)(ws + L.flags + 128);
  for (int k0 = 0; k0 < n_mat; k0 += L.group) {
    const int nb = std::min(L.group, n_mat - k0);
    auto src = [&](const double* p, long st, int rows, int cj) {
      G64Src x{};
      x.base = p + k0 * st * (long)cs;
      x.stride = st;
      x.ld = N;
      x.by_rows = rows;
      x.conj = cj;
      x.nb = nb;
      x.R = x.K = N;
      return x;
    };
    G64Op a{}, b{};
    a.planes = (uint16_t*)(ws + L.pa);
    a.e = (int*)(ws + L.ea);
    a.stride = (long)(g64_plane_bytes(cplx, 0, N, N, 1) / 2);
    a.Rpad = g64_rpad(cplx, 0, N);
    b.planes = (uint16_t*)(ws + L.pb);
    b.e = (int*)(ws + L.eb);
    b.stride = (long)(g64_plane_bytes(cplx, 1, N, N, 1) / 2);
    b.Rpad = g64_rpad(cplx, 1, N);
    a.n_kb = b.n_kb = g64_nkb(cplx, N);
    if (cudaError_t x = g64_slice(cplx, 0, src(A, sa, a_rows, a_conj), a, flag, 0, s)) return x;
    if (cudaError_t x = g64_slice(cplx, 1, src(B, sb, 1, 0), b, flag, 0, s)) return x;
    G64Out o{};
    o.base = out + k0 * so * (long)cs;
    o.stride = so;
    o.s0 = 1;
    o.t0 = N;
    o.rd = o.cd = 1 << 30;
    o.R = o.C = N;
    o.add = add;
    if (cudaError_t x = g64_product(cplx, a, b, G64Index{nullptr, nullptr, 1, 1}, o, nb, 0, nullptr, 0, flag, 0, status,
                                    nl, s))
      return x;
    *nl += 4;
  }
  return cudaSuccess;
}

// The largest cosine between two columns of W (digit planes: rounding at 2^-55
// of the largest entries), into *cosine, and the products' status word (a wait that
// ran out: the cosine means nothing) into *status_h; M is left with E for V += V E,
// W += W E, the first-order rotations of the pairs that take less than 2e-9 (its
// square, what V then lacks in orthonormality, is below rounding).
static cudaError_t column_cosine(int cplx, int n_mat, int N, int Np, char* ws, const double* W, float* cosine,
                                 int* status_h, uint64_t* nl, cudaStream_t s) {
  const FastLayout L = fast_layout(cplx, n_mat, N);
  double *M = (double*)(ws + L.M), *diag = (double*)(ws + L.diag);
  unsigned* off = (unsigned*)(ws + L.flags);
  const long cols = (long)Np * N;
  cudaError_t e = cudaMemsetAsync(off, 0, sizeof(unsigned), s);
  if (e == cudaSuccess) e = fast_product(cplx, n_mat, N, ws, W, cols, 1, 0, W, cols, M, (long)N * N, 0, nl, s);
  if (e == cudaSuccess) e = launch_proj_corr(cplx, n_mat, N, false, M, diag, 2e-9f, off, s);
  *nl += 2;
  if (e == cudaSuccess) e = cudaMemcpyAsync(cosine, off, sizeof *cosine, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(status_h, ws + L.flags + 128, sizeof *status_h, cudaMemcpyDeviceToHost, s);
  return e == cudaSuccess ? cudaStreamSynchronize(s) : e;
}

// V: eigenvectors of S (= W on entry) to nearly FP64 accuracy, W = S V.  The FP64
// sweeps from V = I took 13 sweeps of 16 ms on 16 overlaps of 256 functions (208
// ms); with this start none is left there (or one, where many columns stay close).
// *ok = false (W = S and V = I again) when the start did not give an
// orthonormal V: columns outside its range (proj_norm_kernel), no convergence.
static rpa_status fast_start(rpa_ctx* ctx, int cplx, int n_mat, int N, int Np, double* W, double* V,
                             const ProjPtrs& P, char* ws, cudaStream_t s, bool* ok,
                             float* cosine) {
  const FastLayout L = fast_layout(cplx, n_mat, N);
  double *S = (double*)(ws + L.S), *M = (double*)(ws + L.M), *diag = (double*)(ws + L.diag);
  const size_t es = cplx ? 16 : 8, cs = cplx ? 2 : 1;
  const long cols = (long)Np * N, full = (long)n_mat * cols * (long)cs;
  float *W32 = (float*)(ws + L.f32), *V32 = (float*)(ws + L.f32 + al256(es / 2 * n_mat * cols));
  unsigned* off = (unsigned*)(ws + L.flags);       // cosines, then |V^H V - I|
  int* status = (int*)(ws + L.flags + 128);
  float* scale = (float*)(ws + L.flags + 256);
  cudaError_t e = cudaSuccess;
  uint64_t nl = 0;
  *ok = false;
  auto fail = [&](const char* what) {
    ctx_set_error(ctx, "projector: %s failed: %s", what, cudaGetErrorString(e));
    return RPA_E_CUDA;
  };
#define CKP(call)                               \
  do {                                          \
    if ((e = (call)) != cudaSuccess) return fail(#call); \
  } while (0)
  CKP(cudaMemsetAsync(ws + L.flags, 0, 256, s));
  CKP(cudaMemcpyAsync(S, W, es * n_mat * cols, cudaMemcpyDeviceToDevice, s));
  CKP(launch_proj_load32(cplx, n_mat, N, Np, W, scale, W32, V32, s));
  nl += 2;
  float off_h = 1.f;
  for (int sweep = 0; sweep < kSweeps32 && off_h > 3e-6f; ++sweep) {
    CKP(cudaMemsetAsync(off, 0, sizeof(unsigned), s));
    const int n = launch_jacobi32_sweep(cplx, n_mat, N, Np, W32, V32, 1e-7f, off, s);
    if (n < 0) CKP((cudaError_t)-n);
    nl += n;
    CKP(cudaMemcpyAsync(&off_h, off, sizeof off_h, cudaMemcpyDeviceToHost, s));
    CKP(cudaStreamSynchronize(s));
    if (!(off_h < 1e30f)) {  // W and V are as they were
      ctx->launches += nl;
      return RPA_OK;
    }
  }
  CKP(launch_proj_widen(full, V32, V, s));
  ++nl;
  auto product = [&](const double* A, long sa, int a_rows, int a_conj, const double* B, long sb, double* out, long so,
                     int add) { return fast_product(cplx, n_mat, N, ws, A, sa, a_rows, a_conj, B, sb, out, so, add, &nl, s); };
  const long NN = (long)N * N;
  auto update = [&]() { return product(V, cols, 0, 1, M, NN, V, cols, 1); };  // V += V M
  auto ortho = [&]() -> cudaError_t {
    cudaError_t x = cudaMemsetAsync(off, 0, sizeof(unsigned), s);
    if (x == cudaSuccess) x = product(V, cols, 1, 0, V, cols, M, NN, 0);
    if (x == cudaSuccess) x = launch_proj_corr(cplx, n_mat, N, true, M, diag, 0.f, off, s);
    ++nl;
    return x == cudaSuccess ? update() : x;
  };
  CKP(ortho());
  CKP(ortho());
  for (int it = 0; it < 3; ++it) {
    CKP(product(S, cols, 1, 0, V, cols, W, cols, 0));  // W = S V
    CKP(product(V, cols, 1, 0, W, cols, M, NN, 0));    // M = V^H S V
    CKP(launch_proj_corr(cplx, n_mat, N, false, M, diag, 0.02f, off, s));
    nl += 2;
    CKP(update());
    if (it < 2) CKP(ortho());
  }
  // orthonormal to rounding: a step squares what it finds
  float dev = 1.f;
  for (int it = 0; it < 4 && !(dev < 1e-9f); ++it) {
    CKP(ortho());
    CKP(cudaMemcpyAsync(&dev, off, sizeof dev, cudaMemcpyDeviceToHost, s));
    CKP(cudaStreamSynchronize(s));
  }
  CKP(product(S, cols, 1, 0, V, cols, W, cols, 0));
  // columns of W orthogonal to FP64 rounding: first-order rotations of all
  // pairs that take little, full ones among the few columns that remain
  float last = 2.f;
  int st = 0;
  for (int it = 0; dev < 1e-9f; ++it) {
    CKP(column_cosine(cplx, n_mat, N, Np, ws, W, cosine, &st, &nl, s));
    if (st || *cosine <= kOrthogonal || it == kPolish || !(*cosine < 0.5f * last)) break;
    last = *cosine;
    CKP(update());
    CKP(product(W, cols, 0, 1, M, NN, W, cols, 1));
    CKP(product(W, cols, 1, 0, W, cols, M, NN, 0));
    CKP(launch_proj_cluster(cplx, n_mat, N, Np, M, W, V, 1e-15, s));
    ++nl;
  }
  CKP(cudaMemcpyAsync(&st, status, sizeof st, cudaMemcpyDeviceToHost, s));
  CKP(cudaStreamSynchronize(s));
  ctx->launches += nl;
  if (st) return decode_status(ctx, st, 1);
  if (dev < 1e-9f) {
    *ok = true;
    return RPA_OK;
  }
  CKP(launch_proj_load(cplx, P, n_mat, N, Np, W, V, s));
  ctx->launches += 1;
  return RPA_OK;
#undef CKP
}

rpa_status run_projector(rpa_ctx* ctx, Exec* pex, int cplx, int n_mat, int N, int n_mo, const void* const* S,
                         const double* const* c, double* const* out, double eps_d, char* region, cudaStream_t s,
                         int* m_out, double* eig_host, char* fast) {
  if (n_mat > ProjPtrs::kMax) {
    ctx_set_error(ctx, "projector: at most %d k-points", ProjPtrs::kMax);
    return RPA_E_INVAL;
  }
  const ProjLayout L = proj_layout(cplx, n_mat, N, n_mo);
  ProjPtrs P{};
  for (int k = 0; k < n_mat; ++k) {
    P.S[k] = (const double*)S[k];
    P.c[k] = c[k];
    P.out[k] = out[k];
  }
  double* W = (double*)(region + L.W);
  double* V = (double*)(region + L.V);
  unsigned long long* off = (unsigned long long*)(region + L.flags);
  int* m = (int*)(region + L.flags + 64);
  auto fail = [&](cudaError_t e, const char* what) {
    ctx_set_error(ctx, "projector: %s failed: %s", what, cudaGetErrorString(e));
    return RPA_E_CUDA;
  };
  cudaError_t e = launch_proj_load(cplx, P, n_mat, N, L.Np, W, V, s);
  if (e != cudaSuccess) return fail(e, "load");
  ctx->launches += 1;
  // rotate pairs above the rounding level of a length-N inner product; stop
  // once no pair of a sweep is further from orthogonal than a few times that
  const double rot_thresh = 1e-15;
  const double conv = std::max(1e-14, 4.0 * N * DBL_EPSILON);
  int sweep = 0;
  double off_h = 1.0;
  bool started = false;
  float cosine = 1.f;
  prof_begin(ctx, pex, s);
  if (fast && proj_fast_bytes(cplx, n_mat, N)) {
    if (rpa_status st = fast_start(ctx, cplx, n_mat, N, L.Np, W, V, P, fast, s, &started, &cosine)) return st;
    if (started && cosine <= kOrthogonal) off_h = cosine;
  }

  for (; sweep < kMaxSweeps && off_h > conv; ++sweep) {
    if ((e = cudaMemsetAsync(off, 0, sizeof(unsigned long long), s)) != cudaSuccess) return fail(e, "memset");
    for (int r = 0; r < L.Np - 1; ++r)
      if ((e = launch_jacobi_round(cplx, n_mat, N, L.Np, r, W, V, rot_thresh, off, s)) != cudaSuccess)
        return fail(e, "Jacobi round");
    ctx->launches += L.Np - 1;
    unsigned long long bits = 0;
    if ((e = cudaMemcpyAsync(&bits, off, sizeof bits, cudaMemcpyDeviceToHost, s)) != cudaSuccess)
      return fail(e, "copy");
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return fail(e, "sync");
    memcpy(&off_h, &bits, sizeof off_h);
    // the sweep that would only find the columns orthogonal is a Gram product
    if (started && off_h > conv) {
      uint64_t nl = 0;
      int st = 0;
      if ((e = column_cosine(cplx, n_mat, N, L.Np, fast, W, &cosine, &st, &nl, s)) != cudaSuccess)
        return fail(e, "Gram product");
      ctx->launches += nl;
      if (st) return decode_status(ctx, st, 1);
      if (cosine <= kOrthogonal) off_h = cosine;
    }
  }
  prof_end(ctx, pex, s, RPA_K_PROJ, sweep * (L.Np - 1));
  if (off_h > conv) {
    ctx_set_error(ctx, "projector: Jacobi not converged after %d sweeps (off-orthogonality %.3g)", kMaxSweeps, off_h);
    return RPA_E_TIMEOUT;
  }
  if ((e = cudaMemsetAsync(m, 0, sizeof(int), s)) != cudaSuccess) return fail(e, "memset");
  if ((e = cudaMemsetAsync(region + L.rank, 0xff, sizeof(int) * (size_t)n_mat * N, s)) != cudaSuccess)
    return fail(e, "memset");
  prof_begin(ctx, pex, s);
  e = launch_proj_finish(cplx, P, n_mat, N, L.Np, n_mo, W, V, eps_d, (double*)(region + L.lam),
                         (int*)(region + L.rank), m, (double*)(region + L.X), s);
  if (e != cudaSuccess) return fail(e, "finish");
  prof_end(ctx, pex, s, RPA_K_PROJ, 3);
  ctx->launches += 3;
  int mh = 0;
  if ((e = cudaMemcpyAsync(&mh, m, sizeof(int), cudaMemcpyDeviceToHost, s)) != cudaSuccess) return fail(e, "copy");
  if (eig_host && (e = cudaMemcpyAsync(eig_host, region + L.lam, sizeof(double) * (size_t)n_mat * N,
                                       cudaMemcpyDeviceToHost, s)) != cudaSuccess)
    return fail(e, "copy");
  if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return fail(e, "sync");
  if (m_out) *m_out = mh;
  return RPA_OK;
}

}  // namespace rpa

using namespace rpa;

extern "C" rpa_status rpa_projector(rpa_ctx* ctx, const rpa_job* job, void* const* mo_out, double* eig_out,
                                    int* n_removed, void* stream) {
  if (!ctx) return RPA_E_INVAL;
  std::lock_guard<std::mutex> lk(ctx->mu);
  char msg[512];
  if (validate_job(job, msg, sizeof msg)) {
    ctx_set_error(ctx, "%s", msg);
    return RPA_E_INVAL;
  }
  if (!job->ao || !job->ao->overlap || !mo_out) {
    ctx_set_error(ctx, "rpa_projector: needs an AO-form job with overlap matrices and mo_out");
    return RPA_E_INVAL;
  }
  for (int k = 0; k < job->n_kpts; ++k)
    if (!mo_out[k]) {
      ctx_set_error(ctx, "rpa_projector: mo_out[%d] is NULL", k);
      return RPA_E_INVAL;
    }
  if (cudaSetDevice(ctx->device) != cudaSuccess) {
    ctx_set_error(ctx, "cudaSetDevice failed");
    return RPA_E_CUDA;
  }
  const rpa_ao* a = job->ao;
  int n_bas = 0;
  for (int A = 0; A < a->n_atoms; ++A) n_bas += a->n_bas_atom[A];
  const ProjLayout L = proj_layout(job->is_complex, job->n_kpts, n_bas, a->n_mo);
  Exec& ex = ctx->ex;
  const size_t base = (L.bytes + 1023) & ~(size_t)1023;
  size_t fb = proj_fast_bytes(job->is_complex, job->n_kpts, n_bas);
  if (base + fb > sync_ws_cap(ctx) || (fb && !ex.ensure_ws(base + fb))) fb = 0;
  if (!ex.ensure_ws(L.bytes)) {
    ctx_set_error(ctx, "cannot allocate %zu bytes of workspace", L.bytes);
    return RPA_E_NOMEM;
  }
  std::vector<const double*> c(job->n_kpts);
  std::vector<double*> out(job->n_kpts);
  for (int k = 0; k < job->n_kpts; ++k) {
    c[k] = (const double*)a->mo[k];
    out[k] = (double*)mo_out[k];
  }
  rpa_status st = run_projector(ctx, &ex, job->is_complex, job->n_kpts, n_bas, a->n_mo, a->overlap, c.data(),
                                out.data(), a->eps_d, (char*)ex.ws, (cudaStream_t)stream, n_removed, eig_out,
                                fb ? (char*)ex.ws + base : nullptr);
  prof_collect(ctx, &ex);
  return st;
}
