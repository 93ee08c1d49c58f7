// Host side of AO-form jobs (rpa_job.ao, Sec. 2.2): validation, the layout of
// the AO part of a lane's workspace, and the enqueue of the two transform
// kernels of kernels_ao.cu.
//
// Workspace region (offsets from Bufs.ao):
//   fit table   int4 per fit function gamma (see launch_ao_assemble)
//   PADF        lattice form only: one k-point's k-dependent PADF array
//   projector   with overlap matrices: the projector's workspace and the
//               regularised MO coefficients c~ of every k-point
//   H_occ       one S x n_occ slot per k-point that appears as k (pair_k)
//   H_virt      one S x n_virt slot per k-point that appears as k+q (pair_kq)
//   C           qb x n_k blocks n_aux x n_occ*n_virt: the MO-basis
//               coefficients of the q batch being processed (read by chi0)
// The half-transforms depend on the k-point only, so rpa_energy forms them
// once per job; each q then costs one assembly launch.
#include <cuda_runtime.h>
#include <math.h>
#include <stdio.h>

#include <algorithm>
#include <vector>

#include "ao_internal.h"
#include "g64.h"
#include "proj_internal.h"
#include "rpa_internal.h"
#include "rpa_runtime.h"

namespace rpa {

namespace {
size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }
}  // namespace

int ao_validate(const rpa_job* j, char* msg, size_t len) {
  auto fail = [&](const char* m) {
    if (msg && len) snprintf(msg, len, "%s", m);
    return RPA_E_INVAL;
  };
  const rpa_ao* a = j->ao;
  if (j->C) return fail("AO-form job: C must be NULL (the coefficients are formed from ao)");
  if (j->mem != RPA_MEM_DEVICE) return fail("AO-form job: inputs must be in device memory");
  if (a->n_atoms <= 0 || !a->n_bas_atom || !a->n_fit_atom || !a->mo)
    return fail("AO-form job: n_atoms must be positive and the ao arrays non-NULL");
  if (a->n_R < 0 || a->n_R > PadfLattice::kMax)
    return fail("AO-form job: n_R must lie in [0, 128]");
  if (a->n_R > 0) {
    if (a->padf) return fail("AO-form job: give padf or the lattice form (n_R > 0), not both");
    if (!a->lattice || !a->kfrac || !a->padf_R) return fail("AO-form job: lattice form needs lattice, kfrac, padf_R");
    for (int r = 0; r < a->n_R; ++r)
      if (!a->padf_R[r]) return fail("AO-form job: a padf_R pointer is NULL");
    for (int k = 0; k < 3 * j->n_kpts; ++k) {
      if (!isfinite(a->kfrac[k])) return fail("AO-form job: kfrac not finite");
      if (!j->is_complex && a->kfrac[k] != floor(a->kfrac[k]))
        return fail("AO-form job: real (Gamma-only) lattice-form jobs need integer kfrac");
    }
  } else if (!a->padf) {
    return fail("AO-form job: padf is NULL and no lattice form given");
  }
  long nb = 0, nf = 0, S = 0;
  for (int A = 0; A < a->n_atoms; ++A) {
    if (a->n_bas_atom[A] <= 0 || a->n_fit_atom[A] <= 0)
      return fail("AO-form job: every atom needs at least one basis and one fit function");
    nb += a->n_bas_atom[A];
    nf += a->n_fit_atom[A];
    S += (long)a->n_bas_atom[A] * a->n_fit_atom[A];
  }
  if (nf != j->n_aux) return fail("AO-form job: fit functions per atom must sum to n_aux");
  if (a->overlap) {
    if (j->n_kpts > ProjPtrs::kMax) return fail("AO-form job: the projector takes at most 256 k-points");
    if (nb > 6144) return fail("AO-form job: the projector takes n_bas <= 6144");
    if (!isfinite(a->eps_d) || a->eps_d < 0.0) return fail("AO-form job: eps_d must be finite and >= 0");
    for (int k = 0; k < j->n_kpts; ++k)
      if (!a->overlap[k]) return fail("AO-form job: an overlap pointer is NULL");
  }
  if (a->n_mo < j->n_occ + j->n_virt || a->n_mo > nb)
    return fail("AO-form job: n_mo must lie in [n_occ + n_virt, n_bas]");
  if (nb > 65536 || S > (1L << 30)) return fail("AO-form job: basis or PADF array too large");
  for (int k = 0; k < j->n_kpts; ++k)
    if ((a->n_R == 0 && !a->padf[k]) || !a->mo[k]) return fail("AO-form job: a padf or mo pointer is NULL");
  return RPA_OK;
}

AoPlan ao_plan(const rpa_job* j, int qb) {
  AoPlan p;
  const rpa_ao* a = j->ao;
  const size_t es = j->is_complex ? 16 : 8;
  for (int A = 0; A < a->n_atoms; ++A) {
    p.n_bas += a->n_bas_atom[A];
    p.S += a->n_bas_atom[A] * a->n_fit_atom[A];
  }
  p.fit.resize(j->n_aux);
  for (int A = 0, b0 = 0, f0 = 0, s0 = 0; A < a->n_atoms; ++A) {
    const int nb = a->n_bas_atom[A], nf = a->n_fit_atom[A];
    for (int g = 0; g < nf; ++g) p.fit[f0 + g] = make_int4(b0, nb, s0 + g, nf);
    b0 += nb;
    f0 += nf;
    s0 += nb * nf;
  }
  p.occ_slot.assign(j->n_kpts, -1);
  p.virt_slot.assign(j->n_kpts, -1);
  for (long i = 0; i < (long)j->n_q * j->n_k; ++i) {
    if (p.occ_slot[j->pair_k[i]] < 0) p.occ_slot[j->pair_k[i]] = p.n_occ_slots++;
    if (p.virt_slot[j->pair_kq[i]] < 0) p.virt_slot[j->pair_kq[i]] = p.n_virt_slots++;
  }
  p.occ_bytes = al256(es * (size_t)p.S * j->n_occ);
  p.virt_bytes = al256(es * (size_t)p.S * j->n_virt);
  p.cblk = es * (size_t)j->n_aux * j->n_occ * j->n_virt;
  p.off_padf = al256(sizeof(int4) * (size_t)j->n_aux);
  p.padf_bytes = a->n_R > 0 ? al256(es * (size_t)p.n_bas * p.S) : 0;
  p.off_proj = p.off_padf + p.padf_bytes;
  size_t proj_bytes = 0;
  if (a->overlap) {
    proj_bytes = al256(proj_layout(j->is_complex, j->n_kpts, p.n_bas, a->n_mo).bytes);
    p.cproj_bytes = al256(es * (size_t)p.n_bas * a->n_mo);
  }
  p.off_cproj = p.off_proj + proj_bytes;
  p.off_hocc = p.off_cproj + p.cproj_bytes * (a->overlap ? j->n_kpts : 0);
  p.off_hvirt = p.off_hocc + p.occ_bytes * p.n_occ_slots;
  p.off_c = p.off_hvirt + p.virt_bytes * p.n_virt_slots;
  p.bytes = p.off_c + al256(p.cblk * j->n_k * (size_t)std::max(qb, 1));
  return p;
}

size_t ao_region_bytes(const rpa_job* j, int qb) { return j->ao ? ao_plan(j, qb).bytes : 0; }

size_t ao_input_bytes(const rpa_job* j) {
  if (!j->ao) return 0;
  const AoPlan p = ao_plan(j, 1);
  const size_t es = j->is_complex ? 16 : 8;
  if (j->ao->n_R > 0)
    return 8 * (size_t)j->ao->n_R * p.n_bas * p.S + es * (size_t)j->n_kpts * p.n_bas * j->ao->n_mo;
  return es * (size_t)j->n_kpts * p.n_bas * ((size_t)p.S + j->ao->n_mo);
}

#define CKA(call)                                                                                    \
  do {                                                                                               \
    cudaError_t e_ = (call);                                                                         \
    if (e_ != cudaSuccess) {                                                                         \
      ctx_set_error(ctx, "%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, __LINE__); \
      return RPA_E_CUDA;                                                                             \
    }                                                                                                \
  } while (0)

const double* ao_mo(const rpa_job* j, const AoPlan& p, const char* region, int k) {
  if (j->ao->overlap) return (const double*)(region + p.off_cproj + p.cproj_bytes * (size_t)k);
  return (const double*)j->ao->mo[k];
}

rpa_status ao_project(rpa_ctx* ctx, Exec* pex, const rpa_job* j, const AoPlan& p, char* region, cudaStream_t s,
                      char* gws) {
  const rpa_ao* a = j->ao;
  if (!a->overlap) return RPA_OK;
  std::vector<const double*> c(j->n_kpts);
  std::vector<double*> out(j->n_kpts);
  for (int k = 0; k < j->n_kpts; ++k) {
    c[k] = (const double*)a->mo[k];
    out[k] = (double*)(region + p.off_cproj + p.cproj_bytes * (size_t)k);
  }
  return run_projector(ctx, pex, j->is_complex, j->n_kpts, p.n_bas, a->n_mo, a->overlap, c.data(), out.data(),
                       a->eps_d, region + p.off_proj, s, nullptr, nullptr, gws ? gws + 1024 : nullptr);
}

// ------------------------------------------------ digit products ----------
// Both transforms are contractions of FP64 arrays whose FP64 form is bound by
// the FP64 pipe (0.98 of it).  One q of 2 x (96 basis, 192 fit), 16 k-points,
// 192 orbitals: 180 ms in FP64, 11.7 ms here (slicing and stores about half of
// it); error against 113-bit sums 9.9e-16 in FP64, 4.0e-16 here.  As digit products
// (g64.cu):
//   half:  H[s][n] = sum_nu P[nu][s] c[nu][n]; left rows s, right rows n; the PADF
//          planes serve the occupied and the virtual columns.
//   C, 1:  sum_mu H_virt[mu][(gamma, a)] conj(c_{mu i}); left rows (gamma, a) (the
//          fit functions of an atom and the virtual states are contiguous in
//          H), right rows i, stored at [gamma][i][a].
//   C, 2:  sum_nu c_{nu a} conj(H_occ[nu][(gamma, i)]); left rows a, right rows
//          (gamma, i), added.
// Planes are bounded by running over panels of PADF columns or fit functions
// and batches of k-points or pairs.  A row outside the split's range makes the
// FP64 kernels redo the batch.

namespace {

constexpr size_t kAoPlanes = (size_t)1 << 30;  // planes of one batch, each side

struct AoAtom {
  int b0, nb, f0, nf, s0;  // first basis function, their count, fit functions, first PADF column
};
std::vector<AoAtom> ao_atoms(const rpa_ao* a) {
  std::vector<AoAtom> v;
  for (int A = 0, b0 = 0, f0 = 0, s0 = 0; A < a->n_atoms; ++A) {
    const int nb = a->n_bas_atom[A], nf = a->n_fit_atom[A];
    v.push_back(AoAtom{b0, nb, f0, nf, s0});
    b0 += nb;
    f0 += nf;
    s0 += nb * nf;
  }
  return v;
}

// One assembly step of an atom: fit functions per panel and pairs per batch.
struct AsmStep {
  int g, np;
};
AsmStep asm_step(const rpa_job* j, const AoAtom& t) {
  const int c = j->is_complex;
  auto bytes = [&](int g) {
    return std::max(g64_plane_bytes(c, 0, g * j->n_virt, t.nb, 1), g64_plane_bytes(c, 1, g * j->n_occ, t.nb, 1));
  };
  // row counts stay far below 2^31 also before the planes' bound applies
  AsmStep s{std::min(t.nf, std::max(1, (1 << 29) / std::max(j->n_virt, j->n_occ))), 1};
  while (s.g > 1 && bytes(s.g) > kAoPlanes) s.g = (s.g + 1) / 2;
  if (s.g == t.nf) s.np = (int)std::max<size_t>(1, std::min<size_t>(G64_TAB, kAoPlanes / bytes(s.g)));
  s.np = std::min(s.np, j->n_k);
  return s;
}

// Planes and exponents of one operand of a batch, carved at planes / e.
G64Op op_of(int cplx, int role, int R, int K, char* planes, char* e) {
  G64Op o{};
  o.planes = (uint16_t*)planes;
  o.e = (int*)e;
  o.stride = (long)(g64_plane_bytes(cplx, role, R, K, 1) / 2);
  o.Rpad = g64_rpad(cplx, role, R);
  o.n_kb = g64_nkb(cplx, K);
  return o;
}

G64Src src_of(int by_rows, int conj, int R, int K, long ld, int nb) {
  G64Src s{};
  s.use_tab = 1;
  s.by_element = 1;
  s.by_rows = by_rows;
  s.conj = conj;
  s.R = R;
  s.K = K;
  s.ld = ld;
  s.nb = nb;
  return s;
}

}  // namespace

// The FP64 kernels stay for contractions shorter than 32 real terms (the
// split's error is no smaller than theirs there) and for small jobs, whose
// FP64 time is near that of the extra launches: below 2e8 flops, 0.2 ms.
AoG64 ao_g64_plan(const rpa_job* j, const AoPlan& p) {
  AoG64 g;
  const int c = j->is_complex, cm = c ? 2 : 1;
  const double f = c ? 8.0 : 2.0;
  const long n_mo = j->n_occ + j->n_virt;
  g.half = p.n_bas * cm >= 32 && f * p.S * (double)p.n_bas * n_mo >= 2e8;
  int nb_min = 1 << 30;
  const std::vector<AoAtom> at = ao_atoms(j->ao);
  for (const AoAtom& t : at) nb_min = std::min(nb_min, t.nb);
  g.assemble = nb_min * cm >= 32 && f * 2.0 * p.S * j->n_occ * (double)j->n_virt * j->n_k >= 2e8 * at.size();
  if (j->ao->overlap) {  // the projector's fast start uses the region before the transforms
    const size_t f = proj_fast_bytes(c, j->n_kpts, p.n_bas);
    if (f) g.bytes = 1024 + f;
  }
  if (!g.half && !g.assemble) return g;
  if (g.half) {
    g.rows = p.S;
    const size_t all = g64_plane_bytes(c, 0, p.S, p.n_bas, 1);
    if (all > kAoPlanes) {
      const size_t blk = g64_plane_bytes(c, 0, 128, p.n_bas, 1);
      g.rows = (int)(128 * std::max<size_t>(1, kAoPlanes / blk));
    } else if (j->ao->n_R == 0) {
      g.k_batch = (int)std::max<size_t>(1, std::min<size_t>({(size_t)G64_TAB, (size_t)j->n_kpts, kAoPlanes / all}));
    }
    g.a = g64_plane_bytes(c, 0, g.rows, p.n_bas, g.k_batch);
    g.b = g64_plane_bytes(c, 1, std::max(j->n_occ, j->n_virt), p.n_bas, g.k_batch);
    g.e = sizeof(int) * (size_t)g.k_batch * std::max(g64_rpad(c, 0, g.rows), g64_rpad(c, 1, (int)n_mo));
  }
  if (g.assemble)
    for (const AoAtom& t : at) {
      const AsmStep st = asm_step(j, t);
      g.a = std::max({g.a, g64_plane_bytes(c, 0, st.g * j->n_virt, t.nb, st.np), g64_plane_bytes(c, 0, j->n_virt, t.nb, st.np)});
      g.b = std::max({g.b, g64_plane_bytes(c, 1, st.g * j->n_occ, t.nb, st.np), g64_plane_bytes(c, 1, j->n_occ, t.nb, st.np)});
      g.e = std::max(g.e, sizeof(int) * (size_t)st.np * std::max(g64_rpad(c, 0, st.g * j->n_virt), g64_rpad(c, 1, st.g * j->n_occ)));
    }
  g.a = (g.a + 1023) & ~(size_t)1023;
  g.b = (g.b + 1023) & ~(size_t)1023;
  g.e = (g.e + 1023) & ~(size_t)1023;
  g.bytes = std::max(g.bytes, 1024 + g.a + g.b + 2 * g.e);
  return g;
}

rpa_status ao_enqueue_half(rpa_ctx* ctx, Exec* pex, const rpa_job* j, const AoPlan& p, char* region, int q,
                           cudaStream_t s, char* gws, int* status) {
  const rpa_ao* a = j->ao;
  // the fit table (small, pageable source: consumed before the call returns)
  CKA(cudaMemcpyAsync(region, p.fit.data(), sizeof(int4) * p.fit.size(), cudaMemcpyHostToDevice, s));
  std::vector<char> need_o(j->n_kpts, 0), need_v(j->n_kpts, 0);
  const int q0 = q < 0 ? 0 : q, q1 = q < 0 ? j->n_q : q + 1;
  for (int qq = q0; qq < q1; ++qq)
    for (int jj = 0; jj < j->n_k; ++jj) {
      need_o[j->pair_k[(size_t)qq * j->n_k + jj]] = 1;
      need_v[j->pair_kq[(size_t)qq * j->n_k + jj]] = 1;
    }
  PadfLattice lat{};
  if (a->n_R > 0) {
    lat.n_R = a->n_R;
    for (int r = 0; r < a->n_R; ++r) {
      for (int d = 0; d < 3; ++d) lat.R[r][d] = a->lattice[3 * r + d];
      lat.C0[r] = (const double*)a->padf_R[r];
    }
  }
  int n = 0;
  const AoG64 g = gws ? ao_g64_plan(j, p) : AoG64{};
  int* flag = (int*)gws;
  prof_begin(ctx, pex, s);
  if (g.half) CKA(cudaMemsetAsync(flag, 0, sizeof(int), s));
  // H of the k-points ks as digit products, PADF arrays Ps
  auto half_g64 = [&](const std::vector<int>& ks, const std::vector<const double*>& Ps) -> rpa_status {
    const int c = j->is_complex, nb = (int)ks.size(), cs = c ? 2 : 1;
    char* pl = gws + 1024;
    uint64_t nl = 0;
    for (int r0 = 0; r0 < p.S; r0 += g.rows) {
      const int R = std::min(g.rows, p.S - r0);
      const G64Op A = op_of(c, 0, R, p.n_bas, pl, pl + g.a + g.b);
      G64Src sa = src_of(0, 1, R, p.n_bas, p.S, nb);  // conjugated: the product conjugates its left side
      for (int b = 0; b < nb; ++b) sa.tab[b] = Ps[b] + (long)r0 * cs;
      CKA(g64_slice(c, 0, sa, A, flag, 0, s));
      nl += 2;
      for (int side = 0; side < 2; ++side) {
        const int n0 = side ? j->n_occ : 0, nc = side ? j->n_virt : j->n_occ;
        std::vector<short> ia;
        G64Src sb = src_of(0, 0, nc, p.n_bas, a->n_mo, 0);
        G64Out o{};
        o.use_tab = 1;
        o.rd = o.cd = 1 << 30;
        o.s0 = nc;
        o.t0 = 1;
        o.R = R;
        o.C = nc;
        for (int b = 0; b < nb; ++b) {
          const int k = ks[b];
          if (!(side ? need_v[k] : need_o[k])) continue;
          sb.tab[sb.nb] = ao_mo(j, p, region, k) + (long)n0 * cs;
          o.tab[sb.nb] = (double*)(region + (side ? p.off_hvirt + p.virt_bytes * p.virt_slot[k]
                                                  : p.off_hocc + p.occ_bytes * p.occ_slot[k])) +
                         (long)r0 * nc * cs;
          ia.push_back((short)b);
          ++sb.nb;
        }
        if (sb.nb == 0) continue;
        const G64Op B = op_of(c, 1, nc, p.n_bas, pl + g.a, pl + g.a + g.b + g.e);
        CKA(g64_slice(c, 1, sb, B, flag, 0, s));
        nl += 2;
        CKA(g64_product(c, A, B, G64Index{ia.data(), nullptr, 1, 1}, o, sb.nb, 0, nullptr, 0, flag, 0, status, &nl, s));
      }
    }
    n += (int)nl;
    return RPA_OK;
  };
  std::vector<int> bk;
  std::vector<const double*> bp;
  auto half_fp64 = [&](int k, const double* P, const int* only) -> rpa_status {
    if (need_o[k]) {
      CKA(launch_ao_half(j->is_complex, p.n_bas, p.S, a->n_mo, P, ao_mo(j, p, region, k), 0, j->n_occ,
                         (double*)(region + p.off_hocc + p.occ_bytes * p.occ_slot[k]), s, only));
      ++n;
    }
    if (need_v[k]) {
      CKA(launch_ao_half(j->is_complex, p.n_bas, p.S, a->n_mo, P, ao_mo(j, p, region, k), j->n_occ, j->n_virt,
                         (double*)(region + p.off_hvirt + p.virt_bytes * p.virt_slot[k]), s, only));
      ++n;
    }
    return RPA_OK;
  };
  auto flush = [&]() -> rpa_status {
    if (bk.empty()) return RPA_OK;
    if (rpa_status st = half_g64(bk, bp)) return st;
    for (size_t b = 0; b < bk.size(); ++b)
      if (rpa_status st = half_fp64(bk[b], bp[b], flag)) return st;
    bk.clear();
    bp.clear();
    return RPA_OK;
  };
  for (int k = 0; k < j->n_kpts; ++k) {
    if (!need_o[k] && !need_v[k]) continue;
    const double* P = (const double*)(a->n_R > 0 ? nullptr : a->padf[k]);
    if (a->n_R > 0) {  // this k-point's array as the lattice sum, into the PADF slot
      CKA(launch_padf_k(j->is_complex, lat, a->kfrac + 3 * k, (long)p.n_bas * p.S, (double*)(region + p.off_padf),
                        s));
      P = (const double*)(region + p.off_padf);
      ++n;
    }
    if (!g.half) {
      if (rpa_status st = half_fp64(k, P, nullptr)) return st;
      continue;
    }
    bk.push_back(k);
    bp.push_back(P);
    if ((int)bk.size() == g.k_batch)
      if (rpa_status st = flush()) return st;
  }
  if (rpa_status st = flush()) return st;
  prof_end(ctx, pex, s, RPA_K_AO2MO, n);
  ctx->launches += n;
  return RPA_OK;
}

rpa_status ao_enqueue_assemble(rpa_ctx* ctx, Exec* pex, const rpa_job* j, const AoPlan& p, const char* region, int q,
                               char* out, cudaStream_t s, char* gws, int* status) {
  const rpa_ao* a = j->ao;
  int n = 0;
  const AoG64 g = gws ? ao_g64_plan(j, p) : AoG64{};
  int* flag = g.assemble ? (int*)gws + 1 : nullptr;
  prof_begin(ctx, pex, s);
  if (g.assemble) {
    CKA(cudaMemsetAsync(flag, 0, sizeof(int), s));
    const int c = j->is_complex, cs = c ? 2 : 1;
    const long nov = (long)j->n_occ * j->n_virt;
    char* pl = gws + 1024;
    char *ea = pl + g.a + g.b, *eb = ea + g.e;
    uint64_t nl = 0;
    for (const AoAtom& t : ao_atoms(a)) {
      const AsmStep st = asm_step(j, t);
      for (int j0 = 0; j0 < j->n_k; j0 += st.np)
        for (int g0 = 0; g0 < t.nf; g0 += st.g) {
          const int np = std::min(st.np, j->n_k - j0), gc = std::min(st.g, t.nf - g0);
          // left rows (gamma, a), right rows i; then left rows a, right rows (gamma, i)
          G64Src a1 = src_of(0, 1, gc * j->n_virt, t.nb, (long)t.nf * j->n_virt, np);
          G64Src b1 = src_of(0, 1, j->n_occ, t.nb, a->n_mo, np);
          G64Src a2 = src_of(0, 1, j->n_virt, t.nb, a->n_mo, np);
          G64Src b2 = src_of(0, 1, gc * j->n_occ, t.nb, (long)t.nf * j->n_occ, np);
          G64Out o1{}, o2{};
          for (int u = 0; u < np; ++u) {
            const size_t i = (size_t)q * j->n_k + j0 + u;
            const int k = j->pair_k[i], kq = j->pair_kq[i];
            a1.tab[u] = (const double*)(region + p.off_hvirt + p.virt_bytes * p.virt_slot[kq]) +
                        ((long)t.s0 + g0) * j->n_virt * cs;
            b1.tab[u] = ao_mo(j, p, region, k) + (long)t.b0 * a->n_mo * cs;
            a2.tab[u] = ao_mo(j, p, region, kq) + ((long)t.b0 * a->n_mo + j->n_occ) * cs;
            b2.tab[u] = (const double*)(region + p.off_hocc + p.occ_bytes * p.occ_slot[k]) +
                        ((long)t.s0 + g0) * j->n_occ * cs;
            o1.tab[u] = (double*)(out + p.cblk * (size_t)(j0 + u)) + (t.f0 + g0) * nov * cs;
            o2.tab[u] = o1.tab[u];
          }
          o1.use_tab = o2.use_tab = 1;
          o1.rd = j->n_virt;
          o1.s1 = nov;
          o1.s0 = 1;
          o1.t0 = j->n_virt;
          o1.R = gc * j->n_virt;
          o1.C = j->n_occ;
          o2.rd = o1.cd = o2.cd = 1 << 30;
          o2.s0 = 1;
          o2.t0 = j->n_virt;
          o2.R = j->n_virt;
          o2.C = gc * j->n_occ;
          o2.add = 1;
          const G64Op A1 = op_of(c, 0, a1.R, t.nb, pl, ea), B1 = op_of(c, 1, b1.R, t.nb, pl + g.a, eb);
          CKA(g64_slice(c, 0, a1, A1, flag, 0, s));
          CKA(g64_slice(c, 1, b1, B1, flag, 0, s));
          CKA(g64_product(c, A1, B1, G64Index{nullptr, nullptr, 1, 1}, o1, np, 0, nullptr, 0, flag, 0, status, &nl, s));
          const G64Op A2 = op_of(c, 0, a2.R, t.nb, pl, ea), B2 = op_of(c, 1, b2.R, t.nb, pl + g.a, eb);
          CKA(g64_slice(c, 0, a2, A2, flag, 0, s));
          CKA(g64_slice(c, 1, b2, B2, flag, 0, s));
          CKA(g64_product(c, A2, B2, G64Index{nullptr, nullptr, 1, 1}, o2, np, 0, nullptr, 0, flag, 0, status, &nl, s));
          nl += 8;
        }
    }
    n += (int)nl;
  }
  for (int j0 = 0; j0 < j->n_k; j0 += AoPairs::kMax) {
    const int np = std::min(AoPairs::kMax, j->n_k - j0);
    AoPairs pr{};
    for (int t = 0; t < np; ++t) {
      const size_t i = (size_t)q * j->n_k + j0 + t;
      const int k = j->pair_k[i], kq = j->pair_kq[i];
      pr.mo_k[t] = ao_mo(j, p, region, k);
      pr.mo_kq[t] = ao_mo(j, p, region, kq);
      pr.h_occ[t] = (const double*)(region + p.off_hocc + p.occ_bytes * p.occ_slot[k]);
      pr.h_virt[t] = (const double*)(region + p.off_hvirt + p.virt_bytes * p.virt_slot[kq]);
      pr.out[t] = (double*)(out + p.cblk * (size_t)(j0 + t));
    }
    CKA(launch_ao_assemble(j->is_complex, pr, np, (const int4*)region, j->n_aux, j->n_occ, j->n_virt, a->n_mo, s,
                           flag));
    ++n;
  }
  prof_end(ctx, pex, s, RPA_K_AO2MO, n);
  ctx->launches += n;
  return RPA_OK;
}

}  // namespace rpa
