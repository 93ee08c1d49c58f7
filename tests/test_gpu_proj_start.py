"""The projector's fast start (FP32 sweeps, refinement by digit products) against
the plain FP64 sweeps (taken when its workspace does not fit the context's cap):
odd and even bases, real and complex, degenerate and nearly diagonal overlaps,
and overlaps outside the FP32 range, which must take the plain sweeps.

Tolerance: both end with the same FP64 sweeps and the same convergence test
(4 N 2^-52 between columns), so eigenvalues agree to that of the largest one and
c~ = c - U_m U_m^H c to a few times it; the eigenvalue gaps at the cut are
above 0.2 here."""
import numpy as np
import pytest

from paper_2505_06021_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rpa():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2505_06021_gb300 as m
    from paper_2505_06021_gb300 import build as b

    b.build()
    return m


def _job(rpa, cplx, nb, ovl):
    grid = synth.regular_kq_grid((2, 2, 1)) if cplx else synth.gamma_grid()
    p = synth.make_ao_problem("ps", is_complex=cplx, n_bas_atom=nb, n_fit_atom=(2,) * len(nb), n_occ=6, n_virt=30,
                              grid=grid, n_w=3, seed=75, eps_d=1e-4)
    t = rpa.upload_ao_problem(p)
    if ovl is not None:
        t["overlap"] = [ovl(k, p.n_bas).contiguous() for k in range(p.n_kpts)]
    return rpa.job_from_ao_problem(p, t), p


def _degenerate(k, n):
    S = torch.eye(n, dtype=torch.complex128, device="cuda")
    S[0, 0] = 1e-6
    S[1, 1] = 1e-6
    S[2, 3], S[3, 2] = 0.3j, -0.3j
    return S


def _banded(k, n):
    i = torch.arange(n, device="cuda")
    S = torch.exp(-3.0 * (i[:, None] - i[None, :]).abs().double()).to(torch.complex128)
    ph = torch.exp(1j * 0.3 * k * i.double())
    S = S * ph[:, None] * ph.conj()[None, :]
    S[n - 1] = 0
    S[:, n - 1] = 0
    S[n - 1, n - 1] = 1e-7
    return S


@pytest.mark.parametrize("cplx,nb,ovl,scale", [
    (True, (40, 45), None, 1.0), (True, (64, 66), None, 1.0), (False, (60, 41), None, 1.0),
    (True, (40, 40), _degenerate, 1.0), (True, (50, 41), _banded, 1.0), (True, (40, 45), None, 1e45)])
def test_projector_start_matches_plain_sweeps(rpa, cplx, nb, ovl, scale):
    job, p = _job(rpa, cplx, nb, ovl)
    if scale != 1.0:
        for S in job.ao_t["overlap"]:
            S.mul_(scale)
        job._ao.eps_d = 1e-4 * scale
    res = []
    for cap in (0, 1 << 18):
        with rpa.Context(0, hbm_cap_bytes=cap) as c:
            n0 = c.launches
            out, m, eig = c.projector(job)
            res.append((out, m, eig, c.launches - n0))
    (a, ma, ea, la), (b, mb, eb, lb) = res
    assert la != lb, "the two caps took the same route"
    assert ma == mb and ma > 0
    tol = 4 * p.n_bas * 2.0 ** -52
    assert np.abs(ea - eb).max() <= tol * eb.max()
    if scale != 1.0:
        assert np.array_equal(ea, eb)
    for k in range(p.n_kpts):
        assert float((a[k] - b[k]).abs().max()) <= 20 * tol


@pytest.mark.parametrize("cplx,nb", [(True, (32, 32)), (False, (33, 32)), (True, (225, 225)), (True, (226, 227)),
                                     (True, (451, 454))])
def test_projector_start_column_blocks(rpa, cplx, nb):
    """The smallest basis of the start, the edge between blocks of 16 and 8
    columns, and columns too long for either."""
    test_projector_start_matches_plain_sweeps(rpa, cplx, nb, None, 1.0)
