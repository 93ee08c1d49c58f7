"""AO -> MO transform as digit products on the tensor cores against its FP64
kernels (taken when the planes do not fit the context's cap): several atoms of
uneven sizes, row and column counts off the tile edges, real and complex, k
form and lattice form, and a PADF entry that sends the transform back to the
FP64 kernels.

Tolerance: entries are sums of n_bas and then 2 nb products of numbers of
random sign.  Both forms are off by a few u = 2^-53 of the root mean square
times sqrt(n_bas) at most; 1e-14 of a block's largest entry is 90 u."""
import numpy as np
import pytest

from paper_2505_06021_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-14


@pytest.fixture(scope="module")
def rpa():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2505_06021_gb300 as m
    from paper_2505_06021_gb300 import build as b

    b.build()
    return m


def _problem(cplx, nb, nf, n_occ, n_virt, lattice=None):
    grid = synth.regular_kq_grid((2, 2, 1)) if cplx else synth.gamma_grid()
    return synth.make_ao_problem("g64ao", is_complex=cplx, n_bas_atom=nb, n_fit_atom=nf, n_occ=n_occ, n_virt=n_virt,
                                 grid=grid, n_w=4, seed=81, lattice=lattice)


def _both(rpa, job, q):
    out = []
    for cap in (0, 1 << 20):
        with rpa.Context(0, hbm_cap_bytes=cap) as c:
            n0 = c.launches
            out.append(c.ao2mo(job, q))
            out.append(c.launches - n0)
    assert out[1] > out[3], "the two caps took the same route"
    return out[0], out[2]


@pytest.mark.parametrize("cplx,nb,nf,n_occ,n_virt,lat", [
    (True, (48, 33, 51), (97, 64, 110), 17, 101, None),
    (True, (64, 64), (128, 128), 32, 96, 1),
    (False, (130, 77), (301, 160), 25, 170, None),
])
def test_ao2mo_matches_fp64_kernels(rpa, cplx, nb, nf, n_occ, n_virt, lat):
    p = _problem(cplx, nb, nf, n_occ, n_virt, None if lat is None else synth.lattice_2d(lat))
    job = rpa.job_from_ao_problem(p, rpa.upload_ao_problem(p))
    a, b = _both(rpa, job, p.n_q - 1)
    assert float((a - b).abs().max()) <= TOL * float(b.abs().max())


def test_ao2mo_spread_rows(rpa):
    """MO columns and a PADF entry somewhat out of the rest: one more digit
    level, the same tolerance."""
    p = _problem(True, (48, 40), (96, 90), 16, 70)
    t = rpa.upload_ao_problem(p)
    for k in range(p.n_kpts):
        t["mo"][k].add_(torch.eye(p.n_bas, p.n_occ + p.n_virt, dtype=torch.complex128, device="cuda"))
        t["padf"][k][5, 7] *= 8.0
    a, b = _both(rpa, rpa.job_from_ao_problem(p, t), 1)
    for g in range(p.n_aux):
        assert float((a[:, g] - b[:, g]).abs().max()) <= TOL * float(b[:, g].abs().max()), g


@pytest.mark.parametrize("far", [2.0 ** 20, 2.0 ** 70])
def test_ao2mo_out_of_range_keeps_the_fp64_result(rpa, far):
    """A far PADF entry: the half-transforms come from the FP64 kernels, and the
    assembly, which its fit function's rows would spoil, too."""
    p = _problem(True, (48, 40), (96, 90), 16, 70)
    t = rpa.upload_ao_problem(p)
    for k in range(p.n_kpts):
        t["mo"][k].mul_(0.01).add_(torch.eye(p.n_bas, p.n_occ + p.n_virt, dtype=torch.complex128, device="cuda"))
        t["padf"][k][5, 7] = far
    a, b = _both(rpa, rpa.job_from_ao_problem(p, t), 1)
    assert np.array_equal(a.cpu().numpy(), b.cpu().numpy())
