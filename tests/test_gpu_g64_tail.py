"""The log-det step's triangular products and the inverse form's Gram product as
digit products on the tensor cores against their FP64 kernels (taken when the
planes do not fit the context's cap), over the edges of the tiles, several
passes, and matrices that must go back to the FP64 kernels.

Tolerance: ln det(1 - Pi) and Tr Pi are sums over N pivots or diagonal entries of
one sign.  Each entry of Y = -L^H chi L is off by a few u = 2^-53 times sqrt(N)
of its largest products in either form, with random signs over the sum: below
1e-13 of the sum for N <= 400."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-13


@pytest.fixture(scope="module")
def rpa():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2505_06021_gb300 as m
    from paper_2505_06021_gb300 import build as b

    b.build()
    return m


def _inputs(cplx, n, n_w, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    dt = torch.complex128 if cplx else torch.float64

    def rnd(*s):
        x = torch.randn(s + (2,), generator=g, device="cuda", dtype=torch.float64) * 0.7
        return torch.view_as_complex(x) if cplx else x[..., 0].contiguous()

    q, _ = torch.linalg.qr(rnd(n, n))
    lam = torch.exp(torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * 4.6 - 2.3)
    V = (q * lam.to(dt)) @ q.conj().T
    V = (0.5 * (V + V.conj().T)).contiguous()
    A = rnd(2 * n, n) / (2 * n) ** 0.5
    chi = torch.stack([-(A.conj().T @ A) * 10.0 ** (0.5 - 6.0 * w / max(1, n_w - 1)) for w in range(n_w)]).contiguous()
    return V, chi


def _job(rpa, cplx, n, n_w, V):
    one = torch.ones((1, 1), dtype=torch.float64, device="cuda")
    C = torch.ones((n, 1), dtype=V.dtype, device="cuda")
    z = np.zeros((1, 1), np.int32)
    return rpa.Job(is_complex=cplx, n_aux=n, n_occ=1, n_virt=1, pair_k=z, pair_kq=z, w_q=np.ones(1), zeta_k=1.0,
                   omega=np.arange(1.0, n_w + 1), zeta_w=np.ones(n_w), eps_occ=-one, eps_virt=one, C=[C], V=[V])


def _both(rpa, cplx, n, n_w, V, chi):
    job = _job(rpa, cplx, n, n_w, V)
    out = []
    for cap in (0, 1 << 20):
        with rpa.Context(0, hbm_cap_bytes=cap) as c:
            n0 = c.launches
            out += [c.logdet(job, 0, chi), c.launches - n0]
    assert out[1] > out[3], "the two caps took the same route"
    return out[0], out[2]


@pytest.mark.parametrize("cplx,n,n_w", [(True, 128, 12), (True, 129, 20), (True, 161, 8), (True, 384, 3),
                                        (False, 193, 16), (False, 400, 5)])
def test_logdet_matches_fp64_kernels(rpa, cplx, n, n_w):
    V, chi = _inputs(cplx, n, n_w, 91)
    a, b = _both(rpa, cplx, n, n_w, V, chi)
    assert np.all(np.abs(a - b) <= TOL * np.abs(b)), np.max(np.abs(a - b) / np.abs(b))


@pytest.mark.parametrize("far", [0.3, 2.0 ** 20])
def test_spread_matrix(rpa, far):
    """One matrix with an entry out of the rest: one more digit level within the
    tolerance, or, far out, the FP64 kernels' result bit for bit; the others agree."""
    V, chi = _inputs(True, 150, 12, 92)
    chi[3, 10, 20] *= far / abs(chi[3, 10, 20].item())
    chi[3, 20, 10] = chi[3, 10, 20].conj()
    chi[3, 10, 10] -= 2.0 * far
    chi[3, 20, 20] -= 2.0 * far
    a, b = _both(rpa, True, 150, 12, V, chi)
    if far > 1.0:
        assert np.array_equal(a[3], b[3])
    assert np.all(np.abs(a - b) <= TOL * np.abs(b))


@pytest.mark.parametrize("n", [130, 260])
def test_inverse_form_energy_matches(rpa, n):
    """Split-precision job: V^-1 by the Gram product of digit planes; E_c
    against the same job with the FP64 kernels' V^-1 (the chi0 plan is the same
    under both caps, so only the tail differs)."""
    from paper_2505_06021_gb300 import synth

    p = synth.make_problem("tailm", is_complex=True, n_aux=n, n_occ=3, n_virt=12, grid=synth.regular_kq_grid((2, 2, 1)),
                           n_w=6, seed=93)
    job = rpa.job_from_problem(p, rpa.upload_problem(p), prec=rpa.PREC_MIXED)
    r = []
    for cap in (0, 1 << 20):
        with rpa.Context(0, hbm_cap_bytes=cap, chi0_freq=1) as c:
            r.append(c.energy(job))
    assert np.max(np.abs(r[0]["lndet"] - r[1]["lndet"])) <= 1e-11
    assert abs(r[0]["Ec"] - r[1]["Ec"]) <= 1e-11 * abs(r[1]["Ec"])


@pytest.mark.parametrize("cplx,n,n_w", [(True, 384, 8), (True, 385, 9), (True, 513, 8), (False, 400, 20), (False, 640, 8)])
def test_block_columns_match_fp64_kernels(rpa, cplx, n, n_w):
    """Sizes whose Cholesky factors take their block columns as digit products
    (twice the tolerance: N to 640)."""
    V, chi = _inputs(cplx, n, n_w, 94)
    a, b = _both(rpa, cplx, n, n_w, V, chi)
    assert np.all(np.abs(a - b) <= 2 * TOL * np.abs(b)), np.max(np.abs(a - b) / np.abs(b))


@pytest.mark.parametrize("far", [2.0 ** 12, 2.0 ** 80])
def test_block_columns_spread_row(rpa, far):
    """V = 1 and a pair of rows whose factor holds one entry far above the others."""
    _, chi = _inputs(True, 400, 8, 95)
    V = torch.eye(400, dtype=torch.complex128, device="cuda")
    chi[2, 5, 300] = chi[2, 300, 5] = -far
    chi[2, 5, 5] -= 2.0 * far
    chi[2, 300, 300] -= 2.0 * far
    a, b = _both(rpa, True, 400, 8, V, chi)
    assert np.all(np.abs(a - b) <= 2 * TOL * np.abs(b)), np.max(np.abs(a - b) / np.abs(b))


@pytest.mark.parametrize("n,n_w", [(400, 25), (512, 16)])
def test_inverse_form_block_columns(rpa, n, n_w):
    """Split-precision job with digit-product block columns against the FP64
    kernels' tail on the same chi0 plan; the float-float updates of the latter keep
    about 2^-45 of each update: 400 pivots of 2^-45 at most, 1e-11 of ln det."""
    from paper_2505_06021_gb300 import synth

    p = synth.make_problem("tailb", is_complex=True, n_aux=n, n_occ=3, n_virt=12, grid=synth.regular_kq_grid((2, 2, 1)),
                           n_w=n_w, seed=96)
    job = rpa.job_from_problem(p, rpa.upload_problem(p), prec=rpa.PREC_MIXED)
    r = []
    for cap in (0, 1 << 20):
        with rpa.Context(0, hbm_cap_bytes=cap, chi0_freq=1) as c:
            r.append(c.energy(job))
    assert np.max(np.abs(r[0]["lndet"] - r[1]["lndet"])) <= 2e-11 * max(1.0, np.max(np.abs(r[1]["lndet"])))
