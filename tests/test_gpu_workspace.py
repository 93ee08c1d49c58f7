"""Device memory of the calls: what a call reserves, and calls on a device whose
memory is nearly used up."""
import numpy as np
import pytest

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


@pytest.fixture(autouse=True)
def give_back():
    yield
    torch.cuda.empty_cache()  # what _leave held


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _big_job(rpa, n_q=1):
    """Jobs whose chi0 planes are about 3 GB: N_aux 768, 9 k-points, 1536 band pairs."""
    n_aux, n_occ, n_virt, n_k, n_w = 768, 16, 96, 9, 16
    g = torch.Generator(device="cuda").manual_seed(3)
    nov = n_occ * n_virt
    C = [torch.view_as_complex(torch.randn((n_aux, nov, 2), generator=g, device="cuda", dtype=torch.float64) /
                               (2.0 * nov) ** 0.5) for _ in range(n_k)] * n_q
    eo = torch.rand((n_k, n_occ), generator=g, device="cuda", dtype=torch.float64) - 1.3
    ev = torch.rand((n_k, n_virt), generator=g, device="cuda", dtype=torch.float64) + 0.1
    pair = np.tile(np.arange(n_k, dtype=np.int32), (n_q, 1))
    om = np.linspace(0.1, 4.0, n_w)
    return rpa.Job(is_complex=True, n_aux=n_aux, n_occ=n_occ, n_virt=n_virt, pair_k=pair, pair_kq=pair,
                   w_q=np.ones(n_q) / n_q, zeta_k=1.0 / n_k, omega=om, zeta_w=np.full(n_w, 0.25), eps_occ=eo,
                   eps_virt=ev, C=C, V=[torch.eye(n_aux, dtype=torch.complex128, device="cuda")] * n_q)


def test_calls_reserve_only_the_planes_they_use(rpa):
    """The log-det step holds no chi0 planes (16 frequencies' chi0, chi0 L and factors
    are 0.3 GB, its own planes 1 GB at most), the chi0 step no tail planes."""
    job = _big_job(rpa)
    with rpa.Context(0) as c:
        chi = c.chi0(job, 0)
        torch.cuda.empty_cache()
    with rpa.Context(0) as c:
        f0 = _free()
        c.logdet(job, 0, chi)
        used = f0 - _free()
    assert used < 1.6 * 2 ** 30, used


def _leave(n):
    """Holds the device's memory but for n bytes."""
    torch.cuda.empty_cache()
    return torch.empty(_free() - n, dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("left", [0.75, 0.95])
def test_calls_fit_beside_what_the_caller_holds(rpa, left):
    """With less memory left than the digit planes need (3 GB for chi0, 1 GB for the
    log-det, which itself needs 0.35), the calls run without them; the results
    agree to rounding (1e-13 of sums over 13824 transitions and 768 pivots)."""
    job = _big_job(rpa)

    def calls(hold):
        out = []
        for what in (lambda c: c.chi0(job, 0, out=chi).clone().cpu(), lambda c: torch.from_numpy(c.logdet(job, 0, chi0)),
                     lambda c: torch.from_numpy(c.energy(job)["eps"]), lambda c: torch.from_numpy(c.energy_batch([job]))):
            with rpa.Context(0) as c:
                c.logdet(small, 0, torch.zeros((1, 8, 8), dtype=torch.complex128, device="cuda"))  # kernels loaded
                h = _leave(int(left * 2 ** 30)) if hold else None
                out.append(what(c))
                del h
        return out

    one = torch.ones((1, 1), dtype=torch.float64, device="cuda")
    z = np.zeros((1, 1), np.int32)
    small = rpa.Job(is_complex=True, n_aux=8, n_occ=1, n_virt=1, pair_k=z, pair_kq=z, w_q=np.ones(1), zeta_k=1.0,
                    omega=np.ones(1), zeta_w=np.ones(1), eps_occ=-one, eps_virt=one,
                    C=[torch.ones((8, 1), dtype=torch.complex128, device="cuda")],
                    V=[torch.eye(8, dtype=torch.complex128, device="cuda")])
    chi = torch.empty((16, 768, 768), dtype=torch.complex128, device="cuda")
    with rpa.Context(0) as c:
        chi0 = c.chi0(job, 0)
    for a, b in zip(calls(False), calls(True)):
        assert float((a - b).abs().max()) <= 1e-13 * float(a.abs().max())


@pytest.mark.parametrize("left,same", [(0.75, False), (1.9, True)])
def test_served_job_fits_beside_what_the_caller_holds(rpa, left, same):
    """A lane that cannot hold a job's planes runs it with the smallest ones (the same
    bits: 1.1 GB here) or without them."""
    job = _big_job(rpa)
    with rpa.Context(0) as c:
        ref = c.energy(job)
    with rpa.Context(0) as c:
        h = _leave(int(left * 2 ** 30))
        Ec, eps = c.wait(c.submit(job), 300.0, job)
        del h
    eps = eps.reshape(ref["eps"].shape)
    if same:
        assert Ec == ref["Ec"] and np.array_equal(eps, ref["eps"])
    else:
        assert not np.array_equal(eps, ref["eps"])
        assert np.abs(eps - ref["eps"]).max() <= 1e-13 * np.abs(ref["eps"]).max()
