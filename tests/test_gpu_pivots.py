"""The reciprocal pivot of the Cholesky factorisation: correctly rounded, like the
division.

With V = 1 the log-det step factorises 1 + Y, Y = -chi, itself.  For the matrix
[[p, x], [x, 1 + y]], x a power of two, the second pivot is 1 + y - x (x / p).  y =
x^2 r + 1 with r = 1 / p correctly rounded, scaled so that x^2 times one unit in
the last place of r is 1/2 or 1, makes that 2 exactly (no step but the reciprocal
rounds), and half or twice as far off per unit that the reciprocal misses: ln det is
ln p + ln 2, or off by 0.2 and more."""
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


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("e", [-24, -2, 0, 2, 30, 200, 1000])
def test_reciprocal_pivot_is_correctly_rounded(rpa, cplx, e):
    n = 20000
    r = np.random.default_rng(100 + e)
    m = r.uniform(1.0 + 2.0 ** -40, 2.0, n)
    m[:2000] = 2.0 - np.arange(1, 2001) * 2.0 ** -52  # and the significands next to 2 and 1
    m[2000:4000] = 1.0 + np.arange(8, 2008) * 2.0 ** -52
    u = np.ldexp(m, e) - 1.0
    p = 1.0 + u  # what the kernel divides by
    x = np.ldexp(1.0, 26 + e // 2)
    y = np.ldexp(1.0 / p, 52 + e) + 1.0
    chi = np.zeros((n, 2, 2))
    chi[:, 0, 0], chi[:, 1, 1] = -u, -y
    chi[:, 0, 1] = chi[:, 1, 0] = -x
    dt = torch.complex128 if cplx else torch.float64
    out = torch.empty((n, 2), dtype=torch.float64, device="cuda")
    rpa.logdet_noalloc(cplx, 2, n, torch.eye(2, dtype=dt, device="cuda"), torch.from_numpy(chi).to("cuda").to(dt), out)
    torch.cuda.synchronize()
    want = np.log(p) + np.log(2.0)
    off = np.abs(out[:, 0].cpu().numpy() - want) > 1e-9 * np.maximum(1.0, np.abs(want))
    assert not off.any(), (int(off.sum()), n)
