"""FP64 chi0 by exact digit products on the tensor cores against the FP64
kernel (taken when the digit planes do not fit the context's cap), over the
edges of its tiles (128 rows, 32 complex or 64 real columns), of its exact
accumulation (384 complex, 768 real transitions) and of its ranges.

Tolerance: both sum K products of the same numbers.  The FP64 kernel's chain of
K additions is off by at most about u sqrt(K) of sqrt(chi_PP chi_QQ) (u =
2^-53; rounding errors of random sign), the digit products by less; with K
up to 8000 that is 1e-14, and the bound is four times that."""
import numpy as np
import pytest

from paper_2505_06021_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 4e-14


@pytest.fixture(scope="module")
def rpa():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2505_06021_gb300 as m
    from paper_2505_06021_gb300 import build as b

    b.build()
    return m


def _close(a, b):
    d = torch.sqrt(torch.abs(torch.diagonal(b, dim1=-2, dim2=-1)).double())
    return float((torch.abs(a - b) / (d[:, :, None] * d[:, None, :])).max())


def _both(rpa, job, q):
    """(digit products, FP64 kernel): a cap of 1 MB leaves no room for the planes."""
    with rpa.Context(0) as c:
        a = c.chi0(job, q)
        n_a = c.launches
    with rpa.Context(0, hbm_cap_bytes=1 << 20) as c:
        b = c.chi0(job, q)
        n_b = c.launches
    assert n_b == 2 and n_a > 4, (n_a, n_b)
    return a, b


@pytest.mark.parametrize("cplx,n_aux,n_occ,n_virt,kdims,n_w", [
    (True, 128, 8, 96, (2, 2, 1), 16),   # whole tiles, 8 whole accumulations (3072 t)
    (True, 129, 7, 55, (2, 2, 1), 20),   # one row and one column over, odd K
    (True, 161, 5, 77, (2, 1, 1), 33),   # two frequency passes (32 + 1)
    (True, 97, 13, 59, (3, 2, 1), 9),    # less than one row tile, uneven K
    (False, 200, 24, 200, (1, 1, 1), 16),
    (False, 257, 12, 321, (1, 1, 1), 5),
])
def test_chi0_matches_fp64_kernel(rpa, cplx, n_aux, n_occ, n_virt, kdims, n_w):
    grid = synth.regular_kq_grid(kdims) if cplx else synth.gamma_grid()
    p = synth.make_problem("g64", is_complex=cplx, n_aux=n_aux, n_occ=n_occ, n_virt=n_virt, grid=grid, n_w=n_w, seed=71)
    job = rpa.job_from_problem(p, rpa.upload_problem(p))
    a, b = _both(rpa, job, p.n_q - 1)
    assert _close(a, b) <= TOL
    assert torch.equal(a, a.transpose(-1, -2).conj())


@pytest.mark.parametrize("spike", [24.0, 2.0 ** 12, 2.0 ** 70, float("inf"), float("nan"), 2.0 ** -130])
def test_rows_outside_the_split(rpa, spike):
    """A row with one entry somewhat out of the others takes one more digit level
    and stays within the tolerance; far out, beyond 2^60, and with infinities and
    NaN, the q goes through the FP64 kernel: the same bits.  A tiny entry alone
    changes nothing."""
    p = synth.make_problem("g64", is_complex=True, n_aux=130, n_occ=8, n_virt=60, grid=synth.regular_kq_grid((2, 2, 1)),
                           n_w=12, seed=72)
    t = rpa.upload_problem(p)
    q = 1
    blk = t["C"][q * p.n_k + 2]
    blk[77, 31] = blk[77, 31] * spike if abs(spike) < 1e30 else complex(spike, 0.0)
    a, b = _both(rpa, rpa.job_from_problem(p, t), q)
    if spike < 100.0:
        assert _close(a, b) <= TOL
    else:
        assert np.array_equal(a.cpu().numpy(), b.cpu().numpy(), equal_nan=True)


def test_batch_and_alone_agree_bit_for_bit(rpa):
    p = synth.make_problem("g64", is_complex=True, n_aux=150, n_occ=6, n_virt=60, grid=synth.regular_kq_grid((2, 2, 1)),
                           n_w=12, seed=73)
    job = rpa.job_from_problem(p, rpa.upload_problem(p))
    with rpa.Context(0) as c:
        one = c.energy(job)["Ec"]
        b1 = c.energy_batch([job, job])
        b2 = c.energy_batch([job, job])
    assert np.array_equal(b1, [one, one]) and np.array_equal(b1, b2)
