"""FP64 jobs above the sizes from which their products run as digit products: the
same bits through rpa_energy, rpa_energy_batch and rpa_submit, whatever the
workspace cap leaves for the digit planes, until it leaves no room for the smallest
ones (then the FP64 kernels' result, the same to rounding)."""
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


def _problem(cplx, n_aux, n_occ, n_virt, kdims, n_w, gap=None):
    grid = synth.regular_kq_grid(kdims) if cplx else synth.gamma_grid()
    p = synth.make_problem("rt", is_complex=cplx, n_aux=n_aux, n_occ=n_occ, n_virt=n_virt, grid=grid, n_w=n_w, seed=77)
    if gap is not None:
        # one transition far below the others: at low frequencies its weight stands out of
        # every row, which then takes one more digit level; at high ones it does not
        p.eps_virt[0, 0] = p.eps_occ.max() + gap
    return p


@pytest.mark.parametrize("cplx,n_aux,n_occ,n_virt,kdims,n_w", [
    (True, 150, 6, 60, (2, 2, 1), 12),   # chi0, sandwich
    (True, 392, 4, 28, (2, 1, 1), 8),    # sandwich and block columns of the Cholesky
    (False, 400, 12, 160, (1, 1, 1), 20),
])
@pytest.mark.parametrize("mem", ["device", "host"])
def test_served_equals_energy_bit_for_bit(rpa, cplx, n_aux, n_occ, n_virt, kdims, n_w, mem):
    p = _problem(cplx, n_aux, n_occ, n_virt, kdims, n_w)
    t = rpa.upload_problem(p, device="cpu" if mem == "host" else "cuda", pin=mem == "host")
    job = rpa.job_from_problem(p, t, mem=rpa.MEM_HOST if mem == "host" else rpa.MEM_DEVICE)
    with rpa.Context(0) as c:
        alone = c.energy(job)
        if mem == "device":
            assert np.array_equal(c.energy_batch([job, job]), [alone["Ec"]] * 2)
    with rpa.Context(0, max_inflight=8) as c:
        for tk in [c.submit(job) for _ in range(4)]:
            Ec, eps = c.wait(tk, 300.0, job)
            assert Ec == alone["Ec"]
            assert np.array_equal(eps.reshape(alone["eps"].shape), alone["eps"])


@pytest.mark.parametrize("call", ["chi0", "energy"])
def test_room_for_the_planes_changes_no_bit(rpa, call):
    """Caps from below the smallest planes to above the largest: the bits of the
    digit products from some cap on, those of the FP64 kernels below it, and caps in
    between that take more launches for the same bits."""
    p = _problem(True, 260, 9, 56, (2, 2, 1), 18, gap=0.05)
    job = rpa.job_from_problem(p, rpa.upload_problem(p))

    def one(cap):
        with rpa.Context(0, hbm_cap_bytes=cap) as c:
            n0 = c.launches
            r = c.chi0(job, 0).cpu().numpy() if call == "chi0" else c.energy(job)["eps"]
            return c.launches - n0, r.tobytes(), r

    n_full, full, vf = one(0)
    n_fp64, fp64, vd = one(1 << 20)
    assert full != fp64 and np.abs(vf - vd).max() <= 1e-12 * np.abs(vd).max()
    seen = [one(int(2.0 ** (22 + 0.25 * i))) for i in range(44)]
    bits = [s[1] for s in seen]
    first = bits.index(full)
    assert first > 0 and all(b == full for b in bits[first:])
    # below it, a smaller part of the products (chi0 or the tail alone) may still fit
    assert bits[0] == fp64
    assert {s[0] for s in seen[first:]} - {n_full}, "no cap took the smaller planes"
