"""The projector's sweeps as launches: what a column pair costs its SM, and
contexts that share the device."""
import threading
import time

import pytest

from paper_2505_06021_gb300 import synth
from test_gpu_proj_start import test_projector_start_matches_plain_sweeps as start_matches_plain_sweeps

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


def _job(rpa, n_bas, kdims):
    p = synth.make_ao_problem("sw", is_complex=True, n_bas_atom=(n_bas,), n_fit_atom=(2,), n_occ=4,
                              n_virt=n_bas - 4, grid=synth.regular_kq_grid(kdims), n_w=3, seed=76, eps_d=1e-4)
    return rpa.job_from_ao_problem(p, rpa.upload_ao_problem(p))


def test_small_basis_pairs_share_an_sm(rpa):
    """63 functions take the FP64 sweeps, a CTA per column pair: 31 pairs at one
    k-point (an SM each), 496 at 16 (up to four per SM).  Of a CTA's time only its
    share of the FP64 pipe adds up over the CTAs of an SM.  With the rotation
    computed by one warp that is the smaller part of a round (1.7 times the time at 16
    k-points), computed by all eight it is nearly all of it (3.1 times)."""
    with rpa.Context(0) as c:
        per_launch = []
        for kdims in ((1, 1, 1), (4, 4, 1)):
            job = _job(rpa, 63, kdims)
            c.projector(job)
            best = 1e9
            for _ in range(5):
                torch.cuda.synchronize()
                n0, t0 = c.launches, time.perf_counter()
                c.projector(job)
                torch.cuda.synchronize()
                best = min(best, (time.perf_counter() - t0) / (c.launches - n0))
            per_launch.append(best)
    assert per_launch[1] <= 2.3 * per_launch[0], per_launch


def test_two_contexts_with_different_bases(rpa):
    """Two contexts in two threads on one device, a block kernel launch of 16
    columns each with other shared memory: every call succeeds and gives what it
    gives alone."""
    jobs = [_job(rpa, n, (2, 1, 1)) for n in (256, 64)]
    alone, errors, results = [], [], [[], []]
    for job in jobs:
        with rpa.Context(0) as c:
            alone.append(c.projector(job)[2].tobytes())
    torch.cuda.synchronize()
    gate = threading.Barrier(2)

    def work(i):
        try:
            with rpa.Context(0) as c, torch.cuda.stream(torch.cuda.Stream()):
                gate.wait(60)
                for _ in range(60):
                    results[i].append(c.projector(jobs[i])[2].tobytes())
        except Exception as e:
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    assert all(r == a for a, rs in zip(alone, results) for r in rs)


@pytest.mark.parametrize("scale", [1e21, 1e30, 1e-22])
def test_overlaps_beyond_the_start(rpa, scale):
    """Overlaps whose squares leave the FP32 range while their entries do not (and
    such as leave the digit products' range) take the plain sweeps, bit for bit."""
    start_matches_plain_sweeps(rpa, True, (40, 45), None, scale)
