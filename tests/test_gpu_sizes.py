"""Sizes at which the launches of the log-det step, the FP64 chi0 and the
frequency-batched chi0 change shape: panel and tile edges, one matrix and many,
groups of frequencies, more energy bins than rpa_freq_plan describes, and the V
side that starts before the frequency plan.

Tolerances (from the arithmetic, u = 2^-53):
* ln det and Tr by Cholesky of a matrix A with 1 <= A <= c: backward error at
  most (N + 1) u of the diagonal per column, so |d ln det| <= N (N + 1) u c;
  with c = 8 and N <= 200 below 4e-11, typically its square root.  Bar: 1e-11
  per matrix, relative to ln det (which is above 1 for every N >= 4; absolute
  below).
* inverse form (V^-1 - chi) against the sandwich form on the same chi0: the
  inverse adds cond(V) u per entry: 1e-9 of ln det for cond(V) below 1e4.
* FP64 chi0: K <= 400 products of one sign on the diagonal, K u = 5e-14 and a
  few u from the weights: 2e-13 of max |chi|.
* split-precision chi0: 8e-7 of max |chi| (coefficient sum 16 times the bar
  5e-8 of one contraction).
"""
import numpy as np
import pytest

import oracle
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


def _chi(cplx, n, n_w, seed):
    """-chi with eigenvalues within 0..7, one scale per frequency."""
    r = np.random.default_rng(seed)
    out = []
    for w in range(n_w):
        a = r.standard_normal((n, n))
        if cplx:
            a = a + 1j * r.standard_normal((n, n))
        q, _ = np.linalg.qr(a)
        lam = r.uniform(0.0, 7.0, n) * 2.0 ** (-w)
        x = (q * lam) @ q.conj().T
        out.append(-0.5 * (x + x.conj().T))
    return np.array(out)


def _unit_v_job(rpa, cplx, n, n_w):
    one = torch.ones((1, 1), dtype=torch.float64, device="cuda")
    dt = torch.complex128 if cplx else torch.float64
    z = np.zeros((1, 1), np.int32)
    return rpa.Job(is_complex=cplx, n_aux=n, n_occ=1, n_virt=1, pair_k=z, pair_kq=z, w_q=np.ones(1), zeta_k=1.0,
                   omega=np.arange(1.0, n_w + 1), zeta_w=np.ones(n_w), eps_occ=-one, eps_virt=one,
                   C=[torch.ones((n, 1), dtype=dt, device="cuda")], V=[torch.eye(n, dtype=dt, device="cuda")])


@pytest.mark.parametrize("cplx", [True, False])
@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 32, 33, 63, 64, 65, 96, 97, 200])
@pytest.mark.parametrize("n_w", [1, 13])
def test_logdet_panel_edges(rpa, cplx, n, n_w):
    chi = _chi(cplx, n, n_w, 1000 * n + n_w)
    ref = np.array([[np.log(np.linalg.eigvalsh(np.eye(n) - c)).sum(), np.trace(c).real] for c in chi])
    job = _unit_v_job(rpa, cplx, n, n_w)
    t = torch.from_numpy(chi).cuda()
    with rpa.Context(0) as c:
        got = c.logdet(job, 0, t)
    bar = 1e-11 * np.maximum(np.abs(ref), 1.0)
    assert np.all(np.abs(got - ref) <= bar), np.abs(got - ref).max()
    out = torch.full((n_w, 2), float("nan"), dtype=torch.float64, device="cuda")
    rpa.logdet_noalloc(cplx, n, n_w, torch.eye(n, dtype=t.dtype, device="cuda"), t, out)
    torch.cuda.synchronize()
    assert np.all(np.abs(out.cpu().numpy() - ref) <= bar)


@pytest.mark.parametrize("n", [15, 16, 17, 33, 63, 64, 65, 97, 130])
@pytest.mark.parametrize("cplx", [True, False])
def test_inverse_form_edges(rpa, cplx, n):
    grid = synth.regular_kq_grid((2, 2, 1)) if cplx else synth.gamma_grid()
    p = synth.make_problem("inv", is_complex=cplx, n_aux=n, n_occ=3, n_virt=40, grid=grid, n_w=4, seed=300 + n)
    t = rpa.upload_problem(p)
    job = rpa.job_from_problem(p, t, prec=rpa.PREC_MIXED)
    job64 = rpa.job_from_problem(p, t)
    with rpa.Context(0, chi0_freq=1) as c:
        r = c.energy(job)
        for q in range(p.n_q):
            ref = c.logdet(job64, q, c.chi0(job, q))
            assert np.all(np.abs(r["lndet"][q] - ref[:, 0]) <= 1e-9 * np.maximum(np.abs(ref[:, 0]), 1e-3)), q


def test_batch_over_panel_edges(rpa):
    """One ragged batch of Cholesky launches over the panel edges."""
    probs = [synth.make_problem("b%d" % n, is_complex=bool(n % 2), n_aux=n, n_occ=2, n_virt=50,
                                grid=synth.regular_kq_grid((2, 1, 1)) if n % 2 else synth.gamma_grid(), n_w=3,
                                seed=400 + n) for n in (15, 16, 17, 31, 32, 33, 64, 65, 96, 97, 130, 201)]
    jobs = [rpa.job_from_problem(p, rpa.upload_problem(p)) for p in probs]
    with rpa.Context(0) as c:
        one = np.array([c.energy(j)["Ec"] for j in jobs])
        for _ in range(2):  # eager, then the replayed graph
            e = np.array(c.energy_batch(jobs))
            assert np.all(np.abs(e - one) <= 1e-11 * np.abs(one)), np.abs(e / one - 1).max()
    ref = np.array([oracle.energy(p)["Ec"] for p in probs])
    assert np.all(np.abs(one - ref) <= 1e-10 * np.abs(ref))


@pytest.mark.parametrize("cplx", [True, False])
@pytest.mark.parametrize("n,n_w", [(1, 1), (16, 3), (17, 8), (33, 5), (65, 10), (40, 17), (130, 16), (300, 2)])
def test_fp64_chi0_tiles(rpa, cplx, n, n_w):
    grid = synth.regular_kq_grid((2, 2, 1)) if cplx else synth.gamma_grid()
    p = synth.make_problem("t", is_complex=cplx, n_aux=n, n_occ=3, n_virt=31 if cplx else 127, grid=grid, n_w=n_w,
                           seed=500 + n)
    job = rpa.job_from_problem(p, rpa.upload_problem(p))
    q = p.n_q - 1
    C = [p.C(q, j) for j in range(p.n_k)]
    eo = [p.eps_pair(q, j)[0] for j in range(p.n_k)]
    ev = [p.eps_pair(q, j)[1] for j in range(p.n_k)]
    with rpa.Context(0) as c:
        chi = c.chi0(job, q).cpu().numpy()
    for w in range(n_w):
        ref = oracle.chi0(C, eo, ev, p.grid.zeta_k, float(p.omega[w]))
        assert np.abs(chi[w] - ref).max() <= 2e-13 * np.abs(ref).max(), w


def _binned(rpa, p, freq):
    job = rpa.job_from_problem(p, rpa.upload_problem(p), prec=rpa.PREC_MIXED)
    q = p.n_q - 1
    C = [p.C(q, j) for j in range(p.n_k)]
    eo = [p.eps_pair(q, j)[0] for j in range(p.n_k)]
    ev = [p.eps_pair(q, j)[1] for j in range(p.n_k)]
    with rpa.Context(0, chi0_freq=freq) as c:
        chi = c.chi0(job, q).cpu().numpy()
    for w in sorted({0, p.n_w // 2, p.n_w - 1}):
        ref = oracle.chi0(C, eo, ev, p.grid.zeta_k, float(p.omega[w]))
        assert np.abs(chi[w] - ref).max() <= 8e-7 * np.abs(ref).max(), w
        assert np.array_equal(chi[w], chi[w].conj().T)


@pytest.mark.parametrize("cplx", [True, False])
@pytest.mark.parametrize("n_w", [2, 6, 7, 9, 10, 11, 17, 32])
def test_recombination_group_widths(rpa, cplx, n_w):
    grid = synth.regular_kq_grid((2, 2, 1)) if cplx else synth.gamma_grid()
    _binned(rpa, synth.make_problem("g", is_complex=cplx, n_aux=130, n_occ=5, n_virt=37 if cplx else 150, grid=grid,
                                    n_w=n_w, seed=600 + n_w), 2)


def test_many_bins(rpa):
    """64000 transitions at one q and 10 frequencies: 52 bins of rank 5."""
    _binned(rpa, synth.make_problem("n", is_complex=False, n_aux=40, n_occ=40, n_virt=1600, grid=synth.gamma_grid(),
                                    n_w=10, seed=51), 0)


def test_v_side_before_the_plan(rpa):
    """The first call of a context allocates its workspace after the plan, later
    calls factor V before it: the same bits, also after a larger job, a smaller
    one and one of another shape have used the workspace."""
    def prob(n, n_w, kd, seed):
        p = synth.make_problem("v", is_complex=True, n_aux=n, n_occ=4, n_virt=30, grid=synth.regular_kq_grid(kd),
                               n_w=n_w, seed=seed)
        t = rpa.upload_problem(p)
        return rpa.job_from_problem(p, t, prec=rpa.PREC_MIXED), t

    specs = [(200, 16, (2, 2, 1), 1), (90, 16, (2, 1, 1), 2), (260, 12, (2, 2, 1), 3), (131, 20, (3, 1, 1), 4)]
    jobs = [prob(*s) for s in specs]
    first = []
    for j, _ in jobs:
        with rpa.Context(0, chi0_freq=2) as c:
            first.append(c.energy(j))
    with rpa.Context(0, chi0_freq=2) as c:
        for i in (2, 0, 1, 0, 3, 2, 3, 1):
            r = c.energy(jobs[i][0])
            assert r["Ec"] == first[i]["Ec"] and np.array_equal(r["lndet"], first[i]["lndet"]), i
