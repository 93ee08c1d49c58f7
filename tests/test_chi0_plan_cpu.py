"""The frequency-batched plan that the chi0 runs (rpa_chi0_plan, host-only): up to
64 bins, the bounds of rpa_freq_plan, and the factorised chi0 against the oracle
as in test_freq_plan_cpu.  Long contractions (many transitions per q) take more
and narrower bins than short ones."""
import numpy as np
import pytest

import oracle
from paper_2505_06021_gb300 import synth
from test_freq_plan_cpu import _factorised, _host_job

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def rpa():
    import paper_2505_06021_gb300 as m
    from paper_2505_06021_gb300 import build as b

    b.build()
    return m


@pytest.mark.parametrize("is_complex,kdims,n_occ,n_virt,n_w", [
    (True, (2, 2, 1), 6, 40, 16), (False, (1, 1, 1), 6, 60, 16), (True, (4, 4, 1), 8, 64, 20), (False, (1, 1, 1), 4, 28, 5)])
def test_executed_plan_matches_oracle(rpa, is_complex, kdims, n_occ, n_virt, n_w):
    grid = synth.regular_kq_grid(kdims) if is_complex else synth.gamma_grid()
    p = synth.make_problem("xp", is_complex=is_complex, n_aux=12, n_occ=n_occ, n_virt=n_virt, grid=grid, n_w=n_w, seed=5)
    plan = _host_job(rpa, p).chi0_plan(mode=2)
    assert 1 <= plan["n_bins"] <= 64 and np.all(plan["rank"] <= n_w)
    assert np.all(plan["err"] <= 1e-10) and np.all(np.diff(plan["edges"]) > 0)
    for b in range(plan["n_bins"]):
        r = plan["rank"][b]
        assert np.allclose(plan["coef"][b][:r][:, plan["skel"][b][:r]], np.eye(r), atol=1e-12)
        assert np.all(plan["skel"][b][r:] == -1)
    q = p.n_q - 1
    C = [p.C(q, j) for j in range(p.n_k)]
    eo = [p.eps_pair(q, j)[0] for j in range(p.n_k)]
    ev = [p.eps_pair(q, j)[1] for j in range(p.n_k)]
    ws = [0, n_w // 2, n_w - 1]
    fac = _factorised(p, plan, q, C, ws)
    lo = min((v[None, :] - o[:, None]).min() for o, v in zip(eo, ev))
    hi = max((v[None, :] - o[:, None]).max() for o, v in zip(eo, ev))
    # (the residual is relative to a bin's largest weight: one bin ratio more, as in test_freq_plan_cpu)
    rho = (hi / lo) ** (1.5 / plan["n_bins"])
    for w in ws:
        ref = oracle.chi0(C, eo, ev, p.grid.zeta_k, float(p.omega[w]))
        err = np.abs(fac[w] - ref).max() / np.abs(np.diag(ref)).max()
        assert err <= 2.0 * plan["err"].max() * rho + 1e-14, (w, err)


def test_long_contractions_take_more_bins(rpa):
    short = _host_job(rpa, synth.config1(n_aux=8, n_occ=8, n_virt=40, kdims=(2, 1, 1))).chi0_plan(mode=2)
    p = synth.config1(n_aux=8, n_occ=32, n_virt=224)
    long_, base = _host_job(rpa, p).chi0_plan(), _host_job(rpa, p).freq_plan()
    assert 0 < short["n_bins"] < long_["n_bins"] and long_["n_bins"] > 32
    assert long_["work_ratio"] < base["work_ratio"]


@pytest.mark.parametrize("n_w", [24, 32])
@pytest.mark.parametrize("mode", [0, 2])
def test_gap_so_small_that_no_plan_fits(rpa, n_w, mode):
    """A gap of 1e-16 puts 17 decades of transition energies into the bins: even at
    the widest ratio their coefficients exceed the recombination's shared memory,
    and every frequency is contracted on its own."""
    p = synth.make_problem("gap", is_complex=False, n_aux=12, n_occ=4, n_virt=28, grid=synth.gamma_grid(), n_w=n_w, seed=5)
    t = rpa.upload_problem(p, device="cpu")
    t["eps_occ"] -= t["eps_occ"].max()
    t["eps_virt"] += 1e-16 - t["eps_virt"].min()
    t["eps_virt"][0, int(t["eps_virt"][0].argmin())] = 1e-16
    job = rpa.job_from_problem(p, t, prec=rpa.PREC_MIXED, mem=rpa.MEM_HOST)
    assert job.chi0_plan(mode)["n_bins"] == 0
    assert job.freq_plan(mode)["n_bins"] == 0
