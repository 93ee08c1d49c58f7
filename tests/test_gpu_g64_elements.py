"""Element-wise accuracy of the FP64 chi0 by digit products: rows whose large entries
meet the small ones of the other row, so that an element is 2^-g of |C_P| |C_Q|.

All band pairs have the energy 2 and the frequencies are 0 and 2, so every weight is
exactly -2 or -1 and an element is an exact product sum, summed here in extended
precision.  Errors are taken relative to sum_t |C_Pt C_Qt d|, root mean square over
the elements.  Bounds (u = 2^-53): a chain of K additions of random sign is off by about
u / 2; the digit products by up to 2.6 u for K = 128 (rows just below the gap from which
level 8 is multiplied) and less above, and never by more than about twice the chain's from
K = 2048 on."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def rpa():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2505_06021_gb300 as m
    from paper_2505_06021_gb300 import build as b

    b.build()
    return m


@pytest.mark.parametrize("K,n_w", [(128, 64), (512, 16), (2048, 4), (8192, 2)])
@pytest.mark.parametrize("g", [0, 2, 4, 6, 8, 11, 20])
def test_elements_of_complementary_rows(rpa, K, n_w, g):
    N, n_occ, m = 256, 8, 24
    r = np.random.default_rng(1000 * g + K)
    C = r.standard_normal((N, K))
    half = r.random(K) < 0.5
    C[:m, half] *= 2.0 ** -g
    C[m:2 * m, ~half] *= 2.0 ** -g
    one = torch.ones((1, 1), dtype=torch.float64, device="cuda")
    z = np.zeros((1, 1), np.int32)
    om = np.array([0.0, 2.0] * (n_w // 2))
    job = rpa.Job(is_complex=False, n_aux=N, n_occ=n_occ, n_virt=K // n_occ, pair_k=z, pair_kq=z, w_q=np.ones(1),
                  zeta_k=1.0, omega=om, zeta_w=np.ones(n_w), eps_occ=-one.expand(1, n_occ).contiguous(),
                  eps_virt=one.expand(1, K // n_occ).contiguous(), C=[torch.from_numpy(C).cuda()],
                  V=[torch.eye(N, dtype=torch.float64, device="cuda")])
    A, B = C[:m].astype(np.longdouble), C[m:2 * m].astype(np.longdouble)
    exact = -(A[:, None, :] * B[None, :, :]).sum(2)
    size = (np.abs(C[:m])[:, None, :] * np.abs(C[m:2 * m])[None, :, :]).sum(2)
    rms = []
    for cap in (0, 1 << 20):
        with rpa.Context(0, hbm_cap_bytes=cap) as c:
            chi = c.chi0(job, 0).cpu().numpy()
        e = [((chi[w, :m, m:2 * m].astype(np.longdouble) - d * exact) / (d * size)).astype(np.float64)
             for w, d in ((0, 2), (1, 1))]
        rms.append(float(np.sqrt(np.mean(np.square(e)))))
    split, chain = rms
    assert chain <= 2.0 * U
    assert split <= 3.5 * U, rms
    if K >= 2048:
        assert split <= 2.5 * chain, rms
