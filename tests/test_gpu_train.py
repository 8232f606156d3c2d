"""GPU training kernels (a7) against the CPU oracle's training pieces, through
the C ABI: residuals and reverse-mode Jacobian, the Gram reduction, one LM
step, and a full fit showing what training gains over the untrained SP2
sequence (Sec. II A 1, Fig. 2 in spirit)."""
import numpy as np
import pytest

from oracle import sp2, tables, train

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ft():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_2605_08523_gb300 as ft
    return ft


@pytest.mark.parametrize("target", ["fermi", "entropy"])
def test_residual_and_jacobian_match_oracle(ft, target):
    rng = np.random.default_rng(1)
    L = 26
    th = np.array(tables.PRINTED_B1500) + 1e-6 * rng.standard_normal((L, 4))
    beta0, mu0, alpha = 1500.0, 1 / 3, 0.842704
    x = train.sample_grid(5000, beta0, mu0)
    tcode = ft.TARGET_ENTROPY if target == "entropy" else ft.TARGET_FERMI
    xd = torch.from_numpy(x).cuda()
    r, M = ft.ftsp2_train_residual_jacobian(tcode, beta0, mu0, th, xd, alpha=alpha)
    y, J = train.forward_jacobian(th, x, target, alpha if target == "entropy" else 1.0, mu0)
    r_or = y - train.target(x, target, beta0, mu0)
    r = r.cpu().numpy()
    M = M.cpu().numpy()
    assert np.max(np.abs(r - r_or)) < 1e-12
    assert np.max(np.abs(M[-1] - r)) == 0.0
    scale = np.max(np.abs(J), axis=0) + 1e-300
    assert np.max(np.abs(M[:-1].T - J) / scale) < 1e-11


def test_gram_matches_numpy(ft):
    rng = np.random.default_rng(2)
    L = 9
    ns = 20011
    M = rng.standard_normal((4 * L + 1, ns))
    G = ft.ftsp2_train_normal_equations(torch.from_numpy(M).cuda(), L).cpu().numpy()
    ref = M @ M.T
    assert np.max(np.abs(G - ref)) < 1e-10 * np.max(np.abs(ref))
    assert np.max(np.abs(G - G.T)) == 0.0


@pytest.mark.parametrize("seed", [0, 5])
def test_one_lm_step_matches_oracle(ft, seed):
    # theta_init = NULL: the library builds the samples (nsamples, seed) and
    # the SP2 start itself; the oracle takes the same steps from its own
    L, beta0, mu0 = 12, 40.0, 1 / 3
    x = train.sample_grid(4000, beta0, mu0, seed=seed)
    th0 = train.init_from_sp2(L, beta0, mu0)
    th_or, hist = train.lm_fit(th0, x, beta0=beta0, mu0=mu0, iters=1, accel=False)
    th_gpu, rep = ft.ftsp2_train_coeffs(ft.TARGET_FERMI, beta0, mu0, L=L, nsamples=4000, seed=seed,
                                        iterations=1, accel=False)
    assert rep["accepted"] == int(hist[0][2])
    assert np.max(np.abs(th_gpu - th_or)) < 1e-8 * max(1.0, np.max(np.abs(th_or)))
    assert abs(rep["cost"] - hist[0][0]) < 1e-9 * hist[0][0]


@pytest.mark.parametrize("L, ns", [(3, 255), (3, 257), (12, 256), (16, 2000), (45, 300), (46, 300), (47, 700),
                                   (48, 1021), (64, 257)])
def test_one_accelerated_step_matches_oracle(ft, L, ns):
    # the right-hand side of the second solve at the edges of the 256-sample blocks
    # and on either side of the width up to which slices hold 16 samples.  Damping
    # 1e-3 of the diagonal bounds the scaled condition number by 4 L / 1e-3 = 2e5;
    # the second difference at h = 0.1 multiplies rounding by 200: 2e5 x 200 x 1e-16
    # of the correction, held to 1e-6 of the table.
    beta0, mu0 = 40.0, 1 / 3
    x = train.sample_grid(ns, beta0, mu0, seed=1)
    th0 = train.init_from_sp2(L, beta0, mu0)
    th_or, _ = train.lm_fit(th0, x, beta0=beta0, mu0=mu0, iters=1, accel=True)
    th_gpu, _ = ft.ftsp2_train_coeffs(ft.TARGET_FERMI, beta0, mu0, L=L, nsamples=ns, seed=1, iterations=1, accel=True)
    assert np.max(np.abs(th_gpu - th_or)) < 1e-6 * max(1.0, np.max(np.abs(th_or)))


def test_training_gain_over_sp2(ft):
    # beta0 = 40, mu0 = 1/3, 12 layers: the SP2-mu table misses the Fermi
    # function by ~0.3; LM with geodesic acceleration on the GPU brings the
    # max error on [0, 1] below 1e-4, like the oracle's own fit.
    L, beta0, mu0 = 12, 40.0, 1 / 3
    x = train.sample_grid(20000, beta0, mu0)
    th0 = train.init_from_sp2(L, beta0, mu0)
    th, rep = ft.ftsp2_train_coeffs(ft.TARGET_FERMI, beta0, mu0, L=L, nsamples=20000, iterations=150, accel=True)
    e_sp2 = train.max_error(np.array(sp2.sp2_table(mu0, L)), beta0=beta0, mu0=mu0, grid=20001)
    e_tr = train.max_error(th, beta0=beta0, mu0=mu0, grid=20001)
    assert e_sp2 > 1e-1 and e_tr < 1e-4
    assert rep["cost"] < rep["cost0"] * 1e-6
    assert abs(rep["max_err"] - np.max(np.abs(train.forward(th, x) - train.fermi_target(x, beta0, mu0)))) < 1e-12
