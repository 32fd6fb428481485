"""The regressions of the fast fit against the oracle's on the same cloud, for
cloud lengths around a warp, around what fits in shared memory, and the shortest.

A sum of m terms in another order differs by up to m eps = 2.3e-13 (m = 1,025) of
the terms' size; the regressions on h in [1e-3, 1e-2] amplify that by the squared
ratio of h to its spread, below 20, twice for the weighted one: 1e-10 is allowed,
of the data's size for the intercept and over the spread of h for the slope."""
import numpy as np
import pytest

from paper_1512_02818_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import oracle
    from paper_1512_02818_gb300 import build, pdd
    build.build()
    oracle.build()
    ctx = pdd.Context(0)
    prob = pdd.Problem(ctx, pdd.PDD_PROBLEM_CFG0_2D)
    prob.set_control_grid(0, W.control_grid(0, 65, 1.0) - W.control_grid(0, 65, 0.0))
    yield oracle, pdd, prob
    ctx.close()


@pytest.mark.parametrize("grid", [False, True])
@pytest.mark.parametrize("m", [2, 3, 31, 32, 33, 100, 1024, 1025])
def test_fits(env, m, grid):
    oracle, pdd, prob = env
    nodes = W.workload_nodes("c0")[::5]
    g = prob.fit_constants(nodes, 200, 1e-3, 1e-2, m, grid_id=0 if grid else pdd.PDD_CV_NONE,
                           seed=5)
    x = g["cloud"][0, :, 0]
    fits = [("E_phi", "beta", 1, oracle.ols_fit), ("E_tau", None, 3, oracle.ols_fit),
            ("V_phi", "alpha", 2, oracle.gamma_identity_fit)]
    if grid:
        fits += [("cov_phi_psi", None, 4, oracle.ols_fit),
                 ("V_psi", None, 5, oracle.gamma_identity_fit)]
    else:
        assert np.all(np.isnan(g["cov_phi_psi"])) and np.all(np.isnan(g["V_psi"]))
    for i in range(len(nodes)):
        for at0, at1, col, fit in fits:
            y = g["cloud"][i, :, col]
            a, b = fit(x, y)
            size = np.abs(y).max()
            assert abs(g[at0][i] - a) <= 1e-10 * size, (i, at0)
            if at1:
                assert abs(g[at1][i] - b) <= 1e-10 * size / np.std(x), (i, at1)
