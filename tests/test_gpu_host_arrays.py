"""Host arrays in and out give what device arrays give, at the sizes around
which the copies change (through page-locked memory, or array by array), with
several levels, and with results the caller does not ask for."""
import numpy as np
import pytest

from paper_1512_02818_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1512_02818_gb300 import build, pdd
    build.build()
    ctx = pdd.Context(0)
    yield torch, pdd, pdd.Problem(ctx, pdd.PDD_PROBLEM_CFG0_2D), pdd.Problem(ctx, pdd.PDD_PROBLEM_CUBE_3D)
    ctx.close()


def _same(pdd, host, dev):
    for f in pdd.STAT_FIELDS + pdd.COUNT_FIELDS:
        a, b = host[f].numpy(), dev[f].cpu().numpy()
        assert np.array_equal(a, b, equal_nan=a.dtype.kind == "f"), f


@pytest.mark.parametrize("n", [1, 31, 33, 2336, 2337, 8192, 8193])
def test_sizes(env, n):
    torch, pdd, prob, prob3 = env
    rng = np.random.default_rng(n)
    for p, dim in ((prob, 2), (prob3, 3)):
        nodes = rng.uniform(0.2, 0.8, (n, dim)).astype(np.float32)
        a = p.estimate(nodes, 3, 1e-2, host_inputs=True, device_out=False)
        b = p.estimate(nodes, 3, 1e-2)
        _same(pdd, a, b)


def test_levels_and_missing_results(env):
    torch, pdd, prob, _ = env
    rng = np.random.default_rng(5)
    levels = [dict(nodes=rng.uniform(0.2, 0.8, (n, 2)).astype(np.float32), n_paths=5, dt=1e-2,
                   stream_tag=n) for n in (1, 700, 40, 1200)]
    _, host = prob.estimate_levels(levels, device_out=False, host_inputs=True)
    _, dev = prob.estimate_levels(levels)
    for a, b in zip(host, dev):
        _same(pdd, a, b)
    args, out, res = prob._prepare(levels[1]["nodes"], 5, 1e-2, pdd.PDD_CV_NONE, 1234, 700, 1.0, False,
                                   False, True, False)
    before = res["var_phi"].fill_(-7.0)
    out.var_phi = None
    assert pdd.pdd_estimate_nodes(prob.handle, args, out) == 0
    assert bool((before == -7.0).all())
    assert np.array_equal(res["mean_steps"].numpy(), host[1]["mean_steps"].numpy())
