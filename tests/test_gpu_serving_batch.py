"""Requests that enter and end in one launch are staged and finalised together:
results equal those of each request alone, for batches around the lengths of the
finalisation's table and for requests around the size whose results are copied."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1512_02818_gb300 import build, pdd
    build.build()
    ctx = pdd.Context(0)
    yield torch, pdd, ctx
    ctx.close()


def _check(pdd, ctx, prob, sizes, paths, **kw):
    rng = np.random.default_rng(len(sizes))
    srv = pdd.Server(ctx, **kw)
    try:
        nodes = [rng.uniform(0.2, 0.8, (n, prob.dim)).astype(np.float32) for n in sizes]
        tickets = [srv.submit(prob, x, paths, 1e-2, seed=7, stream_tag=i, kappa=1.0 + i)
                   for i, x in enumerate(nodes)]
        for i, (t, x) in enumerate(zip(tickets, nodes)):
            status, got = srv.poll(t, len(x), 60_000_000)
            assert status == pdd.PDD_OK
            alone = prob.estimate(x, paths, 1e-2, seed=7, stream_tag=i, kappa=1.0 + i)
            for f in pdd.STAT_FIELDS + pdd.COUNT_FIELDS:
                want = alone[f].cpu().numpy()
                assert np.array_equal(got[f], want, equal_nan=want.dtype.kind == "f"), (i, f)
    finally:
        srv.close()


@pytest.mark.parametrize("three", [False, True])
@pytest.mark.parametrize("count", [1, 2, 16, 17, 18, 128])
def test_batch_lengths(env, three, count):
    _, pdd, ctx = env
    prob = pdd.Problem(ctx, pdd.PDD_PROBLEM_CUBE_3D if three else pdd.PDD_PROBLEM_CFG0_2D)
    sizes = [(1, 31, 64, 129, 1000)[i % 5] for i in range(count)]
    # a first large request keeps the device busy while the others queue up
    _check(pdd, ctx, prob, [20_000] + sizes, 40, max_active=128)


@pytest.mark.parametrize("n", [(1 << 18) - 1, 1 << 18, (1 << 18) + 1])
def test_results_written_or_copied(env, n):
    _, pdd, ctx = env
    _check(pdd, ctx, pdd.Problem(ctx, pdd.PDD_PROBLEM_CFG0_2D), [5, n, 33], 2)
