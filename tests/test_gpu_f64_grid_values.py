"""FP64 paths read the FP32 control table by its bits: every kind of value.

One step of one path from a grid point, whose cell has the interpolation weights
1, 0, 0, 0: a value that is not finite ends in PDD_ERR_OVERFLOW wherever it
stands in the cell (0 x NaN and 0 x infinity are NaN), in FP32 and FP64 paths
alike, and scaling the table by a power of two scales xi by it exactly.
"""
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
    yield pdd, ctx
    ctx.close()


def _one_step(pdd, ctx, kind, precision, grid):
    prob = pdd.Problem(ctx, kind, precision=precision, max_steps=1)
    try:
        prob.set_control_grid(0, grid, pdd.PDD_GRID_GRADIENT)
        node = np.full((1, grid.ndim - 1), 0.5, np.float32)
        return prob.estimate(node, 1, 1e-4, grid_id=0, emit_paths=True)
    finally:
        prob.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("kind,precision", [(0, 0), (0, 1), (2, 1)])
def test_values_that_are_not_finite(env, kind, precision, bad):
    pdd, ctx = env
    dim = 3 if kind == 2 else 2
    # corners of the cell with x_0 > 1/2 (weight 0), then the node's own (weight 1)
    for at in ((2,) * (dim - 1) + (3,), (3,) * dim, (2,) * dim):
        grid = np.full((5,) * dim + (dim,), 0.25)
        grid[at + (dim - 1,)] = bad
        with pytest.raises(pdd.PddError) as e:
            _one_step(pdd, ctx, kind, precision, grid)
        assert e.value.status == pdd.PDD_ERR_OVERFLOW, at


@pytest.mark.parametrize("kind", [0, 2])
def test_powers_of_two(env, kind):
    pdd, ctx = env
    dim = 3 if kind == 2 else 2
    pattern = np.random.default_rng(5).uniform(-1, 1, (5,) * dim + (dim,)).astype(np.float32)
    one = float(_one_step(pdd, ctx, kind, 1, pattern)["xi"].cpu()[0, 0])
    assert one != 0.0
    for e in (-100, -20, 0, 10):
        for sign in (1.0, -1.0):
            got = float(_one_step(pdd, ctx, kind, 1, pattern * (sign * 2.0**e))["xi"].cpu()[0, 0])
            assert got == sign * one * 2.0**e, (e, sign)
