"""Block sizes around those the launcher cuts a caller's choice to: results are
the same bits for every one, single-segment and with a segment table."""
import numpy as np
import pytest

from paper_1512_02818_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt", [1e-3, 5e-3])  # long and short iterations
@pytest.mark.parametrize("kind", ["PDD_PROBLEM_CFG0_2D", "PDD_PROBLEM_ANISO_2D"])
def test_block_sizes(kind, dt):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1512_02818_gb300 import build, pdd
    build.build()
    ctx = pdd.Context(0)
    k = getattr(pdd, kind)
    prob = pdd.Problem(ctx, k)
    prob.set_control_grid(0, W.control_grid(k, 65, 1e-1))
    nodes = np.random.default_rng(3).uniform(0.1, 0.9, (40, 2)).astype(np.float32)
    levels = [dict(nodes=nodes[i::2], n_paths=4000, dt=dt, grid_id=0, stream_tag=i)
              for i in (0, 1)]

    def run():
        one = prob.estimate(nodes, 4000, dt, grid_id=0)
        _, many = prob.estimate_levels(levels)
        return [r[f].cpu().numpy() for r in [one] + list(many)
                for f in pdd.STAT_FIELDS + pdd.COUNT_FIELDS]

    want = run()
    for threads in (32, 416, 448, 480, 512):
        ctx.set_launch(threads, 0)
        for a, b in zip(want, run()):
            assert np.array_equal(a, b, equal_nan=a.dtype.kind == "f"), threads
    ctx.close()
