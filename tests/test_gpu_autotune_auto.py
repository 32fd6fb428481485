"""A tuned context is not slower than an untuned one where the automatic launch
shape beats every explicit one, and says which shape it reports."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_automatic_shape_is_among_the_trials():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1512_02818_gb300 import build, pdd
    build.build()
    ctx = pdd.Context(0)
    prob = pdd.Problem(ctx, pdd.PDD_PROBLEM_CFG0_2D, precision=pdd.PDD_PATH_FP64)
    nodes = np.random.default_rng(2).uniform(0.2, 0.8, (64, 2)).astype(np.float32)

    def run():
        e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        times = []
        for _ in range(5):
            e0.record(ctx.stream)
            r = prob.estimate(nodes, 1000, 1e-3)
            e1.record(ctx.stream)
            torch.cuda.synchronize()
            times.append(e0.elapsed_time(e1))
        return r, min(times), pdd.pdd_debug_last_launch(ctx.handle)

    want, plain, shape = run()
    threads, blocks, ms = prob.autotune(nodes, 1000, 1e-3)
    got, tuned, tuned_shape = run()
    # (FP64 paths: 6 warps an SM or fewer by the launch's size, which no explicit
    # shape of the trials gives)
    assert tuned_shape == shape and tuned < 1.25 * plain
    assert ms < 1.25 * plain
    for f in pdd.STAT_FIELDS + pdd.COUNT_FIELDS:
        assert torch.equal(got[f].nan_to_num(-1.0), want[f].nan_to_num(-1.0)), f
    # the reported shape is an explicit one; asked for, it runs
    assert ctx.get_launch()[:2] == (threads, blocks) and threads in (128, 256, 512)
    ctx.set_launch(threads, blocks)
    assert run()[2]["block_threads"] == threads
    prob.close()
    ctx.close()
