"""Both sides of the launch rules' lines give the same bits, and the launches are
the ones meant: the route of each is read back.

Record copies in shared memory (at most 512 records): a launch with a control
grid leaves them out where its paths are long and the copies would take L1 from
the gathers, a spread launch keeps up to 64.  Spread launches: one batch a warp,
up to 24 paths of long paths and 12 of short ones, none beyond.
"""
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
    yield torch, pdd, ctx
    ctx.close()


def _same(torch, pdd, a, b):
    for f in pdd.STAT_FIELDS + pdd.COUNT_FIELDS:
        assert torch.equal(a[f].nan_to_num(-1.0), b[f].nan_to_num(-1.0)), f


@pytest.mark.parametrize("n_nodes", [480, 512])
def test_records_with_and_without_copies(env, n_nodes):
    torch, pdd, ctx = env
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    prob = pdd.Problem(ctx, pdd.PDD_PROBLEM_CFG0_2D)
    prob.set_control_grid(0, W.control_grid(0, 129, 1e-1))
    nodes = W.random_interface_nodes(np.random.default_rng(1), n_nodes)
    # enough paths for full blocks of 512 threads
    level = dict(nodes=nodes, n_paths=8 * 32 * 24 * sms // n_nodes + 1, dt=1e-3, grid_id=0)
    alone = prob.estimate(**level)
    assert pdd.pdd_debug_last_launch(ctx.handle)["cached_records"] == 0
    # many short paths beside it: mean steps under the line, copies kept
    few = dict(nodes=nodes[:512 - n_nodes], n_paths=2_000_000, dt=2e-2, grid_id=0, stream_tag=5)
    if n_nodes < 512:
        _, (beside, _) = prob.estimate_levels([level, few])
        assert pdd.pdd_debug_last_launch(ctx.handle)["cached_records"] == 512
        _same(torch, pdd, alone, beside)
    # short paths alone: both records in shared memory and, one record more, global
    short = dict(level, dt=2e-2, n_paths=3000)
    kept = prob.estimate(**short)
    assert pdd.pdd_debug_last_launch(ctx.handle)["cached_records"] == n_nodes
    more = np.concatenate([nodes, W.random_interface_nodes(np.random.default_rng(2), 513 - n_nodes)])
    beyond = prob.estimate(**dict(short, nodes=more))
    assert pdd.pdd_debug_last_launch(ctx.handle)["cached_records"] == 0
    for f in pdd.STAT_FIELDS + pdd.COUNT_FIELDS:
        assert torch.equal(kept[f].nan_to_num(-1.0), beyond[f][:n_nodes].nan_to_num(-1.0)), f
    prob.close()


@pytest.mark.parametrize("coupled", [False, True])
def test_records_of_spread_launches(env, coupled):
    torch, pdd, ctx = env
    prob = pdd.Problem(ctx, pdd.PDD_PROBLEM_CFG0_2D)
    prob.set_control_grid(0, W.control_grid(0, 129, 1e-1))
    per = 2 if coupled else 1  # fine and difference records
    nodes = W.random_interface_nodes(np.random.default_rng(4), 64 // per + 1)

    def run(n):
        r = (prob.estimate_coupled if coupled else prob.estimate)(nodes[:n], 20, 1e-3, grid_id=0)
        launch = pdd.pdd_debug_last_launch(ctx.handle)
        assert launch["paths_per_warp"] > 0
        return (r if coupled else (r,)), launch["cached_records"]

    most, n64 = run(64 // per)
    more, n65 = run(64 // per + 1)
    assert (n64, n65) == (64, 0)
    for a, b in zip(most, more):
        for f in pdd.STAT_FIELDS + pdd.COUNT_FIELDS:
            assert torch.equal(a[f].nan_to_num(-1.0), b[f][:64 // per].nan_to_num(-1.0)), f
    prob.close()


@pytest.mark.parametrize("dt", [1e-2, 2e-3])
@pytest.mark.parametrize("kind,precision", [(0, 0), (0, 1), (2, 0)])
def test_lines_of_the_spread_rule(env, kind, precision, dt):
    torch, pdd, ctx = env
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    warps = 10 * sms if precision == 0 else 4 * sms
    most = 24 if dt <= 2e-3 else 12
    prob = pdd.Problem(ctx, kind, precision=precision)
    prob.set_control_grid(0, W.control_grid(kind, 33, 1e-1))
    node = np.full((1, 3 if kind == 2 else 2), 0.5, np.float32)
    counts = {1: 1, warps: 1, warps + 1: 2, 2 * warps + 1: 3, 8 * warps + 1: 9,
              most * warps: most, 24 * 32 * sms + 1: 0}
    # beyond the line: short and FP64 paths in ordinary batches, long FP32 paths
    # 24 a warp as long as the chip has a warp's place for each
    wide = precision == 0 and dt <= 2e-3
    counts[most * warps + 1] = counts[24 * 32 * sms] = 24 if wide else 0
    for n, batch in counts.items():
        a = prob.estimate(node, n, dt, grid_id=0)
        assert pdd.pdd_debug_last_launch(ctx.handle)["paths_per_warp"] == batch, n
        ctx.set_claim(1)  # one path a lane: never spread
        b = prob.estimate(node, n, dt, grid_id=0)
        assert pdd.pdd_debug_last_launch(ctx.handle)["paths_per_warp"] == 0
        ctx.set_claim(0)
        _same(torch, pdd, a, b)
        assert int(a["n_paths"][0]) == n
    prob.close()
