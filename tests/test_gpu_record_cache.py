"""The node records' shared-memory copies change no result.

Launches whose records fit the copies leave them out when the paths are long
and the copies would take L1 from a control grid's gathers.  The same level is
run both ways: alone (no copies), and beside a level of so many short paths
that the launch keeps them.
"""
import numpy as np
import pytest

from paper_1512_02818_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_nodes,h", [(449, 1e-3), (480, 1e-3), (496, 5e-4)])
def test_with_and_without_copies(n_nodes, h):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1512_02818_gb300 import build, pdd
    build.build()
    ctx = pdd.Context(0)
    prob = pdd.Problem(ctx, pdd.PDD_PROBLEM_CFG0_2D)
    prob.set_control_grid(0, W.control_grid(0, 129, 1e-1))
    nodes = W.random_interface_nodes(np.random.default_rng(1), n_nodes)
    level = dict(nodes=nodes, n_paths=400, dt=h, grid_id=0)
    short = dict(nodes=W.workload_nodes("c0")[:16], n_paths=400_000, dt=2e-2, grid_id=0, stream_tag=5)
    alone = prob.estimate(**level)
    _, (beside, few) = prob.estimate_levels([level, short])
    few_alone = prob.estimate(**short)
    for f in pdd.STAT_FIELDS + pdd.COUNT_FIELDS:
        assert torch.equal(alone[f].nan_to_num(-1.0), beside[f].nan_to_num(-1.0)), f
        assert torch.equal(few_alone[f].nan_to_num(-1.0), few[f].nan_to_num(-1.0)), f
    prob.close()
    ctx.close()
