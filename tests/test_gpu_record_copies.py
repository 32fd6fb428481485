"""Launches of many small levels add into copies of their records, which are
merged exactly: every level equals the level alone, with and without room for
the copies, and replayed from a graph."""
import numpy as np
import pytest

from paper_1512_02818_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,n_nodes,n_levels,dt", [(0, 24, 22, 1e-2), (0, 5, 128, 4e-3), (0, 200, 3, 1e-2),
                                                      (2, 33, 16, 1e-2)])
def test_levels_equal_levels_alone(kind, n_nodes, n_levels, dt):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1512_02818_gb300 import build, pdd
    build.build()
    rng = np.random.default_rng(n_nodes)
    dim = 3 if kind == 2 else 2
    levels = [dict(nodes=torch.from_numpy(rng.uniform(0.3, 0.7, (n_nodes, dim)).astype(np.float32)).cuda(),
                   n_paths=50 + i, dt=dt * (1 + i % 3), grid_id=0, stream_tag=i) for i in range(n_levels)]
    v = W.control_grid(kind, 17, 1e-1)
    ctx = pdd.Context(0)
    prob = pdd.Problem(ctx, kind)
    prob.set_control_grid(0, v)
    alone = [prob.estimate(**lv) for lv in levels]
    runs = [prob.estimate_levels(levels)[1], prob.estimate_levels(levels, graph=True)[1]]
    # room for the records and nothing else, and for two copies
    for copies in (1, 2):
        small = pdd.Context(0, mem_budget=1024 + copies * n_nodes * n_levels * 128)
        p2 = pdd.Problem(small, kind)
        p2.set_control_grid(0, v)
        runs.append(p2.estimate_levels(levels)[1])
    for run in runs:
        for a, b in zip(alone, run):
            for f in pdd.STAT_FIELDS + pdd.COUNT_FIELDS:
                assert torch.equal(a[f].nan_to_num(-1.0), b[f].nan_to_num(-1.0)), f
    ctx.close()
