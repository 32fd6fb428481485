"""Coupled pairs end with the same bits in ordinary iterations and in the drain's
batches, for every problem and kind of control variate: the first pairs of a
launch of many against small launches, spread and not, for both Y rules."""
import numpy as np
import pytest

from paper_1512_02818_gb300 import workloads as W

pytestmark = pytest.mark.gpu

KINDS = {"cfg0": (0, 129), "aniso": (1, 129), "cube": (2, 33), "harmonic": (3, 129), "paper": (4, 129)}


@pytest.mark.parametrize("y_exp", [0, 1])
@pytest.mark.parametrize("cv", ["none", "grid", "exact"])
@pytest.mark.parametrize("kind", list(KINDS))
def test_drained_equals_ordinary(kind, cv, y_exp):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1512_02818_gb300 import build, pdd
    build.build()
    ctx = pdd.Context(0)
    k, grid = KINDS[kind]
    prob = pdd.Problem(ctx, k, y_rule=y_exp)
    gid = {"none": pdd.PDD_CV_NONE, "exact": pdd.PDD_CV_EXACT, "grid": 0}[cv]
    if cv == "grid":
        prob.set_control_grid(0, W.control_grid(k, grid, 1e-1))
    node = np.full((1, 3 if kind == "cube" else 2), 0.5, np.float32)
    big = prob.estimate_coupled(node, 130_000, 4e-3, grid_id=gid, emit_paths=True)
    for claim, n in ((1, 1), (1, 9), (1, 14), (1, 32), (0, 1500), (0, 9000)):
        ctx.set_claim(claim)
        small = prob.estimate_coupled(node, n, 4e-3, grid_id=gid, emit_paths=True)
        for a, b in zip(small, big):
            for f in ("phi", "xi", "steps"):
                assert torch.equal(a[f], b[f][:, :n]), (claim, n, f)
    prob.close()
    ctx.close()
