"""Paths finished in the drain's batches equal the same paths run in ordinary iterations.

The drain takes a warp's last paths S steps at a time, S depending on how many
paths the warp still holds, and finds the exits and the truncations afterwards.
One warp is given every number of paths here (a claim of one path per lane
keeps the launch from being spread), with caps on the steps that fall at the
start, inside and at the end of a batch; the same paths of a launch of many
are issued first and run in the ordinary iterations.  Everything is compared
bit for bit, and spread launches with the unspread ones.
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


KINDS = {"cfg0": (0, 129), "aniso": (1, 129), "cube": (2, 33), "harmonic": (3, 129), "paper": (4, 129)}


@pytest.mark.parametrize("kind,precision,y_exp,cv", [
    ("cfg0", 0, 0, "grid"), ("cfg0", 0, 1, "none"), ("cfg0", 1, 0, "grid"), ("aniso", 0, 0, "grid"),
    ("paper", 0, 1, "grid"), ("harmonic", 0, 0, "exact"), ("cube", 0, 0, "grid"),
    ("cube", 0, 0, "none"), ("cube", 1, 0, "grid"), ("cfg0", 0, 0, "exact")])
def test_every_count_and_cap(env, kind, precision, y_exp, cv):
    torch, pdd, ctx = env
    k, grid = KINDS[kind]
    node = np.full((1, 3 if kind == "cube" else 2), 0.5, np.float32)
    many = 40_000 if precision == 0 else 4_000
    for cap in (0, 37, 64):
        prob = pdd.Problem(ctx, k, y_rule=y_exp, precision=precision, max_steps=cap)
        gid = {"none": pdd.PDD_CV_NONE, "exact": pdd.PDD_CV_EXACT, "grid": 0}[cv]
        if cv == "grid":
            prob.set_control_grid(0, W.control_grid(k, grid, 1e-1))
        big = prob.estimate(node, many, 2e-3, grid_id=gid, emit_paths=True)
        ctx.set_claim(1)
        try:
            for n in (1, 2, 3, 5, 7, 8, 9, 11, 15, 16, 17, 20, 32):
                small = prob.estimate(node, n, 2e-3, grid_id=gid, emit_paths=True)
                for f in ("phi", "xi", "steps"):
                    assert torch.equal(small[f], big[f][:, :n]), (cap, n, f)
        finally:
            ctx.set_claim(0)
        prob.close()


@pytest.mark.parametrize("kind,precision", [("cfg0", 0), ("cfg0", 1), ("cube", 0)])
def test_spread_launches(env, kind, precision):
    """Around every line of the rule (paths per warp 1, 2 and 24, and none)."""
    torch, pdd, ctx = env
    k, grid = KINDS[kind]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    warps = 10 * sms if precision == 0 else 4 * sms
    prob = pdd.Problem(ctx, k, precision=precision)
    prob.set_control_grid(0, W.control_grid(k, grid, 1e-1))
    nodes = np.full((1, 3 if kind == "cube" else 2), 0.5, np.float32)
    for n in (1, 31, warps - 1, warps, warps + 1, 2 * warps, 2 * warps + 1, 24 * warps,
              24 * warps + 1, 24 * 32 * sms, 24 * 32 * sms + 1):
        a = prob.estimate(nodes, n, 1e-2, grid_id=0)
        ctx.set_launch(0, 3)  # too few blocks for one claim per warp
        c = prob.estimate(nodes, n, 1e-2, grid_id=0)
        ctx.set_launch(0, 0)
        ctx.set_claim(1)
        b = prob.estimate(nodes, n, 1e-2, grid_id=0)
        ctx.set_claim(0)
        for f in pdd.STAT_FIELDS + pdd.COUNT_FIELDS:
            assert torch.equal(a[f].nan_to_num(-1.0), b[f].nan_to_num(-1.0)), (n, f)
            assert torch.equal(c[f].nan_to_num(-1.0), b[f].nan_to_num(-1.0)), (n, f)
        assert int(a["n_paths"][0]) == n
    prob.close()


@pytest.mark.parametrize("kind,y_exp,cv", [("cfg0", 0, "grid"), ("cfg0", 1, "none"), ("aniso", 0, "grid"),
                                           ("paper", 0, "exact"), ("cube", 0, "grid")])
def test_pairs(env, kind, y_exp, cv):
    """The coupled kernels: every number of pairs in a warp, caps that end one
    path of a pair (the fine path has twice the steps) or both, and spread
    launches; against the first pairs of a large launch."""
    torch, pdd, ctx = env
    k, grid = KINDS[kind]
    node = np.full((1, 3 if kind == "cube" else 2), 0.5, np.float32)
    for cap in (0, 37, 64):
        prob = pdd.Problem(ctx, k, y_rule=y_exp, max_steps=cap)
        gid = {"none": pdd.PDD_CV_NONE, "exact": pdd.PDD_CV_EXACT, "grid": 0}[cv]
        if cv == "grid":
            prob.set_control_grid(0, W.control_grid(k, grid, 1e-1))
        big = prob.estimate_coupled(node, 130_000, 4e-3, grid_id=gid, emit_paths=True)
        for claim, counts in ((1, (1, 2, 3, 5, 7, 8, 9, 11, 14, 15, 28, 32)), (0, (3, 1500, 9000))):
            ctx.set_claim(claim)
            try:
                for n in counts:
                    small = prob.estimate_coupled(node, n, 4e-3, grid_id=gid, emit_paths=True)
                    for a, b in zip(small, big):
                        for f in ("phi", "xi", "steps"):
                            assert torch.equal(a[f], b[f][:, :n]), (cap, claim, n, f)
            finally:
                ctx.set_claim(0)
        prob.close()
