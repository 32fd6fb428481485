"""Requests admitted one after another while others run: a launch waits for the
staging of its own requests, whenever each was admitted, and every result equals
the request alone.  A small quantum makes many launches, whose batches mix
requests of different admissions; polled requests leave room for later ones."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("policy", ["PDD_SERVE_FAIR", "PDD_SERVE_SHORTEST"])
def test_admissions_interleaved(policy):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1512_02818_gb300 import build, pdd
    build.build()
    ctx = pdd.Context(0)
    prob = pdd.Problem(ctx, pdd.PDD_PROBLEM_CFG0_2D)
    rng = np.random.default_rng(8)
    # sizes on both sides of the one (2^18 nodes) above which inputs are copied
    sizes = [500, 1 << 19, 7, 300_000, 64, 2000, 1 << 18, 33] * 3
    nodes = [rng.uniform(0.2, 0.8, (n, 2)).astype(np.float32) for n in sizes]
    paths = [2 if n > 100_000 else 4000 for n in sizes]
    srv = pdd.Server(ctx, max_active=4, policy=getattr(pdd, policy), quantum_path_steps=2_000_000,
                     device_arena_bytes=1 << 30)
    try:
        tickets = [srv.submit(prob, x, p, 1e-2, seed=3, stream_tag=i)
                   for i, (x, p) in enumerate(zip(nodes, paths))]
        for i, (t, x, p) in enumerate(zip(tickets, nodes, paths)):
            status, got = srv.poll(t, len(x), 60_000_000)
            assert status == pdd.PDD_OK
            alone = prob.estimate(x, p, 1e-2, seed=3, stream_tag=i)
            for f in pdd.STAT_FIELDS + pdd.COUNT_FIELDS:
                want = alone[f].cpu().numpy()
                assert np.array_equal(got[f], want, equal_nan=want.dtype.kind == "f"), (i, f)
    finally:
        srv.close()
    prob.close()
    ctx.close()
