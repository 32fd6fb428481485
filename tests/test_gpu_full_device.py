"""Record copies are left out where the device has no room for them.

128 levels of 60 nodes at 10 steps a path take 16 copies of their records, 24 MB
of workspace with its reserve, and 1.5 MB without copies.  With about 10 MB left
on the device the call still runs, with the same results.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_levels_on_a_full_device():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1512_02818_gb300 import build, pdd
    build.build()
    rng = np.random.default_rng(1)
    levels = [dict(nodes=torch.from_numpy(rng.uniform(0.3, 0.7, (60, 2)).astype(np.float32)).cuda(),
                   n_paths=200, dt=1e-2, stream_tag=i) for i in range(128)]
    first = pdd.Context(0)
    p1 = pdd.Problem(first, pdd.PDD_PROBLEM_CFG0_2D)
    want = p1.estimate_levels(levels)[1]  # also loads the kernels
    ctx = pdd.Context(0)
    prob = pdd.Problem(ctx, pdd.PDD_PROBLEM_CFG0_2D)
    prepared = [prob._prepare(lv["nodes"], 200, 1e-2, pdd.PDD_CV_NONE, 1234, lv["stream_tag"], 1.0, False, True,
                              False, False) for lv in levels]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    filler = torch.empty((free // 2**21 - 5) * 2**21, dtype=torch.uint8, device="cuda")
    try:
        assert torch.cuda.mem_get_info()[0] < 20 * 2**20
        for _ in range(2):  # the second call finds its workspace in place
            status = pdd.pdd_estimate_levels(prob.handle, [p[0] for p in prepared], [p[1] for p in prepared])
            assert status == pdd.PDD_OK
    finally:
        del filler
        torch.cuda.empty_cache()
    for a, (_, _, b) in zip(want, prepared):
        for f in pdd.STAT_FIELDS + pdd.COUNT_FIELDS:
            assert torch.equal(a[f].nan_to_num(-1.0), b[f].nan_to_num(-1.0)), f
    for x in (prob, ctx, p1, first):
        x.close()
