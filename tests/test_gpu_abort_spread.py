"""An abort stops the unstarted paths of a launch whose warps take one batch each.

24 paths a warp over the whole chip are more blocks than fit at once, so some
wait for others to end.  The paths take about 1e6 steps each (the launch runs
for over a second), and the abort comes a tenth of a second after it began: the
waiting blocks find the mark and run nothing, and the call reports
PDD_ERR_CANCELLED with the counts of the paths that ran.
"""
import threading
import time

import pytest

from paper_1512_02818_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,coupled,dt", [(1, False, 2e-7), (0, True, 4e-7)])
def test_waiting_blocks_take_no_paths(kind, coupled, dt):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1512_02818_gb300 import build, pdd
    build.build()
    ctx = pdd.Context(0)
    prob = pdd.Problem(ctx, kind)
    prob.set_control_grid(0, W.control_grid(kind, 65, 1e-1))
    node = torch.full((1, 2), 0.5, device="cuda")
    n = 24 * 32 * torch.cuda.get_device_properties(0).multi_processor_count

    def run(paths, h, rec):
        if coupled:
            return prob.accumulate_coupled(node, paths, h, rec[0], rec[1], grid_id=0)
        return prob.accumulate(node, paths, h, rec[0], grid_id=0)

    def records():
        r = [torch.zeros((1, pdd.PDD_RECORD_WORDS), dtype=torch.int64, device="cuda") for _ in range(2)]
        torch.cuda.synchronize()
        return r

    run(n, 1e-3, records())  # workspace and kernels loaded
    rec, out = records(), {}

    def call():
        try:
            out["status"] = run(n, dt, rec)
        except pdd.PddError as e:
            out["status"] = e.status

    th = threading.Thread(target=call)
    th.start()
    time.sleep(0.1)
    ctx.abort()
    th.join(timeout=60)
    assert not th.is_alive()
    assert out["status"] == pdd.PDD_ERR_CANCELLED
    assert 0 < int(rec[0][0, 14]) < n
    # the next call is whole, and its completeness check counts every warp
    assert prob.estimate(node, n, 1e-3, grid_id=0)["n_paths"][0] == n
    prob.close()
    ctx.close()
