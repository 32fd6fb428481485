"""The FP64 paths' normals against extended precision.

r = sqrt(-2 ln u) and the angle come from tables and short polynomials.  Their
roundings add up to under five units of 2^-53 of r: the logarithm and its sum
(1.5, halved by the root), the reciprocal root (2), two products (1), the
rotation (1.5, at most 1 in absolute terms) and its product (0.5).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tag", [0, 7, 0xFFFFFFFF])
def test_normals(tag):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    L = np.longdouble
    if np.finfo(L).nmant < 63:
        pytest.skip("no extended precision on this machine")
    from paper_1512_02818_gb300 import build, pdd
    build.build()
    n = 200_000
    out = torch.zeros(4 * n, dtype=torch.float64, device="cuda")
    pdd.pdd_debug_normals(99, tag, 3, 5, 0, 4 * n, pdd.PDD_PATH_FP64, None, out.data_ptr())
    ctr = torch.zeros((n, 4), dtype=torch.int32, device="cuda")
    ctr[:, 0], ctr[:, 1], ctr[:, 2] = torch.arange(n), 5, 3
    key = torch.zeros((n, 2), dtype=torch.int32, device="cuda")
    key[:, 0], key[:, 1] = 99, tag if tag < 2**31 else tag - 2**32
    w = torch.zeros((n, 4), dtype=torch.int32, device="cuda")
    pdd.pdd_debug_philox(ctr.data_ptr(), key.data_ptr(), w.data_ptr(), n)
    u = ((w.cpu().numpy().view(np.uint32).astype(np.int64) >> 9).astype(L) + L(0.5)) / L(2**23)
    two_pi = 2 * L("3.14159265358979323846264338327950288")
    got = out.cpu().numpy().reshape(n, 4)
    for a, b in ((0, 1), (2, 3)):
        r = np.sqrt(-2 * np.log(u[:, a]))
        for col, f in ((a, np.cos), (b, np.sin)):
            err = np.abs(got[:, col].astype(L) - r * f(two_pi * u[:, b])) / r
            assert float(err.max()) <= 5 * 2.0**-53, float(err.max())
