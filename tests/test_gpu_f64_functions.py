"""The FP64 paths' sin, cos and exp by table, and the grid's cells, at their own accuracy.

The functions add a table value t (in two parts) and a term of at most 1/511 of
it, so their error is half a unit in the last place of the result and what
roundings leave in the term.  sin and cos: half a unit of the remainder's sine
(2^-63), of the term (2^-62) and the cosine's truncation, d^6 / 720 at d = 1/512
(2^-63.5): under 2^-60.5.  exp, with t up to e^2: e^2 times half a unit of the
polynomial (2^-62), of its sum before the last product and the truncation
(2^-63.5 each), and half a unit of the term (2^-60): under 2^-57.5.
"""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _evaluate(x, n):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1512_02818_gb300 import build, pdd
    build.build()
    xd = torch.from_numpy(x).cuda()
    d = [torch.empty_like(xd) for _ in range(4)]
    cell = torch.empty(len(x), dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    pdd.pdd_debug_f64_functions(xd.data_ptr(), len(x), n, d[0].data_ptr(), d[1].data_ptr(),
                                d[2].data_ptr(), cell.data_ptr(), d[3].data_ptr())
    return [t.cpu().numpy() for t in d] + [cell.cpu().numpy()]


def test_sin_cos_exp():
    L = np.longdouble
    if np.finfo(L).nmant < 63:
        pytest.skip("no extended precision on this machine")
    rng = np.random.default_rng(11)
    points = np.arange(513) / 256.0
    middles = (np.arange(512) + 0.5) / 256.0
    x = np.concatenate([points, middles, np.nextafter(middles, 0), np.nextafter(middles, 2),
                        np.nextafter(points[1:], 0), np.nextafter(points[:-1], 2),
                        2.0 ** -np.arange(1, 300), rng.uniform(0, 2, 200_000)])
    s, c, e, _, _ = _evaluate(x, 3)
    for got, f, term in ((s, np.sin, 2.0**-60.5), (c, np.cos, 2.0**-60.5), (e, np.exp, 2.0**-57.5)):
        want = f(x.astype(L))
        err = np.abs(got.astype(L) - want)
        bound = 0.5 * np.spacing(np.abs(want).astype(np.float64)) + term
        assert np.all(err <= bound), (f.__name__, x[np.argmax(err / bound)], float(np.max(err / bound)))


@pytest.mark.parametrize("n", [3, 17, 129, 4097])
def test_cells(n):
    rng = np.random.default_rng(n)
    edges = np.arange(n) / (n - 1)
    edges = edges[rng.permutation(n)[:200]]
    x = np.concatenate([edges, np.nextafter(edges, -1), np.nextafter(edges, 2), [0.0, 1.0, -1e-9, 1 + 1e-9],
                        rng.uniform(0, 1, 1000)])
    *_, frac, cell = _evaluate(x, n)
    for xi, f, i in zip(x, frac, cell):
        assert i == min(max(int(np.floor(xi * (n - 1))), 0), n - 2), xi
        assert f == float(Fraction(float(xi)) * (n - 1) - int(i)), xi  # rounded once
