"""The isclose grid's rtol table where it can go wrong: rtols on and around
table entries, equal and very close rtols, differences equal to atol + rtol |g|,
operands at the ends of the range, goldens of zero, and partial warps."""
import numpy as np
import pytest

from parity_util import to_device

pytestmark = pytest.mark.gpu
RTOLS = {"decades": [10.0 ** -k for k in range(8, 0, -1)], "powers": [2.0 ** -k for k in range(14, -2, -2)],
         "near": [1e-4, 1.1e-4, 1.2e-4, 1.21e-4], "same": [1e-3, 1e-3, 1e-2], "zero": [0.0, 1e-6, 1.0], "one": [1e-4],
         "huge": [1e-30, 1.0, 1e30], "close": [0.0, 0.0, 1.0, 1.0, 1.1, 1.2, 1.3, 1.7]}


@pytest.mark.parametrize("rtols", RTOLS)
@pytest.mark.parametrize("atols", ([0.0], [1e-6, 0.0, 1e-3], [0.0, 1e-40, 1e-20, 1e20]))
@pytest.mark.parametrize("n", (31, 33, 40_003))
def test_grid(peat_gpu, oracle, rtols, atols, n):
    rt = RTOLS[rtols]
    rng = np.random.default_rng(n)
    g = (rng.standard_normal(n) * np.exp2(rng.choice([0, 0, 0, 5, -30, -125, 100], n))).astype(np.float32)
    g[rng.random(n) < 0.02] = 0.0
    r = np.array(rt, np.float32)[rng.integers(0, len(rt), n)]
    with np.errstate(over="ignore", invalid="ignore"):
        c = (g + np.abs(g) * r).astype(np.float32)      # on a boundary, up to rounding
        k = rng.integers(0, 4, n)
        c = np.where(k == 1, np.nextafter(c, np.float32(np.inf)), c)
        c = np.where(k == 2, (g * (1 + 1e-4 * rng.standard_normal(n))).astype(np.float32), c)
        c = np.where(k == 3, g.astype(np.float16).astype(np.float32), c).astype(np.float32)
    gb, cb = g.view(np.uint32), c.view(np.uint32)
    with peat_gpu.Handle(0) as h:
        got = peat_gpu.peat_isclose_grid(h, to_device(gb, "f32"), to_device(cb, "f32"), rt, atols)
    for i, x in enumerate(rt):
        for j, y in enumerate(atols):
            st, _ = oracle.compare(gb, cb, "f32", x, y)
            assert got[i, j] == st["count"][0] + st["count"][1], (rtols, x, y)
