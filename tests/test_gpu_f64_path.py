"""The binary64 compare's integer path against the oracle where it can go wrong:
item and vector edges, crossings of a binade, distances at the ends of the
window, ties of the maxima, equal tensors with NaN, and data whose binades
leave the window so that it has to be placed again."""
import numpy as np
import pytest

from parity_util import assert_hist_equal, assert_stats_equal
from test_gpu_f64 import dev

pytestmark = pytest.mark.gpu


def check(peat_gpu, oracle, g, c, rtol, atol, ctx, offsets=None):
    gb, cb = (np.ascontiguousarray(x, np.float64).view(np.uint64) for x in (g, c))
    with peat_gpu.Handle(0) as h:
        if offsets is None:
            st, hist = peat_gpu.peat_compare(h, dev(gb), dev(cb), rtol, atol)
            ost, oh = oracle.compare(gb, cb, "f64", rtol, atol)
            st, ost = [st], [ost]
        else:
            st, hist = peat_gpu.peat_compare_segmented(h, dev(gb), dev(cb), offsets, rtol, atol)
            ost, oh = oracle.compare_segmented(gb, cb, offsets, "f64", rtol, atol)
    for s, (a, b) in enumerate(zip(st, ost)):
        assert_stats_equal(a, b, f"{ctx} segment {s}")
    assert_hist_equal(hist, oh, ctx)


def step(g, k):
    return (g.view(np.int64) + k.astype(np.int64)).view(np.float64)


@pytest.mark.parametrize("n", (1, 2, 511, 512, 513, 4096, 4097, 70_001))
@pytest.mark.parametrize("bits", (0, 1, 28, 31, 32, 33, 45, 50, 51, 52))
def test_distances(peat_gpu, oracle, n, bits):
    rng = np.random.default_rng(n + bits)
    g = rng.standard_normal(n)
    g[::5] = 2.0 ** rng.integers(-3, 3, g[::5].size)  # on a binade's edge
    k = rng.integers(-(2 ** bits), 2 ** bits + 1, n)
    check(peat_gpu, oracle, g, step(g, k), 1e-7, 0.0, f"n={n} bits={bits}")


@pytest.mark.parametrize("cast", (np.float32, np.float16))
@pytest.mark.parametrize("rtol,atol", ((1e-7, 0.0), (2.0 ** -25, 0.0), (0.0, 0.0), (1e-4, 1e-9)))
def test_casts(peat_gpu, oracle, cast, rtol, atol):
    rng = np.random.default_rng(1)
    g = rng.standard_normal(100_003)
    check(peat_gpu, oracle, g, g.astype(cast).astype(np.float64), rtol, atol, f"{cast} {rtol} {atol}")


def test_ties_and_equal_pairs(peat_gpu, oracle):
    g = np.full(60_000, 1.7)
    c = g.copy()
    c[777:] = np.nextafter(1.7, 2.0)
    check(peat_gpu, oracle, g, c, 1e-7, 0.0, "every pair ties")
    c = g.copy()
    c[5] = g[5] = np.nan
    g[0] = np.nan
    check(peat_gpu, oracle, g, c, 1e-7, 0.0, "equal pairs and NaN")
    g = np.zeros(50_000)
    c = -g
    c[::2] = 0.0
    check(peat_gpu, oracle, g, c, 1e-7, 0.0, "zeros of both signs")


def test_window_moves(peat_gpu, oracle):
    """Blocks of very different magnitude in one tensor, and segments of them."""
    rng = np.random.default_rng(2)
    g = rng.standard_normal(120_000) * np.repeat(np.exp2([0.0, 90.0, -200.0, 900.0, -990.0, 10.0]), 20_000)
    c = step(g, rng.integers(-5, 6, g.size))
    check(peat_gpu, oracle, g, c, 1e-7, 0.0, "blocks")
    check(peat_gpu, oracle, g, c, 1e-7, 0.0, "segments", [0, 3, 20_000, 20_000, 50_001, 120_000])
