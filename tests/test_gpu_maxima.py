"""Merging the maxima of warps, CTAs and segments, and the general pairs' sums:
records that tie, that differ only in the rounding error of |d|, overflow
float32, divide by zero or lie among the subnormals, spread over all CTAs, and
more general pairs per CTA than its digit words hold without a flush."""
import numpy as np
import pytest
import torch

import paper_2609_13544_gb300 as peat
from parity_util import assert_hist_equal, assert_stats_equal, to_device

pytestmark = pytest.mark.gpu


def spread(kind, n, rng):
    """A quiet tensor with about one special pair in every 700."""
    g = rng.standard_normal(n).astype(np.float32)
    c = g.copy()
    idx = np.flatnonzero(rng.random(n) < 1 / 700)
    m = idx.size
    if kind == "ties":  # one ratio, one |d|, one ULP distance
        g[idx], c[idx] = np.float32(3.0), np.float32(7.5)
    elif kind == "lo":  # |d| equal in float32, apart in the rounding error only
        g[idx] = -np.float32(2.0) ** -rng.integers(3, 9, m).astype(np.float32)
        c[idx] = np.float32(2 ** 24 + 2)
    elif kind == "ratio":  # ratios within a few units of each other
        g[idx] = np.float32(1.0) + rng.integers(0, 4, m).astype(np.float32) * np.float32(2.0 ** -23)
        c[idx] = -g[idx] * np.float32(2 ** 20) + rng.integers(0, 3, m).astype(np.float32)
    elif kind == "overflow":
        g[idx] = -np.float32(3e38)
        c[idx] = np.float32(3e38) + rng.integers(0, 2, m).astype(np.float32) * np.float32(2e31)
    elif kind == "zero":  # infinite ratios
        g[idx] = np.float32(0.0)
        c[idx] = rng.integers(1, 4, m).astype(np.float32)
    elif kind == "subnormal":
        g = (rng.integers(1, 50, n)).astype(np.uint32).view(np.float32).copy()
        c = g.copy()
        c[idx] = rng.integers(1, 1 << 24, m).astype(np.uint32).view(np.float32)
    return g.view(np.uint32), c.view(np.uint32)


@pytest.mark.parametrize("kind", ("ties", "lo", "ratio", "overflow", "zero", "subnormal"))
@pytest.mark.parametrize("n", (700, 40_001, 1_200_007))
def test_records(peat_gpu, oracle, kind, n):
    g, c = spread(kind, n, np.random.default_rng(n))
    with peat.Handle(0) as h:
        gd, cd = to_device(g, "f32"), to_device(c, "f32")
        one, hist = peat.peat_compare(h, gd, cd, 1e-3, 0.0)
        off = np.array([0, n // 3, n // 3, n // 3 + 5, n], np.int64)
        many, hists = peat.peat_compare_segmented(h, gd, cd, off, 1e-3, 0.0)
    want, wh = oracle.compare(g, c, "f32", 1e-3, 0.0)
    assert_stats_equal(one, want, f"{kind} n={n}")
    assert_hist_equal(hist, wh, f"{kind} n={n}")
    want, wh = oracle.compare_segmented(g, c, off, "f32", 1e-3, 0.0)
    for s in range(4):
        assert_stats_equal(many[s], want[s], f"{kind} n={n} segment {s}")
        assert_hist_equal(hists[s], wh[s], f"{kind} n={n} segment {s}")


def test_many_general_pairs_per_cta(peat_gpu):
    """Every pair general (golden 0): d = +-c with known counts, summed in integers."""
    n = 304 * 256 * 300
    rng = np.random.default_rng(1)
    vals = np.array([0xFFFFFF, -0xFFFFFF, 0xABCDEF, -0x800001, 0xFF00FF], np.int64)
    which = rng.integers(0, vals.size, n)
    c = vals[which].astype(np.float32)
    with peat.Handle(0) as h:
        got = peat.peat_compare(h, torch.zeros(n, dtype=torch.float32, device="cuda"), torch.from_numpy(c).cuda(),
                                rtol=1e-3, atol=0.0)[0]
    cnt = [int(x) for x in np.bincount(which, minlength=vals.size)]
    v = [int(x) for x in vals]
    assert got["sum_signed"] == float(sum(k * x for k, x in zip(cnt, v)))
    assert got["sum_abs"] == float(sum(k * abs(x) for k, x in zip(cnt, v)))
    assert got["sum_sq"] == float(sum(k * x * x for k, x in zip(cnt, v)))
