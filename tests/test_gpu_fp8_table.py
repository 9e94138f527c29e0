"""The 8-bit compare, short items pair by pair and longer ones (from about
4 M elements) through a table of (golden, candidate) combinations, against
the oracle: every pair of patterns, ties of the maxima in many places, item and
vector edges, opposite signs, all-equal tensors and segments."""
import numpy as np
import pytest
import torch

from parity_util import assert_hist_equal, assert_stats_equal

pytestmark = pytest.mark.gpu
TDT = {"f8e4m3": torch.float8_e4m3fn, "f8e5m2": torch.float8_e5m2}


def check(peat_gpu, oracle, g, c, dtype, rtol, atol, ctx, offsets=None, shift=0):
    def dev(x):
        buf = torch.empty(x.size + shift, dtype=torch.uint8, device="cuda")
        buf[shift:].copy_(torch.from_numpy(x))
        return buf[shift:].view(TDT[dtype])
    with peat_gpu.Handle(0) as h:
        if offsets is None:
            st, hist = peat_gpu.peat_compare(h, dev(g), dev(c), rtol, atol)
            ost, oh = oracle.compare(g, c, dtype, rtol, atol)
            st, ost = [st], [ost]
        else:
            st, hist = peat_gpu.peat_compare_segmented(h, dev(g), dev(c), offsets, rtol, atol)
            ost, oh = oracle.compare_segmented(g, c, offsets, dtype, rtol, atol)
    for s, (a, b) in enumerate(zip(st, ost)):
        assert_stats_equal(a, b, f"{ctx} segment {s}")
    assert_hist_equal(hist, oh, ctx)


@pytest.mark.parametrize("dtype", TDT)
@pytest.mark.parametrize("rtol,atol", ((0.125, 0.0), (0.0, 0.0), (0.1, 0.01)))
@pytest.mark.parametrize("least", (131_072, 1 << 22))
def test_every_pair(peat_gpu, oracle, dtype, rtol, atol, least):
    """All 65536 combinations in a random order; then those of one sign, and without the non-finite ones; those of
    opposite signs, and a few of them among the others."""
    rng = np.random.default_rng(1)
    idx = np.arange(65536)
    g, c = (idx >> 8).astype(np.uint8), (idx & 255).astype(np.uint8)

    def run(k, ctx):
        i = rng.permutation(np.tile(idx[k], -(-least // int(k.sum()))))
        check(peat_gpu, oracle, g[i], c[i], dtype, rtol, atol, ctx)
    run(idx >= 0, "all")
    one = ((g ^ c) & 0x80) == 0
    run(~one, "opposite signs")
    run(one | (idx % 101 == 0), "few of opposite signs")
    run(one, "one sign")
    one &= ((g & 0x7F) < 0x78) & ((c & 0x7F) < 0x78)
    run(one, "finite")
    run(one & ((g & 0x7F) != 0), "no zero golden")


@pytest.mark.parametrize("dtype", TDT)
@pytest.mark.parametrize("n", (1, 15, 16, 17, 4095, 4096, 4097, 16385, 700_001, (1 << 22) - 1, (1 << 22) + 77))
@pytest.mark.parametrize("shift", (0, 5))
def test_edges(peat_gpu, oracle, dtype, n, shift):
    rng = np.random.default_rng(n)
    g = rng.integers(0x20, 0x50, n).astype(np.uint8) | (rng.integers(0, 2, n).astype(np.uint8) << 7)
    c = g + rng.integers(-2, 3, n).astype(np.uint8)
    check(peat_gpu, oracle, g, c, dtype, 0.125, 0.0, f"n={n}", shift=shift)
    check(peat_gpu, oracle, g, g, dtype, 0.125, 0.0, f"equal n={n}", shift=shift)


@pytest.mark.parametrize("dtype", TDT)
@pytest.mark.parametrize("scale", (1, 15))
def test_segments_and_ties(peat_gpu, oracle, dtype, scale):
    rng = np.random.default_rng(3)
    n = 300_000 * scale
    g = np.full(n, 0x41, np.uint8)
    c = g.copy()
    c[100_001 * scale:] = 0x42
    c[250_000 * scale:] = 0xC1
    off = [0, 0, 7, 100_000 * scale, 100_003 * scale, 250_000 * scale, 250_000 * scale, n]
    check(peat_gpu, oracle, g, c, dtype, 0.01, 0.0, "constant", off)
    g = rng.integers(0, 256, n).astype(np.uint8)
    check(peat_gpu, oracle, g, rng.permutation(g), dtype, 0.01, 0.0, "random", off)


@pytest.mark.parametrize("dtype", TDT)
def test_many_segments(peat_gpu, oracle, dtype):
    """More segments than CTAs and more pairs than a table call needs: short items, evaluated pair by pair."""
    rng = np.random.default_rng(5)
    off = np.concatenate([[0], np.cumsum(rng.integers(0, 20_000, 460))])
    n = int(off[-1])
    assert n > 1 << 22
    g = rng.integers(0x20, 0x50, n).astype(np.uint8) | (rng.integers(0, 2, n).astype(np.uint8) << 7)
    c = g + rng.integers(-2, 3, n).astype(np.uint8)
    check(peat_gpu, oracle, g, c, dtype, 0.125, 0.0, "many segments", list(map(int, off)))
