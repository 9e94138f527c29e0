"""The mean of the top errors through its table pass: short exact differences
(rounding modes, steps of the spacing, a cast to half precision) from the size
at which the pass is offered, with pairs that its table does not take (NaN,
infinities, overflowing and inexact differences, values beyond the table, long
keys) among them, at the places a sample looks at and only elsewhere."""
import numpy as np
import pytest
import torch

import paper_2609_13544_gb300 as peat
from parity_util import NP_BITS, to_device

pytestmark = pytest.mark.gpu
N0 = 1 << 20


def pair(dtype, kind, n, rng):
    """Bit patterns of golden and candidate."""
    x = (rng.standard_normal(n) * 2).astype(np.float32)
    if dtype == "f32":
        g = x.view(np.uint32).copy()
    elif dtype == "bf16":
        g = (x.view(np.uint32) >> 16).astype(np.uint16)
    else:
        g = x.astype(np.float16).view(np.uint16).copy()
    if kind == "rounding":  # up to one spacing
        c = g + rng.integers(0, 2, n).astype(g.dtype)
    elif kind == "steps":   # some spacings either way
        c = (g.astype(np.int64) + np.rint(rng.standard_normal(n) * 9).astype(np.int64)).astype(g.dtype)
    elif kind == "cast":
        v = g.view(np.float32).astype(np.float16).astype(np.float32)
        c = v.view(np.uint32)
    elif kind == "same":
        c = g.copy()
    elif kind == "sparse":  # most pairs equal
        c = g + (rng.random(n) < 0.03).astype(g.dtype)
    return g, c


def spoil(g, c, idx, rng):
    """Pairs the table cannot hold at the given places."""
    big = {np.dtype(np.uint32): [0x7F800000, 0x7FC00001, 0xFF7FFFFF, 0x7F7FFFFF, 0x4B800001, 0x00000001, 0xFF800000],
           np.dtype(np.uint16): [0x7F80, 0x7FC1, 0xFF7F, 0x7F7F, 0x7BFF, 0xFBFF, 0x0001]}[g.dtype]
    c[idx] = rng.choice(np.array(big, np.uint64), idx.size).astype(g.dtype)
    half = idx[: idx.size // 2]
    g[half] = rng.choice(np.array(big, np.uint64), half.size).astype(g.dtype)


CASES = [(d, k) for d in ("f32", "f16", "bf16") for k in ("rounding", "steps", "same", "sparse")] + [("f32", "cast")]


@pytest.mark.parametrize("dtype,kind", CASES)
@pytest.mark.parametrize("n,shift", ((N0 - 1, 0), (N0, 0), (N0 + 24, 3), (3 * N0 + 5, 1)))
@pytest.mark.parametrize("bad", ("none", "few", "many", "unsampled"))
def test_table(peat_gpu, oracle, dtype, kind, n, shift, bad):
    rng = np.random.default_rng(n + 7 * shift)
    g, c = pair(dtype, kind, n, rng)
    if bad == "few":
        spoil(g, c, rng.choice(n, 40, replace=False), rng)
    elif bad == "many":
        spoil(g, c, rng.choice(n, n // 50, replace=False), rng)
    elif bad == "unsampled":  # everything outside the runs of a sample of 2^18 pairs
        vec = 16 // g.itemsize
        runs = min((n // vec + 31) // 32, (1 << 18) // (32 * vec))
        seen = np.zeros(n + 64 * vec, bool)
        for r in range(runs):
            a = (r * (n // vec) // runs) * vec
            seen[a:a + 32 * vec] = True
        free = np.flatnonzero(~seen[:n])
        if free.size:
            spoil(g, c, rng.choice(free, free.size // 9, replace=False), rng)
    gd, cd = to_device(g, dtype, shift), to_device(c, dtype, shift)
    with peat.Handle(0) as h:
        for num, den in ((1, 10), (1, 1), (1, 1000)):
            for _ in range(2):  # the state is clean for the next call
                got = peat.peat_topk_mean(h, gd, cd, num, den)
            want = oracle.topk_mean(g, c, dtype, num, den)
            for k in ("n_finite", "k", "threshold", "sum", "mean"):
                assert got[k] == want[k], (num, den, k, got[k], want[k])


@pytest.mark.parametrize("n", (65_535, 65_536, 65_537))
def test_inexact_pairs_up_to_the_list(peat_gpu, oracle, n):
    """Every pair tied in float32 and inexact, at the length of the list of rounding errors: up to it the passes
    for an overflowing list are not launched."""
    rng = np.random.default_rng(n)
    g = -(rng.integers(1, 3000, n).astype(np.float32) * np.float32(2.0 ** -12))
    c = np.full(n, np.float32(2 ** 24 + 2), np.float32)
    gb, cb = g.view(np.uint32), c.view(np.uint32)
    with peat.Handle(0) as h:
        for num, den in ((1, 10), (1, 1), (1, 1000)):
            got = peat.peat_topk_mean(h, to_device(gb, "f32"), to_device(cb, "f32"), num, den)
            want = oracle.topk_mean(gb, cb, "f32", num, den)
            for k in ("n_finite", "k", "threshold", "sum", "mean"):
                assert got[k] == want[k], (num, den, k, got[k], want[k])
