"""The compare's window tables at the places where they can go wrong: tile and
vector edges, vectors with a few unequal lanes, equal pairs that hold NaN or
infinity inside them, ties of a maximum across the whole tensor, values at the
ends of the window, and a nonzero atol.  Everything exact against the oracle."""
import numpy as np
import pytest

from parity_util import NP_BITS, assert_hist_equal, assert_stats_equal, oracle_segmented, random_pairs, to_device

pytestmark = pytest.mark.gpu
DTYPES = ("f32", "f16", "bf16")


def encode(x, dtype):
    if dtype == "f32":
        return np.asarray(x, np.float32).view(np.uint32)
    if dtype == "f16":
        return np.asarray(x, np.float16).view(np.uint16)
    return (np.ascontiguousarray(np.asarray(x, np.float32)).view(np.uint32) >> 16).astype(np.uint16)


def check(peat_gpu, oracle, gb, cb, dtype, rtol, atol, ctx, shift=0):
    with peat_gpu.Handle(0) as h:
        st, hist = peat_gpu.peat_compare(h, to_device(gb, dtype, shift), to_device(cb, dtype, shift), rtol, atol)
    ost, oh = oracle.compare(gb, cb, dtype, rtol, atol)
    assert_stats_equal(st, ost, ctx)
    assert_hist_equal(hist, oh, ctx)


def steps(gb, k):
    """Patterns k steps away, inside the finite range and the same sign."""
    w = gb.dtype.itemsize * 8
    mag = gb & ((1 << (w - 1)) - 1)
    return np.where(mag > 4096 if w == 32 else mag > 300, gb + k.astype(gb.dtype), gb).astype(gb.dtype)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("n", (1, 7, 8, 9, 255, 256, 511, 512, 513, 8191, 8192, 8193, 65537))
@pytest.mark.parametrize("shift", (0, 3))
def test_edges(peat_gpu, oracle, dtype, n, shift):
    rng = np.random.default_rng(n + shift)
    gb = encode(rng.standard_normal(n), dtype)
    cb = steps(gb, rng.integers(-3, 4, n))
    check(peat_gpu, oracle, gb, cb, dtype, 1e-3, 0.0, f"{dtype} n={n} shift={shift}", shift)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("share", (0.0, 0.0005, 0.01, 0.05, 0.3, 1.0))
def test_shares_of_unequal_pairs(peat_gpu, oracle, dtype, share):
    """Sparse and dense vectors, with NaN and infinity in equal and unequal pairs of both."""
    rng = np.random.default_rng(int(share * 1e4))
    n = 200_003
    gb = encode(rng.standard_normal(n) * 3.0, dtype)
    k = np.where(rng.random(n) < share, rng.integers(-2, 3, n), 0)
    cb = steps(gb, k)
    special = [np.nan, np.inf, -np.inf, 0.0, -0.0]
    for i in rng.integers(0, n, 60):
        gb[i] = cb[i] = encode([special[int(rng.integers(0, 5))]], dtype)[0]
    for i in rng.integers(0, n, 20):
        cb[i] = encode([special[int(rng.integers(0, 5))]], dtype)[0]
    check(peat_gpu, oracle, gb, cb, dtype, 1e-3, 0.0, f"{dtype} share={share}")


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("value", (1.0, 1.3, -777.0, 3e-5, 60000.0))
def test_one_value_everywhere(peat_gpu, oracle, dtype, value):
    """Every pair ties for all three maxima: the first one wins."""
    n = 150_001
    gb = np.repeat(encode([value], dtype), n)
    cb = gb.copy()
    cb[1234:] += 1
    check(peat_gpu, oracle, gb, cb, dtype, 1e-2, 0.0, f"{dtype} value={value}")


@pytest.mark.parametrize("dtype,lo,hi", (("f32", -120, 120), ("f32", -12, 3), ("f16", -24, -10), ("f16", -24, 15),
                                         ("f16", 8, 15), ("bf16", -120, 120), ("bf16", -60, 4), ("bf16", -126, -100)))
@pytest.mark.parametrize("width", (1, 20, 63, 64, 127, 128, 400))
def test_window_ends(peat_gpu, oracle, dtype, lo, hi, width):
    """Goldens over a range of binades, differences up to `width` steps: inside and outside of the window."""
    rng = np.random.default_rng(width)
    n = 60_000
    x = np.exp2(rng.uniform(lo, hi, n)) * rng.choice([-1.0, 1.0], n)
    gb = encode(x, dtype)
    cb = (gb.astype(np.int64) + rng.integers(-width, width + 1, n)).clip(0, 2 ** (8 * gb.dtype.itemsize) - 1).astype(
        NP_BITS[dtype])
    check(peat_gpu, oracle, gb, cb, dtype, 1e-2, 0.0, f"{dtype} 2^{lo}..2^{hi} width={width}")


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("rtol,atol", ((1e-3, 1e-5), (0.0, 1e-3), (2.0 ** -7, 2.0 ** -12), (0.0, 0.0), (1.0, 1e30)))
def test_tolerances(peat_gpu, oracle, dtype, rtol, atol):
    rng = np.random.default_rng(3)
    n = 100_001
    gb = encode(rng.standard_normal(n), dtype)
    cb = steps(gb, rng.integers(-9, 10, n))
    check(peat_gpu, oracle, gb, cb, dtype, rtol, atol, f"{dtype} rtol={rtol} atol={atol}")


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("share", (0.02, 0.6))
@pytest.mark.parametrize("lead", (0.0, 1e-3))
def test_magnitudes_above_the_first_ones(peat_gpu, oracle, dtype, share, lead):
    """Equal and unequal pairs far above the elements that a CTA's range starts with: each segment, one CTA's work,
    begins with zeros or small values, as a padded batch does, then holds data over many binades."""
    rng = np.random.default_rng(int(share * 100) + int(lead * 1e4))
    m, nseg = 18_000, 200
    x = np.exp2(rng.uniform(-3, 15, (nseg, m))) * rng.choice([-1.0, 1.0], (nseg, m))
    x[:, :9000] = lead * rng.standard_normal((nseg, 9000))
    gb = encode(x.reshape(-1), dtype)
    cb = steps(gb, np.where(rng.random(gb.size) < share, rng.integers(-2, 3, gb.size), 0))
    off = np.arange(nseg + 1, dtype=np.int64) * m
    with peat_gpu.Handle(0, max_segments=nseg) as h:
        st, hist = peat_gpu.peat_compare_segmented(h, to_device(gb, dtype), to_device(cb, dtype), off, 1e-3, 0.0)
    ost, oh = oracle_segmented(gb, cb, off, dtype, 1e-3, 0.0)
    for s in range(nseg):
        assert_stats_equal(st[s], ost[s], f"{dtype} share={share} lead={lead} segment {s}")
        assert_hist_equal(hist[s], oh[s], f"{dtype} share={share} lead={lead} segment {s}")


@pytest.mark.parametrize("dtype,umax", (("f32", 2 ** 23 - 1), ("f16", 127), ("bf16", 63)))
@pytest.mark.parametrize("flip", (None, 5, 150_000))
def test_steps_at_the_limit(peat_gpu, oracle, dtype, umax, flip):
    """Pairs exactly as many steps apart as the window allows, tied all over the tensor, beside none or one that is far
    outside of it (in the window's sample or not): the largest ULP distance and difference and their first indices."""
    n = 200_001
    rng = np.random.default_rng(umax)
    gb = encode(1.0 + rng.random(n), dtype)
    cb = gb.copy()
    for i in rng.integers(300, n, 2000):
        cb[i] += umax if rng.random() < 0.5 else umax - 1
    if flip is not None:
        cb[flip] ^= 1 << (8 * gb.itemsize - 3)
    check(peat_gpu, oracle, gb, cb, dtype, 1e-3, 0.0, f"{dtype} flip={flip}")
    cb[-1] = gb[-1] + umax + 1  # one step more, at the very end
    check(peat_gpu, oracle, gb, cb, dtype, 1e-3, 0.0, f"{dtype} flip={flip}, one past the limit")


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("seed", (1, 2))
def test_short_segments(peat_gpu, oracle, dtype, seed):
    """Segments of about as many pairs as a CTA has threads (at most a pair per thread is a path of its own), of any
    bit patterns and of close pairs, between longer and empty ones, at odd offsets."""
    rng = np.random.default_rng(seed)
    sizes = rng.choice([0, 1, 2, 31, 33, 255, 256, 257, 511, 512, 513, 700, 5000], 300)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n = int(off[-1])
    gb, cb = random_pairs(dtype, n, seed) if seed == 1 else (None, None)
    if gb is None:
        gb = encode(rng.standard_normal(n), dtype)
        cb = steps(gb, np.where(rng.random(n) < 0.6, rng.integers(-3, 4, n), 0))
    with peat_gpu.Handle(0, max_segments=300) as h:
        st, hist = peat_gpu.peat_compare_segmented(h, to_device(gb, dtype, 1), to_device(cb, dtype, 1), off, 1e-3, 1e-6)
    ost, oh = oracle.compare_segmented(gb, cb, off, dtype, 1e-3, 1e-6)
    for s in range(300):
        assert_stats_equal(st[s], ost[s], f"{dtype} segment {s} of {sizes[s]}")
        assert_hist_equal(hist[s], oh[s], f"{dtype} segment {s} of {sizes[s]}")
