"""Calls whose data is laid out in a way that once cost many times an ordinary
call of the same size: each against that ordinary call, timed in turn on the
same GPU.  The limits lie between the two and leave room for noise."""
import pytest

pytestmark = pytest.mark.gpu
EPS = {"f32": 2.0 ** -23, "f16": 2.0 ** -10, "bf16": 2.0 ** -7}


def median_us(torch, f):
    f()
    torch.cuda.synchronize()
    a, b, t = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True), []
    for _ in range(9):
        a.record()
        for _ in range(5):
            f()
        b.record()
        torch.cuda.synchronize()
        t.append(a.elapsed_time(b) * 200.0)
    return sorted(t)[4]


def compare_us(peat, golden, candidate, rtol=1e-3, atol=0.0):
    import torch
    stats = torch.zeros(peat.STATS_BYTES, dtype=torch.uint8, device="cuda")
    hist = torch.zeros(peat.HIST_BINS, dtype=torch.int64, device="cuda")
    with peat.Handle(0) as h:
        return median_us(torch, lambda: peat.peat_compare_raw(h, golden, candidate, rtol, atol, stats, hist))


def activation(dtype, rows=1 << 13, cols=1 << 12):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    dt = getattr(torch, {"f32": "float32", "f16": "float16", "bf16": "bfloat16"}[dtype])
    return dt, torch.randn(rows, cols, generator=gen, device="cuda"), torch.randn(rows, cols, generator=gen, device="cuda")


def noisy(x, noise, dtype, dt):
    g = x.to(dt)
    return g.view(-1), (g.float() * (1.0 + EPS[dtype] * noise)).to(dt).view(-1)


@pytest.mark.parametrize("dtype", ("f16", "bf16"))
def test_zero_padding(peat_gpu, dtype):
    """Rows and parts of rows of zeros before the data (25 and 4 times the ordinary call, with a window placed by
    the first elements of a CTA's range)."""
    dt, x, noise = activation(dtype)
    plain = compare_us(peat_gpu, *noisy(x, noise, dtype, dt))
    for pad in ("sequences", "rows"):
        y = x.clone()
        if pad == "sequences":
            y.view(8, -1)[:, : y.numel() // 16] = 0.0
        else:
            y[:, :2048] = 0.0
        t = compare_us(peat_gpu, *noisy(y, noise, dtype, dt))
        assert t < 1.7 * plain, f"{dtype} {pad}: {t:.1f} us against {plain:.1f}"


@pytest.mark.parametrize("dtype,limit", (("f16", 15), ("bf16", 12)))
def test_most_pairs_outside_the_window(peat_gpu, dtype, limit):
    """Additive noise of a tenth of the scale: a third of the pairs and more are general, every piece is rescanned
    (20 times the ordinary 16-bit call when the rescan ran a round for every 32 elements)."""
    dt, x, noise = activation(dtype)
    plain = compare_us(peat_gpu, *noisy(x, noise, dtype, dt))
    t = compare_us(peat_gpu, x.to(dt).view(-1), (x + 0.1 * noise).to(dt).view(-1))
    assert t < limit * plain, f"{dtype}: {t:.1f} us against {plain:.1f}"


@pytest.mark.parametrize("dtype", ("f16", "bf16"))
def test_additive_noise(peat_gpu, dtype):
    """Errors of absolute size: small values differ by hundreds of steps, nearly every vector holds such a pair, and
    1 to 8 % of all are general (25 times the ordinary binary16 call when each went the slow path)."""
    dt, x, noise = activation(dtype)
    plain = compare_us(peat_gpu, *noisy(x, noise, dtype, dt))
    for sigma, limit in ((0.001, 2.7), (0.01, 4.5)):
        t = compare_us(peat_gpu, x.to(dt).view(-1), (x + sigma * noise).to(dt).view(-1))
        assert t < limit * plain, f"{dtype} {sigma}: {t:.1f} us against {plain:.1f}"


@pytest.mark.parametrize("rtols", ("decades", "close"))
def test_isclose_large_noise(peat_gpu, rtols):
    """An isclose grid over errors as large as the values, most of which are not float32 numbers, with rtols a decade
    or a tenth apart (4.5 times the grid over small errors when each test of such a difference took the margins of two roundings)."""
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    decades = [10.0 ** -k for k in range(8, 0, -1)]
    g = torch.randn(1 << 24, generator=gen, device="cuda")
    c = g + torch.randn(1 << 24, generator=gen, device="cuda")
    counts = torch.zeros(64, dtype=torch.int64, device="cuda")
    atols = [0.0] + [10.0 ** -k for k in range(8, 1, -1)]
    with peat_gpu.Handle(0) as h:
        plain = median_us(torch, lambda: peat_gpu.peat_isclose_grid_raw(h, g, g.half().float(), decades, atols, counts))
        rt = decades if rtols == "decades" else [1.0 + 0.1 * k for k in range(8)]
        t = median_us(torch, lambda: peat_gpu.peat_isclose_grid_raw(h, g, c, rt, atols, counts))
    assert t < 3.7 * plain, f"{t:.1f} us against {plain:.1f}"


def test_opposite_signs_8bit(peat_gpu):
    """E5M2 with noise as large as the values: 16 % of the pairs have opposite signs (2.2 times the call with 0.04 %
    of them when each lane took its own in turn)."""
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    x, noise = (torch.randn(9_000_000, generator=gen, device="cuda") for _ in range(2))
    g = (2.0 * x).to(torch.float8_e5m2)
    plain, t = (compare_us(peat_gpu, g, (g.float() * (1.0 + s * noise)).to(torch.float8_e5m2), rtol=0.125) for s in (0.3, 1.0))
    assert t < 1.95 * plain, f"{t:.1f} us against {plain:.1f}"
