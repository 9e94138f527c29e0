"""The binary16 context statistics against the oracle at the edges of their
vector rounds and with every kind of vector: values below 1/4, any finite
values, NaN and infinities among them, both zeros, the smallest and largest
values."""
import numpy as np
import pytest
import torch

import paper_2609_13544_gb300 as peat

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", (1, 7, 8, 9, 255, 2048, 4095, 4096, 4097, 8191, 8192, 8200, 300_001))
@pytest.mark.parametrize("kind", ("small", "mixed", "wide", "special", "constant", "zeros", "largest"))
@pytest.mark.parametrize("shift", (0, 3))
def test_f16(peat_gpu, oracle, n, kind, shift):
    rng = np.random.default_rng(n)
    x = {"small": lambda: rng.laplace(0, 0.02, n).clip(-0.2499, 0.2499),
         "mixed": lambda: rng.standard_normal(n) * 0.2,
         "wide": lambda: rng.standard_normal(n) * np.exp2(rng.integers(-24, 15, n)),
         "special": lambda: np.where(rng.random(n) < 0.01, rng.choice([np.nan, np.inf, -np.inf, -0.0, 6e-8], n), rng.standard_normal(n)),
         "constant": lambda: np.full(n, -0.25), "zeros": lambda: rng.choice([0.0, -0.0], n),
         "largest": lambda: rng.choice([65504.0, -65504.0, 6e-8], n)}[kind]()
    with np.errstate(over="ignore"):
        b = x.astype(np.float16).view(np.uint16)
    buf = torch.empty(n + shift, dtype=torch.int16, device="cuda")
    buf[shift:].copy_(torch.from_numpy(b.view(np.int16)))
    off = [0, n // 3, n // 3, n]
    with peat.Handle(0) as h:
        got = peat.peat_tensor_stats(h, buf.view(torch.float16)[shift:], off)
    for s in range(3):
        want = oracle.tensor_stats(b[off[s]:off[s + 1]], "f16")
        for k in ("n", "n_finite", "n_nan", "n_inf", "sum", "sum_sq", "mean", "var", "min", "max"):
            assert got[s][k] == want[k], (kind, n, s, k, got[s][k], want[k])
