"""The argmax of tensors whose every error is zero is the first finite pair (for
the ULP distance: the first pair without NaN).  Tensors and segments that start
with NaN or infinite pairs, as many as a CTA has threads and around it, the
rest bitwise equal: the search for that pair takes one or more rounds of the
whole CTA, which must all leave after the same one."""
import numpy as np
import pytest

from parity_util import NP_BITS, assert_hist_equal, assert_stats_equal, to_device

pytestmark = pytest.mark.gpu
NAN = {"f32": 0x7FC00000, "f16": 0x7E00, "bf16": 0x7FC0}
INF = {"f32": 0x7F800000, "f16": 0x7C00, "bf16": 0x7F80}
ONE = {"f32": 0x3F800000, "f16": 0x3C00, "bf16": 0x3F80}
LEADS = (1, 255, 256, 257, 511, 512, 513, 5000)


def tensor(dtype, n, lead, kind):
    """n equal pairs, the first `lead` of them NaN ("nan"), infinite ("inf"), or infinite and then NaN ("mixed")."""
    g = np.full(n, ONE[dtype], NP_BITS[dtype])
    g[:lead] = NAN[dtype] if kind == "nan" else INF[dtype]
    if kind == "mixed":
        g[lead // 2:lead] = NAN[dtype]
    return g


@pytest.mark.parametrize("dtype", ("f32", "f16", "bf16"))
@pytest.mark.parametrize("kind", ("nan", "inf", "mixed"))
def test_one_tensor(peat_gpu, oracle, dtype, kind):
    with peat_gpu.Handle(0) as h:
        for lead in LEADS:
            for n in (lead, lead + 1, lead + 700):
                g = tensor(dtype, n, lead, kind)
                st, hist = peat_gpu.peat_compare(h, to_device(g, dtype), to_device(g, dtype), 1e-3, 0.0)
                ost, oh = oracle.compare(g, g, dtype, 1e-3, 0.0)
                assert_stats_equal(st, ost, f"{dtype} {kind} n={n} lead={lead}")
                assert_hist_equal(hist, oh, f"{dtype} {kind} n={n} lead={lead}")


@pytest.mark.parametrize("dtype", ("f32", "f16", "bf16"))
def test_segments(peat_gpu, oracle, dtype):
    """A segment of each kind and length: the pieces after it in the same CTA start from a clean state."""
    parts = [tensor(dtype, lead + 300, lead, kind) for lead in LEADS for kind in ("nan", "inf", "mixed")]
    g = np.concatenate(parts)
    off = np.concatenate([[0], np.cumsum([p.size for p in parts])]).astype(np.int64)
    c = g.copy()
    c[off[1:] - 100] += 1  # one pair of each segment's equal part differs
    for cand in (g, c):
        with peat_gpu.Handle(0, max_segments=64) as h:
            st, hist = peat_gpu.peat_compare_segmented(h, to_device(g, dtype), to_device(cand, dtype), off, 1e-3, 0.0)
        ost, oh = oracle.compare_segmented(g, cand, off, dtype, 1e-3, 0.0)
        for s in range(len(parts)):
            assert_stats_equal(st[s], ost[s], f"{dtype} segment {s}")
            assert_hist_equal(hist[s], oh[s], f"{dtype} segment {s}")
