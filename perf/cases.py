"""The workloads that the library's speed is measured on.

Each case is one call that a fault-assessment program makes on tensors it
already holds on the GPU: the signature of a recorded tensor pair, of a whole
parameter list, the mean of the top errors, the context statistics, the
isclose acceptance grid, and the fused injection.  The inputs are the
synthetic recipes of ``paper_2609_13544_gb300.workloads`` (activations,
parameter lists of two model families, a playback step) and generic tensors
of the same kind.

Every result is defined exactly (integers, or an exact real number rounded
once), so two correct implementations agree bit for bit: the tolerance is
"exact" throughout.
"""
import math

import numpy as np
import torch

import paper_2609_13544_gb300 as peat
from paper_2609_13544_gb300 import workloads as W

DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16, "f8e4m3": torch.float8_e4m3fn,
          "f8e5m2": torch.float8_e5m2, "f64": torch.float64}
SIZE = {"f32": 4, "f16": 2, "bf16": 2, "f8e4m3": 1, "f8e5m2": 1, "f64": 8}
# relative spacing of the type at 1, in which the noise of a replayed tensor is stated
EPS = {"f32": 2.0 ** -23, "f16": 2.0 ** -10, "bf16": 2.0 ** -7, "f8e4m3": 2.0 ** -3, "f8e5m2": 2.0 ** -2,
       "f64": 2.0 ** -52}
# the tolerance that a program of that precision passes
RTOL = {"f32": 1e-5, "f16": 1e-3, "bf16": 2.0 ** -7, "f8e4m3": 0.125, "f8e5m2": 0.125, "f64": 1e-7}

# the tolerance grid of an isclose acceptance map (8 x 8 cells)
GRID_RTOLS = [10.0 ** -k for k in range(8, 0, -1)]
GRID_ATOLS = [0.0] + [10.0 ** -k for k in range(8, 1, -1)]


def listed():
    return [
        # a bias or normalisation vector: the smallest recorded tensors, where a call is all latency
        {"name": "compare_f32_vector", "op": "compare", "dtype": "f32", "n": 10007, "kind": "noise", "sigma": 1e-6,
         "scale": 1.0, "flips": 4, "shift": 0},
        # one float32 layer weight after a few bit flips
        {"name": "compare_f32_1m", "op": "compare", "dtype": "f32", "n": 1048576, "kind": "noise", "sigma": 1e-6,
         "scale": 1.0, "flips": 16, "shift": 0},
        # a bf16 activation [8, 2048, 4096], rounded to nearest against truncated: half of the pairs differ by one step
        {"name": "compare_bf16_activation", "op": "compare", "dtype": "bf16", "n": 67108864, "kind": "rtz",
         "sigma": 0.0, "scale": 2.0, "flips": 0, "shift": 0},
        # every parameter of a convolutional network in one call: 161 tensors from 64 to 2.4 million values
        {"name": "segmented_f32_resnet50", "op": "segmented", "dtype": "f32", "model": "resnet50"},
        # every parameter of a language model's half-precision checkpoint in one call: 292 tensors
        {"name": "segmented_f16_gpt2", "op": "segmented", "dtype": "f16", "model": "gpt2_medium"},
        # one late step of a playback sweep over a large bf16 tensor: about one pair in eleven differs
        {"name": "compare_bf16_playback", "op": "compare", "dtype": "bf16", "n": 268435456, "kind": "noise",
         "sigma": 1e-4 * math.sqrt(63.0), "scale": 1.0, "flips": 0, "shift": 0},
        # the mean of the top 10 % errors of the same activation
        {"name": "topk_bf16_activation", "op": "topk", "dtype": "bf16", "n": 67108864, "kind": "rtz", "sigma": 0.0,
         "scale": 2.0, "flips": 0, "shift": 0},
        # means and variances of every tensor of the checkpoint
        {"name": "context_f16_gpt2", "op": "context", "dtype": "f16", "model": "gpt2_medium", "n": 0, "shift": 0},
        # the isclose acceptance map of a float32 output against its half-precision version; an odd size
        {"name": "isclose_f32_cast", "op": "isclose", "dtype": "f32", "n": 16777259, "kind": "cast_f16",
         "sigma": 0.0, "scale": 1.0, "flips": 0, "shift": 0},
        # injection and assessment of Gaussian noise in one call over the activation
        {"name": "inject_bf16_activation", "op": "inject_compare", "dtype": "bf16", "n": 67108864,
         "model": "rel_gauss", "x": 1e-3, "scale": 2.0, "shift": 0},
        # an 8-bit activation [4, 2048, 4096] against a noisy replay
        {"name": "compare_fp8_activation", "op": "compare", "dtype": "f8e4m3", "n": 33554432, "kind": "noise",
         "sigma": 0.0625, "scale": 2.0, "flips": 0, "shift": 0},
        # a binary64 output against the float32 one, widened: the second half of a precision study; an odd size
        {"name": "compare_f64_cast", "op": "compare", "dtype": "f64", "n": 12345679, "kind": "cast_f32",
         "sigma": 0.0, "scale": 1.0, "flips": 0, "shift": 0},
    ]


def _log_size(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return n | 1 if rng.random() < 0.5 else n


def draw(rng):
    """Another case: any operation, its types, sizes over the whole range (odd ones among them), noise from a
    fraction of the type's spacing to some tens of it, a few flipped bits, tensors inside a packed buffer."""
    op = rng.choice(["compare", "compare", "compare", "segmented", "topk", "context", "isclose", "inject_compare"])
    shift = rng.choice([0, 0, 0, 1, 3])  # elements before the tensor in its buffer
    if op == "segmented":
        dt = rng.choice(["f32", "f16", "bf16"])
        return {"op": op, "dtype": dt, "model": "list", "nseg": rng.randint(3, 400),
                "n": _log_size(rng, 20000, 40000000), "sigma": EPS[dt] * 10.0 ** rng.uniform(-1.0, 1.0),
                "scale": 10.0 ** rng.uniform(-2.0, 1.0)}
    if op == "context":
        dt = rng.choice(["f32", "f16", "bf16"])
        return {"op": op, "dtype": dt, "model": "one", "n": _log_size(rng, 2000, 100000000),
                "scale": 10.0 ** rng.uniform(-2.0, 1.0), "shift": shift}
    if op == "inject_compare":
        dt = rng.choice(["f32", "f16", "bf16"])
        model = rng.choice(["rel_gauss", "add_gauss", "bias", "nan_inf", "signflip"])
        x = 10.0 ** rng.uniform(-6.0, -3.0) if model in ("nan_inf", "signflip") else 10.0 ** rng.uniform(-4.0, -2.0)
        return {"op": op, "dtype": dt, "n": _log_size(rng, 2000, 60000000), "model": model, "x": x,
                "scale": 10.0 ** rng.uniform(-1.0, 1.0), "shift": shift}
    dts = {"compare": ["f32", "f16", "bf16", "bf16", "f8e4m3", "f8e5m2", "f64"], "topk": ["f32", "f16", "bf16"],
           "isclose": ["f32", "f16", "bf16"]}[op]
    dt = rng.choice(dts)
    most = {"f64": 10000000, "f32": 50000000}.get(dt, 100000000) if op != "isclose" else 16000000
    case = {"op": op, "dtype": dt, "n": _log_size(rng, 2000, min(most, 33000000) if SIZE[dt] == 1 else most),
            "kind": "noise", "sigma": EPS[dt] * 10.0 ** rng.uniform(-1.0, 1.0),
            "scale": 10.0 ** rng.uniform(-1.0, 1.0), "flips": rng.choice([0, 0, 16]), "shift": shift}
    if dt == "f64" or (dt == "f32" and rng.random() < 0.4):
        case.update(kind="cast_f32" if dt == "f64" else rng.choice(["cast_f16", "cast_bf16"]), sigma=0.0, flips=0)
    elif dt == "bf16" and rng.random() < 0.3:
        case.update(kind="rtz", sigma=0.0)
    elif rng.random() < 0.2:
        case.update(kind="same", sigma=0.0, flips=16)  # only the flipped bits differ
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _pair(case, seed):
    """Golden and candidate of one tensor, each `shift` elements into its own buffer."""
    n, dt, kind, shift = case["n"], DTYPES[case["dtype"]], case["kind"], case["shift"]
    gen = _gen(seed)
    wide = torch.float64 if case["dtype"] == "f64" else torch.float32
    g = torch.empty(n + shift, dtype=dt, device="cuda")[shift:]
    c = torch.empty(n + shift, dtype=dt, device="cuda")[shift:]
    x = torch.randn(n, generator=gen, device="cuda", dtype=wide) * case["scale"]
    g.copy_(x)
    if kind == "noise":
        c.copy_(g.to(wide) * (1.0 + case["sigma"] * torch.randn(n, generator=gen, device="cuda", dtype=wide)))
    elif kind == "rtz":
        c.copy_(W.truncate_to_bf16(x))
    elif kind == "same":
        c.copy_(g)
    else:
        c.copy_(x.to({"cast_f16": torch.float16, "cast_bf16": torch.bfloat16, "cast_f32": torch.float32}[kind]))
    if case["flips"]:
        k, bits = case["flips"], 8 * SIZE[case["dtype"]]
        pos = torch.randint(0, n, (k,), generator=gen, device="cuda").tolist()
        bit = torch.randint(0, bits, (k,), generator=gen, device="cuda").tolist()
        iv = c.view({8: torch.uint8, 16: torch.int16, 32: torch.int32, 64: torch.int64}[bits])
        for p, b in zip(pos, bit):
            m = (1 << b) - (1 << bits if b == bits - 1 and bits > 8 else 0)
            iv[p] = iv[p] ^ m
    return g, c


def _offsets(case, seed):
    """A ragged list of tensors: many small ones, a few large ones, some empty."""
    rng = np.random.default_rng(seed)
    w = np.exp(rng.normal(0.0, 2.5, case["nseg"]))
    w[rng.random(case["nseg"]) < 0.02] = 0.0
    off = np.concatenate([[0.0], np.cumsum(w)])
    off = np.floor(off / max(off[-1], 1e-300) * case["n"]).astype(np.int64)
    off[-1] = case["n"]
    return off


def _inputs(case, seed):
    """(golden, candidate or None, offsets)."""
    op = case["op"]
    if op in ("segmented", "context") and case["model"] in ("resnet50", "gpt2_medium"):
        w = (W.c3_resnet50 if case["model"] == "resnet50" else W.c4_gpt2_medium)(seed=seed, device="cuda")
        return w.golden, w.candidate if op == "segmented" else None, w.offsets
    if op == "segmented":
        g, c = _pair({**case, "kind": "noise", "flips": 0, "shift": 0}, seed)
        return g, c, _offsets(case, seed)
    if op in ("context", "inject_compare"):
        x = torch.empty(case["n"] + case["shift"], dtype=DTYPES[case["dtype"]], device="cuda")[case["shift"]:]
        x.copy_(torch.randn(case["n"], generator=_gen(seed), device="cuda") * case["scale"])
        return x, None, np.array([0, case["n"]], np.int64)
    g, c = _pair(case, seed)
    return g, c, np.array([0, case["n"]], np.int64)


def _stats_views(raw):
    """The fields of peat_stats_t records as tensors on the same memory."""
    i, f = raw.view(torch.int64).view(-1, 20), raw.view(torch.float64).view(-1, 20)
    return {"counts": i[:, 0:7], "max_abs": f[:, 7], "argmax_abs": i[:, 8], "max_rel": f[:, 9],
            "argmax_rel": i[:, 10], "max_ulp": i[:, 11], "argmax_ulp": i[:, 12], "sums": f[:, 13:16],
            "tolerance": f[:, 16:18], "mean_var": f[:, 18:20]}


def prepare(case, seed):
    """The tensors, a handle, and the output buffers that the program reuses."""
    op = case["op"]
    g, c, off = _inputs(case, seed)
    nseg = len(off) - 1
    st = {"case": case, "g": g, "c": c, "off": off, "seed": seed, "h": peat.Handle(0)}

    def zeros(k):
        return torch.zeros(k, dtype=torch.uint8, device="cuda")

    if op in ("compare", "segmented", "inject_compare"):
        st["stats"], st["hist"] = zeros(peat.STATS_BYTES * nseg), zeros(8 * peat.HIST_BINS * nseg).view(torch.int64)
        st["out"] = {**_stats_views(st["stats"]), "hist": st["hist"].view(nseg, peat.HIST_BINS)}
        st["rtol"] = RTOL[case["dtype"]]
        if op == "inject_compare":
            st["models"] = [peat.inject_model(case["model"], x=case["x"])]
    elif op == "topk":
        st["stats"] = zeros(peat.TOPK_BYTES)
        i, f = st["stats"].view(torch.int64), st["stats"].view(torch.float64)
        st["out"] = {"counts": i[0:2], "threshold": f[2:3], "sum_mean": f[3:5]}
    elif op == "context":
        st["stats"] = zeros(peat.TSTATS_BYTES * nseg)
        i, f = st["stats"].view(torch.int64).view(-1, 10), st["stats"].view(torch.float64).view(-1, 10)
        st["out"] = {"counts": i[:, 0:4], "sums": f[:, 4:6], "mean_var": f[:, 6:8], "min_max": f[:, 8:10]}
    else:
        st["stats"] = zeros(8 * len(GRID_RTOLS) * len(GRID_ATOLS)).view(torch.int64)
        st["out"] = {"counts": st["stats"]}
    return st


def run(st):
    """One call; its outputs are the program's own buffers."""
    op, h = st["case"]["op"], st["h"]
    if op == "compare":
        peat.peat_compare_raw(h, st["g"], st["c"], st["rtol"], 0.0, st["stats"], st["hist"])
    elif op == "segmented":
        peat.peat_compare_segmented_raw(h, st["g"], st["c"], st["off"], st["rtol"], 0.0, st["stats"], st["hist"])
    elif op == "inject_compare":
        peat.peat_inject_compare_raw(h, st["g"], st["models"], st["seed"], st["rtol"], 0.0, st["stats"], st["hist"])
    elif op == "topk":
        peat.peat_topk_mean_raw(h, st["g"], st["c"], 1, 10, st["stats"])
    elif op == "context":
        peat.peat_tensor_stats_raw(h, st["g"], st["off"], st["stats"])
    else:
        peat.peat_isclose_grid_raw(h, st["g"], st["c"], GRID_RTOLS, GRID_ATOLS, st["stats"])
    return st["out"]


def _elements(case):
    if case.get("model") == "resnet50":
        return int(W.offsets_of(W.resnet50_param_shapes())[-1]), 161
    if case.get("model") == "gpt2_medium":
        return int(W.offsets_of(W.gpt2_medium_param_shapes())[-1]), 292
    return case["n"], case.get("nseg", 1)


def work(case):
    """Each input once, each output once; the operations of the definitions, a few per element."""
    n, nseg = _elements(case)
    op = case["op"]
    out = {"topk": 48, "context": 80 * nseg, "isclose": 512}.get(op, (160 + 1024) * nseg)
    reads = 1 if op in ("context", "inject_compare") else 2
    # compare: difference, ratio, tolerance, three sums, three maxima, two bins
    flops = {"topk": 3, "context": 3, "isclose": 2 + 2 * len(GRID_RTOLS) * len(GRID_ATOLS), "inject_compare": 40}
    return {"bytes": reads * n * SIZE[case["dtype"]] + out, "flops": n * flops.get(op, 12)}


def tolerance(case):
    """Integers, and exact real numbers rounded once: nothing may differ."""
    return "exact"


# ---------------------------------------------------------------------------
# the definitions in binary64, plain torch
# ---------------------------------------------------------------------------
def _keys(x):
    """Ordered-integer keys: the pattern without its sign, negated below zero."""
    iv = x.view({1: torch.int8, 2: torch.int16, 4: torch.int32, 8: torch.int64}[x.element_size()]).to(torch.int64)
    mag = iv & ((1 << (8 * x.element_size() - 1)) - 1)
    return torch.where(iv < 0, -mag, mag)


def _first_max(v, ok):
    """The largest of v where ok, and its lowest index (0.0 and the first ok index when all are zero)."""
    if not bool(ok.any()):
        return 0.0, -1
    v = torch.where(ok, v, torch.full_like(v, -1))
    m = v.max()
    return m.item(), int((v == m).nonzero()[0])


def _signature(gt, ct, rtol):
    n = gt.numel()
    if n == 0:
        return [0] * 7, (0.0, -1), (0.0, -1), (0, -1), [0.0] * 3, [0.0] * 2, torch.zeros(128, dtype=torch.int64)
    g, c, u = gt.double(), ct.double(), (_keys(ct) - _keys(gt)).abs()
    gn, cn = torch.isnan(g), torch.isnan(c)
    fin = torch.isfinite(g) & torch.isfinite(c)
    d = torch.where(fin, c - g, torch.zeros_like(g))
    a, ag = d.abs(), torch.where(fin, g.abs(), torch.ones_like(g))
    asym = ~fin & ~((gn & cn) | (~gn & ~cn & (g == c)))
    exact = ~asym & (a == 0)
    within = fin & ~exact & (a <= rtol * ag)
    flip = fin & ~exact & ~within & (g != 0) & (c != 0) & (torch.signbit(g) != torch.signbit(c))
    nf = int(fin.sum())
    counts = [int(v.sum()) for v in (exact, within, fin & ~exact & ~within & ~flip, asym, flip)]
    ratio = torch.where(exact, torch.zeros_like(a), a / ag)
    k = torch.frexp(torch.where(ratio > 0, ratio, torch.ones_like(ratio)))[1] - 1 + 48
    k = torch.where(exact, torch.zeros_like(k), k.clamp(1, 62))
    k = torch.where(asym | (fin & (ag == 0) & (a > 0)), torch.full_like(k, 63), k)
    ub = torch.where(gn | cn, torch.where(gn & cn, torch.zeros_like(u), torch.full_like(u, 63)), u.clamp(max=63))
    hist = torch.cat([torch.bincount(k.long(), minlength=64), torch.bincount(ub, minlength=64)]).cpu()
    s1, s2, s = a.sum().item(), (a * a).sum().item(), d.sum().item()
    mean = s1 / nf if nf else 0.0
    var = ((torch.where(fin, a - mean, torch.zeros_like(a)) ** 2).sum().item() / nf) if nf else 0.0
    return ([n] + counts + [nf], _first_max(a, fin), _first_max(ratio, fin), _first_max(u, ~(gn | cn)), [s1, s2, s],
            [mean, var], hist)


def exact(case, seed):
    """What run returns, from binary64 arithmetic; None for the injection, whose candidate exists only as the
    generator's own bit pattern."""
    op = case["op"]
    if op == "inject_compare":
        return None
    gt, ct, off = _inputs(case, seed)
    if op in ("compare", "segmented"):
        rtol = float(np.float32(RTOL[case["dtype"]]))
        rs = [_signature(gt[a:b], ct[a:b], rtol) for a, b in zip(off[:-1].tolist(), off[1:].tolist())]
        i64, f64 = torch.int64, torch.float64
        return {"counts": torch.tensor([r[0] for r in rs], dtype=i64),
                "max_abs": torch.tensor([r[1][0] for r in rs], dtype=f64),
                "argmax_abs": torch.tensor([r[1][1] for r in rs], dtype=i64),
                "max_rel": torch.tensor([r[2][0] for r in rs], dtype=f64),
                "argmax_rel": torch.tensor([r[2][1] for r in rs], dtype=i64),
                "max_ulp": torch.tensor([int(r[3][0]) for r in rs], dtype=i64),
                "argmax_ulp": torch.tensor([r[3][1] for r in rs], dtype=i64),
                "sums": torch.tensor([r[4] for r in rs], dtype=f64),
                "tolerance": torch.tensor([[rtol, 0.0]] * len(rs), dtype=f64),
                "mean_var": torch.tensor([r[5] for r in rs], dtype=f64), "hist": torch.stack([r[6] for r in rs])}
    if op == "topk":
        g, c = gt.double(), ct.double()
        fin = torch.isfinite(g) & torch.isfinite(c)
        a = (c - g).abs()[fin]
        nf = a.numel()
        k = -(-nf // 10)
        top = torch.sort(a, descending=True).values[:k]
        s = top.sum().item()
        return {"counts": torch.tensor([nf, k]), "threshold": torch.tensor([top[-1].item() if k else 0.0],
                                                                         dtype=torch.float64),
                "sum_mean": torch.tensor([s, s / k if k else 0.0], dtype=torch.float64)}
    if op == "context":
        rows = []
        for a, b in zip(off[:-1].tolist(), off[1:].tolist()):
            x = gt[a:b].double()
            f = x[torch.isfinite(x)]
            nf = f.numel()
            mean = f.sum().item() / nf if nf else 0.0
            rows.append(([b - a, nf, int(torch.isnan(x).sum()), int(torch.isinf(x).sum())],
                         [f.sum().item(), (f * f).sum().item()],
                         [mean, ((f - mean) ** 2).sum().item() / nf if nf else 0.0],
                         [f.min().item(), f.max().item()] if nf else [0.0, 0.0]))
        return {"counts": torch.tensor([r[0] for r in rows]),
                "sums": torch.tensor([r[1] for r in rows], dtype=torch.float64),
                "mean_var": torch.tensor([r[2] for r in rows], dtype=torch.float64),
                "min_max": torch.tensor([r[3] for r in rows], dtype=torch.float64)}
    g, c = gt.double(), ct.double()
    a, ag = (c - g).abs(), g.abs()
    same = (g == c) | (torch.isnan(g) & torch.isnan(c))
    fin = torch.isfinite(g) & torch.isfinite(c)
    cells = [int((same | (fin & (a <= float(np.float32(at)) + float(np.float32(rt)) * ag))).sum())
             for rt in GRID_RTOLS for at in GRID_ATOLS]
    return {"counts": torch.tensor(cells)}
