"""What a user of this library has it do: whole layer solves, and the quantize step on a ready state.

A case is a dict of plain values:

    kind    "solve"     reset, accumulate every token batch, factor, build_P, quantize on one handle
            "host"      the same through the host entry points (pinned host activations and weights in,
                        codes and grids back in host memory)
            "quantize"  quantize alone: several weight matrices share one calibrated state
            "static"    gptaq_quantize_static: U and P as plain inputs, no handle and no workspace
    m, n    output channels and input channels of the layer;  tokens, batches: tokens per accumulate call
            and number of calls (the calibration that `prepare` runs for "quantize" and "static")
    act     activation recipe: "gauss", "student" (heavy tails and outlier channels), "gated" (most entries
            near zero, lognormal rest) or "layernorm";  noise: relative difference of the two streams
    bits, group, sym, block, damp, alpha       arguments of the entry points
    bf16    bfloat16 weights (else float32);  act_order, static_groups, clip   options of the handle

`run` returns the quantized layer and, of a solve, the factor and the correction matrix: codes, scales, zero
points and, from 4 bits on, the dequantized float32 weights.  (At 2 and 3 bits these are left out: they are
scale * (code - zero) of the other three, and one code that falls to the other side of a rounding tie moves
such a weight by more than the weights' own root mean square.)
"""
import math

import torch

import paper_2504_02692_b200 as g

_BASE = dict(kind="solve", act="student", noise=0.05, bits=4, group=128, sym=False, block=128, damp=0.01,
             alpha=0.25, bf16=False, act_order=False, static_groups=False, clip=0)


def _case(name=None, **kw):
    c = dict(_BASE, **kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one small linear layer, per-channel grids: every call is a handful of short launches
        _case("small_linear", m=128, n=128, tokens=512, batches=1, act="gauss", group=0, block=32),
        # a narrow layer with groups, calibrated on a few sequences
        _case("narrow_groups", m=512, n=1024, tokens=4096, batches=4),
        # first layer of a vision transformer's MLP: 16 images of 257 tokens a batch, symmetric 3-bit per-channel
        # grids and the stronger damping that goes with them
        _case("vision_mlp", m=4096, n=1024, tokens=4112, batches=8, act="layernorm", noise=0.08, bits=3, group=0,
              sym=True, damp=0.1),
        # attention projection of a language model on 128 sequences of 2048 tokens: the ordinary layer
        _case("attention_projection", m=4096, n=4096, tokens=8192, batches=32),
        # down projection of a gated MLP: the largest layer, 3-bit groups
        _case("mlp_down", m=4096, n=14336, tokens=8192, batches=32, act="gated", bits=3),
        # odd sizes in every direction, little calibration data (both fp16 parts of X are used)
        _case("ragged_few_tokens", m=1003, n=1416, tokens=3001, batches=2, group=64, block=64),
        # a width that is a multiple of 4 only, one short batch, 8-bit per-channel grids
        _case("ragged_width", m=777, n=2052, tokens=2777, batches=1, bits=8, group=0, sym=True),
        # columns in the order of the Hessian's diagonal, grids that survive it, bfloat16 weights
        _case("act_order_static_groups", m=4096, n=4096, tokens=8192, batches=4, bf16=True, act_order=True,
              static_groups=True),
        # second and later matrices on one state: a wide bfloat16 up projection
        _case("shared_state_wide", kind="quantize", m=16384, n=4096, tokens=8192, batches=2, bf16=True),
        # ... and one with searched clipping ranges
        _case("shared_state_clip", kind="quantize", m=4096, n=4096, tokens=8192, batches=2, bits=3, clip=80),
        # a caller that may not allocate
        _case("no_workspace", kind="static", m=1024, n=1024, tokens=4096, batches=1),
        # activations and weights in host memory
        _case("from_host", kind="host", m=1024, n=1024, tokens=4112, batches=2, act="layernorm"),
    ]


def _spread(rng, lo, hi, multiple):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / multiple)) * multiple))


def draw(rng):
    """One more case: sizes spread over their logarithm, widths aligned and odd, every option in use."""
    kind = rng.choice(["solve"] * 6 + ["quantize"] * 2 + ["static", "host"])
    multiple = rng.choice([128, 128, 64, 8, 4, 1])
    top = {"solve": 14336, "quantize": 8192, "static": 2048, "host": 2048}[kind]
    # a width that is not a multiple of 8 has the plain float32 products for its large ones
    n = _spread(rng, 96, top if multiple >= 8 else 2600, multiple)
    m = _spread(rng, 64, {"quantize": 16384, "static": 2048}.get(kind, 4096), rng.choice([64, 1]))
    if kind == "static":
        m = min(m, g.GPTAQ_STATIC_SCRATCH_FLOATS // 256)
    # enough tokens for a full-rank H, at most 128 sequences of 2048
    tokens = _spread(rng, max(512, min(n, 8192)), 8192, rng.choice([64, 1]))
    need = max(1, -(-2 * n // tokens))
    batches = rng.randint(need, max(need, min(32, 2 ** rng.randint(0, 5)))) if kind == "solve" else need
    block = rng.choice([128, 128, 128, 64, 32])
    group = rng.choice([gr for gr in (0, 32, 64, 128, 128) if gr <= block])
    act_order = kind == "solve" and rng.random() < 0.2
    act = rng.choice(["gauss", "student", "gated", "layernorm"])
    if act_order:
        act = "student"     # channels that differ in scale: what the option is for, and few ties in the order
        n = min(n, 4096)
    return _case(kind=kind, m=m, n=n, tokens=tokens, batches=batches, act=act,
                 noise=rng.choice([0.05, 0.08]), bits=rng.choice([3, 4, 4, 8]), group=group, sym=rng.random() < 0.3, block=block,
                 damp=rng.choice([0.01, 0.01, 0.1]), bf16=kind != "host" and rng.random() < 0.4, act_order=act_order,
                 static_groups=act_order and group > 0, clip=80 if kind == "quantize" and rng.random() < 0.3 else 0)


def _activations(c, gen, device):
    """One token batch of the two streams: (X of the quantized model, X of the full-precision model)."""
    shape = (c["tokens"], c["n"])

    def randn():
        return torch.randn(shape, generator=gen, device=device)

    z = randn()
    if c["act"] == "student":
        chi = randn().square_()
        for _ in range(3):
            chi += randn().square_()
        z /= chi.mul_(0.25).sqrt_()
    elif c["act"] == "gated":
        u = torch.rand(shape, generator=gen, device=device)
        big = torch.exp(z - 1.0)
        big = torch.where(u > 0.8, big, -big)
        z = torch.where(u < 0.6, 1e-3 * z, big)
    elif c["act"] == "layernorm":
        z = (z - z.mean(dim=1, keepdim=True)) / z.std(dim=1, keepdim=True)
    if c["act"] != "gated":
        # one channel in a hundred carries outliers
        ch = torch.randperm(c["n"], generator=gen, device=device)[: max(1, c["n"] // 100)]
        z[:, ch] *= 30.0
    return z + randn() * (c["noise"] * z.abs()), z


def _groups(c):
    return 1 if c["group"] <= 0 else -(-c["n"] // c["group"])


def prepare(case, seed):
    c = dict(case)
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    m, n, G = c["m"], c["n"], _groups(c)
    W = torch.randn((m, n), generator=gen, device=dev) * 0.02
    if c["bf16"]:
        W = W.to(torch.bfloat16)
    batches = [_activations(c, gen, dev) for _ in range(c["batches"])]
    st = g.LayerState(n, m, c["tokens"], c["block"], dev, total_tokens=c["tokens"] * c["batches"])
    if c["act_order"]:
        g.gptaq_set_act_order(st.handle, True)
    if c["static_groups"]:
        g.gptaq_set_static_groups(st.handle, True)
    if c["clip"]:
        g.gptaq_set_clip_search(st.handle, c["clip"], 0.2)
    host = c["kind"] == "host"
    kw = dict(pin_memory=True) if host else dict(device=dev)
    s = {"case": c, "st": st, "h": st.handle,
         "codes": torch.empty((m, n), dtype=torch.uint8, **kw), "scales": torch.empty((m, G), **kw),
         "zeros": torch.empty((m, G), **kw), "Wq": torch.empty((m, n), **kw)}
    if host:
        s["batches"] = [(x.cpu().pin_memory(), f.cpu().pin_memory()) for x, f in batches]
        s["W"] = W.cpu().pin_memory()
        need = max(2 * c["tokens"] * n * 4, g.gptaq_quantize_stage_bytes(m, n, c["group"]))
        s["stage"] = torch.empty(need, dtype=torch.uint8, device=dev)
    else:
        s["batches"], s["W"] = batches, W
    if c["kind"] in ("quantize", "static"):
        for x, f in s.pop("batches"):
            g.gptaq_accumulate(st.handle, x, f)
        g.gptaq_factor(st.handle, c["damp"])
        g.gptaq_build_P(st.handle, c["alpha"])
        if c["kind"] == "static":
            s["U"], s["P"] = st.H().clone(), st.D().clone()
            s["status"] = torch.zeros(2, dtype=torch.int64, device=dev)
    return s


def run(s):
    c, h = s["case"], s["h"]
    how = (c["bits"], c["group"], c["sym"], c["block"])
    out = [s["codes"], s["scales"], s["zeros"]] + ([s["Wq"]] if c["bits"] >= 4 else [])
    if c["kind"] == "quantize":
        g.gptaq_quantize(h, s["W"], *how, s["codes"], s["scales"], s["zeros"], s["Wq"])
        return out
    if c["kind"] == "static":
        g.gptaq_quantize_static(s["U"], s["P"], s["W"], *how, s["codes"], s["scales"], s["zeros"], s["Wq"], s["status"])
        return out + [s["status"]]
    g.gptaq_reset(h)
    for x, f in s["batches"]:
        if c["kind"] == "host":
            g.gptaq_accumulate_host(h, x, f, s["stage"])
        else:
            g.gptaq_accumulate(h, x, f)
    g.gptaq_factor(h, c["damp"])
    g.gptaq_build_P(h, c["alpha"])
    if c["kind"] == "host":
        g.gptaq_quantize_host(h, s["W"], *how, s["codes"], s["scales"], s["zeros"], s["stage"], s["Wq"])
    else:
        g.gptaq_quantize(h, s["W"], *how, s["codes"], s["scales"], s["zeros"], s["Wq"])
    if c["act_order"]:
        return out      # U and P are in sorted order, and the order of two inputs with nearly the same diagonal entry is a tie
    return out + [s["st"].H(), s["st"].D()]


def work(case):
    c = case
    m, n, G, t = float(c["m"]), float(c["n"]), float(_groups(c)), float(c["tokens"] * c["batches"])
    # U and P (upper triangles) once more to read; weights in, codes, grids and dequantized weights out
    by = 4.0 * n * n + m * n * ((2 if c["bf16"] else 4) + 1 + 4) + 8.0 * m * G
    fl = 2.0 * m * n * n                                 # both terms of the update, columns to the right only
    if c["kind"] in ("solve", "host"):
        # both streams in, U and P out; H (a triangle) and what P needs of dXX^T, the factor with its
        # inverse, the two triangular products of P
        by += 8.0 * n * t
        fl += (3.0 if c["act_order"] else 2.0) * n * n * t + 4.0 * n ** 3 / 3.0
    return {"bytes": by, "flops": fl}


def tolerance(case):
    # About four times what the same path shows with its sums in another order (the tokens of every batch permuted,
    # all listed cases and ten drawn ones): U, P and per-channel grids differ by at most 2e-6 (2-norm) and 6e-5 (one
    # value).  Codes differ by ties of the rounding and by what follows a flipped code in its row (up to 2e-4 of the
    # codes, 3e-4 at 8 bits); each carries its dequantized weight (5e-3, up to half the weights' rms) and the grids of the row's
    # later groups (3e-3, a zero point by one) with it.
    if case["bits"] < 4 and case["group"] <= 0:
        return {"rel": 1e-5, "max": 3e-4, "differ": 2e-3}
    # (act_order: two inputs that swap places take the codes of a few columns with them)
    return {"rel": 0.02, "max": 0.99, "differ": 4e-3 if case["bits"] == 8 or case["act_order"] else 2e-3}
