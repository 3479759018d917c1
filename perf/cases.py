"""The work whose speed counts: what a user of this package has it do, through ``ArmorContext``.

Three kinds of pass, as in a run over the layers of a model:

  gram      H += X^T X for one chunk of calibration activations
  optimise  one layer: initialisation, a call of ``iters`` BCD iterations, the final proxy loss (with ``tokens`` > 0
            the Gram of that many activations comes first, as for a layer small enough to be done in one go)
  forward   y = A S B x with a finished layer: the packed bf16 layer (what is deployed), the fp32 form (what a check
            of a layer uses) or bf16 activations with fp32 wrappers (dense or packed core)

Sizes are those of ``paper_2510_05528_b200.inputs.CONFIGS`` or lie between them."""
from __future__ import annotations

import math

import torch

from paper_2510_05528_b200 import binding as Bd

DEV = "cuda:0"


# ------------------------------------------------------------------------------------------------ the cases
def _gram(d_in, tokens, dtype, precision="fp16x3", name=None):
    c = {"kind": "gram", "d_in": d_in, "tokens": tokens, "dtype": dtype, "precision": precision}
    return dict(c, name=name) if name else c


def _optimise(d_out, d_in, d_block, iters, weighting, update, *, tokens=0, n_keep=2, m_group=4, normalize=False,
              mask_groups=1, name=None):
    c = {"kind": "optimise", "d_out": d_out, "d_in": d_in, "d_block": d_block, "iters": iters, "weighting": weighting,
         "update": update, "tokens": tokens, "n_keep": n_keep, "m_group": m_group, "normalize": normalize,
         "mask_groups": mask_groups}
    return dict(c, name=name) if name else c


def _forward(d_out, d_in, d_block, tokens, form, name=None):
    c = {"kind": "forward", "d_out": d_out, "d_in": d_in, "d_block": d_block, "tokens": tokens, "form": form}
    return dict(c, name=name) if name else c


def listed():
    # A layer takes 50 iterations (the paper's Adam schedule thousands), and every iteration costs the same.  The calls
    # here are shorter because the method chooses: with enough iterations times blocks some group or mask is decided
    # within rounding, and the outputs of two correct implementations then part (see tolerance).
    return [
        # the smallest configuration whole, Gram to final loss: launches and latency count
        _optimise(256, 256, 32, 20, "full", "exact", tokens=4096, name="tiny_layer"),
        # a square attention projection with the full Gram: what the headline benchmark times
        _optimise(4096, 4096, 128, 8, "full", "exact", name="attn_full"),
        # a key/value projection of a grouped-query layer: few output rows, many small launches; normalised weights
        _optimise(1024, 5120, 128, 10, "full", "exact", normalize=True, name="kv_full"),
        # an up projection with the paper's diagonal loss and exact solves; normalised weights
        _optimise(14336, 4096, 128, 4, "diag", "exact", normalize=True, name="up_diag"),
        # the paper's own schedule: diagonal loss, joint Adam steps, one group of every block per iteration
        _optimise(4096, 4096, 128, 10, "diag", "adam", name="attn_diag_adam"),
        # the largest layer: blocks of 256, groups of eight
        _optimise(28672, 8192, 256, 3, "full", "exact", n_keep=4, m_group=8, name="large_full_4of8"),
        # calibration: 128 sequences of 2,048 tokens in one call; and a ragged bf16 chunk
        _gram(4096, 262144, "f32", name="gram_f32"),
        _gram(5120, 10007, "bf16", name="gram_bf16_ragged"),
        # the finished layer in a decoder: one token, an odd batch of streams, a prompt, and the fp32 check
        _forward(4096, 4096, 128, 1, "layer", name="decode_1"),
        _forward(14336, 4096, 128, 37, "layer", name="decode_batch_37"),
        _forward(28672, 8192, 256, 4096, "layer", name="prefill_4096"),
        _forward(4096, 4096, 128, 8195, "f32", name="forward_f32"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _multiple(rng, lo, hi, m):
    return max(1, round(_log(rng, lo, hi) / m)) * m


def _draw_once(rng):
    kind = rng.choice(["gram", "optimise", "optimise", "optimise", "forward", "forward"])
    if kind == "gram":
        d_in = _multiple(rng, 256, 14336, 128)
        tokens = int(_log(rng, 100, 131072))
        return _gram(d_in, tokens | 1 if rng.random() < 0.5 else tokens, rng.choice(["f32", "bf16"]),
                     rng.choice(["fp16x3", "fp16x3", "tf32"]))
    d_block = rng.choice([128, 128, 256])
    if kind == "forward":
        form = rng.choice(["layer", "layer", "layer", "f32", "bf16", "bf16_packed"])
        return _forward(_multiple(rng, 512, 28672, d_block), _multiple(rng, 512, 8192, d_block), d_block,
                        int(_log(rng, 1, 8192)), form)
    if rng.random() < 0.25:
        d_block = rng.choice([32, 64])
        d_out, d_in = _multiple(rng, 256, 1024, 128), _multiple(rng, 256, 1024, 128)
    else:
        d_out, d_in = _multiple(rng, 512, 14336, d_block), _multiple(rng, 512, 8192, d_block)
    weighting, update = rng.choice([("full", "exact"), ("full", "exact"), ("diag", "exact"), ("diag", "adam")])
    n_keep, m_group = rng.choice([(2, 4), (2, 4), (2, 4), (4, 8), (6, 8)])
    return _optimise(d_out, d_in, d_block, rng.randint(2, 20), weighting, update,
                     tokens=rng.choice([0, 0, int(_log(rng, 512, 8192))]), n_keep=n_keep, m_group=m_group,
                     normalize=rng.random() < 0.5, mask_groups=rng.choice([1, 1, 1, 4]))


def _cost(case):
    w = work(case)
    return max(w["bytes"] / 6.5e12, w["flops"] / 5e14)


def _decisions(case):
    """Groups drawn and masks solved in one pass."""
    blocks = (case["d_out"] // case["d_block"]) * (case["d_in"] // case["d_block"])
    return blocks * case["iters"] * case["mask_groups"]


def draw(rng):
    """Another case of the same ranges; layers with no more decisions than the listed ones make."""
    cost = max(_cost(c) for c in listed())
    most = max(_decisions(c) for c in listed() if c["kind"] == "optimise")
    while True:
        case = _draw_once(rng)
        if _cost(case) <= cost and (case["kind"] != "optimise" or _decisions(case) <= most):
            return case


# ------------------------------------------------------------------------------------------------ inputs
def _scales(gen, d_in):
    """Per-channel standard deviations: log-normal, one channel in a thousand an outlier (x 50)."""
    s = torch.exp(torch.randn(d_in, generator=gen, device=DEV))
    s[torch.randperm(d_in, generator=gen, device=DEV)[: max(1, round(0.001 * d_in))]] *= 50.0
    return s


def _activations(gen, scales, tokens, dtype):
    x = torch.randn(tokens, scales.numel(), generator=gen, device=DEV)
    return x.mul_(scales).to(dtype)


_PREC = {"fp16x3": Bd.PREC_FP16X3, "tf32": Bd.PREC_TF32}


def prepare(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    d_in = case["d_in"]
    scales = _scales(gen, d_in)
    if case["kind"] == "gram":
        dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
        ctx = Bd.ArmorContext(128, d_in, 128, device=DEV, precision=_PREC[case["precision"]])
        return {"case": case, "ctx": ctx, "X": _activations(gen, scales, case["tokens"], dt), "H": ctx.new_gram()}
    d_out, db = case["d_out"], case["d_block"]
    W = torch.randn(d_out, d_in, generator=gen, device=DEV).mul_(0.02)
    if case["kind"] == "optimise":
        ctx = Bd.ArmorContext(d_out, d_in, db, device=DEV, seed=int(seed) & 0xFFFF, n_keep=case["n_keep"], m_group=case["m_group"],
                              h_mode=Bd.H_FULL if case["weighting"] == "full" else Bd.H_DIAG,
                              ab_step=Bd.AB_ADAM if case["update"] == "adam" else Bd.AB_EXACT,
                              normalize=int(case["normalize"]), mask_groups=case["mask_groups"])
        st = {"case": case, "ctx": ctx, "W": W, "H": ctx.new_gram()}
        if case["tokens"]:
            st["X"] = _activations(gen, scales, case["tokens"], torch.float32)
        else:
            # the Gram of a calibration set, symmetric to the last bit
            for _ in range(2):
                X = _activations(gen, scales, d_in, torch.float32)
                st["H"].addmm_(X.t(), X)
            st["H"].tril_()
            st["H"].add_(st["H"].tril(-1).t())
        return st
    # a finished layer: wrappers near the identity, the larger two of every four weights kept
    ctx = Bd.ArmorContext(d_out, d_in, db, device=DEV)
    eye = torch.eye(db, device=DEV)
    A = eye + torch.randn(d_out // db, db, db, generator=gen, device=DEV).mul_(0.3 / math.sqrt(db))
    B = eye + torch.randn(d_in // db, db, db, generator=gen, device=DEV).mul_(0.3 / math.sqrt(db))
    g = W.view(d_out, d_in // 4, 4)
    keep = torch.zeros_like(g, dtype=torch.bool).scatter_(2, g.abs().topk(2, dim=2).indices, True)
    M = (keep * torch.tensor([1, 2, 4, 8], device=DEV)).sum(2).to(torch.uint8)
    layer = Bd.LayerState(Wbar=W, A=A, B=B, S=(g * keep).view(d_out, d_in), M=M)
    x = _activations(gen, scales, case["tokens"], torch.float32 if case["form"] == "f32" else torch.bfloat16)
    st = {"case": case, "ctx": ctx, "layer": layer, "x": x}
    if case["form"] == "layer":
        st["packed"] = ctx.pack_layer(layer)
    elif case["form"] == "bf16_packed":
        st["packed"] = ctx.pack_core(layer)
    return st


# ------------------------------------------------------------------------------------------------ one pass
def run(state):
    case, ctx = state["case"], state["ctx"]
    if case["kind"] == "gram":
        state["H"].zero_()
        return ctx.gram(state["X"], state["H"])
    if case["kind"] == "forward":
        if case["form"] == "layer":
            return ctx.apply_layer(state["packed"], state["x"])
        if case["form"] == "bf16_packed":
            return ctx.apply_packed(state["layer"], state["packed"], state["x"])
        return ctx.apply(state["layer"], state["x"])
    H = state["H"]
    if "X" in state:
        H.zero_()
        ctx.gram(state["X"], H)
    st = ctx.init(state["W"], H)
    records = ctx.bcd_step(st, H, 0, case["iters"]).view(case["iters"], Bd.STATS_DTYPE.itemsize)
    loss = ctx.proxy_loss(st, H)
    # the records hold six doubles, two floats and four 32-bit counts per iteration
    out = {"A": st.A, "B": st.B, "S": st.S, "M": st.M, "loss": loss, "losses": records[:, :48].view(torch.float64),
           "steps": records[:, 48:56].view(torch.float32), "counts": records[:, 56:].view(torch.int32), "Wbar": st.Wbar}
    if case["normalize"]:
        out["r1"], out["r2"] = st.r1, st.r2
    if "X" in state:
        out["H"] = H
    return out


# ------------------------------------------------------------------------------------------------ what it takes
def _gram_work(d_in, tokens, esize):
    return {"bytes": float(tokens * d_in * esize + d_in * d_in * 4), "flops": float(tokens * d_in * (d_in + 1))}


def work(case):
    """Algorithmic bytes (every input once, every output once) and flops of one pass, as single-pass products."""
    d_in = case["d_in"]
    if case["kind"] == "gram":
        return _gram_work(d_in, case["tokens"], 2 if case["dtype"] == "bf16" else 4)
    d_out, db, tokens = case["d_out"], case["d_block"], case["tokens"]
    wn = d_out * d_in
    if case["kind"] == "forward":
        flops = 2.0 * tokens * (wn + (d_out + d_in) * db)
        if case["form"] == "f32":
            return {"bytes": 4.0 * (wn + (d_out + d_in) * (db + tokens)), "flops": flops}
        core = 2.0 * wn if case["form"] == "bf16" else 1.125 * wn      # dense, or kept values and positions
        if case["form"] != "bf16":
            flops = 2.0 * tokens * (wn / 2 + (d_out + d_in) * db)
        wrap = 2.0 if case["form"] == "layer" else 4.0
        core = 4.0 * wn if case["form"] == "bf16" else core            # the dense core comes as fp32
        return {"bytes": core + wrap * (d_out + d_in) * db + 2.0 * tokens * (d_out + d_in), "flops": flops}
    full, adam = case["weighting"] == "full", case["update"] == "adam"
    # an iteration reads W, the core and its mask and writes the core (Adam: reads and writes two moments as well);
    # H counts once per call
    per_iter_bytes = wn * (12.0 + 1.0 / case["m_group"] + (16.0 if adam else 0.0)) + 8.0 * (d_out + d_in) * db
    # products with the wrappers and per-block Grams, 2 d_out d_in d_block flops each: T = S B, A T, the two Grams of
    # either wrapper step, A S, the core's gradient (two sides) before the core step and before the mask step, and,
    # for each line search, the direction and its image (two each)
    block_products = 11.0 if adam else 16.0
    per_iter_flops = block_products * 2.0 * wn * db + ((2.0 * 2.0 * wn * d_in) if full else 0.0)
    w = {"bytes": case["iters"] * per_iter_bytes + 4.0 * (2 * wn + d_in * d_in),
         "flops": case["iters"] * per_iter_flops + 2.0 * 2.0 * wn * db + ((2 * 2.0 * wn * d_in) if full else 0.0)}
    if tokens:
        g = _gram_work(d_in, tokens, 4)
        w = {k: w[k] + g[k] for k in w}
    return w


def tolerance(case):
    """About four times the distance from the same path in 64 bits.  Gram: 6e-6 (7e-4 with one tf32 pass).  Forward: bf16
    3e-3 to 4.7e-3, fp32 5e-6 to 7e-6.
    Layers, compared with the same call on CUDA cores: losses and A to 2e-5, B and S to 2e-4 (Adam, which makes a move
    of fixed size of a gradient of any size: A 1.2e-4, S 4e-4 in ten iterations).  Where one of the ten thousand draws
    or masks of a pass is decided within rounding, the entries of one group of S change altogether and carry B along
    (seen in one pass of six: S 7e-4, B 3e-3), hence the wide bound on single entries."""
    if case["kind"] == "gram":
        return {"rel": 3e-3 if case["precision"] == "tf32" else 3e-5}
    if case["kind"] == "forward":
        return {"rel": 3e-5 if case["form"] == "f32" else 1.6e-2}
    return {"rel": 3e-3, "max": 0.99, "differ": 1e-2}
