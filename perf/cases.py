"""What the speed of this framework is judged by: calls as a user's program makes them, over the sizes, data types, block
patterns and padding that multimodal sentiment data brings.  Shapes follow the workloads of this repository (aligned and
unaligned MOSI / MOSEI, CH-SIMS, MIntRec, a scaled stress shape); `draw` spreads over the ranges between them.

Kinds of case (the `kind` of a case):
  attend     shared QKV projection, then IM attention on the views of its fused buffer
  attention  IM attention on three separate tensors, optionally with the log-sum-exp a backward pass needs
  layer      one IM encoder layer
  stack      the whole fusion stack (both ring encoders, intra encoder) and the read-out of its last steps
  pipeline   the stack on batches in pinned host memory, results back to pinned host memory
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2505_01068_b200 as g

_OPEN = {"fwd": ((0, 1), (1, 2), (2, 0)), "bwd": ((0, 2), (1, 0), (2, 1)), "intra": ((0, 0), (1, 1), (2, 2)),
         "all": tuple((s, r) for s in range(3) for r in range(3))}   # "all": the unmasked naive graph
_PHASE = {"fwd": g.PHASE_INTER_FWD, "bwd": g.PHASE_INTER_BWD, "intra": g.PHASE_INTRA, "all": g.PHASE_CUSTOM}


def _case(kind, dtype, batch, seg, d, heads, phase="fwd", padding="half", lse=False, raw=(0, 0, 0), depth=(0, 0), intra_heads=0):
    return {"kind": kind, "dtype": dtype, "batch": batch, "seg0": seg[0], "seg1": seg[1], "seg2": seg[2], "d": d, "heads": heads,
            "phase": phase, "padding": padding, "lse": lse, "raw0": raw[0], "raw1": raw[1], "raw2": raw[2], "rings": depth[0],
            "intra": depth[1], "intra_heads": intra_heads}


def listed():
    mosi, mosei = (50, 375, 500), (50, 500, 500)
    mosi_raw, mosei_raw = (768, 5, 20), (768, 74, 35)
    named = {
        # one layer on a toy problem in single precision: what a unit test or a notebook calls, all launches and host path
        "tiny_layer_f32": _case("layer", "f32", 2, (8, 12, 10), 32, 4, "fwd", "none"),
        # word-aligned data (all modalities resampled to 50 steps), no padding: short segments, launch-bound
        "aligned_attend": _case("attend", "bf16", 32, (50, 50, 50), 32, 4, "fwd", "none", raw=mosi_raw),
        # one utterance at a time through the whole model: the latency a serving process sees
        "single_stack": _case("stack", "bf16", 1, mosei, 64, 8, raw=mosei_raw, depth=(4, 2), intra_heads=8),
        # one cross-modal layer on an unaligned MOSI batch
        "mosi_layer": _case("layer", "bf16", 32, mosi, 64, 8, "bwd", raw=mosi_raw),
        # the same batch in single precision (evaluation against a float model)
        "mosi_layer_f32": _case("layer", "f32", 32, mosi, 64, 8, "intra", raw=mosi_raw),
        # the whole model on an unaligned MOSEI batch, lengths between half and full: the benchmark's step, issued call by call
        "mosei_stack": _case("stack", "bf16", 64, mosei, 64, 8, raw=mosei_raw, depth=(4, 2), intra_heads=8),
        # the same model at the data set's own length statistics: three quarters of the positions are padding
        "mosei_stats_stack": _case("stack", "bf16", 32, mosei, 64, 8, padding="stats", raw=mosei_raw, depth=(4, 2), intra_heads=8),
        # the model end to end from and to host memory, copies overlapped
        "mosei_pipeline": _case("pipeline", "bf16", 64, mosei, 64, 8, raw=mosei_raw, depth=(4, 2), intra_heads=8),
        # intra-modal attention on a CH-SIMS-shaped batch with wider heads
        "chsims_attend": _case("attend", "bf16", 32, (39, 55, 400), 128, 4, "intra", raw=(768, 33, 709)),
        # the unmasked graph (the ablation every masked variant is compared with), with the log-sum-exp of each row
        "mintrec_unmasked_lse": _case("attention", "bf16", 32, (30, 480, 230), 128, 8, "all", lse=True),
        # long sequences, wide model: projection and cross-modal attention
        "scaled_attend": _case("attend", "bf16", 128, (128, 1024, 1024), 512, 8, "fwd", "quarter"),
        # ... and one whole intra-modal layer of that model
        "scaled_layer": _case("layer", "bf16", 128, (128, 1024, 1024), 512, 8, "intra", "quarter"),
    }
    return [dict(c, name=n) for n, c in named.items()]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case of the same ranges: batches of 1 to 128, segments of 8 to 1024 steps (one of the three usually shorter, as
    text is), widths 32 to 512 with heads of 8 to 64, every block pattern, every kind of padding."""
    kind = rng.choice(("attend", "attend", "attention", "attention", "layer", "layer", "layer", "stack", "stack", "pipeline"))
    dtype = "f32" if kind in ("attend", "attention", "layer") and rng.random() < 0.2 else "bf16"
    if kind in ("stack", "pipeline"):
        d, heads, intra_heads = rng.choice(((64, 8, 8), (64, 8, 8), (64, 4, 8), (64, 2, 4), (32, 4, 4)))
        depth = (rng.randint(1, 4), rng.randint(1, 3))
    else:
        hd = rng.choice((8, 16, 32, 64))
        d = rng.choice([w for w in ((32, 64, 128) if dtype == "f32" else (32, 64, 128, 192, 256, 512)) if hd <= w <= 16 * hd and w % hd == 0])
        heads, intra_heads, depth = d // hd, 0, (0, 0)
    top = 1024 if kind in ("attend", "attention", "layer") else 500
    seg = [_log_int(rng, 8, min(top, 128)), _log_int(rng, 16, top), _log_int(rng, 16, top)]
    if rng.random() < 0.25:
        rng.shuffle(seg)
    phase = rng.choice(("fwd", "bwd", "intra", "fwd", "bwd", "intra", "all"))
    padding = rng.choice(("half", "half", "quarter", "stats", "none")) if kind != "pipeline" else rng.choice(("half", "stats"))
    lse = kind == "attention" and rng.random() < 0.5
    case = _case(kind, dtype, _log_int(rng, 1, 128), seg, d, heads, phase, padding, lse, depth=depth, intra_heads=intra_heads)
    while case["batch"] > 1 and _cost(case) > _most(case):
        case["batch"] = max(1, case["batch"] * 3 // 4)
    return case


def _most(case):
    """What a drawn case may cost: as much as the largest listed one; float cases as much as the float one, host cases and
    stacks as much as the listed stack."""
    name = "mosi_layer_f32" if case["dtype"] == "f32" else "mosei_stack" if case["kind"] in ("stack", "pipeline") else "scaled_layer"
    return _cost(next(c for c in listed() if c["name"] == name))


def _cost(case):
    w = work(case)
    pairs, _ = _sizes(case)
    exps = case["heads"] * pairs(case["phase"]) if case["kind"] not in ("stack", "pipeline") else 0
    return w["flops"] / 1e15 + w["bytes"] / 5e12 + exps / 2e12


def _seg(case):
    return (case["seg0"], case["seg1"], case["seg2"])


def _lengths(case, seed):
    """Valid lengths [B, 3]: uniform between half and full, every fourth sample at half, or clipped normals around the averages
    of the MOSEI training split (in proportion to the maxima); None where nothing is padded."""
    rng, seg, b = np.random.default_rng(int(seed) + 17), np.asarray(_seg(case)), case["batch"]
    if case["padding"] == "none":
        return None
    if case["padding"] == "half":
        return np.stack([rng.integers((n + 1) // 2, n + 1, size=b) for n in seg], axis=1).astype(np.int32)
    if case["padding"] == "quarter":
        n = np.tile(seg, (b, 1))
        n[np.arange(b) % 4 == 3] = np.maximum(1, seg // 2)
        return n.astype(np.int32)
    share, spread = np.array([24 / 50, 149 / 500, 94 / 500]), np.array([148 ** 0.5 / 50, 8105 ** 0.5 / 500, 5115 ** 0.5 / 500])
    return np.clip(np.rint(rng.normal(share * seg, spread * seg, size=(b, 3))), 1, seg).astype(np.int32)


def _sizes(case):
    """(pairs of a block pattern -> open (query, key) pairs of real positions per head, real positions)."""
    n = _lengths(case, 0)
    n = np.tile(np.asarray(_seg(case)), (case["batch"], 1)) if n is None else n
    n = n.astype(np.int64)
    return (lambda phase: int(sum((n[:, s] * n[:, r]).sum() for s, r in _OPEN[phase]))), int(n.sum())


# ---------------------------------------------------------------------------------------------------------- inputs

def _uniform(gen, rows, cols):
    a = (6.0 / (rows + cols)) ** 0.5   # Xavier
    return (torch.rand((rows, cols), device="cuda", generator=gen) * 2 - 1) * a


def _layer_weights(gen, d, dtype):
    """One trained-looking layer: Xavier matrices, small biases, LayerNorm scales around one."""
    t = torch.float32 if dtype == "f32" else torch.bfloat16
    vec = lambda n: torch.randn(n, device="cuda", generator=gen) * 0.1
    return {"w_qkv": torch.cat([_uniform(gen, d, d) for _ in range(3)]).to(t), "b_qkv": vec(3 * d), "w_o": _uniform(gen, d, d).to(t), "b_o": vec(d),
            "w_1": _uniform(gen, 4 * d, d).to(t), "b_1": vec(4 * d), "w_2": _uniform(gen, d, 4 * d).to(t), "b_2": vec(d),
            "ln1_g": 1 + vec(d), "ln1_b": vec(d), "ln2_g": 1 + vec(d), "ln2_b": vec(d)}


def _sequence(gen, case):
    """X [B, L, d]: raw features N(0, 1) of each modality through its own Xavier map, or N(0, 1) where no raw width is given."""
    b, d = case["batch"], case["d"]
    parts = []
    for i, n in enumerate(_seg(case)):
        raw = case["raw%d" % i]
        x = torch.randn((b, n, raw or d), device="cuda", generator=gen)
        parts.append(x @ _uniform(gen, d, raw).T if raw else x)
    x = torch.cat(parts, dim=1)
    return x.bfloat16() if case["dtype"] == "bf16" else x


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    d, b, kind = case["d"], case["batch"], case["kind"]
    n = _lengths(case, seed)
    s = {"case": case, "seg": _seg(case), "valid": None if n is None else torch.from_numpy(n).cuda(),
         "mask": 0x1FF if case["phase"] == "all" else 0}
    if kind == "attention":
        t = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
        s["qkv"] = [torch.randn((b, sum(s["seg"]), case["heads"], d // case["heads"]), device="cuda", generator=gen).to(t) for _ in range(3)]
        return s
    s["x"] = _sequence(gen, case)
    if kind == "attend":
        w = _layer_weights(gen, d, case["dtype"])
        s["w_qkv"], s["b_qkv"] = w["w_qkv"], w["b_qkv"]
        return s
    s["x"] = s["x"].float()   # the residual stream is float whatever the weights are
    if kind == "layer":
        s["w"] = _layer_weights(gen, d, case["dtype"])
        return s
    ring = lambda: [_layer_weights(gen, d, "bf16") for _ in range(case["rings"])]
    head = (_uniform(gen, 128, 6 * d).bfloat16(), torch.randn(128, device="cuda", generator=gen) * 0.1)
    s["stack"] = g.GsitStack(ring(), ring(), [_layer_weights(gen, 2 * d, "bf16") for _ in range(case["intra"])], s["seg"], case["heads"],
                             case["intra_heads"], head=head)
    if kind == "pipeline":
        s["x"] = s["x"].cpu().pin_memory()
        s["valid"] = torch.from_numpy(n).pin_memory()
        s["y"] = torch.empty((b, sum(s["seg"]), 2 * d), dtype=torch.float32, pin_memory=True)
        s["pipe"] = g.HostPipeline(s["stack"], tuple(s["x"].shape))
    return s


# ---------------------------------------------------------------------------------------------------------- one pass

def run(s):
    c, seg, valid, mask = s["case"], s["seg"], s["valid"], s["mask"]
    phase = _PHASE[c["phase"]]
    if c["kind"] == "attention":
        return g.im_attention_fwd(*s["qkv"], seg, valid, phase, mask, want_lse=c["lse"])
    if c["kind"] == "attend":
        qkv = g.im_qkv_proj(s["x"], s["w_qkv"], s["b_qkv"], seg, c["heads"], valid)
        return qkv, g.im_attention_fwd(qkv[:, :, 0], qkv[:, :, 1], qkv[:, :, 2], seg, valid, phase, mask)
    if c["kind"] == "layer":
        return g.im_layer_fwd(s["x"], s["w"], seg, c["heads"], valid, phase, mask)
    if c["kind"] == "stack":
        y = s["stack"].forward(s["x"], valid)
        return y, s["stack"].read_out(y, valid)
    s["pipe"].step(s["x"], s["y"], valid)   # queued; complete once the device is synchronised
    return s["y"]


# ---------------------------------------------------------------------------------------------------------- what it takes

def work(case):
    """Real positions read once, whole outputs (padded positions included, they are written as zero) written once, weights read
    once; multiplications and additions of the open blocks of real positions."""
    pairs, real = _sizes(case)
    d, es, rows = case["d"], 4 if case["dtype"] == "f32" else 2, case["batch"] * sum(_seg(case))
    layer_flops = lambda w, phase: real * 2.0 * 12 * w * w + 4.0 * w * pairs(phase)
    if case["kind"] == "attention":
        return {"bytes": 3.0 * real * d * es + rows * d * es + (4.0 * rows * case["heads"] if case["lse"] else 0), "flops": 4.0 * d * pairs(case["phase"])}
    if case["kind"] == "attend":
        return {"bytes": real * d * es + 3.0 * d * d * es + 4.0 * rows * d * es, "flops": real * 6.0 * d * d + 4.0 * d * pairs(case["phase"])}
    if case["kind"] == "layer":
        return {"bytes": 4.0 * real * d + 4.0 * rows * d + 12.0 * d * d * es, "flops": layer_flops(d, case["phase"])}
    flops = case["rings"] * (layer_flops(d, "fwd") + layer_flops(d, "bwd")) + case["intra"] * layer_flops(2 * d, "intra")
    weights = 12.0 * 2 * (2 * case["rings"] * d * d + case["intra"] * 4 * d * d)
    return {"bytes": 4.0 * real * d + 8.0 * rows * d + weights, "flops": flops + case["batch"] * 2.0 * 128 * 6 * d}


def tolerance(case):
    if case["dtype"] == "f32":
        return {"rel": 1e-5}
    return {"rel": 1e-2, "max": 0.15}   # bf16 operands and storage, float accumulation
