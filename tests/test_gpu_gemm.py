"""The tcgen05 linear layers at both tilings (pairs of CTAs, one CTA per tile) and at their edges: row counts that are no multiple
of a tile, column counts of one box, of partial boxes and of several tiles, tiles of padding only, float output with a residual."""
import numpy as np
import pytest
import torch

import workloads as wk
from gpu_util import pad_mask, to_dev, weights_to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import paper_2505_01068_b200 as lib
    lib.load()
    return lib


@pytest.mark.parametrize("d,heads,seg,B", [(64, 1, (3, 5, 9), 1), (64, 8, (50, 301, 190), 3), (128, 2, (129, 500, 333), 40), (192, 3, (128, 256, 260), 30),
                                           (256, 4, (100, 300, 411), 21), (512, 8, (60, 511, 700), 18), (320, 5, (40, 255, 257), 60)])
@pytest.mark.parametrize("padded", [False, True])
def test_projection_against_matmul(g, d, heads, seg, B, padded):
    rng = np.random.default_rng(d + B)
    L = sum(seg)
    x = torch.randn((B, L, d), device="cuda", generator=torch.Generator("cuda").manual_seed(B)).bfloat16()
    w = to_dev(wk.xavier_uniform(rng, 3 * d, d), "bf16")
    bias = to_dev(rng.standard_normal(3 * d + 1).astype(np.float32))[1:].clone() if d != 192 else to_dev(rng.standard_normal(3 * d + 1).astype(np.float32))[1:]
    valid = np.stack([rng.integers(0, n + 1, size=B) for n in seg], axis=1).astype(np.int32) if padded else None
    if padded:
        valid[B // 2:B // 2 + 3] = 0   # whole tiles of padding
    vl = None if valid is None else torch.from_numpy(valid).cuda()
    pm = torch.from_numpy(pad_mask(seg, valid, B)).cuda()
    x[pm] = float("nan")
    ref = torch.nan_to_num(x.float()) @ w.float().T + bias
    ref[pm] = 0
    out = torch.full((B, L, 3, heads, d // heads), float("nan"), device="cuda", dtype=torch.bfloat16)
    first = None
    for _ in range(5):
        got = g.im_qkv_proj(x, w, bias, seg, heads, vl, out=out).clone()
        first = got if first is None else first
        assert torch.equal(got, first)
    got = first.reshape(B, L, 3 * d).float()
    assert bool((got[pm] == 0).all())
    assert float((got - ref).abs().max()) <= 1e-2 * float(ref.abs().max())
    assert g.last_device_status() == (0, 0)


@pytest.mark.parametrize("d,heads,d_ff,seg,B", [(192, 3, 448, (37, 129, 300), 1), (256, 4, 1024, (100, 300, 411), 25), (512, 8, 2048, (60, 511, 700), 20)])
def test_wide_layer_against_legacy_kernels(g, d, heads, d_ff, seg, B):
    """Every linear layer of a wide layer (bf16 output, ReLU, float output with residual and strided rows) on tcgen05 against the
    mma.sync kernels."""
    rng = np.random.default_rng(d)
    L = sum(seg)
    x = torch.randn((B, L, d), device="cuda", generator=torch.Generator("cuda").manual_seed(B))
    w = weights_to_dev(wk.draw_layer_weights(rng, d, d_ff, "bf16", affine=True), "bf16")
    valid = np.stack([rng.integers(0, n + 1, size=B) for n in seg], axis=1).astype(np.int32)
    pm = torch.from_numpy(pad_mask(seg, valid, B)).cuda()
    x[pm] = float("nan")
    vl = torch.from_numpy(valid).cuda()
    wide = torch.full((B, L, 2 * d), 7.0, device="cuda")
    out = wide[:, :, d:]
    g.im_layer_fwd(x, w, seg, heads, vl, g.PHASE_INTER_FWD, out=out)
    assert bool((wide[:, :, :d] == 7.0).all()) and bool((out[pm] == 0).all())
    first = out.clone()
    for _ in range(5):
        g.im_layer_fwd(x, w, seg, heads, vl, g.PHASE_INTER_FWD, out=out)
        assert torch.equal(out, first)
    g.tune_attention(g.ATTN_LEGACY)
    try:
        ref = g.im_layer_fwd(x, w, seg, heads, vl, g.PHASE_INTER_FWD)
    finally:
        g.tune_attention(g.ATTN_DEFAULT)
    err = (first - ref).abs()
    assert float(err.max()) <= 4e-2 and float(err.mean()) <= 4e-3, (float(err.max()), float(err.mean()))
    assert g.last_device_status() == (0, 0)


@pytest.mark.parametrize("d,heads,seg,B", [(64, 8, (9, 50, 30), 2), (128, 8, (50, 300, 270), 60), (192, 3, (37, 129, 300), 5), (512, 8, (60, 511, 700), 18)])
def test_projection_on_packed_rows(g, d, heads, seg, B):
    """Tiles inside a call's rows, tiles shared with the samples before and after, tiles outside; one CTA per tile and pairs.  Same
    bits as the padded layout; nothing written beyond the call's rows."""
    rng = np.random.default_rng(d + B)
    L, cap = sum(seg), B * sum(seg) + 128
    x = torch.randn((B, L, d), device="cuda", generator=torch.Generator("cuda").manual_seed(B)).bfloat16()
    w, bias = to_dev(wk.xavier_uniform(rng, 3 * d, d), "bf16"), to_dev(rng.standard_normal(3 * d).astype(np.float32))
    valid = np.stack([rng.integers(0, n + 1, size=B) for n in seg], axis=1).astype(np.int32)
    valid[B // 2] = 0
    vl = torch.from_numpy(valid).cuda()
    plan = g.plan_rows(vl, seg)
    want = torch.empty((cap, 3 * d), device="cuda")
    g.pack_rows(g.im_qkv_proj(x, w, bias, seg, heads, vl).reshape(B, L, 3 * d).float(), want, seg, vl, plan)
    xp = torch.full((cap, d), float("nan"), device="cuda")
    xp = g.pack_rows(x.float(), xp, seg, vl, plan).bfloat16()
    starts = plan.cpu().numpy()
    for lo, hi in {(0, B), (0, 1), (B - 1, B), (1, (B + 1) // 2), (B // 3, B)}:
        if lo >= hi:
            continue
        for bare in (False, True):
            out = torch.full((cap, 3, heads, d // heads), 7.0, dtype=torch.bfloat16, device="cuda")
            g.im_qkv_proj(xp, w, None if bare else bias, seg, heads, vl[lo:hi], out=out, row_start=plan[3 * lo:])
            first = out.clone()
            for _ in range(3):
                g.im_qkv_proj(xp, w, None if bare else bias, seg, heads, vl[lo:hi], out=out, row_start=plan[3 * lo:])
                assert torch.equal(out, first)
            a, b = int(starts[3 * lo]), int(starts[3 * hi])
            flat = out.reshape(cap, 3 * d).float()
            assert bool((flat[:a] == 7.0).all()) and bool((flat[b:] == 7.0).all()), (lo, hi)
            if bare:
                ref = xp[a:b].float() @ w.float().T
                assert a == b or float((flat[a:b] - ref).abs().max()) <= 1e-2 * float(ref.abs().max())
            else:
                assert torch.equal(flat[a:b], want[a:b]), (lo, hi)
    assert g.last_device_status() == (0, 0)
