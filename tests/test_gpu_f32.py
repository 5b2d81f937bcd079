"""Float kernels at the sizes where their tiles end: head widths around the slices of a row, key counts around the key tiles,
batches that use one, two and four key splits, and layer widths around the 32-feature slices of the fused halves."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wk
from gpu_util import check_close, pad_mask, to_dev, to_np64, weights_to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import paper_2505_01068_b200 as lib
    lib.load()
    return lib


@pytest.mark.parametrize("H,hd", [(2, 1), (3, 5), (2, 8), (1, 12), (2, 16), (1, 24), (2, 32), (1, 40), (1, 64), (1, 100), (1, 128), (1, 200), (1, 256)])
def test_attention_every_head_width(g, H, hd):
    rng = np.random.default_rng(hd)
    seg = (9, 129, 66)
    valid = np.array([[9, 129, 66], [1, 64, 65], [8, 0, 17]], dtype=np.int32)
    q, k, v = wk.draw_qkv(rng, 3, sum(seg), H, hd, "f32")
    pm = pad_mask(seg, valid, 3)
    dev = [to_dev(np.where(pm[:, :, None, None], np.nan, t).astype(np.float32)) for t in (q, k, v)]
    for phase, mask in ((g.PHASE_INTER_FWD, 0), (g.PHASE_INTRA, 0), (g.PHASE_CUSTOM, 0x1FF), (g.PHASE_CUSTOM, 0b000100011)):
        out, lse = g.im_attention_fwd(*dev, seg, torch.from_numpy(valid).cuda(), phase, mask, want_lse=True)
        ref, ref_lse = oracle.im_attention_dense(q, k, v, seg, valid, phase, custom_mask=mask, want_lse=True)
        check_close(to_np64(out), ref, "f32", pm, f"hd {hd} phase {phase}")
        a, b = to_np64(lse), np.asarray(ref_lse)
        assert np.array_equal(np.isneginf(a), np.isneginf(b)) and np.abs(a[np.isfinite(b)] - b[np.isfinite(b)]).max() <= 1e-4


@pytest.mark.parametrize("B", [1, 24, 96])
def test_attention_key_splits(g, B):
    rng = np.random.default_rng(B)
    seg = (5, 130, 257)
    q, k, v = wk.draw_qkv(rng, B, sum(seg), 4, 8, "f32")
    q *= 6.0   # the running maximum moves
    valid = np.stack([rng.integers(0, n + 1, size=B) for n in seg], axis=1).astype(np.int32)
    out = g.im_attention_fwd(*[to_dev(t) for t in (q, k, v)], seg, torch.from_numpy(valid).cuda(), g.PHASE_INTER_BWD)
    ref = oracle.im_attention_dense(q, k, v, seg, valid, g.PHASE_INTER_BWD)
    check_close(to_np64(out), ref, "f32", pad_mask(seg, valid, B), f"B {B}")


@pytest.mark.parametrize("hd", [3, 8, 40])
@pytest.mark.parametrize("masked", [1, 8, 40, 199])
def test_keys_with_scores_of_minus_infinity(g, hd, masked):
    """Keys that an infinite feature takes out of the softmax: whole groups of them, first in their segment, weigh nothing."""
    rng = np.random.default_rng(masked)
    seg, H, B = (10, 200, 90), 2, 2
    q, k, v = wk.draw_qkv(rng, B, sum(seg), H, hd, "f32")
    q[..., 0] = np.abs(q[..., 0]) + 0.1
    k[:, 10:10 + masked, :, 0] = -np.inf
    out, lse = g.im_attention_fwd(*[to_dev(t) for t in (q, k, v)], seg, None, g.PHASE_INTER_FWD, want_lse=True)
    # rows of segment 0 attend to segment 1
    s = np.einsum("bqhe,bkhe->bhqk", q[:, :10].astype(np.float64), k[:, 10:210].astype(np.float64)) / np.sqrt(hd)
    m = s.max(-1, keepdims=True)
    p = np.exp(s - m)
    want = np.einsum("bhqk,bkhe->bqhe", p / p.sum(-1, keepdims=True), v[:, 10:210].astype(np.float64))
    assert np.abs(to_np64(out)[:, :10].reshape(B, 10, H, hd) - want).max() <= 1e-4
    assert np.abs(to_np64(lse)[:, :, :10] - (m + np.log(p.sum(-1, keepdims=True)))[..., 0]).max() <= 1e-4
    assert np.isfinite(to_np64(out)).all()


@pytest.mark.parametrize("B,H", [(65535, 2), (65536, 2), (131072, 2), (2, 65537)])
def test_batches_and_heads_beyond_one_grid_dimension(g, B, H):
    """A grid's y and z hold 65535 blocks each; attention and layer take larger batches, and attention more heads."""
    rng = np.random.default_rng(B)
    seg, hd = (1, 2, 1), 4
    q, k, v = wk.draw_qkv(rng, B, sum(seg), H, hd, "f32")
    valid = rng.integers(0, 3, size=(B, 3)).astype(np.int32).clip(None, seg).astype(np.int32)
    vl = torch.from_numpy(valid).cuda()
    out, lse = g.im_attention_fwd(*[to_dev(t) for t in (q, k, v)], seg, vl, g.PHASE_CUSTOM, 0x1FF, want_lse=True)
    ref, ref_lse = oracle.im_attention_dense(q, k, v, seg, valid, g.PHASE_CUSTOM, custom_mask=0x1FF, want_lse=True)
    check_close(to_np64(out), ref, "f32", pad_mask(seg, valid, B), f"B {B}")
    a, b = to_np64(lse), np.asarray(ref_lse)
    assert np.array_equal(np.isneginf(a), np.isneginf(b)) and np.abs(a[np.isfinite(b)] - b[np.isfinite(b)]).max() <= 1e-4
    if H > 2:
        return
    x = rng.standard_normal((B, sum(seg), H * hd), dtype=np.float32)
    w = wk.draw_layer_weights(rng, H * hd, 16, "f32", affine=True)
    y = to_np64(g.im_layer_fwd(to_dev(x), weights_to_dev(w, "f32"), seg, H, vl, g.PHASE_INTRA)[-70:])
    check_close(y, oracle.im_layer_fwd(x[-70:], w, seg, H, valid[-70:], g.PHASE_INTRA), "f32", pad_mask(seg, valid[-70:], 70), f"layer B {B}")


@pytest.mark.parametrize("d,heads,d_ff,seg,B", [(32, 4, 128, (8, 12, 10), 2), (36, 3, 100, (64, 64, 0), 1), (64, 8, 256, (50, 75, 100), 3),
                                                (96, 4, 200, (1, 63, 1), 2), (128, 2, 512, (33, 64, 31), 2), (4, 1, 4, (3, 2, 1), 1),
                                                (160, 4, 320, (33, 64, 31), 2), (30, 3, 62, (33, 64, 31), 1), (64, 8, 256, (50, 375, 500), 40)])
def test_layer_widths(g, d, heads, d_ff, seg, B):
    """d <= 128 with whole 16-byte rows takes the fused halves, the others (160; 30 and 62) the separate kernels."""
    rng = np.random.default_rng(d + d_ff)
    L = sum(seg)
    x = rng.standard_normal((B, L, d), dtype=np.float32)
    w = wk.draw_layer_weights(rng, d, d_ff, "f32", affine=True)
    valid = np.stack([rng.integers(0, n + 1, size=B) for n in seg], axis=1).astype(np.int32)
    pm = pad_mask(seg, valid, B)
    xd = to_dev(np.where(pm[:, :, None], np.nan, x).astype(np.float32))
    if d % 4:   # rows of whole 16-byte pieces are required: give the rows a stride of 32
        wide = torch.full((B, L, 32), float("nan"), device="cuda")
        wide[:, :, :d] = xd
        y = torch.full((B, L, 32), float("nan"), device="cuda")
        g.im_layer_fwd(wide[:, :, :d], weights_to_dev(w, "f32"), seg, heads, torch.from_numpy(valid).cuda(), g.PHASE_INTER_FWD, out=y[:, :, :d])
        y = y[:, :, :d]
    else:
        y = g.im_layer_fwd(xd, weights_to_dev(w, "f32"), seg, heads, torch.from_numpy(valid).cuda(), g.PHASE_INTER_FWD)
    n = min(B, 4)
    ref = oracle.im_layer_fwd(x[-n:], w, seg, heads, valid[-n:], g.PHASE_INTER_FWD)
    check_close(to_np64(y)[-n:], ref, "f32", pm[-n:], f"d {d}")
    assert bool((y[torch.from_numpy(pm).cuda()] == 0).all())


@pytest.mark.parametrize("d,heads", [(30, 5), (64, 8), (129, 3)])
def test_projection_odd_widths(g, d, heads):
    rng = np.random.default_rng(d)
    seg, valid = (7, 70, 52), np.array([[7, 70, 52], [3, 0, 51]], dtype=np.int32)
    x, w = rng.standard_normal((2, sum(seg), d), dtype=np.float32), wk.xavier_uniform(rng, 3 * d, d)
    b = rng.standard_normal(3 * d).astype(np.float32)
    qkv = g.im_qkv_proj(to_dev(x), to_dev(w), to_dev(b), seg, heads, torch.from_numpy(valid).cuda())
    ref = x.astype(np.float64) @ w.T.astype(np.float64) + b
    ref[pad_mask(seg, valid, 2)] = 0
    check_close(to_np64(qkv).reshape(ref.shape), ref, "f32", pad_mask(seg, valid, 2), f"d {d}")


@pytest.mark.parametrize("d,heads,d_ff,B", [(32, 4, 128, 3), (64, 8, 256, 40), (128, 8, 320, 9)])
def test_separate_kernels_on_request(g, d, heads, d_ff, B):
    """Kernel choice ATTN_UNFUSED: the separate float kernels at widths that the fused halves cover.  Both within the float
    tolerance of the oracle; other orders of summation, so within its sum of each other and not equal."""
    rng = np.random.default_rng(d)
    seg = (20, 170, 133)
    x = rng.standard_normal((B, sum(seg), d), dtype=np.float32)
    w = wk.draw_layer_weights(rng, d, d_ff, "f32", affine=True)
    valid = np.stack([rng.integers(0, n + 1, size=B) for n in seg], axis=1).astype(np.int32)
    vl, pm, wd, ys = torch.from_numpy(valid).cuda(), pad_mask(seg, valid, B), weights_to_dev(w, "f32"), []
    for choice in (g.ATTN_DEFAULT, g.ATTN_UNFUSED):
        g.tune_attention(choice)
        try:
            ys.append(to_np64(g.im_layer_fwd(to_dev(x), wd, seg, heads, vl, g.PHASE_INTRA)))
        finally:
            g.tune_attention(g.ATTN_DEFAULT)
        ref = oracle.im_layer_fwd(x[:2], w, seg, heads, valid[:2], g.PHASE_INTRA)
        check_close(ys[-1][:2], ref, "f32", pm[:2], f"choice {choice}")
    diff = np.abs(ys[0] - ys[1]).max()
    assert 0 < diff <= 2e-4
