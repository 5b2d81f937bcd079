"""The mma.sync attention at head_dim 8 in every tile form that its dispatch can choose, on long walks: rings of key tiles that are refilled, rows
whose scores outgrow their reference (the second walk), NaN in every padded row, log-sum-exp, packed rows and two problems in one launch."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import workloads as wk
from gpu_util import pad_mask, to_dev, to_np64, weights_to_dev

pytestmark = pytest.mark.gpu
SEG = (50, 500, 449)   # 1 + 8 + 8 tiles of 64 rows; intra walks one or eight key tiles, every block open seventeen


@pytest.fixture(scope="module")
def g():
    import paper_2505_01068_b200 as lib
    lib.load()
    return lib


def batch_for(per_sm, seg=SEG):
    """Samples that make about `per_sm` CTAs of 64 rows per SM, in which the dispatch counts."""
    return max(1, round(per_sm * torch.cuda.get_device_properties(0).multi_processor_count / sum((n + 63) // 64 for n in seg)))


def growing(rng, B, H, seg):
    """q, k, v whose keys, in every third sample, grow along the sequence by far more than a row's reference allows."""
    L = sum(seg)
    q, k, v = wk.draw_qkv(rng, B, L, H, 8, "bf16")
    k[::3] *= (np.arange(L, dtype=np.float32) / L * 400.0)[None, :, None, None]
    valid = np.stack([rng.integers((n + 1) // 2, n + 1, size=B) for n in seg], axis=1).astype(np.int32)
    valid[0], valid[-1] = seg, [1, seg[1], 65]
    return q, wk.storage_round(k, "bf16"), v, valid


# 8 heads: 16 rows up to 1.5 CTAs of 64 rows per SM, 32 (two CTAs per SM) up to 3, 32 (three) beyond, 64 beyond 8 where walks are short (the cross
# pattern); 4 heads: 32 (three) up to 4.5, 64 (two) up to 5.5, 64 (three) beyond
@pytest.mark.parametrize("H,per_sm", [(8, 1.2), (8, 2.2), (8, 3.6), (8, 8.7), (4, 1.2), (4, 5.0), (4, 6.2)])
@pytest.mark.parametrize("pattern", ["fwd", "intra", "all"])
def test_forms_on_long_walks(g, H, per_sm, pattern):
    rng = np.random.default_rng(int(10 * per_sm) + H)
    B = batch_for(per_sm)
    phase, mask = {"fwd": (g.PHASE_INTER_FWD, 0), "intra": (g.PHASE_INTRA, 0), "all": (g.PHASE_CUSTOM, 0x1FF)}[pattern]
    q, k, v, valid = growing(rng, B, H, SEG)
    pm = pad_mask(SEG, valid, B)
    dev = [torch.where(torch.from_numpy(pm).cuda()[:, :, None, None], float("nan"), to_dev(t, "bf16")) for t in (q, k, v)]
    vl = torch.from_numpy(valid).cuda()
    out, lse = g.im_attention_fwd(*dev, SEG, vl, phase, mask, want_lse=True)
    assert bool((out[torch.from_numpy(pm).cuda()] == 0).all())
    for b in range(B):   # one sample alone takes the smallest form: the same bits, but where all rows of a CTA walk again because one of them has to
        if b % 3 == 0:
            continue
        o1, l1 = g.im_attention_fwd(*(t[b:b + 1] for t in dev), SEG, vl[b:b + 1], phase, mask, want_lse=True)
        assert torch.equal(out[b:b + 1], o1) and torch.equal(lse[b:b + 1], l1), b
    for b in sorted({0, 1, 3 * (B // 6), B // 2, B - 1}):
        s = slice(b, b + 1)
        ref, ref_lse = oracle.im_attention_dense(q[s], k[s], v[s], SEG, valid[s], phase, custom_mask=mask, want_lse=True)
        err = np.abs(to_np64(out[s]) - ref)
        assert err.max() <= 4e-2 and err.mean() <= 2e-3, (b, err.max(), err.mean())   # one weight of 1 leaves V whole: |V| reaches 4
        fin, a = np.isfinite(ref_lse), to_np64(lse[s])
        assert np.array_equal(np.isfinite(a), fin) and (np.abs(a[fin] - ref_lse[fin]) <= 1.2e-2 + 1e-5 * np.abs(ref_lse[fin])).all()
    assert g.last_device_status() == (0, 0)


# Every length full: where the long walks of the 32-row form make one wave of CTAs and a bit, the 64-row form is taken (its bits are the same)
@pytest.mark.parametrize("H,pattern,per_row_block", [(8, "fwd", 18), (4, "intra", 32), (4, "all", 34)])
@pytest.mark.parametrize("waves", [0.95, 1.05, 1.2, 1.45])
def test_full_lengths_around_one_wave_of_long_walks(g, H, pattern, per_row_block, waves):
    rng = np.random.default_rng(H)
    seg = (50, 500, 500)
    B = round(waves * 3 * torch.cuda.get_device_properties(0).multi_processor_count / per_row_block)
    phase, mask = {"fwd": (g.PHASE_INTER_FWD, 0), "intra": (g.PHASE_INTRA, 0), "all": (g.PHASE_CUSTOM, 0x1FF)}[pattern]
    gen = torch.Generator("cuda").manual_seed(B)
    dev = [torch.randn((B, sum(seg), H, 8), device="cuda", generator=gen).bfloat16() for _ in range(3)]
    out = g.im_attention_fwd(*dev, seg, None, phase, mask)
    for b in range(B):
        assert torch.equal(out[b:b + 1], g.im_attention_fwd(*(t[b:b + 1] for t in dev), seg, None, phase, mask)), b
    b = int(rng.integers(B))
    ref = oracle.im_attention_dense(*(to_np64(t[b:b + 1]).astype(np.float32) for t in dev), seg, None, phase, mask)
    err = np.abs(to_np64(out[b:b + 1]) - ref)
    assert err.max() <= 2e-2 and err.mean() <= 2e-3, (err.max(), err.mean())
    assert g.last_device_status() == (0, 0)


@pytest.mark.parametrize("H,per_sm", [(8, 3.6), (4, 6.2)])
def test_forms_on_packed_rows(g, H, per_sm):
    rng = np.random.default_rng(H)
    B, d = batch_for(per_sm), 8 * H
    q, k, v, valid = growing(rng, B, H, SEG)
    valid[B // 2] = 0
    vl, L = torch.from_numpy(valid).cuda(), sum(SEG)
    qkv = torch.stack([to_dev(t, "bf16") for t in (q, k, v)], dim=2).contiguous()
    want = g.im_attention_fwd(qkv[:, :, 0], qkv[:, :, 1], qkv[:, :, 2], SEG, vl, g.PHASE_INTRA).reshape(B * L, d)
    real = torch.from_numpy(~pad_mask(SEG, valid, B).reshape(-1)).cuda()
    plan, cap = g.plan_rows(vl, SEG), B * L + 128
    n = int(real.sum())
    assert plan.cpu()[-1] == n
    packed = torch.full((cap, 3 * d), float("nan"), dtype=torch.bfloat16, device="cuda")
    packed[:n] = qkv.reshape(B * L, 3 * d)[real]
    out = torch.full((cap, d), 7.0, dtype=torch.bfloat16, device="cuda")
    shape = g.make_shape(B, SEG, d, H, vl, g.DTYPE_BF16, g.PHASE_INTRA, row_start=plan, capacity=cap)
    ws = torch.empty(256, dtype=torch.uint8, device="cuda")
    assert g.load().gsit_im_attention_fwd(ctypes.byref(shape), packed.data_ptr(), packed.data_ptr() + 2 * d, packed.data_ptr() + 4 * d, 3 * d,
                                          out.data_ptr(), None, ws.data_ptr(), ws.numel(), None) == 0
    assert torch.equal(out[:n], want[real]) and bool((out[n:] == 7.0).all())
    assert g.last_device_status() == (0, 0)


def test_two_problems_in_one_launch(g):
    """The pair counts twice as many CTAs as each layer by itself, and so takes another form."""
    rng = np.random.default_rng(5)
    B, d = batch_for(2.2), 64
    valid = np.stack([rng.integers((n + 1) // 2, n + 1, size=B) for n in SEG], axis=1).astype(np.int32)
    vl = torch.from_numpy(valid).cuda()
    w = [weights_to_dev(wk.draw_layer_weights(rng, d, 4 * d, "bf16", affine=True), "bf16") for _ in range(2)]
    xa, xb = (torch.randn((B, sum(SEG), d), device="cuda", generator=torch.Generator("cuda").manual_seed(i)) for i in range(2))
    ya, yb = g.im_layer_pair_fwd(xa, xb, w[0], w[1], SEG, 8, vl)
    assert torch.equal(ya, g.im_layer_fwd(xa, w[0], SEG, 8, vl, g.PHASE_INTER_FWD))
    assert torch.equal(yb, g.im_layer_fwd(xb, w[1], SEG, 8, vl, g.PHASE_INTER_BWD))
    assert g.last_device_status() == (0, 0)
