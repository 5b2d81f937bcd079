"""Tensor-memory attention for head_dim 8 / 16 / 32 at the edges of its 64-key tiles and of the 16-key groups in them, where the
one-pass walk of the later tiles ends, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wk
from gpu_util import to_dev, to_np64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,hd", [(8, 8), (4, 16), (2, 32)])
@pytest.mark.parametrize("seg", [(1, 64, 128), (16, 65, 129), (63, 80, 193), (145, 17, 256), (33, 0, 288)])
def test_key_tile_edges(seg, H, hd):
    import paper_2505_01068_b200 as g
    rng = np.random.default_rng(sum(seg) + hd)
    B = 5
    q, k, v = wk.draw_qkv(rng, B, sum(seg), H, hd, "bf16")
    valid = np.array([[max(0, n - cut) for n in seg] for cut in (0, 1, 15, 16, 100)], dtype=np.int32)
    vl = torch.from_numpy(valid).cuda()
    dev = [to_dev(wk.fill_padding(t.reshape(B, sum(seg), H * hd), seg, valid, np.nan).reshape(t.shape), "bf16") for t in (q, k, v)]
    g.tune_attention(g.ATTN_TMEM)
    try:
        for phase in (g.PHASE_INTER_FWD, g.PHASE_INTRA):
            out, lse = g.im_attention_fwd(*dev, seg, vl, phase, want_lse=True)
            ref, ref_lse = oracle.im_attention_dense(q, k, v, seg, valid, phase, want_lse=True)
            err = np.abs(to_np64(out) - ref)
            assert err.max() <= 4e-2 and err.mean() <= 2e-3, (phase, err.max(), err.mean())
            fin, a = np.isfinite(ref_lse), to_np64(lse)
            assert np.array_equal(np.isfinite(a), fin) and (np.abs(a[fin] - ref_lse[fin]) <= 1.2e-2).all()
    finally:
        g.tune_attention(g.ATTN_DEFAULT)
    assert g.last_device_status() == (0, 0)
