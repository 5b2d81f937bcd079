"""Float attention at head widths up to 16, whose key tiles hold 256 or 128 keys where a segment is longer than half of one: numbers of real
keys around the rounds in which a tile is filled, its groups of eight and its end, with NaN in every padded row."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wk
from gpu_util import check_close, pad_mask, to_dev, to_np64

pytestmark = pytest.mark.gpu
KEYS = (1, 7, 8, 9, 31, 32, 33, 63, 64, 65, 95, 96, 97, 127, 128, 129, 160, 191, 192, 193, 255, 256, 257, 300)


@pytest.mark.parametrize("H,hd", [(4, 8), (2, 5), (2, 16), (2, 12)])
@pytest.mark.parametrize("seg", [(11, 300, 64), (3, 128, 129), (300, 70, 65)])
def test_key_counts_around_the_rounds_of_a_tile(H, hd, seg):
    import paper_2505_01068_b200 as g
    rng = np.random.default_rng(hd + sum(seg))
    B = len(KEYS)
    valid = np.array([[min(n, k) for n in seg] for k in KEYS], dtype=np.int32)
    q, k, v = wk.draw_qkv(rng, B, sum(seg), H, hd, "f32")
    pm = pad_mask(seg, valid, B)
    dev = [to_dev(np.where(pm[:, :, None, None], np.nan, t).astype(np.float32)) for t in (q, k, v)]
    vl = torch.from_numpy(valid).cuda()
    for phase, mask in ((g.PHASE_INTER_FWD, 0), (g.PHASE_INTRA, 0), (g.PHASE_CUSTOM, 0x1FF)):
        out, lse = g.im_attention_fwd(*dev, seg, vl, phase, mask, want_lse=True)
        ref, ref_lse = oracle.im_attention_dense(q, k, v, seg, valid, phase, custom_mask=mask, want_lse=True)
        check_close(to_np64(out), ref, "f32", pm, f"hd {hd} phase {phase}")
        a, b = to_np64(lse), np.asarray(ref_lse)
        assert np.array_equal(np.isneginf(a), np.isneginf(b)) and np.abs(a[np.isfinite(b)] - b[np.isfinite(b)]).max() <= 1e-4
    assert g.last_device_status() == (0, 0)
