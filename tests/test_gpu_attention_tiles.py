"""The mma.sync attention at head_dim 8 in each of the tile heights its dispatch chooses by the number of CTAs: the bits of a sample do
not depend on the batch it is in, and the first and the last sample agree with the oracle."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wk
from gpu_util import to_dev, to_np64

pytestmark = pytest.mark.gpu


# (70, 130, 33) are six tiles of 64 rows: with 148 SMs 16 rows per CTA up to 30 samples, 32 (two CTAs per SM) up to 61, 32 (three) beyond, and
# 64 from 198 on where a tile walks fewer than six key tiles (here at most three); four heads: 16 rows per warp pair up to 98, then 32.
@pytest.mark.parametrize("H,batches", [(8, (1, 20, 30, 31, 61, 62, 110, 198, 230)), (16, (31, 62, 130)), (4, (1, 98, 99, 150))])
@pytest.mark.parametrize("pattern", ["fwd", "all"])
def test_tile_heights(H, batches, pattern):
    import paper_2505_01068_b200 as g
    rng = np.random.default_rng(H)
    seg, most = (70, 130, 33), max(batches)
    phase, mask = (g.PHASE_INTER_FWD, 0) if pattern == "fwd" else (g.PHASE_CUSTOM, 0x1FF)
    q, k, v = wk.draw_qkv(rng, most, sum(seg), H, 8, "bf16")
    valid = np.stack([rng.integers(0, n + 1, size=most) for n in seg], axis=1).astype(np.int32)
    valid[0] = seg
    dev, vl = [to_dev(t, "bf16") for t in (q, k, v)], torch.from_numpy(valid).cuda()
    one = torch.cat([g.im_attention_fwd(*(t[b:b + 1] for t in dev), seg, vl[b:b + 1], phase, mask) for b in range(most)])
    for B in batches:
        out = g.im_attention_fwd(*(t[:B] for t in dev), seg, vl[:B], phase, mask)
        assert torch.equal(out, one[:B]), B
    for b in (0, most - 1):
        ref = oracle.im_attention_dense(q[b:b + 1], k[b:b + 1], v[b:b + 1], seg, valid[b:b + 1], phase, mask)
        err = np.abs(to_np64(one[b:b + 1]) - ref)
        assert err.max() <= 2e-2 and err.mean() <= 2e-3, (b, err.max(), err.mean())
    assert g.last_device_status() == (0, 0)
