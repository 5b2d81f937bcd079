"""A linear layer whose CTAs have more tiles each than the table of tile states holds (512): the states beyond it are looked up tile by
tile, by every role for itself.  Some ten million rows of width 64; the same rows in parts, which the table covers, give the same bits."""
import numpy as np
import pytest
import torch

import workloads as wk
from gpu_util import pad_mask, to_dev

pytestmark = pytest.mark.gpu


def test_projection_beyond_the_table():
    import paper_2505_01068_b200 as g
    seg, d, heads = (50, 500, 500), 64, 8
    L, pairs = sum(seg), torch.cuda.get_device_properties(0).multi_processor_count // 2
    inside = pairs * 512 * 256              # rows that the tables of all pairs of CTAs cover
    B = (inside + 8 * pairs * 256) // L     # eight tiles more for each pair
    if torch.cuda.mem_get_info()[0] < 24 << 30:
        pytest.skip("needs 24 GB of device memory")
    rng = np.random.default_rng(3)
    valid = np.tile(np.asarray(seg, dtype=np.int32), (B, 1))
    tail = inside // L
    valid[tail + 10:tail + 20] = 0          # tiles of padding beyond the table
    valid[tail + 30:tail + 40] = np.stack([rng.integers(0, n + 1, size=10) for n in seg], axis=1)
    valid[B // 2:B // 2 + 10] = 0
    x = torch.randn((B, L, d), device="cuda", generator=torch.Generator("cuda").manual_seed(1), dtype=torch.bfloat16)
    w, bias = to_dev(wk.xavier_uniform(rng, 3 * d, d), "bf16"), to_dev(rng.standard_normal(3 * d).astype(np.float32))
    vl, pm = torch.from_numpy(valid).cuda(), torch.from_numpy(pad_mask(seg, valid, B)).cuda()
    x[pm] = float("nan")
    out = torch.full((B, L, 3, heads, d // heads), float("nan"), dtype=torch.bfloat16, device="cuda")
    g.im_qkv_proj(x, w, bias, seg, heads, vl, out=out)
    for lo in range(0, B, 3000):
        hi = min(B, lo + 3000)
        assert torch.equal(out[lo:hi], g.im_qkv_proj(x[lo:hi], w, bias, seg, heads, vl[lo:hi])), lo
    rows = out.reshape(B * L, 3 * d)
    ref = x[-4:].reshape(-1, d).float() @ w.float().T + bias
    assert float((rows[-4 * L:].float() - ref).abs().max()) <= 1e-2 * float(ref.abs().max())

    # the packed layout: shared tiles and tiles outside the call beyond the table as well
    plan = g.plan_rows(vl, seg)
    starts = plan.cpu().numpy()
    real = ~pm.reshape(-1)
    total = int(real.sum())
    assert int(starts[0]) == 0 and int(starts[3 * B]) == total and total > inside + 2 * pairs * 256
    xp = torch.full((B * L, d), float("nan"), dtype=torch.bfloat16, device="cuda")
    xp[:total] = x.reshape(B * L, d)[real]
    want = rows[real]
    del out, rows, x
    lo, hi = 1, B - 1
    packed = torch.full((B * L, 3, heads, d // heads), 7.0, dtype=torch.bfloat16, device="cuda")
    g.im_qkv_proj(xp, w, bias, seg, heads, vl[lo:hi], out=packed, row_start=plan[3 * lo:])
    flat, a, b = packed.reshape(B * L, 3 * d), int(starts[3 * lo]), int(starts[3 * hi])
    assert b > inside and torch.equal(flat[a:b], want[a:b])
    assert bool((flat[:a] == 7.0).all()) and bool((flat[b:] == 7.0).all())
    assert g.last_device_status() == (0, 0)
