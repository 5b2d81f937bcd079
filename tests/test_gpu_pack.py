"""Row plan and gather in one launch against the two separate calls, on both sides of the number of samples that one
CTA can scan (1024)."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch, seg_len, cols", [(1, (1, 0, 3), 4), (3, (50, 500, 500), 64), (86, (5, 0, 9), 32), (1024, (3, 2, 4), 8), (1025, (3, 2, 4), 8)])
def test_plan_pack_matches_separate_calls(batch, seg_len, cols):
    import paper_2505_01068_b200 as g
    gen = torch.Generator().manual_seed(batch)
    L = sum(seg_len)
    vl = torch.stack([torch.randint(0, n + 1, (batch,), generator=gen) for n in seg_len], 1).int().cuda()
    x = torch.randn((batch, L, cols), generator=gen).cuda()
    want_plan = g.plan_rows(vl, seg_len)
    want = torch.full((batch * L, cols), -7.0, device="cuda")
    g.pack_rows(x, want, seg_len, vl, want_plan)
    plan = torch.full((3 * batch + 1,), -1, dtype=torch.int32, device="cuda")
    got = torch.full((batch * L, cols), -7.0, device="cuda")
    shape = g.make_shape(batch, seg_len, 16, 1, vl, g.DTYPE_F32, g.PHASE_INTRA)
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    st = g.load().gsit_plan_pack_rows(ctypes.byref(shape), p(plan), p(x), ctypes.c_int64(cols), p(got), ctypes.c_int64(cols), ctypes.c_int32(cols),
                                      ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0
    assert torch.equal(plan, want_plan) and torch.equal(got, want)
