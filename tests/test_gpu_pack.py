"""Row plan and gather in one launch against the two separate calls, on both sides of the number of samples that one
CTA can scan (1024); the stack whose last layer writes the padded result itself."""
import ctypes

import numpy as np
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


@pytest.mark.parametrize("intra_depth", [1, 2])
@pytest.mark.parametrize("d", [32, 64])
def test_stack_result_in_the_padded_layout(d, intra_depth):
    """Above the row limit of the small tiles the stack packs rows; at width 64 its last layer (128 wide) writes the padded result itself, at
    32 a scatter does.  Padded layout throughout and packed: equal bit for bit, padding +0 in a buffer that held NaN, input a view
    of the result buffer of the call before."""
    import paper_2505_01068_b200 as g
    import workloads as wk
    from gpu_util import weights_to_dev
    rng = np.random.default_rng(d)
    seg, B = (50, 300, 270), 12
    layers = lambda width, n: [weights_to_dev(wk.draw_layer_weights(rng, width, 2 * width, "bf16", affine=True), "bf16") for _ in range(n)]
    fwd, bwd, intra = layers(d, 1), layers(d, 1), layers(2 * d, intra_depth)
    valid = np.stack([rng.integers(0, n + 1, size=B) for n in seg], axis=1).astype(np.int32)
    valid[3], valid[7] = 0, seg
    vl = torch.from_numpy(valid).cuda()
    x = torch.from_numpy(rng.standard_normal((B, sum(seg), d), dtype=np.float32)).cuda()
    want = g.GsitStack(fwd, bwd, intra, seg, 4, 4, packed=False).forward(x, vl).clone()
    out = torch.full((B, sum(seg), 2 * d), float("nan"), device="cuda")
    out[:, :, d:] = x
    st = g.GsitStack(fwd, bwd, intra, seg, 4, 4)
    got = st.forward(out[:, :, d:], vl, out=out)
    assert st.packed and torch.equal(got, want)
    assert not torch.signbit(got[torch.from_numpy(wk.padded_row_mask(seg, valid, B)).cuda()]).any()
    assert g.last_device_status() == (0, 0)


@pytest.mark.parametrize("B,intra_depth", [(12, 1), (2, 0), (2, 1), (12, 0)])
@pytest.mark.parametrize("padded", [False, True])
def test_stack_input_anywhere_in_the_result(B, intra_depth, padded):
    """The input of a stack may lie in its result, row for row or in any other mapping: packed rows (12 samples; the last layer at width
    128 could write the padded result itself), layers of one launch (2 samples), rings whose only layer also writes the result."""
    import paper_2505_01068_b200 as g
    import workloads as wk
    from gpu_util import weights_to_dev
    rng = np.random.default_rng(B)
    seg, d = (50, 300, 270), 64
    layers = lambda width, n: [weights_to_dev(wk.draw_layer_weights(rng, width, 2 * width, "bf16", affine=True), "bf16") for _ in range(n)]
    st = g.GsitStack(layers(d, 1), layers(d, 1), layers(2 * d, intra_depth), seg, 4, 4, packed=not padded)
    vl = torch.from_numpy(np.stack([rng.integers(0, n + 1, size=B) for n in seg], axis=1).astype(np.int32)).cuda()
    x = torch.from_numpy(rng.standard_normal((B, sum(seg), d), dtype=np.float32)).cuda()
    for valid in (vl, None):
        want = st.forward(x, valid).clone()
        out = torch.empty((B, sum(seg), 2 * d), device="cuda")
        flat = out.view(-1)
        views = [out[:, :, :d], out[:, :, d:], flat[:x.numel()].view(x.shape), flat[x.numel():].view(x.shape), flat[d // 2 * 3:][:x.numel()].view(x.shape)]
        for v in views:
            out.fill_(float("nan"))
            v.copy_(x)
            assert torch.equal(st.forward(v, valid, out=out), want)
        mine = st.forward(x, valid)   # the object's own buffer
        view = mine.view(-1)[x.numel():].view(x.shape)
        view.copy_(x)
        assert torch.equal(st.forward(view, valid), want)
    assert g.last_device_status() == (0, 0)
