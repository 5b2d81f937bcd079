"""Kernels of the library may start while the kernel before them still runs; they must not read what that one writes before it has
ended.  Each call is issued right behind a kernel that lets its successor start at once and writes the call's inputs -- all of
them: weights, biases, activations, lengths -- late."""
import numpy as np
import pytest
import torch

import workloads as wk
from gpu_util import to_dev, weights_to_dev

pytestmark = pytest.mark.gpu
SEG = (9, 70, 33)


@pytest.fixture(scope="module")
def g():
    import paper_2505_01068_b200 as lib
    lib.load()
    return lib


class Late:
    """Tensors in one buffer, which a late write fills: `old` contents (other values of the same kind) until then."""

    def __init__(self, g, tensors):
        self.g, sizes = g, [(t.numel() * t.element_size() + 255) // 256 * 256 for t in tensors]
        self.new = torch.zeros(sum(sizes), dtype=torch.uint8, device="cuda")
        self.now, views, off = torch.zeros_like(self.new), [], 0
        for t, n in zip(tensors, sizes):
            at = lambda buf: buf[off:off + t.numel() * t.element_size()].view(t.dtype).view(t.shape)
            at(self.new).copy_(t)
            views.append(at(self.now))
            off += n
        self.views = views
        # old values: the new ones scaled by a half (lengths: one)
        for v, t in zip(views, tensors):
            v.copy_(torch.ones_like(t) if t.dtype == torch.int32 else t * 0.5)
        self.old = self.now.clone()

    def check(self, call):
        """call() must see the new values on every one of several tries."""
        self.now.copy_(self.new)
        want = [t.clone() for t in call()]
        for _ in range(3):
            self.now.copy_(self.old)
            torch.cuda.synchronize()
            self.g.late_write(self.now, self.new)
            got = call()
            torch.cuda.synchronize()
            for a, b in zip(got, want):
                assert torch.equal(a, b)
        assert self.g.last_device_status() == (0, 0)


def _layer(rng, d, dtype):
    w = weights_to_dev(wk.draw_layer_weights(rng, d, 4 * d, dtype, affine=True), dtype)
    return list(w), list(w.values())


@pytest.mark.parametrize("dtype,d,heads,B", [("f32", 32, 4, 2), ("f32", 128, 8, 40), ("f32", 160, 4, 2), ("bf16", 32, 4, 2), ("bf16", 64, 8, 2),
                                             ("bf16", 64, 8, 90), ("bf16", 128, 8, 2), ("bf16", 128, 8, 90), ("bf16", 192, 3, 4)])
def test_layer_behind_a_kernel_that_writes_late(g, dtype, d, heads, B):
    rng = np.random.default_rng(d + B)
    keys, ws = _layer(rng, d, dtype)
    x = torch.randn((B, sum(SEG), d), device="cuda")
    valid = torch.from_numpy(np.stack([rng.integers(1, n + 1, size=B) for n in SEG], axis=1).astype(np.int32)).cuda()
    late = Late(g, [x, valid] + ws)
    xl, vl, w = late.views[0], late.views[1], dict(zip(keys, late.views[2:]))
    late.check(lambda: [g.im_layer_fwd(xl, w, SEG, heads, vl, g.PHASE_INTER_FWD)])


@pytest.mark.parametrize("B", [2, 90])
def test_pair_and_stack_behind_a_kernel_that_writes_late(g, B):
    rng = np.random.default_rng(B)
    keys, wa = _layer(rng, 64, "bf16")
    _, wb = _layer(rng, 64, "bf16")
    _, wi = _layer(rng, 128, "bf16")
    head = [torch.randn((16, 384), device="cuda").bfloat16(), torch.randn(16, device="cuda")]
    x = torch.randn((B, sum(SEG), 64), device="cuda")
    valid = torch.from_numpy(np.stack([rng.integers(1, n + 1, size=B) for n in SEG], axis=1).astype(np.int32)).cuda()
    late = Late(g, [x, valid] + head + wa + wb + wi)
    xl, vl, hl, n = late.views[0], late.views[1], late.views[2:4], len(keys)
    a, b, i = (dict(zip(keys, late.views[4 + k * n:4 + (k + 1) * n])) for k in range(3))
    late.check(lambda: list(g.im_layer_pair_fwd(xl, xl, a, b, SEG, 8, vl)))
    for kw in (dict(), dict(packed=False)):
        stack = g.GsitStack([a], [b], [i], SEG, 8, 8, head=tuple(hl), **kw)
        late.check(lambda: [stack.forward(xl, vl)])
    y = torch.randn((B, sum(SEG), 128), device="cuda")
    rd = Late(g, [y, valid] + head)
    late_stack = g.GsitStack([a], [b], [i], SEG, 8, 8, head=tuple(rd.views[2:4]))
    rd.check(lambda: [late_stack.read_out(rd.views[0], rd.views[1])])


@pytest.mark.parametrize("dtype,d,heads", [("f32", 30, 5), ("f32", 64, 8), ("bf16", 32, 4), ("bf16", 64, 8), ("bf16", 64, 4), ("bf16", 128, 4), ("bf16", 128, 2)])
def test_projection_and_attention_behind_a_kernel_that_writes_late(g, dtype, d, heads):
    rng = np.random.default_rng(d)
    t = torch.float32 if dtype == "f32" else torch.bfloat16
    x = torch.randn((3, sum(SEG), d), device="cuda").to(t)
    w, b = to_dev(wk.xavier_uniform(rng, 3 * d, d), dtype), to_dev(rng.standard_normal(3 * d).astype(np.float32))
    valid = torch.tensor([[9, 70, 33], [2, 41, 1], [1, 64, 17]], dtype=torch.int32, device="cuda")
    late = Late(g, [x, w, b, valid])
    late.check(lambda: [g.im_qkv_proj(late.views[0], late.views[1], late.views[2], SEG, heads, late.views[3])])
    qkv = torch.randn((3, 3, sum(SEG), heads, d // heads), device="cuda").to(t)
    att = Late(g, [qkv, valid])
    for choice in (g.ATTN_DEFAULT, g.ATTN_TMEM):
        g.tune_attention(choice)
        try:
            q = att.views[0]
            att.check(lambda: list(g.im_attention_fwd(q[0], q[1], q[2], SEG, att.views[1], g.PHASE_INTER_BWD, want_lse=True)))
        finally:
            g.tune_attention(g.ATTN_DEFAULT)
