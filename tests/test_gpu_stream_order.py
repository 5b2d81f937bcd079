"""Kernels of the library may start while the kernel before them still runs; they must not read what that one writes before it has
ended.  Each call is issued right behind a kernel that lets its successor start at once and writes the call's inputs -- all of
them: weights, biases, activations, lengths -- late."""
import ctypes

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


@pytest.mark.parametrize("B", [2, 90])
def test_deep_stack_behind_a_kernel_that_writes_late(g, B):
    """Three ring layers and two intra layers with weights of their own.  Two samples: every layer behind the first projection is one launch,
    which reads its parameters above its wait while the launch before it runs; 90: packed rows, the last layer writes the padded result."""
    rng = np.random.default_rng(B)
    sets = [_layer(rng, 64, "bf16") for _ in range(6)] + [_layer(rng, 128, "bf16") for _ in range(2)]
    keys, n = sets[0][0], len(sets[0][0])
    x = torch.randn((B, sum(SEG), 64), device="cuda")
    valid = torch.from_numpy(np.stack([rng.integers(1, n + 1, size=B) for n in SEG], axis=1).astype(np.int32)).cuda()
    late = Late(g, [x, valid] + [t for _, ws in sets for t in ws])
    w = [dict(zip(keys, late.views[2 + k * n:2 + (k + 1) * n])) for k in range(8)]
    stack = g.GsitStack(w[0:3], w[3:6], w[6:8], SEG, 8, 8)
    ring = [g.make_shape(B, SEG, 64, 8, late.views[1], g.DTYPE_BF16, p) for p in (g.PHASE_INTER_FWD, g.PHASE_INTER_BWD)]
    intra = g.make_shape(B, SEG, 128, 8, late.views[1], g.DTYPE_BF16, g.PHASE_INTRA)
    for shapes, d_ff in ((ring, 256), ([intra], 512)):
        p = (ctypes.c_void_p * len(shapes))(*[ctypes.addressof(s) for s in shapes])
        assert g.load().gsit_encoder_runs_chained(p, len(shapes), d_ff) == (B == 2)
    if B == 90:
        plan = g.plan_rows(late.views[1], SEG)
        packed = g.make_shape(B, SEG, 128, 8, late.views[1], g.DTYPE_BF16, g.PHASE_INTRA, row_start=plan, capacity=B * sum(SEG) + 128)
        assert g.load().gsit_layer_scatters(ctypes.byref(packed), 512) == 1
    late.check(lambda: [stack.forward(late.views[0], late.views[1])])


# more items than CTAs are resident, so that the kernel hands them out through the counter in its scratch
@pytest.mark.parametrize("d,heads,choice", [(256, 4, "ATTN_DEFAULT"), (64, 4, "ATTN_TMEM"), (64, 2, "ATTN_TMEM"), (64, 8, "ATTN_TMEM")])
def test_counter_of_the_attention_behind_a_kernel_that_writes_late(g, d, heads, choice):
    """The counter is cleared by a kernel of the call: behind one that leaves something else there late, and behind an attention that is
    still counting."""
    B, hd = 150, d // heads
    rng = np.random.default_rng(d)
    valid = torch.from_numpy(np.stack([rng.integers(1, n + 1, size=B) for n in SEG], axis=1).astype(np.int32)).cuda()
    qkv = torch.randn((3, B, sum(SEG), heads, hd), device="cuda").bfloat16()
    late = Late(g, [qkv, valid, torch.full((64,), 1 << 20, dtype=torch.int32, device="cuda")])
    q, vl, ws = late.views[0], late.views[1], late.views[2].view(torch.uint8)
    g.tune_attention(getattr(g, choice))
    try:
        shape = g.make_shape(B, SEG, d, heads, vl, g.DTYPE_BF16, g.PHASE_INTER_BWD)
        assert g.load().gsit_attention_uses_workspace(ctypes.byref(shape)) == 1
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        tiles = 3 * B   # every segment is one tile of 128 rows
        assert tiles * heads > 8 * sms if hd == 64 else tiles * heads // 2 > 2 * sms
        late.now.copy_(late.new)
        want = g.im_attention_fwd(q[0], q[1], q[2], SEG, vl, g.PHASE_INTER_BWD, out=torch.empty((B, sum(SEG), d), dtype=q.dtype, device="cuda"),
                                  workspace=torch.zeros(256, dtype=torch.uint8, device="cuda")).clone()
        outs = [torch.empty_like(want) for _ in range(2)]
        for _ in range(3):
            late.now.copy_(late.old)
            for o in outs:
                o.fill_(float("nan"))
            torch.cuda.synchronize()
            g.late_write(late.now, late.new)
            for o in outs:
                g.im_attention_fwd(q[0], q[1], q[2], SEG, vl, g.PHASE_INTER_BWD, out=o, workspace=ws)
            torch.cuda.synchronize()
            assert all(torch.equal(o, want) for o in outs)
    finally:
        g.tune_attention(g.ATTN_DEFAULT)
    assert g.last_device_status() == (0, 0)
