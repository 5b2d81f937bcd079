"""What the native argument marshalling passes on and accepts: torch's own exception types, weights in any mapping, a type per layer."""
import collections

import numpy as np
import pytest
import torch

import workloads as wk
from gpu_util import weights_to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import paper_2505_01068_b200 as lib
    lib.load()
    return lib


def test_failed_allocation_raises_torch_out_of_memory_error(g):
    """Callers catch torch.OutOfMemoryError to go on with a smaller batch.  The limit is one of this process's allocator."""
    seg, d = (1024, 2048, 1024), 512
    x = torch.zeros((8, sum(seg), d), device="cuda", dtype=torch.bfloat16)
    w = torch.zeros((3 * d, d), device="cuda", dtype=torch.bfloat16)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    torch.cuda.set_per_process_memory_fraction((torch.cuda.memory_reserved() + (16 << 20)) / torch.cuda.get_device_properties(0).total_memory)
    try:
        with pytest.raises(torch.OutOfMemoryError):
            g.im_qkv_proj(x, w, None, seg, 8)                       # the result is 100 MB
        half = g.im_qkv_proj(x[:1, :], w, None, seg, 8)             # 12.6 MB: fits
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert bool((half == 0).all()) and g.last_device_status() == (0, 0)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_weights_in_any_mapping(g, dtype):
    """An nn.ParameterDict without the optional vectors, an OrderedDict, and a mapping that makes its tensors when asked."""
    rng = np.random.default_rng(0)
    seg, d = (5, 40, 21), 64
    w = {k: t for k, t in weights_to_dev(wk.draw_layer_weights(rng, d, 4 * d, dtype), dtype).items() if t is not None}
    x = torch.randn((2, sum(seg), d), device="cuda")
    call = lambda m: g.im_layer_fwd(x, m, seg, 8)

    class Made(collections.abc.Mapping):
        __len__, __iter__ = (lambda self: len(w)), (lambda self: iter(w))
        __getitem__ = lambda self, k: w[k].clone()

    ref = call(w)
    assert torch.equal(ref, call(torch.nn.ParameterDict({k: torch.nn.Parameter(t, requires_grad=False) for k, t in w.items()})))
    assert torch.equal(ref, call(collections.OrderedDict(w)))
    for _ in range(3):
        assert torch.equal(ref, call(Made()))
    ya, yb = g.im_layer_pair_fwd(x, x, Made(), torch.nn.ParameterDict(w), seg, 8, None, g.PHASE_INTER_FWD, g.PHASE_INTER_FWD)
    assert torch.equal(ya, ref) and torch.equal(yb, ref)
    for m in (dict, collections.OrderedDict):
        with pytest.raises(KeyError):
            call(m({k: t for k, t in w.items() if k != "w_o"}))
    with pytest.raises(TypeError):
        call([w])


@pytest.mark.parametrize("types", [("f32", "f32", "bf16"), ("bf16", "bf16", "f32"), ("bf16", "f32", "bf16"), ("f32", "bf16", "f32")])
@pytest.mark.parametrize("padded", [False, True])
def test_stack_runs_every_layer_in_the_type_of_its_weights(g, types, padded):
    """Rings and intra encoder of different types, and MLP widths that differ from layer to layer: the bits of the layers called
    one by one, whichever way the stack issues them."""
    rng = np.random.default_rng(1)
    seg, d, B, H, IH = (5, 70, 33), 32, 3, 4, 4
    layers = lambda width, t, ffs: [weights_to_dev(wk.draw_layer_weights(rng, width, f, t, affine=True), t) for f in ffs]
    fwd, bwd, intra = layers(d, types[0], (64, 128)), layers(d, types[1], (64, 192)), layers(2 * d, types[2], (128, 256))
    x = torch.randn((B, sum(seg), d), device="cuda")
    vl = torch.tensor([[5, 70, 33], [2, 41, 0], [1, 64, 17]], dtype=torch.int32, device="cuda") if padded else None

    def chain(cur, ws, heads, phase):
        for w in ws:
            cur = g.im_layer_fwd(cur, w, seg, heads, vl, phase)
        return cur

    want = chain(torch.cat([chain(x, fwd, H, g.PHASE_INTER_FWD), chain(x, bwd, H, g.PHASE_INTER_BWD)], dim=2), intra, IH, g.PHASE_INTRA)
    for kw in (dict(), dict(packed=False), dict(paired_rings=False), dict(paired_rings=False, concurrent_rings=False)):
        got = g.GsitStack(fwd, bwd, intra, seg, H, IH, **kw).forward(x, vl).clone()
        torch.cuda.synchronize()
        assert torch.equal(got, want), kw
    assert g.last_device_status() == (0, 0)


def test_weights_of_two_types_in_one_layer_are_refused(g):
    """The type of w_qkv is the type every matrix of the call is read in."""
    seg, d = (5, 9, 3), 32
    w = [weights_to_dev(wk.draw_layer_weights(np.random.default_rng(2), d, 64, "bf16"), t) for t in ("bf16", "f32")]
    x = torch.randn((1, sum(seg), d), device="cuda")
    with pytest.raises(AssertionError):
        g.im_layer_fwd(x, dict(w[1], w_2=w[0]["w_2"]), seg, 4)
    with pytest.raises(AssertionError):
        g.im_layer_pair_fwd(x, x, w[0], w[1], seg, 4)


def test_projection_and_read_out_refuse_other_types(g):
    """The projection reads its weights in the type of x, biases are float32: anything else would be read past its end."""
    seg, d = (5, 9, 3), 64
    x, w, b = torch.randn((1, sum(seg), d), device="cuda"), torch.randn((3 * d, d), device="cuda"), torch.randn(3 * d, device="cuda")
    g.im_qkv_proj(x, w, b, seg, 8)
    g.im_qkv_proj(x.bfloat16(), w.bfloat16(), b, seg, 8)
    for args in ((x, w.bfloat16(), b), (x.bfloat16(), w, b), (x, w, b.bfloat16()), (x, w, torch.randn(6 * d, device="cuda")[::2])):
        with pytest.raises(AssertionError):
            g.im_qkv_proj(*args, seg, 8)
    w_f = torch.randn((7, 3 * d), device="cuda")
    g.stack_head_fwd(x, w_f, b[:7].contiguous(), seg)
    with pytest.raises(AssertionError):
        g.stack_head_fwd(x, w_f, b[:7].bfloat16(), seg)
