"""A layer behind its projection in one launch (attention, out-projection, LN2, MLP, the next layer's first half): the same bits as the
separate kernels, which serve the same samples inside a batch whose walks are too long for it, at both heights of its row tiles."""
import ctypes

import numpy as np
import pytest
import torch

import workloads as wk
from gpu_util import to_dev, weights_to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import paper_2505_01068_b200 as lib
    lib.load()
    return lib


# segments around tile edges (16, 32, 64 rows) with one of more than eight key tiles: nine samples are two waves of long walks
@pytest.mark.parametrize("seg", [(33, 577, 47), (16, 640, 15), (1, 560, 65)])
@pytest.mark.parametrize("d,heads,d_ff", [(64, 8, 256), (64, 4, 64), (64, 2, 192), (128, 8, 512), (128, 4, 64), (32, 4, 128), (32, 2, 512), (32, 1, 64)])
def test_same_bits_as_separate_kernels(g, d, heads, d_ff, seg):
    rng = np.random.default_rng(d + heads + seg[0])
    B = 30 if d == 32 else 9
    x = to_dev(rng.standard_normal((B, sum(seg), d), dtype=np.float32))
    w = weights_to_dev(wk.draw_layer_weights(rng, d, d_ff, "bf16", affine=True), "bf16")
    valid = np.stack([rng.integers(n // 2, n + 1, size=B) for n in seg], axis=1).astype(np.int32)
    valid[1] = [seg[0], 0, seg[2]]
    valid[2] = 0
    vl = torch.from_numpy(valid).cuda()
    for phase in (g.PHASE_INTER_FWD, g.PHASE_INTER_BWD, g.PHASE_INTRA):
        want = g.im_layer_fwd(x, w, seg, heads, vl, phase)
        for lo, hi in ((0, 1), (1, 3), (3, 7)):   # one sample: small tiles; four: large ones
            assert torch.equal(g.im_layer_fwd(x[lo:hi], w, seg, heads, vl[lo:hi], phase), want[lo:hi]), (phase, lo)
    assert g.last_device_status() == (0, 0)


@pytest.mark.parametrize("d,heads,intra_heads", [(64, 8, 8), (64, 2, 4), (32, 4, 4)])
@pytest.mark.parametrize("B", [1, 5])
def test_chained_layers_equal_layer_calls(g, d, heads, intra_heads, B):
    """Rings and intra encoder of depth 3 in one call each, without biases and with: the bits of one call per layer."""
    rng = np.random.default_rng(B)
    seg = (17, 130, 64)
    for affine in (True, False):
        layers = lambda width: [weights_to_dev(wk.draw_layer_weights(rng, width, 2 * width, "bf16", affine=affine), "bf16") for _ in range(3)]
        fwd, bwd, intra = layers(d), layers(d), layers(2 * d)
        x = to_dev(rng.standard_normal((B, sum(seg), d), dtype=np.float32))
        vl = torch.from_numpy(np.stack([rng.integers(1, n + 1, size=B) for n in seg], axis=1).astype(np.int32)).cuda()
        a, b = x, x
        for wa, wb in zip(fwd, bwd):
            a, b = (g.im_layer_fwd(a, wa, seg, heads, vl, g.PHASE_INTER_FWD), g.im_layer_fwd(b, wb, seg, heads, vl, g.PHASE_INTER_BWD))
        want = torch.cat([a, b], dim=2)
        for wi in intra:
            want = g.im_layer_fwd(want, wi, seg, intra_heads, vl, g.PHASE_INTRA)
        for packed in (True, False):
            assert torch.equal(g.GsitStack(fwd, bwd, intra, seg, heads, intra_heads, packed=packed).forward(x, vl), want)
    assert g.last_device_status() == (0, 0)


# Beyond one wave of the one-launch kernel's CTAs; (phases, with no valid_len: one launch?) -- a second wave of long walks costs more than
# the launches it saves, one of short walks behind them does not
@pytest.mark.parametrize("B,seg,d,heads,routes", [
    (6, (50, 500, 500), 64, 8, {(2,): 0, (0,): 1, (0, 1): 0}), (32, (50, 52, 52), 64, 4, {(2,): 0}), (4, (50, 500, 500), 64, 8, {(0, 1): 1}),
    (25, (50, 52, 52), 128, 8, {(2,): 0}), (5, (50, 500, 500), 128, 8, {(2,): 1}), (54, (50, 52, 52), 32, 4, {(2,): 0}), (8, (50, 500, 500), 32, 4, {(0, 1): 1})])
def test_full_lengths_known_to_the_host(g, B, seg, d, heads, routes):
    """Without valid_len every length is full and the launch is chosen by the walks that follow from it; with lengths that are full as
    well, by what padding usually leaves.  The same bits either way."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("sizes chosen for 148 SMs")
    rng = np.random.default_rng(B)
    full = torch.tensor([seg] * B, dtype=torch.int32, device="cuda")
    x = to_dev(rng.standard_normal((B, sum(seg), d), dtype=np.float32))
    w = [weights_to_dev(wk.draw_layer_weights(rng, d, 2 * d, "bf16", affine=True), "bf16") for _ in range(2)]
    fn = g.load().gsit_encoder_runs_chained
    for phases, one_launch in routes.items():
        shapes = [g.make_shape(B, seg, d, heads, None, g.DTYPE_BF16, p) for p in phases]
        assert fn((ctypes.c_void_p * 2)(*[ctypes.addressof(s) for s in shapes]), len(phases), 2 * d) == one_launch, phases
        if len(phases) == 1:
            a, b = (g.im_layer_fwd(x, w[0], seg, heads, v, phases[0]) for v in (None, full))
        else:
            a, b = (torch.cat(g.im_layer_pair_fwd(x, x, w[0], w[1], seg, heads, v), 2) for v in (None, full))
        assert torch.equal(a, b), phases
    assert g.last_device_status() == (0, 0)


# Beyond one wave with lengths that only the device knows: by walks of two thirds of the segments.  Segments of one tile keep their CTAs
# however few rows are real; at width 128 an encoder's other choice are packed rows.
@pytest.mark.parametrize("B,seg,d,phases,one_launch", [
    (54, (50, 52, 52), 32, (2,), 0), (23, (50, 180, 180), 32, (2,), 1), (30, (50, 52, 52), 32, (2,), 1), (42, (21, 43, 34), 64, (0, 1), 0),
    (5, (50, 500, 500), 64, (0, 1), 1), (25, (30, 26, 146), 128, (2,), 0), (5, (50, 500, 500), 128, (2,), 1)])
def test_lengths_only_the_device_knows(g, B, seg, d, phases, one_launch):
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("sizes chosen for 148 SMs")
    rng = np.random.default_rng(B)
    vl = torch.from_numpy(np.stack([rng.integers(0, n + 1, size=B) for n in seg], axis=1).astype(np.int32)).cuda()
    shapes = [g.make_shape(B, seg, d, 8 if d > 32 else 4, vl, g.DTYPE_BF16, p) for p in phases]
    assert g.load().gsit_encoder_runs_chained((ctypes.c_void_p * 2)(*[ctypes.addressof(s) for s in shapes]), len(phases), 64) == one_launch
    x = to_dev(rng.standard_normal((B, sum(seg), d), dtype=np.float32))
    w = [weights_to_dev(wk.draw_layer_weights(rng, d, 64, "bf16", affine=True), "bf16") for _ in phases]
    run = lambda x, v: torch.cat([g.im_layer_fwd(x, w[0], seg, shapes[0].heads, v, phases[0])] if len(phases) == 1 else
                                 g.im_layer_pair_fwd(x, x, w[0], w[1], seg, shapes[0].heads, v), 2)
    want = torch.cat([run(x[b:b + 1], vl[b:b + 1]) for b in range(B)])
    assert torch.equal(run(x, vl), want)
    assert g.last_device_status() == (0, 0)
