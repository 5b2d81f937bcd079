"""The encoder call, the layer call that writes the padded result and the plan that prepares it, called as a C program would: results against
the layer calls, and what they refuse."""
import ctypes

import numpy as np
import pytest
import torch

import workloads as wk
from gpu_util import to_dev, weights_to_dev

pytestmark = pytest.mark.gpu
OK, INVALID, UNSUPPORTED, WORKSPACE = 0, 1, 2, 3
W_FIELDS = ("ln1_g", "ln1_b", "w_qkv", "b_qkv", "w_o", "b_o", "ln2_g", "ln2_b", "w_1", "b_1", "w_2", "b_2")


@pytest.fixture(scope="module")
def g():
    import paper_2505_01068_b200 as lib
    lib.load()
    return lib


def ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def i64(v):
    return ctypes.c_int64(v)


def stream():
    return ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)


def c_weights(g, w, eps=1e-5):
    p = [None if w[k] is None else w[k].data_ptr() for k in W_FIELDS]
    return g.binding.LayerWeights(*p, w["w_1"].shape[0], eps)


def pointers(items):
    return (ctypes.c_void_p * len(items))(*items)


class Encoder:
    """Arguments of gsit_im_encoder_fwd for `problems` x `depth` layers; out[i][j] receives what layer j of problem i writes."""

    def __init__(self, g, seg, d, heads, valid, d_ffs, phases, eps=None, seed=0):
        self.g, self.seg, self.d, self.heads, self.valid, self.phases = g, seg, d, heads, valid, phases
        rng = np.random.default_rng(seed)
        B, n, depth = valid.shape[0], len(phases), len(d_ffs)
        self.x = to_dev(rng.standard_normal((B, sum(seg), d), dtype=np.float32))
        self.w = [[weights_to_dev(wk.draw_layer_weights(rng, d, f, "bf16", affine=True), "bf16") for f in d_ffs] for _ in range(n)]
        self.eps = eps or [[1e-5] * depth for _ in range(n)]
        self.out = [[torch.full_like(self.x, float("nan")) for _ in range(depth)] for _ in range(n)]
        self.shapes = [g.make_shape(B, seg, d, heads, valid, g.DTYPE_BF16, p) for p in phases]
        self.need = n * g.workspace_bytes(self.shapes[0], g.CALL_LAYER, max(d_ffs))

    def call(self, ws_bytes=None, **change):
        self.keep = [[c_weights(self.g, w, e) for w, e in zip(ws, es)] for ws, es in zip(self.w, self.eps)]
        rows = [pointers([ctypes.addressof(w) for w in ws]) for ws in self.keep]
        outs = [pointers([t.data_ptr() for t in o]) for o in self.out]
        n, depth = len(self.phases), len(self.w[0])
        lds = (ctypes.c_int64 * depth)(*[self.d] * depth)
        ws = torch.empty((self.need if ws_bytes is None else ws_bytes) + 256, dtype=torch.uint8, device="cuda")
        base = (ws.data_ptr() + 255) // 256 * 256
        a = dict(shapes=pointers([ctypes.addressof(s) for s in self.shapes]), problems=n, weights=pointers([ctypes.addressof(r) for r in rows]),
                 depth=depth, x=pointers([self.x.data_ptr()] * n), x_stride=(ctypes.c_int64 * n)(*[self.d] * n),
                 y=pointers([ctypes.addressof(o) for o in outs]), y_stride=pointers([ctypes.addressof(lds)] * n))
        a.update(change)
        st = self.g.load().gsit_im_encoder_fwd(a["shapes"], a["problems"], a["weights"], a["depth"], a["x"], a["x_stride"], a["y"], a["y_stride"],
                                               ctypes.c_void_p(base), ctypes.c_size_t(self.need if ws_bytes is None else ws_bytes), stream())
        torch.cuda.synchronize()
        return st

    def want(self):
        res = []
        for p, ws, es in zip(self.phases, self.w, self.eps):
            cur, mine = self.x, []
            for w, e in zip(ws, es):
                cur = self.g.im_layer_fwd(cur, w, self.seg, self.heads, self.valid, p, ln_eps=e)
                mine.append(cur)
            res.append(mine)
        return res


def lengths(seg, B, seed=1):
    rng = np.random.default_rng(seed)
    return torch.from_numpy(np.stack([rng.integers(0, n + 1, size=B) for n in seg], axis=1).astype(np.int32)).cuda()


SEG = (17, 130, 64)


# (width, heads, samples): layers of one launch, row tiles with head_dim 64, tcgen05 halves
@pytest.mark.parametrize("d,heads,B", [(64, 8, 2), (32, 4, 3), (64, 1, 2), (64, 8, 80)])
@pytest.mark.parametrize("problems", [1, 2])
def test_encoder_equals_layer_calls(g, d, heads, B, problems):
    """Equal widths of the MLP, widths that differ in depth, and an eps that differs in depth (one per layer) or between two problems
    (then the layers run one by one)."""
    phases = [g.PHASE_INTER_FWD, g.PHASE_INTER_BWD][:problems]
    cases = [((128, 128, 128), None), ((128, 64, 192), None), ((64,), None), ((128, 64), [[1e-5, 1e-3]] * problems)]
    if problems == 2:
        cases.append(((128, 128), [[1e-5, 1e-5], [1e-5, 1e-2]]))
    for d_ffs, eps in cases:
        e = Encoder(g, SEG, d, heads, lengths(SEG, B), d_ffs, phases, eps, seed=len(d_ffs))
        assert e.call() == OK
        for got, want in zip(e.out, e.want()):
            assert all(torch.equal(a, b) for a, b in zip(got, want)), (d_ffs, eps)
    assert g.last_device_status() == (0, 0)


def test_encoder_refuses(g):
    phases = [g.PHASE_INTER_FWD, g.PHASE_INTER_BWD]
    new = lambda **kw: Encoder(g, SEG, 64, 8, lengths(SEG, 2), (128, 128), phases, **kw)
    e = new()
    assert g.load().gsit_encoder_runs_chained(pointers([ctypes.addressof(s) for s in e.shapes]), 2, 128) == 1
    for name in ("shapes", "weights", "x", "x_stride", "y", "y_stride"):
        assert e.call(**{name: None}) == INVALID, name
    for change in (dict(problems=0), dict(problems=3), dict(depth=0), dict(x=pointers([e.x.data_ptr(), None])), dict(x=pointers([e.x.data_ptr(), e.x.data_ptr() + 4])),
                   dict(x_stride=(ctypes.c_int64 * 2)(64, 60)), dict(x_stride=(ctypes.c_int64 * 2)(66, 66)), dict(shapes=pointers([ctypes.addressof(e.shapes[0]), None]))):
        assert e.call(**change) == INVALID, change
    assert e.call(ws_bytes=e.need - 1) == WORKSPACE
    assert new().call(ws_bytes=0) == WORKSPACE
    other = new()
    other.shapes[1] = g.make_shape(2, (17, 130, 63), 64, 8, other.valid, g.DTYPE_BF16, phases[1])   # not the same geometry
    assert other.call() == INVALID
    widths = new()
    widths.w[1][1] = weights_to_dev(wk.draw_layer_weights(np.random.default_rng(0), 64, 64, "bf16"), "bf16")   # d_ff differs between the problems
    assert widths.call() == INVALID
    odd = new()
    odd.out[1][0] = torch.empty(odd.x.numel() + 1, device="cuda")[1:]   # not 16-byte aligned
    assert odd.call() == INVALID
    assert all(torch.isnan(t).all() for t in e.out[0] + e.out[1]) and g.last_device_status() == (0, 0)   # nothing was launched


def scatter_args(g, B, seg=(50, 300, 270), d=128, heads=4):
    rng = np.random.default_rng(B)
    vl = lengths(seg, B, seed=B)
    x = to_dev(rng.standard_normal((B, sum(seg), d), dtype=np.float32))
    w = weights_to_dev(wk.draw_layer_weights(rng, d, 2 * d, "bf16", affine=True), "bf16")
    return seg, vl, x, w, B * sum(seg) + 128


def test_layer_on_packed_rows_that_writes_the_padded_result(g):
    seg, vl, x, w, cap = scatter_args(g, 12)
    B, L, d = x.shape
    lib, plain = g.load(), g.make_shape(B, seg, 16, 1, vl, g.DTYPE_F32, g.PHASE_INTRA)
    plan = torch.full((3 * B + 1,), -1, dtype=torch.int32, device="cuda")
    row_map = torch.full((cap,), -1, dtype=torch.int32, device="cuda")
    # the plan's own columns are half as wide as the result it clears
    half = x[:, :, :64].contiguous()
    xp = torch.zeros((cap, 64), device="cuda")
    y = torch.full((B, L, d), float("nan"), device="cuda")
    args = lambda **kw: [kw.get("shape", ctypes.byref(plain)), kw.get("plan", ptr(plan)), kw.get("row_map", ptr(row_map)), kw.get("x", ptr(half)), i64(64), ptr(xp),
                         i64(64), ctypes.c_int32(64), kw.get("y", ptr(y)), i64(kw.get("y_stride", d)), stream()]
    fn = lib.gsit_plan_pack_map_rows
    for bad in (dict(row_map=None), dict(y=None), dict(y=ctypes.c_void_p(y.data_ptr() + 4)), dict(y_stride=127), dict(y_stride=130), dict(plan=None), dict(x=None), dict(shape=None)):
        assert fn(*args(**bad)) == INVALID, bad
    assert fn(*args()) == OK
    assert torch.equal(plan, g.plan_rows(vl, seg))
    pad = torch.from_numpy(wk.padded_row_mask(seg, vl.cpu().numpy(), B)).cuda()
    real = (~pad).view(-1).nonzero().view(-1).int()
    assert torch.equal(row_map[:real.numel()], real) and torch.equal(xp[:real.numel()], half.view(-1, 64)[real.long()])
    assert bool((y[pad] == 0).all()) and not bool(torch.signbit(y[pad]).any()) and bool(torch.isnan(y[~pad]).all())

    packed = g.make_shape(B, seg, d, 4, vl, g.DTYPE_BF16, g.PHASE_INTRA, row_start=plan, capacity=cap)
    assert lib.gsit_layer_scatters(ctypes.byref(packed), 2 * d) == 1
    rows = torch.zeros((cap, d), device="cuda")
    g.pack_rows(x, rows, seg, vl, plan)
    cw, n = c_weights(g, w), g.workspace_bytes(packed, g.CALL_LAYER, 2 * d)
    ws = torch.empty(n, dtype=torch.uint8, device="cuda")
    call = lambda shape, m, size: lib.gsit_im_layer_scatter_fwd(ctypes.byref(shape), ctypes.byref(cw), ptr(rows), i64(d), m, ptr(y), i64(d), ptr(ws), ctypes.c_size_t(size), stream())
    assert call(packed, None, n) == INVALID
    assert call(packed, ptr(row_map), n - 1) == WORKSPACE
    padded = g.make_shape(B, seg, d, 4, vl, g.DTYPE_BF16, g.PHASE_INTRA)
    assert lib.gsit_layer_scatters(ctypes.byref(padded), 2 * d) == 0 and call(padded, ptr(row_map), n) == UNSUPPORTED
    assert call(packed, ptr(row_map), n) == OK
    assert torch.equal(y, g.im_layer_fwd(x, w, seg, 4, vl, g.PHASE_INTRA))
    assert g.last_device_status() == (0, 0)


def test_a_layer_on_small_row_tiles_does_not_scatter(g):
    seg, vl, x, w, cap = scatter_args(g, 2)
    plan = g.plan_rows(vl, seg)
    packed = g.make_shape(2, seg, 128, 4, vl, g.DTYPE_BF16, g.PHASE_INTRA, row_start=plan, capacity=cap)
    n = g.workspace_bytes(packed, g.CALL_LAYER, 256)
    ws, rows, y = torch.empty(n, dtype=torch.uint8, device="cuda"), torch.zeros((cap, 128), device="cuda"), torch.full_like(x, 3.0)
    m = torch.zeros(cap, dtype=torch.int32, device="cuda")
    cw = c_weights(g, w)
    assert g.load().gsit_layer_scatters(ctypes.byref(packed), 256) == 0
    assert g.load().gsit_im_layer_scatter_fwd(ctypes.byref(packed), ctypes.byref(cw), ptr(rows), i64(128), ptr(m), ptr(y), i64(128), ptr(ws), ctypes.c_size_t(n),
                                              stream()) == UNSUPPORTED
    assert bool((y == 3.0).all())


def test_map_of_more_samples_than_one_cta_can_scan_is_refused(g):
    B, seg = 1025, (3, 2, 4)
    vl = lengths(seg, B)
    x, xp, y = torch.zeros((B, 9, 8), device="cuda"), torch.zeros((B * 9, 8), device="cuda"), torch.full((B, 9, 16), 3.0, device="cuda")
    plan, m = torch.zeros(3 * B + 1, dtype=torch.int32, device="cuda"), torch.zeros(B * 9, dtype=torch.int32, device="cuda")
    shape = g.make_shape(B, seg, 16, 1, vl, g.DTYPE_F32, g.PHASE_INTRA)
    assert g.load().gsit_plan_pack_map_rows(ctypes.byref(shape), ptr(plan), ptr(m), ptr(x), i64(8), ptr(xp), i64(8), ctypes.c_int32(8), ptr(y), i64(16), stream()) == UNSUPPORTED
    assert bool((y == 3.0).all()) and not bool(plan.any())
