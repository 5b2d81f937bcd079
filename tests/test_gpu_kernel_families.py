"""Small problems run on other kernels than large ones: mma.sync attention instead of the tensor-memory kernels, row tiles instead of
the tcgen05 layer halves.  The checks that other files make at small sizes are made here on the kernels of the large ones:
attention with the tensor-memory family selected, layers above 43 rows per SM."""
import numpy as np
import pytest
import torch

import test_gpu_edge as edge
import test_gpu_rows as rows
import workloads as wk
from gpu_util import to_dev, weights_to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import paper_2505_01068_b200 as lib
    lib.load()
    return lib


@pytest.fixture
def tmem(g):
    g.tune_attention(g.ATTN_TMEM)
    yield
    g.tune_attention(g.ATTN_DEFAULT)


@pytest.mark.parametrize("H,hd", [(8, 8), (2, 8), (4, 16), (8, 16), (2, 32), (4, 32), (2, 64), (1, 64)])
def test_tensor_memory_attention_patterns_and_packed_rows(g, tmem, H, hd):
    edge.test_custom_block_patterns_every_head_width(g, H, hd)
    edge.test_attention_on_packed_rows_equals_padded_layout(g, H, hd)


def test_tensor_memory_attention_random_shapes(g, tmem):
    edge.test_random_shapes_property(g)


def test_tensor_memory_attention_with_and_without_scratch(g, tmem):
    edge.test_attention_with_and_without_scratch_gives_the_same_bits(g)


ABOVE = dict(seg=(50, 300, 271), B=11)   # 6831 rows: above the limit, no multiple of a tile, whole tiles of padding in between


@pytest.mark.parametrize("d,heads,d_ff", [(64, 8, 256), (64, 4, 64), (64, 2, 128), (64, 8, 192), (128, 8, 512), (128, 4, 64), (128, 8, 320)])
def test_tcgen05_halves(g, d, heads, d_ff):
    """Oracle, strided rows, NaN in the padding, the packed layout and the pair call, as for the row tiles."""
    assert ABOVE["B"] * sum(ABOVE["seg"]) > 43 * torch.cuda.get_device_properties(0).multi_processor_count
    rows.check_layer(g, d, heads, d_ff, ABOVE["seg"], ABOVE["B"], tile=128)


@pytest.mark.parametrize("d,heads,d_ff", [(64, 8, 256), (128, 8, 512)])
def test_tcgen05_halves_against_mma_sync_halves(g, d, heads, d_ff):
    rng = np.random.default_rng(d)
    seg, B = ABOVE["seg"], ABOVE["B"]
    x = to_dev(rng.standard_normal((B, sum(seg), d), dtype=np.float32))
    w = weights_to_dev(wk.draw_layer_weights(rng, d, d_ff, "bf16", affine=True), "bf16")
    vl = torch.from_numpy(np.stack([rng.integers(1, n + 1, size=B) for n in seg], axis=1).astype(np.int32)).cuda()
    new = g.im_layer_fwd(x, w, seg, heads, vl, g.PHASE_INTER_BWD)
    g.tune_attention(g.ATTN_LEGACY)
    try:
        err = (new - g.im_layer_fwd(x, w, seg, heads, vl, g.PHASE_INTER_BWD)).abs()
    finally:
        g.tune_attention(g.ATTN_DEFAULT)
    assert 0 < float(err.max()) <= 2e-2 and float(err.mean()) <= 1e-3   # rounding points as in the small test; other kernels: not equal
    assert g.last_device_status() == (0, 0)
