"""-m gpu: expert GEMMs on CTA pairs, with weights on M and tokens on N (turned) or, for gate/up, token-major, at the edges of their tiles."""
import numpy as np
import pytest

from paper_2502_04416_b200 import binding, workloads as wl
from tests import parity

pytestmark = pytest.mark.gpu

# token tiles: one group below, at and above 256 rows, equal tiles with a shorter last one; columns in steps of 32.  Neurons: fewer than
# one tile, halves of 8, 16 and 56 neurons per CTA, a last tile that ends early; d: k and output channels that fill no block.
CASES = [
    (256, 16, (257, 300, 400)),
    (256, 24, (256, 257, 300, 511, 513)),
    (328, 200, (287, 1030)),
    (1032, 448, (1000,)),
    (512, 384, (2049, 4100)),
]


@pytest.mark.parametrize("skew", [0.0, 1.0], ids=["even", "skewed"])
@pytest.mark.parametrize("d,m,tokens", CASES, ids=[f"d{c[0]}-m{c[1]}" for c in CASES])
def test_pair_tiles(d, m, tokens, skew):
    shape = wl.LayerShape(d, m * 8, 8, 2, 2, "bf16")
    inp = wl.make_inputs(wl.Workload("pair_tiles", shape, tokens, seed=11))
    lay = inp.layers[0]
    # skewed: one expert takes every row, others a handful or none
    lay.select_bias_b = (skew * np.array([2.0, 0.3, 0.0, -0.3, -2.0, 0.1])).astype(np.float32)
    lay.gate_scale_u = np.random.default_rng(2).normal(scale=0.5, size=6).astype(np.float32)
    layer = parity.gpu_layer(lay, max(tokens))
    layer.set_gemm_path(binding.GEMM_TENSOR_PAIRS)
    for t in tokens:
        st = parity.check_plain_layer(layer, lay, inp.x[:t])
        assert st["differing"] <= st["near_tie"]
    assert layer.status() == 0
    layer.destroy()


# The tiles change which rows are multiplied together, not the sums of one output: same bits as single-CTA tiles, whatever form the
# forced pairs take (see below for each form by itself).
@pytest.mark.parametrize("tokens", [256, 700, 1111])
def test_pair_tiles_have_the_bits_of_single_tiles(tokens):
    import torch
    shape = wl.LayerShape(512, 200 * 8, 8, 2, 2, "bf16")
    inp = wl.make_inputs(wl.Workload("pair_bits", shape, (tokens,), seed=5))
    layer = parity.gpu_layer(inp.layers[0], tokens)
    x = parity.to_device(inp.x, "bf16")
    got = []
    for path in (binding.GEMM_TENSOR, binding.GEMM_TENSOR_PAIRS):
        layer.set_gemm_path(path)
        got.append(layer.forward(x).view(torch.int16).clone())
    assert torch.equal(*got)
    layer.destroy()


def _bits_on_single_tiles_and_pairs(lay, x, forms, path=binding.GEMM_TENSOR_PAIRS):
    import torch
    layer = parity.gpu_layer(lay, len(x))
    xd = parity.to_device(x, "bf16")
    layer.set_gemm_path(binding.GEMM_TENSOR)
    want = layer.forward(xd).view(torch.int16).clone()
    layer.set_gemm_path(path)
    assert layer.gemm_forms(len(x)) == forms
    assert torch.equal(layer.forward(xd).view(torch.int16), want)
    st = parity.check_plain_layer(layer, lay, x)
    assert st["differing"] <= st["near_tie"]
    counts = layer.routing(len(x), lay.shape.n_routed)["counts"]
    assert layer.status() == 0
    layer.destroy()
    return counts


# turned gate/up tiles: one, two (both whole), three and five per group, the last one shorter; neurons that end inside the second tile,
# and halves of 8 per CTA
@pytest.mark.parametrize("m,tokens", [(248, 257), (248, 512), (248, 520), (248, 600), (248, 700), (248, 1111), (16, 257), (16, 300)])
def test_turned_gate_up_has_the_bits_of_single_tiles(m, tokens):
    shape = wl.LayerShape(328, m * 8, 8, 2, 2, "bf16")
    inp = wl.make_inputs(wl.Workload("turned_bits", shape, (tokens,), seed=5))
    _bits_on_single_tiles_and_pairs(inp.layers[0], inp.x, ("turned", "turned"))


# token-major gate/up: the forced choice is made for even loads, so skewed ones bring groups with odd and even numbers of 128-row
# tiles, a single one and none; m as neurons that fill their tiles and end inside them
@pytest.mark.parametrize("m", [200, 448, 864])
@pytest.mark.parametrize("tokens", [1000, 1024, 2048])
def test_token_major_gate_up_has_the_bits_of_single_tiles(tokens, m):
    shape = wl.LayerShape(264, m * 8, 8, 2, 3, "bf16")
    inp = wl.make_inputs(wl.Workload("token_major_bits", shape, (tokens,), seed=8))
    lay = inp.layers[0]
    lay.select_bias_b = np.array([0.5, 0.01, 0.0, -0.01, -0.02, -0.5], np.float32)
    counts = _bits_on_single_tiles_and_pairs(lay, inp.x, ("pair", "turned"))
    tiles = (counts + 127) // 128
    assert counts[5] == 0 and (tiles % 2 == 1).any() and ((tiles % 2 == 0) & (tiles > 0)).any(), counts


# the down GEMM too: large batches whose groups are expected to fill 256-row tiles; K that ends inside a block, channels inside a tile
@pytest.mark.parametrize("skewed", [False, True])
@pytest.mark.parametrize("tokens,m", [(2304, 512), (2300, 520), (3071, 576)])
def test_token_major_down_has_the_bits_of_single_tiles(tokens, m, skewed):
    shape = wl.LayerShape(264, m * 8, 8, 2, 2, "bf16")
    inp = wl.make_inputs(wl.Workload("token_major_down_bits", shape, (tokens,), seed=13))
    lay = inp.layers[0]
    if skewed:
        lay.select_bias_b = np.array([0.5, 0.01, 0.0, -0.01, -0.02, -0.5], np.float32)
    counts = _bits_on_single_tiles_and_pairs(lay, inp.x, ("pair", "pair"), binding.GEMM_AUTO)
    assert not skewed or counts[5] == 0
