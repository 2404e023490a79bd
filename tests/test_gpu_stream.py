"""-m gpu: the weight streamers of plain bf16 layers for 2 to 64 rows (gates folded into the hidden activations, down
projection over all active experts at once), at the edges of their tiles, k blocks, runs and token columns."""
import numpy as np
import pytest

from paper_2502_04416_b200 import workloads as wl
from tests import parity
from tests.test_gpu_fp8 import _quantised

pytestmark = pytest.mark.gpu


def _check(d, m, n_experts, n_shared, top_k, tokens, seed=5, fp8=False):
    shape = wl.LayerShape(d, m * n_experts, n_experts, n_shared, top_k, "bf16")
    inp = wl.make_inputs(wl.Workload("stream_edges", shape, (max(tokens),), seed=seed))
    lay = inp.layers[0]
    rng = np.random.default_rng(seed)
    lay.gate_scale_u = rng.normal(scale=0.5, size=shape.n_routed).astype(np.float32)
    layer = parity.gpu_layer(lay, max(tokens))
    weights = None
    if fp8:
        layer.quantise_fp8()
        weights = _quantised(lay)
    for t in tokens:
        for _ in range(2):                   # the tickets are back at zero after a forward
            st = parity.check_plain_layer(layer, lay, inp.x[:t], expert_weights=weights)
        if top_k:
            assert st["differing"] <= st["near_tie"]
        if top_k and t <= 64:                # router, up and down kernel, FP8: two splits; no combine
            assert st["launches"] == (5 if fp8 else 3)
    layer.destroy()


# token columns 16 / 32 / 64 and their neighbours; few and nearly all experts active
@pytest.mark.parametrize("tokens", [(2, 3, 15, 16, 17), (31, 32, 33), (63, 64)])
@pytest.mark.parametrize("n_experts,n_shared,top_k", [(8, 2, 2), (32, 4, 4)])
def test_stream_token_columns(n_experts, n_shared, top_k, tokens):
    _check(256, 176, n_experts, n_shared, top_k, tokens)


@pytest.mark.parametrize("d,m,n_experts,n_shared,top_k", [
    (72, 200, 8, 2, 2),          # k and channel tails, group width neither a multiple of 16 nor of 64
    (1032, 24, 9, 1, 8),         # groups narrower than a tile
    (64, 800, 33, 1, 8),         # more tiles than SMs: several rounds of the up kernel, both accumulators in use
    (4096, 32, 4, 1, 1),         # two k blocks per channel tile: a run of the down kernel spans whole tiles
    (2048, 64, 4, 0, 2),         # no shared expert
    (192, 640, 6, 4, 1),         # wide shared expert
])
def test_stream_shapes(d, m, n_experts, n_shared, top_k):
    _check(d, m, n_experts, n_shared, top_k, (2, 9, 40))


def test_stream_shared_only():
    _check(320, 136, 4, 4, 0, (5, 50))


# FP8 codes: group widths of whole and partial 128-wide k blocks, token boxes of 16 to 64 rows, and the batches of
# 65 to 128 rows that read the bf16 copies
@pytest.mark.parametrize("d,m,n_experts,n_shared,top_k,tokens", [
    (256, 176, 8, 2, 2, (2, 16, 17, 33, 48, 49, 64, 65, 128)),
    (1040, 448, 32, 4, 4, (3, 64)),
    (64, 800, 33, 1, 8, (5, 64)),
    (4096, 32, 4, 1, 1, (2, 40)),
    (2048, 64, 4, 0, 2, (9,)),
    (320, 144, 4, 4, 0, (5, 50)),
])
def test_stream_fp8(d, m, n_experts, n_shared, top_k, tokens):
    _check(d, m, n_experts, n_shared, top_k, tokens, fp8=True)
