"""-m gpu: the clustered router (up to 1024 rows) with its fused permutation and the tile router, at the edges of
its 16-row tiles and row limit, of its 32-wide k slices and of its column tiles."""
import numpy as np
import pytest

from paper_2502_04416_b200 import binding, workloads as wl
from tests import parity

pytestmark = pytest.mark.gpu


def _layer(n_experts, n_shared, top_k, d, tokens, seed=11):
    shape = wl.LayerShape(d, 32 * n_experts, n_experts, n_shared, top_k, "bf16")
    inp = wl.make_inputs(wl.Workload("router_edges", shape, (tokens,), seed=seed))
    lay = inp.layers[0]
    rng = np.random.default_rng(seed)
    lay.gate_scale_u = rng.normal(scale=0.5, size=shape.n_routed).astype(np.float32)
    lay.select_bias_b = rng.normal(scale=0.05, size=shape.n_routed).astype(np.float32)
    return lay, inp.x


# routed experts 1, 8 | 9, 16 | 17, 32 (column tiles 2, 4, 8 and a partly filled one), k slices cut by d = 72, 1032
@pytest.mark.parametrize("n_experts,n_shared,top_k,d", [(3, 2, 1, 256), (9, 1, 8, 72), (11, 2, 3, 1032), (17, 1, 4, 320),
                                                        (18, 1, 4, 2056), (33, 1, 8, 256), (32, 0, 1, 64)])
def test_router_shapes(n_experts, n_shared, top_k, d):
    lay, x = _layer(n_experts, n_shared, top_k, d, 300)
    layer = parity.gpu_layer(lay, 300)
    for t in (1, 15, 16, 17, 300):
        st = parity.check_plain_layer(layer, lay, x[:t])
        assert st["differing"] <= st["near_tie"]
    layer.destroy()


# 384 rows of 8 or 1024 rows of 3 selections: the limit of the fused permutation; 1024 rows: the limit of the router
@pytest.mark.parametrize("top_k,tokens", [(8, (383, 384, 385)), (3, (1023, 1024, 1025))])
def test_router_row_limits(top_k, tokens):
    lay, x = _layer(14, 2, top_k, 128, max(tokens))
    layer = parity.gpu_layer(lay, max(tokens))
    for t in tokens:
        for _ in range(2):                      # the ticket is back at zero after a forward
            st = parity.check_plain_layer(layer, lay, x[:t])
        assert st["differing"] <= st["near_tie"]
    layer.destroy()


@pytest.mark.parametrize("n_routed,n_outer", [(6, 8), (12, 5), (20, 3), (6, 12)])
def test_router_hierarchical_tiles(n_routed, n_outer):
    """Row tiles that span one, several or all outer experts; 12 x 6 groups are too many for the fused permutation."""
    shape = wl.LayerShape(192, 16 * (n_routed + 2), n_routed + 2, 2, 2, "bf16")
    w = wl.Workload("hier_router", shape, (200,), seed=7, n_outer=n_outer, outer_top_k=2)
    inp = wl.make_inputs(w)
    inners = [parity.gpu_layer(lay, 8) for lay in inp.layers]
    layer = binding.Layer.create_hier(parity.to_device(inp.w_router, "bf16"), inners, 2, 200)
    for t in (1, 7, 8, 60, 200):
        st = parity.check_hier_layer(layer, inp, inp.x[:t])
        assert st["differing"] <= st["near_tie"]
    layer.destroy()


# outer experts 1, 8 | 9, 32 (one column tile, four), d cut inside a 32-wide slice, and the 1024 outer rows up to which
# the routers run clustered and the inner one copies the rows
@pytest.mark.parametrize("n_outer,outer_k,d,tokens", [(1, 1, 64, (1, 17)), (8, 2, 192, (16, 512, 513)), (9, 3, 72, (15, 341, 342)),
                                                      (32, 4, 264, (1, 33))])
def test_router_outer_edges(n_outer, outer_k, d, tokens):
    shape = wl.LayerShape(d, 16 * 6, 6, 2, 2, "bf16")
    w = wl.Workload("hier_outer", shape, (max(tokens),), seed=5, n_outer=n_outer, outer_top_k=outer_k)
    inp = wl.make_inputs(w)
    inners = [parity.gpu_layer(lay, 8) for lay in inp.layers]
    layer = binding.Layer.create_hier(parity.to_device(inp.w_router, "bf16"), inners, outer_k, max(tokens))
    for t in tokens:
        st = parity.check_hier_layer(layer, inp, inp.x[:t])
        assert st["differing"] <= st["near_tie"]
    layer.destroy()


# tile routers: rows at the edges of a 64-row tile, of the line at 512 rows, and for clusters of 8, 4, 2 and 1 CTAs; k cut inside
# a block; 32832 rows of 32 experts: more row masks than the one-launch permutation takes
@pytest.mark.parametrize("n_experts,n_shared,top_k,d,tokens", [(20, 2, 4, 1032, (512, 513, 576, 577)), (9, 1, 2, 1032, (1025, 2400)),
                                                               (33, 1, 8, 520, (4800,)), (12, 1, 3, 520, (9601,)),
                                                               (33, 1, 2, 64, (32832,))])
def test_router_tiles(n_experts, n_shared, top_k, d, tokens):
    lay, x = _layer(n_experts, n_shared, top_k, d, max(tokens))
    layer = parity.gpu_layer(lay, max(tokens))
    for t in tokens:
        st = parity.check_plain_layer(layer, lay, x[:t])
        assert st["differing"] <= st["near_tie"]
    layer.destroy()


# outer rows past 1024 (tiles that begin at every expert's first row), tokens past 1024 (top-level router on tiles)
@pytest.mark.parametrize("n_outer,outer_k,tokens", [(9, 2, (520, 1025)), (20, 4, (300, 1090)), (3, 1, (1024, 1025))])
def test_router_tiles_hierarchical(n_outer, outer_k, tokens):
    shape = wl.LayerShape(200, 16 * 6, 6, 2, 2, "bf16")
    w = wl.Workload("hier_tiles", shape, (max(tokens),), seed=3, n_outer=n_outer, outer_top_k=outer_k)
    inp = wl.make_inputs(w)
    inners = [parity.gpu_layer(lay, 8) for lay in inp.layers]
    layer = binding.Layer.create_hier(parity.to_device(inp.w_router, "bf16"), inners, outer_k, max(tokens))
    for t in tokens:
        st = parity.check_hier_layer(layer, inp, inp.x[:t])
        assert st["differing"] <= st["near_tie"]
    layer.destroy()
