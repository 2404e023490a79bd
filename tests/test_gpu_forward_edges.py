"""-m gpu: forwards at the edges of what the entry points take."""
import pytest

from oracle import cmoe_oracle as oracle
from paper_2502_04416_b200 import workloads as wl
from tests import parity
from tests.test_gpu_fp8 import _quantised

pytestmark = pytest.mark.gpu


# A top-level router over one outer expert is no plain layer: the layer's copy of the rows is written by its own launches, and
# the weight streamers (experts of at least 128 neurons in all) have no buffers there.
@pytest.mark.parametrize("m,fp8", [(16, False), (16, True), (176, False), (176, True)])
def test_one_outer_expert(m, fp8):
    shape = wl.LayerShape(256, m * 6, 6, 2, 2, "bf16")
    inp = wl.make_inputs(wl.Workload("one_outer", shape, (300,), seed=8, n_outer=1, outer_top_k=1))
    layer = parity.torch_io.layer_from_workload(inp, 300)
    weights = None
    if fp8:
        layer.quantise_fp8()
        weights = [_quantised(lay) for lay in inp.layers]
    for t in (1, 2, 16, 64, 65, 128, 300):
        for x in (inp.x[-t:], inp.x[:t]):           # other rows in the copy than the forward before left there
            st = parity.check_hier_layer(layer, inp, x, expert_weights=weights)
            assert st["differing"] <= st["near_tie"]
    layer.destroy()


# 65535 row tiles of 64 and one more: past what a grid's second dimension can hold
def test_more_rows_than_a_grid_dimension_of_tiles():
    import torch
    tokens, ends = 65535 * 64 + 70, 300
    shape = wl.LayerShape(64, 16 * 2, 2, 1, 1, "bf16")      # one routed expert: nothing to tie
    inp = wl.make_inputs(wl.Workload("many_rows", shape, (2 * ends,), seed=6))
    lay = inp.layers[0]
    layer = parity.gpu_layer(lay, tokens)
    x = torch.zeros(tokens, 64, dtype=torch.bfloat16, device="cuda")
    edge = parity.to_device(inp.x, "bf16")
    x[:ends], x[-ends:] = edge[:ends], edge[ends:]
    out = layer.forward(x)
    torch.cuda.synchronize()
    assert layer.status() == 0
    got = parity.to_host(torch.cat([out[:ends], out[-ends:]]))
    parity.check_output(got, oracle.cmoe_layer_forward(inp.x, **parity.oracle_kwargs(lay))[0])
    assert torch.count_nonzero(out[ends:-ends]) == 0
    layer.destroy()
