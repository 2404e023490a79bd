"""-m gpu: forwards at the edges of what the entry points take."""
import pytest

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
