"""-m gpu: one row of a plain layer on both sides of the width up to which two warps share a pair of output channels."""
import pytest

from paper_2502_04416_b200 import workloads as wl
from tests import parity
from tests.test_gpu_fp8 import _quantised

pytestmark = pytest.mark.gpu


# 4 blocks of 8 warps on every SM, two channels per pair of warps: 16 channels per SM and block
@pytest.mark.parametrize("fp8", [False, True])
@pytest.mark.parametrize("side", [-1, 0, 1])
def test_single_row(side, fp8):
    import torch
    d = 32 * torch.cuda.get_device_properties(0).multi_processor_count + 16 * side
    inp = wl.make_inputs(wl.Workload("single_row", wl.LayerShape(d, 48 * 8, 8, 2, 2, "bf16"), (2,), seed=12))
    lay = inp.layers[0]
    layer = parity.gpu_layer(lay, 2)
    if fp8:
        layer.quantise_fp8()
    for x in (inp.x[:1], inp.x[1:]):
        st = parity.check_plain_layer(layer, lay, x, expert_weights=_quantised(lay) if fp8 else None)
        assert st["differing"] <= st["near_tie"]
    layer.destroy()
