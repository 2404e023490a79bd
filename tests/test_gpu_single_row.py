"""-m gpu: one row of a plain layer on both sides of the width up to which the down kernel gives every output channel a warp."""
import numpy as np
import pytest

from paper_2502_04416_b200 import workloads as wl
from tests import parity
from tests.test_gpu_fp8 import _quantised

pytestmark = pytest.mark.gpu


def _channels_per_chip():
    import torch
    return 32 * torch.cuda.get_device_properties(0).multi_processor_count       # 4 blocks of 8 warps on every SM, a channel each


@pytest.mark.parametrize("fp8", [False, True])
@pytest.mark.parametrize("side", [-1, 0, 1])
def test_single_row(side, fp8):
    d = _channels_per_chip() + 16 * side
    inp = wl.make_inputs(wl.Workload("single_row", wl.LayerShape(d, 48 * 8, 8, 2, 2, "bf16"), (2,), seed=12))
    lay = inp.layers[0]
    layer = parity.gpu_layer(lay, 2)
    if fp8:
        layer.quantise_fp8()
    for x in (inp.x[:1], inp.x[1:]):
        st = parity.check_plain_layer(layer, lay, x, expert_weights=_quantised(lay) if fp8 else None)
        assert st["differing"] <= st["near_tie"]
    layer.destroy()


def _lane_order_sums(w_down, h, groups):
    """W_down . h in fp32 in the order of one warp: lane l adds the chunks l, l + 32, ... of eight neurons of a group one after the
    other (products of two bf16 values are exact), the groups' sums follow in order, the lanes meet in a butterfly."""
    out = np.zeros((w_down.shape[0], 32), np.float32)
    for cols in groups:
        chunks = len(cols) // 8
        acc = np.zeros_like(out)
        for run in range(0, chunks, 32):
            n = min(32, chunks - run)
            at = np.asarray(cols)[8 * run:8 * (run + n)].reshape(n, 8)
            for q in range(8):
                acc[:, :n] += w_down[:, at[:, q]] * h[at[:, q]]
        out += acc
    for o in (16, 8, 4, 2, 1):
        out = out + out[:, np.arange(32) ^ o]
    return out[:, 0]


@pytest.mark.parametrize("fp8", [False, True])
@pytest.mark.parametrize("wide", [False, True])
def test_sums_of_a_channel_do_not_depend_on_the_width(wide, fp8):
    m, n, ns = 560, 4, 2                        # rounds of loads that end early: 140 chunks shared, 70 per routed expert
    d = _channels_per_chip() + 128 if wide else m * n
    shape = wl.LayerShape(d, m * n, n, ns, n - ns, "bf16")                       # every expert selected, gates 1
    inp = wl.make_inputs(wl.Workload("single_row_order", shape, (8,), seed=6))
    lay = inp.layers[0]
    lay.gate_scale_u = None
    x = parity.to_device(inp.x, "bf16")

    def forward(w_down):                        # row by row
        lay.w_down = w_down
        layer = parity.gpu_layer(lay, 1)
        if fp8:
            layer.quantise_fp8()                # scales are powers of two: they commute with every rounding
        y = np.stack([parity.to_host(layer.forward(x[t:t + 1].clone()))[0] for t in range(8)])
        layer.destroy()
        return y

    w_down = lay.w_down.copy()
    weights = (_quantised(lay)["w_down"] if fp8 else w_down).astype(np.float32)
    unit = np.zeros_like(w_down)
    unit[np.arange(m * n), np.arange(m * n)] = 1.0
    h = forward(unit)[:, :m * n].astype(np.float32)     # channel c of this layer is hidden activation c itself
    slices = np.asarray(lay.neuron_perm).reshape(n, m)
    want = np.stack([_lane_order_sums(weights, h[t], [slices[:ns].ravel(), *slices[ns:]]) for t in range(8)])
    np.testing.assert_array_equal(forward(w_down), wl.round_to_storage(want, "bf16"))
