"""-m gpu: forwards at the edges of what the entry points take."""
import numpy as np
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


# An expert's weights reach only the tokens that selected it, whatever they hold: 0 x Inf is NaN, so a sum over all active
# experts would carry a single Inf of W_down to every token of the batch.
@pytest.mark.parametrize("fp8,value", [(False, np.inf), (False, np.nan), (True, np.nan)])
def test_non_finite_down_weight_stays_with_its_expert(fp8, value):
    import torch
    shape = wl.LayerShape(256, 176 * 8, 8, 2, 2, "bf16")
    inp = wl.make_inputs(wl.Workload("non_finite", shape, (65,), seed=3))
    lay, expert, channel = inp.layers[0], 3, 5
    clean = lay.w_down.copy()
    lay.w_down[channel, lay.neuron_perm[(shape.n_shared + expert) * shape.m + 7]] = value
    layer = parity.gpu_layer(lay, 65)
    lay.w_down = clean
    if fp8:
        layer.quantise_fp8()
    ew = _quantised(lay) if fp8 else dict(w_gate=lay.w_gate, w_up=lay.w_up, w_down=clean)
    for t in (1, 2, 16, 33, 64, 65):
        out = layer.forward(parity.to_device(inp.x[:t], "bf16"))
        torch.cuda.synchronize()
        got, r = parity.to_host(out), layer.routing(t, shape.n_routed)
        hit = (r["topk_idx"] == expert).any(axis=1)
        want = oracle.moe_forward(inp.x[:t], ew["w_gate"], ew["w_up"], ew["w_down"], lay.neuron_perm, shape.n_experts,
                                  shape.n_shared, r["topk_idx"].astype(np.int32), r["topk_gate"].astype(np.float64))
        assert not np.isfinite(got[hit, channel]).any()
        got[hit, channel] = want[hit, channel] = 0.0
        parity.check_output(got, want)
        assert t < 16 or 0 < hit.sum() < t
    layer.destroy()


# The hidden activations of the shared experts 2^20 times those of the routed ones, their down rows smaller by as much: both
# contribute alike, and every expert's channels have scales of their own.
@pytest.mark.parametrize("n_experts,n_shared,top_k", [(8, 2, 2), (32, 4, 4)])
def test_fp8_experts_of_different_magnitude(n_experts, n_shared, top_k):
    shape = wl.LayerShape(256, 176 * n_experts, n_experts, n_shared, top_k, "bf16")
    inp = wl.make_inputs(wl.Workload("fp8_magnitudes", shape, (64,), seed=4))
    lay = inp.layers[0]
    shared = lay.neuron_perm[:n_shared * shape.m]
    lay.w_up[shared] *= 2.0 ** 20
    lay.w_down[:, shared] *= 2.0 ** -20
    layer = parity.gpu_layer(lay, 64)
    layer.quantise_fp8()
    for t in (1, 2, 16, 17, 48, 64):
        parity.check_plain_layer(layer, lay, inp.x[:t], expert_weights=_quantised(lay))
    layer.destroy()
