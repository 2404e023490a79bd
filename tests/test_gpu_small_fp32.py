"""-m gpu: fp32 layers of a few rows (gate/up product of all experts beside the router; down product, combine and permutation in one launch)."""
import numpy as np
import pytest

from paper_2502_04416_b200 import binding, workloads as wl
from tests import parity

pytestmark = pytest.mark.gpu

# d: less than a slice of 64, slices that end early, more slices than warps; m: one quad, parts of a slice, more than two; experts: one routed,
# 32 routed, none shared, everything selected; rows on both sides of the tiles of 8 and 16 and of the path's end
CASES = [
    (8, 4, 3, 1, 1, (1, 8, 9)),
    (72, 20, 8, 2, 3, (1, 7, 16, 17, 64)),
    (256, 128, 8, 2, 2, (63, 255, 256, 257)),
    (320, 132, 5, 0, 2, (2, 33)),
    (512, 24, 34, 2, 8, (5, 40)),
    (128, 68, 4, 2, 2, (100,)),
]


@pytest.mark.parametrize("d,m,n,ns,k,tokens", CASES, ids=[f"d{c[0]}-m{c[1]}-n{c[2]}" for c in CASES])
def test_small_fp32(d, m, n, ns, k, tokens):
    inp = wl.make_inputs(wl.Workload("small_fp32", wl.LayerShape(d, m * n, n, ns, k, "fp32"), tokens, seed=4))
    lay = inp.layers[0]
    rng = np.random.default_rng(1)
    lay.gate_scale_u = rng.normal(scale=0.5, size=n - ns).astype(np.float32)
    lay.select_bias_b = rng.normal(scale=0.05, size=n - ns).astype(np.float32)
    layer = parity.gpu_layer(lay, max(tokens))
    for t in tokens:
        st = parity.check_plain_layer(layer, lay, inp.x[:t])
        assert st["differing"] <= st["near_tie"]
        assert st["max_rel"] < 1e-4 and st["mean_rel"] < 1e-4      # fp32 end to end
    layer.destroy()


def test_same_rows_on_the_general_path():
    import torch
    inp = wl.make_inputs(wl.Workload("small_fp32", wl.LayerShape(256, 1024, 8, 2, 2, "fp32"), (400,), seed=9))
    layer = parity.gpu_layer(inp.layers[0], 400)
    x = parity.to_device(inp.x, "fp32")
    whole = layer.forward(x)[:200].clone()                # 400 rows: per-expert products, permuted rows
    few = layer.forward(x[:200].contiguous())
    # two orders of fp32 sums over at most 1024 terms each: sqrt(1024) roundings of 6e-8
    assert ((whole - few).norm() / whole.norm()).item() < 2e-6
    assert torch.isfinite(few).all()
    layer.destroy()


def test_the_general_path_can_be_forced():
    import torch
    inp = wl.make_inputs(wl.Workload("small_fp32", wl.LayerShape(256, 1024, 8, 2, 2, "fp32"), (256,), seed=10))
    layer = parity.gpu_layer(inp.layers[0], 256)
    x = parity.to_device(inp.x, "fp32")
    for t in (1, 64, 256):
        got = []
        for path, launches in ((binding.GEMM_AUTO, 3), (binding.GEMM_SIMT, 5)):
            layer.set_gemm_path(path)
            got.append(layer.forward(x[:t].contiguous()))
            assert layer.launch_count() == launches
        # as above: two orders of fp32 sums over at most 1024 terms each
        assert ((got[0] - got[1]).norm() / got[1].norm()).item() < 2e-6
    st = parity.check_plain_layer(layer, inp.layers[0], inp.x[:64])
    assert st["differing"] == 0 and st["max_rel"] < 1e-4
    layer.destroy()


# many unselected experts: their slices (one row), their slices and tiles, rows, weights; beside each a batch that gains by the path
@pytest.mark.parametrize("d,m,n,k,general,three", [(128, 256, 34, 2, 16, None), (2048, 256, 34, 2, 1, 6), (256, 64, 34, 1, 192, 16),
                                                   (384, 96, 18, 2, 192, 24), (64, 512, 12, 2, 128, 16)])
def test_layers_of_many_unselected_experts_take_the_general_path(d, m, n, k, general, three):
    inp = wl.make_inputs(wl.Workload("small_fp32", wl.LayerShape(d, m * n, n, 2, k, "fp32"), (256,), seed=14))
    layer = parity.gpu_layer(inp.layers[0], 256)
    for t, launches in ((general, 5), (three, 3)):
        if t:
            st = parity.check_plain_layer(layer, inp.layers[0], inp.x[:t])
            assert st["differing"] <= st["near_tie"] and st["max_rel"] < 1e-4
            assert layer.launch_count() == launches
    layer.destroy()


@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_non_finite_weight_stays_with_its_expert(value):
    import torch
    shape = wl.LayerShape(128, 48 * 8, 8, 2, 2, "fp32")
    inp = wl.make_inputs(wl.Workload("small_fp32", shape, (60,), seed=3))
    lay, expert, channel = inp.layers[0], 3, 5
    lay.w_down[channel, lay.neuron_perm[(shape.n_shared + expert) * shape.m + 7]] = value
    layer = parity.gpu_layer(lay, 60)
    out = layer.forward(parity.to_device(inp.x, "fp32"))
    torch.cuda.synchronize()
    got, hit = parity.to_host(out), (layer.routing(60, shape.n_routed)["topk_idx"] == expert).any(axis=1)
    assert 0 < hit.sum() < 60
    assert not np.isfinite(got[hit, channel]).any() and np.isfinite(got[~hit]).all()
    layer.destroy()


@pytest.mark.parametrize("path", [binding.GEMM_AUTO, binding.GEMM_SIMT], ids=["three_launches", "general"])
def test_small_fp32_stack_is_the_same_chained_or_not(path):
    import torch
    inp = wl.make_inputs(wl.Workload("small_fp32", wl.LayerShape(256, 512, 8, 2, 2, "fp32"), (64,), seed=7))
    layers = [parity.gpu_layer(inp.layers[0], 64) for _ in range(3)]
    for layer in layers:
        layer.set_gemm_path(path)
    x = parity.to_device(inp.x, "fp32")

    def run(chain):
        outs = []
        for layer in layers:
            layer.set_launch_chaining(chain)
        for t in (64, 3, 64, 17, 1, 64):
            y = x[:t].contiguous()
            for layer in layers:
                y = layer.forward(y)
            outs.append(y)
        torch.cuda.synchronize()
        return outs

    for a, b in zip(run(False), run(True)):
        assert torch.equal(a, b)
    for layer in layers:
        layer.destroy()
