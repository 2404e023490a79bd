"""-m gpu: forwards enqueued back to back without synchronising, each reading what the one before it wrote (a stack of
layers), against the same calls with a synchronisation after each.  Launch chaining lets a forward's first kernel become
resident while the preceding layer's last kernel still runs."""
import numpy as np
import pytest

from paper_2502_04416_b200 import binding, workloads as wl
from tests import parity

pytestmark = pytest.mark.gpu


def _stack(dtype, fp8, tokens, n_layers=3, d=512, m=176, n=8, n_shared=2, top_k=2):
    shape = wl.LayerShape(d, m * n, n, n_shared, top_k, dtype)
    rng = np.random.Generator(np.random.PCG64(3))
    layers = []
    for _ in range(n_layers):
        lay = wl.draw_layer(rng, shape)
        for w in (lay.w_gate, lay.w_up, lay.w_down):       # a layer's output is of its input's size
            w *= 2.0
        layers.append(parity.gpu_layer(lay, tokens))
        if fp8:
            layers[-1].quantise_fp8()
    return layers, wl.draw_tokens(rng, tokens, shape)


@pytest.mark.parametrize("dtype,fp8,tokens", [("bf16", False, t) for t in (1, 2, 16, 64, 100, 300, 1100)] +
                         [("bf16", True, t) for t in (1, 16, 64)] + [("fp32", False, t) for t in (1, 64, 700)])
def test_layer_stack_matches_synchronised_calls(dtype, fp8, tokens):
    _check_stack(*_stack(dtype, fp8, tokens), dtype)


# the shared experts' tiles run ahead of the routing: more of them than CTAs (single CTAs and pairs), none, only them, and a router
# too large to share an SM with the GEMM
@pytest.mark.parametrize("n,n_shared,top_k,m,tokens", [(8, 6, 2, 512, 1030), (8, 6, 2, 512, 2100), (8, 0, 2, 176, 300), (4, 4, 0, 176, 300),
                                                       (32, 4, 4, 48, 300), (32, 4, 4, 48, 700)])
def test_layer_stack_shared_tiles(n, n_shared, top_k, m, tokens):
    _check_stack(*_stack("bf16", False, tokens, m=m, n=n, n_shared=n_shared, top_k=top_k), "bf16")


# under a top-level router: rows copied by the inner router (up to 1024 outer rows), by a launch of their own, both routers on
# tiles; FP8 planes made from the copied rows
@pytest.mark.parametrize("fp8,tokens", [(False, 7), (False, 300), (False, 700), (False, 1100), (True, 7), (True, 30)])
def test_hierarchical_stack(fp8, tokens):
    shape = wl.LayerShape(512, 176 * 8, 8, 2, 2, "bf16")
    rng = np.random.Generator(np.random.PCG64(5))
    layers = []
    for _ in range(3):
        inners = []
        for _ in range(4):
            lay = wl.draw_layer(rng, shape)
            for w in (lay.w_gate, lay.w_up, lay.w_down):
                w *= 2.0
            inners.append(parity.gpu_layer(lay, 8))
        w_router = wl.round_to_storage(rng.normal(scale=0.02, size=(4, 512)).astype(np.float32), "bf16")
        layers.append(binding.Layer.create_hier(parity.to_device(w_router, "bf16"), inners, 2, tokens))
        if fp8:
            layers[-1].quantise_fp8()
    _check_stack(layers, wl.draw_tokens(rng, tokens, shape), "bf16")


# batches of all kinds in turn on one layer: the streamers' down kernel, which lets its successor start at once, followed by kernels
# that allocate tensor memory ahead of their wait, and the other way round
@pytest.mark.parametrize("fp8", [False, True])
def test_mixed_batches_back_to_back(fp8):
    import torch
    (layer,), x = _stack("bf16", fp8, 2300, n_layers=1)
    xd = parity.to_device(x, "bf16")
    sizes = (64, 1100, 16, 2300, 64, 300, 48, 700, 1, 1100, 33, 100, 64, 2300)
    starts = [(97 * i) % (2300 - t + 1) for i, t in enumerate(sizes)]
    want = []
    for t, a in zip(sizes, starts):
        want.append(layer.forward(xd[a:a + t]).clone())
        torch.cuda.synchronize()
    for _ in range(5):
        got = [layer.forward(xd[a:a + t]) for t, a in zip(sizes, starts)]
        torch.cuda.synchronize()
        for g, w in zip(got, want):
            assert torch.equal(g, w)
    assert layer.status() == 0
    layer.destroy()


def _check_stack(layers, x, dtype):
    import torch
    xs = [parity.to_device(x, dtype)]
    xs += [torch.roll(xs[0], k, 1).contiguous() for k in (1, 2, 3)]
    bufs = [torch.empty_like(xs[0]) for _ in range(3)]

    def step(k, sync):
        src = xs[k]
        for layer, dst in zip(layers, bufs):
            layer.forward(src, dst)
            if sync:
                torch.cuda.synchronize()
            src = dst
        return src.clone()

    want = [step(k, True) for k in range(4)]
    assert not torch.equal(want[0], want[1])
    for _ in range(5):
        got = [step(k, False) for k in range(4)]
        torch.cuda.synchronize()
        for g, w in zip(got, want):
            assert torch.equal(g, w)
    for layer in layers:
        assert layer.status() == 0
        layer.destroy()


# the shared experts' down GEMM combines (a narrow shared block always qualifies): columns cut inside a tile and a 32-column step,
# rows inside a tile, one to four selections, five (combined by its own kernel), and rows past one tile per CTA
@pytest.mark.parametrize("d,top_k,tokens", [(272, 1, 129), (512, 2, 300), (304, 3, 257), (1040, 4, 700), (272, 5, 300), (2064, 4, 2600)])
def test_combine_in_the_down_gemm(d, top_k, tokens):
    shape = wl.LayerShape(d, 16 * 8, 8, 2, top_k, "bf16")
    inp = wl.make_inputs(wl.Workload("fold", shape, (tokens,), seed=9))
    layer = parity.gpu_layer(inp.layers[0], tokens)
    for _ in range(2):
        st = parity.check_plain_layer(layer, inp.layers[0], inp.x)
        assert st["differing"] <= st["near_tie"]
    assert layer.status() == 0
    layer.destroy()
