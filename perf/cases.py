"""The work that users of this library have it do, as timed cases.

A case is one call on one prepared layer: the forward of a restructured SwiGLU FFN (plain or
hierarchical, bf16 / fp32, FP8 expert weights, launched directly or replayed from a CUDA graph),
or one chunk of the activation profiling that precedes a restructuring.  Shapes are those of
``workloads.WORKLOADS`` or generic ones of the same proportions.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2502_04416_b200 import binding, workloads as wl

TIE_MARGIN = 2e-4     # tokens whose k-th and (k+1)-th key lie closer than this are drawn again


# ------------------------------------------------------------------ the cases
def _case(name, d, m, n, shared, top_k, tokens, *, kind="forward", dtype="bf16", fp8=False, graph=False,
          zipf=0.0, n_outer=0, outer_k=0):
    c = dict(kind=kind, d=d, m=m, n=n, shared=shared, top_k=top_k, tokens=tokens, dtype=dtype, fp8=fp8,
             graph=graph, zipf=zipf, n_outer=n_outer, outer_k=outer_k)
    return dict(c, name=name) if name else c


def _shape(workload):
    w = wl.WORKLOADS[workload]
    s = w.shape
    return dict(d=s.d_model, m=s.m, n=s.n_experts, shared=s.n_shared, top_k=s.top_k, n_outer=w.n_outer,
                outer_k=w.outer_top_k, zipf=w.zipf_s)


def listed():
    tiny, b7, b8, b13, hier = (_shape(k) for k in ("c1_tiny_fp32", "c2_llama2_7b", "c3_llama3_8b", "c5_skew_13b",
                                                  "c4_hier_8x7b"))
    return [
        # a toy layer in fp32, as in unit tests and in checks of a partition: launches and latency only
        _case("tiny_fp32_64", **tiny, tokens=64, dtype="fp32"),
        # one user's token-by-token generation
        _case("decode_7b_1", **b7, tokens=1),
        # a small serving batch, the decode loop captured in a graph as servers do
        _case("decode_7b_graph_16", **b7, tokens=16, graph=True),
        # a serving batch on a weight-quantised layer
        _case("decode_7b_fp8_48", **b7, tokens=48, fp8=True),
        # a serving batch on many narrow experts
        _case("decode_8b_32", **b8, tokens=32),
        # a few users on a restructured mixture-of-experts layer
        _case("decode_hier_7", **hier, tokens=7),
        # a short prompt, or decode of a large batch; not a multiple of any tile
        _case("prompt_7b_300", **b7, tokens=300),
        # a prompt of about a thousand tokens on narrow experts
        _case("prompt_8b_1000", **b8, tokens=1000),
        # one chunk of calibration rows through the dense FFN (activation profiling)
        _case("profile_7b_2048", d=4096, m=11008, n=1, shared=1, top_k=10, tokens=2048, kind="profile"),
        # prefill of a restructured mixture-of-experts layer
        _case("prefill_hier_4096", **hier, tokens=4096),
        # long prefill, many narrow experts
        _case("prefill_8b_8192", **b8, tokens=8192),
        # the largest: prefill of several prompts with skewed expert load
        _case("prefill_13b_skew_16384", **b13, tokens=16384),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plain"] * 6 + ["hier", "profile", "tiny"])
    if kind == "tiny":
        c = _case("", d=64 * rng.randint(2, 8), m=8 * rng.randint(4, 24), n=8, shared=2, top_k=rng.randint(1, 3),
                  tokens=_log_int(rng, 1, 256), dtype="fp32")
    elif kind == "profile":
        c = _case("", d=rng.choice([2048, 4096, 5120]), m=64 * rng.randint(32, 216), n=1, shared=1,
                  top_k=rng.randint(4, 32), tokens=_log_int(rng, 64, 2048), kind="profile")
    elif kind == "hier":
        s = _shape("c4_hier_8x7b")
        s.update(d=rng.choice([1024, 2048, 4096]), m=16 * rng.randint(28, 112))
        c = _case("", **s, tokens=_log_int(rng, 1, 4096), fp8=rng.random() < 0.2)
    else:
        s = _shape(rng.choice(["c2_llama2_7b", "c3_llama3_8b", "c5_skew_13b"]))
        s["zipf"] = rng.choice([0.0, s["zipf"]])
        if rng.random() < 0.5:                    # generic shapes of the same proportions
            s.update(d=64 * rng.randint(16, 80), m=16 * rng.randint(20, {8: 86, 16: 64, 32: 36}[s["n"]]))
        tokens = _log_int(rng, 1, 12000)
        c = _case("", **s, tokens=tokens, fp8=tokens <= 256 and rng.random() < 0.4,
                  graph=tokens <= 512 and rng.random() < 0.3)
    return c


# --------------------------------------------------------------------- inputs
def _zipf_bias(n_routed, top_k, s):
    """A selection bias that skews the load of the routed experts: the log of the target shares, scaled to
    the width of softmax scores."""
    p = wl.zipf_target_shares(n_routed, top_k, s)
    return (0.05 * np.log(p / p.min())).astype(np.float32)


def _near_ties(x, layers, w_router, top_k, outer_k, biases):
    """Tokens for which two experts tie for the last place within rounding: either choice would be right."""
    def close(keys, k):
        if k >= keys.shape[1]:
            return torch.zeros(keys.shape[0], dtype=torch.bool, device=keys.device)
        top = keys.topk(k + 1, dim=1).values
        return (top[:, k - 1] - top[:, k]) < TIE_MARGIN
    xf = x.float()
    bad = torch.zeros(x.shape[0], dtype=torch.bool, device=x.device)
    for (rep_gate, rep_up), b in zip(layers, biases):
        s = torch.nn.functional.silu(xf @ rep_gate.float().T) * (xf @ rep_up.float().T)
        bad |= close(torch.softmax(s, dim=1) + b, top_k)
    if w_router is not None:
        bad |= close(xf @ w_router.float().T, outer_k)
    return bad


def prepare(case, seed):
    """Weights and layer as a model's start-up builds them, and one batch of tokens."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.default_rng(seed)
    dt = torch.float32 if case["dtype"] == "fp32" else torch.bfloat16
    d, m, n, ns, k, T = (case[f] for f in ("d", "m", "n", "shared", "top_k", "tokens"))
    d_ff, nr = m * n, n - ns

    def normal(*shape, std=1.0):
        return torch.randn(*shape, device="cuda", dtype=dt, generator=gen).mul_(std)

    profile = case["kind"] == "profile"
    layers, reps, biases = [], [], []
    for _ in range(max(case["n_outer"], 1)):
        wg, wu, wd = normal(d_ff, d, std=wl.WEIGHT_STD), normal(d_ff, d, std=wl.WEIGHT_STD), normal(d, d_ff, std=wl.WEIGHT_STD)
        perm = np.arange(d_ff, dtype=np.int32) if profile else rng.permutation(d_ff).astype(np.int32)
        rep = perm[(ns + np.arange(nr)) * m]
        u = (0.1 * rng.standard_normal(nr)).astype(np.float32)      # gates as after fine-tuning: near 1
        b = _zipf_bias(nr, k, case["zipf"]) if case["zipf"] else None
        layers.append(binding.Layer.create(wg, wu, wd, perm, rep, n, ns, 0 if profile else k,
                                           8 if case["n_outer"] else T, u, b))
        at = torch.from_numpy(rep.astype(np.int64)).cuda()
        reps.append((wg[at], wu[at]))
        biases.append(0.0 if b is None else torch.from_numpy(b).cuda())
    w_router = None
    layer = layers[0]
    if case["n_outer"]:
        w_router = normal(case["n_outer"], d, std=wl.WEIGHT_STD)
        layer = binding.Layer.create_hier(w_router, layers, case["outer_k"], T)
    if case["fp8"]:
        layer.quantise_fp8()
    x = normal(T, d)
    state = {"layer": layer, "x": x}
    if profile:
        state.update(k_a=k, bits=torch.zeros(d_ff, (T + 31) // 32, dtype=torch.int32, device="cuda"),
                     counts=torch.zeros(d_ff, dtype=torch.int32, device="cuda"))
        return state
    for _ in range(8):
        at = _near_ties(x, reps, w_router, k, case["outer_k"], biases).nonzero().flatten()
        if at.numel() == 0:
            break
        x[at] = normal(at.numel(), d)
    if case["graph"]:
        out = torch.empty_like(x)
        layer.forward(x, out)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            layer.forward(x, out)
        state.update(graph=graph, out=out)
    return state


def run(state):
    if "graph" in state:
        state["graph"].replay()
        return state["out"]
    if "bits" in state:
        state["bits"].zero_()
        state["counts"].zero_()
        state["layer"].profile_activations(state["x"], state["k_a"], state["bits"], state["counts"])
        return state["bits"], state["counts"]
    return state["layer"].forward(state["x"])


# ------------------------------------------------------------ floors and rules
def work(case):
    d, m, n, ns, k, T = (case[f] for f in ("d", "m", "n", "shared", "top_k", "tokens"))
    esz = 4 if case["dtype"] == "fp32" else 2
    wsz = 1 if case["fp8"] else esz
    if case["kind"] == "profile":
        d_ff = m * n
        return {"bytes": 2 * d_ff * d * 2 + T * d * 2 + d_ff * ((T + 31) // 32) * 4 + d_ff * 4,
                "flops": 4.0 * d * d_ff * T}
    rows, outers = T, 1.0
    if case["n_outer"]:                                  # outer experts that at least one token selects
        rows = T * case["outer_k"]
        outers = case["n_outer"] * (1.0 - (1.0 - case["outer_k"] / case["n_outer"]) ** T)
    nr = n - ns
    touched = nr * (1.0 - (1.0 - k / nr) ** (rows / outers))
    io = 2 * T * d * esz
    flops = rows * (6.0 * d * m * (ns + k) + 4.0 * d * nr) + 2.0 * T * d * case["n_outer"]
    return {"bytes": outers * (ns + touched) * 3 * d * m * wsz + io, "flops": flops}


def tolerance(case):
    if case["kind"] == "profile":
        # H is held in bf16 and the cut falls between two values of it: a sum in another order moves a few
        return {"rel": 0.0, "differ": 0.005}
    # 7e-7 / 2.7e-3 against the same forward in 64 bits: fp32 sums, or bf16 hidden activations, partial
    # outputs and result
    return {"rel": 5e-6} if case["dtype"] == "fp32" else {"rel": 1e-2}
