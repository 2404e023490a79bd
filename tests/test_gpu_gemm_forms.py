"""-m gpu: which tiles the automatic choice takes for the gate/up GEMM at sizes where all forms were timed, and that the choice
does not show in the output."""
import numpy as np
import pytest

from paper_2502_04416_b200 import binding, workloads as wl

pytestmark = pytest.mark.gpu

# rows -> forms within 2 % of the fastest forward (single CTAs / token-major pairs / turned pairs, us, at the first size of each
# line: 7B-shaped 1000 rows 160 / 157 / 154, 512 rows 104 / 96 / 95, 1400 rows 201 / 195 / 199, 300 rows 79 / 86 / 80, 8B-shaped 1500 rows
# 182 / 171 / 178, 700 rows 109 / 117 / 114, 3200 rows 322 / 307 / 311, 13B-shaped 600 rows 150 / 142 / 137)
SIZES = [
    ("c2_llama2_7b", (1000, 1024), ("turned",)),
    ("c2_llama2_7b", (512, 400, 600, 850, 1300, 1600), ("turned",)),
    ("c2_llama2_7b", (1400, 1470), ("pair",)),
    ("c2_llama2_7b", (300, 256), ("single",)),
    ("c3_llama3_8b", (1500, 1400), ("pair",)),
    ("c3_llama3_8b", (700, 600, 768, 820), ("single",)),
    ("c5_skew_13b", (600, 400, 512, 1000, 1500), ("turned",)),
    ("c3_llama3_8b", (3200, 14592, 16384), ("pair",)),
]


def _layer(name, rows):
    import torch
    s = wl.WORKLOADS[name].shape
    gen = torch.Generator(device="cuda").manual_seed(3)
    w = [torch.randn(*shape, device="cuda", dtype=torch.bfloat16, generator=gen).mul_(wl.WEIGHT_STD)
         for shape in ((s.d_ff, s.d_model), (s.d_ff, s.d_model), (s.d_model, s.d_ff))]
    perm = np.arange(s.d_ff, dtype=np.int32)
    return s, binding.Layer.create(*w, perm, perm[s.n_shared * s.m::s.m], s.n_experts, s.n_shared, s.top_k, rows)


@pytest.mark.parametrize("name,rows,forms", SIZES, ids=[f"{n}-{r[0]}" for n, r, _ in SIZES])
def test_chosen_forms(name, rows, forms):
    import torch
    s, layer = _layer(name, max(rows))
    for t in rows:
        assert layer.gemm_forms(t)[0] in forms, t
    x = torch.randn(rows[0], s.d_model, device="cuda", dtype=torch.bfloat16, generator=torch.Generator(device="cuda").manual_seed(4))
    got = layer.forward(x)
    layer.set_gemm_path(binding.GEMM_TENSOR)
    assert layer.gemm_forms(rows[0]) == ("single", "single")
    assert torch.equal(got.view(torch.int16), layer.forward(x).view(torch.int16))
    assert layer.status() == 0
    layer.destroy()


# 13B-shaped 16384 rows 2380 / 2426 us with token-major / turned down tiles, 7B-shaped 4096 rows 505 / 497 (1365 rows per expert: 1536 / 1376 columns),
# 448 neurons are too few k blocks for either
@pytest.mark.parametrize("name,rows,form", [("c5_skew_13b", 16384, "pair"), ("c2_llama2_7b", 4096, "turned"), ("c3_llama3_8b", 8192, "single")])
def test_chosen_down_form(name, rows, form):
    _, layer = _layer(name, rows)
    assert layer.gemm_forms(rows)[1] == form
    layer.destroy()


def test_small_batches_have_no_tile_form():
    _, layer = _layer("c2_llama2_7b", 200)
    assert layer.gemm_forms(64) == layer.gemm_forms(128) == ("other", "other")
    assert layer.gemm_forms(129) == ("single", "single")
    layer.set_gemm_path(binding.GEMM_SIMT)
    assert layer.gemm_forms(200) == ("other", "other")
    with pytest.raises(binding.CmoeError):
        layer.gemm_forms(201)
    layer.destroy()
