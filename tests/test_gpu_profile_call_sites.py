"""Work by call site of an fp32 task module: each product under its own role, whether two of them share a launch or not."""
import pytest
import torch

from paper_2204_04179_b200 import binding, synth

pytestmark = pytest.mark.gpu


# 96 and 4000 rows: the two products of a gradient go in one launch; 8000 rows: apart
@pytest.mark.parametrize("B,L", [(6, 16), (40, 100), (80, 100)])
def test_products_are_filed_by_role(B, L):
    d, f, layers = 64, 128, 2
    shape = synth.GramShape(name="p", dtype="f32", n_items=1, l_t=1, vocab=1, d=d, n_heads=1, d_ff=4, n_layers=0, task="kt", task_layers=layers,
                            task_heads=2, task_d_ff=f, task_attn_only=False, B=B, L=L)
    g = binding.Gram(binding.config_from_shape(shape))
    g.set_params(binding.GRAM_MODULE_TASK, synth.flatten(synth.task_params(shape, 3, sigma=0.1, plain=False)))
    E = torch.randn(B, L, d, generator=torch.Generator().manual_seed(1)).cuda()
    lab = torch.from_numpy(synth.labels(5, B, L, 0.6)).cuda()
    dE, loss = torch.empty(B * L, d, device="cuda"), torch.empty(1, device="cuda")
    g.profile(True)
    g.task(E, lab, B, dE, loss)
    sites, kinds = g.profile_dump(), g.profile_read()
    g.close()
    flops = {"qkv": 3 * d * d, "attn_out": d * d, "ffn1": d * f, "ffn2": d * f}
    for role, per_row in flops.items():
        for tag in ("fwd_" + role, "dw_" + role, "dx_" + role + ("_dgelu" if role == "ffn2" else "")):
            assert sites[tag]["work"] == pytest.approx(2 * per_row * B * L * layers, rel=1e-6), tag     # printed with seven digits
            assert sites[tag]["launches"] == layers and sites[tag]["ms"] > 0, tag
    gemm = [s for s in sites.values() if s["kind"] == "gemm"]
    assert sum(s["work"] for s in gemm) == pytest.approx(kinds["gemm"]["work"], rel=1e-6)
    assert sum(s["ms"] for s in gemm) == pytest.approx(kinds["gemm"]["ms"], rel=1e-3)
