"""A feed-forward width that is no multiple of 4 moves the parameters behind it off 16 bytes in fp32 contexts: LayerNorm, which reads
its gain and bias 16 bytes at a time, refuses them; the context stays usable."""
import pytest
import torch

from paper_2204_04179_b200 import binding, synth

pytestmark = pytest.mark.gpu


def test_parameters_off_16_bytes_are_refused():
    B, L, d = 3, 5, 32
    shape = synth.GramShape(name="a", dtype="f32", n_items=1, l_t=1, vocab=1, d=d, n_heads=2, d_ff=64, n_layers=0, task="kt", task_layers=1,
                            task_heads=2, task_d_ff=34, task_attn_only=False, B=B, L=L)
    g = binding.Gram(binding.config_from_shape(shape))
    g.set_params(binding.GRAM_MODULE_TASK, synth.flatten(synth.task_params(shape, 3, sigma=0.1, plain=False)))
    E = torch.randn(B, L, d, generator=torch.Generator().manual_seed(1)).cuda()
    lab = torch.from_numpy(synth.labels(5, B, L, 0.6)).cuda()
    dE, loss = torch.empty(B * L, d, device="cuda"), torch.empty(1, device="cuda")
    with pytest.raises(binding.GramError, match="GRAM_ERR_UNSUPPORTED.*16 bytes"):
        g.task(E, lab, B, dE, loss)
    g.sync()
    g.close()
