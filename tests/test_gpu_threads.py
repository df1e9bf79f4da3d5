"""Contexts of different widths in use by different threads at once: a context is one thread's, the kernels are everybody's."""
import threading

import pytest
import torch

from paper_2204_04179_b200 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths", [(768, 640), (512, 320)])
def test_two_widths_at_once(widths):
    """Both widths of a pair run the same instantiations with other amounts of shared memory."""
    errors, together = [], threading.Barrier(len(widths))

    def work(d):
        shape = synth.GramShape(name="w", dtype="f32", n_items=1, l_t=1, vocab=1, d=d, n_heads=d // 64, d_ff=64, n_layers=0, task="kt",
                                task_layers=2, task_heads=d // 64, task_d_ff=64, task_attn_only=False, B=1, L=3)
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                g = binding.Gram(binding.config_from_shape(shape))
                g.set_params(binding.GRAM_MODULE_TASK, synth.flatten(synth.task_params(shape, 3, sigma=0.1, plain=False)))
                E, lab = torch.randn(1, 3, d, device="cuda"), torch.ones(1, 3, dtype=torch.int32, device="cuda")
                dE, loss = torch.empty(3, d, device="cuda"), torch.empty(1, device="cuda")
                g.task(E, lab, 1, dE, loss)
                g.sync()
                want = dE.clone(), loss.clone()
                together.wait(60)
                for _ in range(1500):
                    g.task(E, lab, 1, dE, loss)
                g.sync()
                assert torch.equal(dE, want[0]) and torch.equal(loss, want[1])
                g.close()
        except Exception as e:                                  # reported by the test's own thread
            errors.append(e)
            together.abort()

    threads = [threading.Thread(target=work, args=(d,)) for d in widths]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
