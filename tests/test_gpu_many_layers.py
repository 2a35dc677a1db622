"""Sums and head statistics of more (layer, head) vectors than SMs in one launch, at the edges of its forms (blocks of
512 keys; all statistics first, or each layer's sums behind its own; three or six CTAs an SM): the bits of the
separate calls."""
import pytest
import torch

from tests.test_gpu_prefill_call import OUT, prompt, step_by_step

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seq,n_layers", [(130, 5), (512, 33), (513, 14), (4097, 13), (8193, 24), (32768, 7),
                                          (33000, 24)])
def test_one_launch_equals_the_separate_calls(cuda_device, seq, n_layers):
    one, args = prompt(cuda_device, seq, n_layers, 100)
    ref, _ = prompt(cuda_device, seq, n_layers, 100)
    for _ in range(2):                                       # the counters are left as they were found
        one.run(*args)
    step_by_step(ref, *args)
    torch.cuda.synchronize()
    assert one.ctx.poll_device_status() == 0 and one.pivot == ref.pivot
    for key in OUT + ("hidden_out", "pos_out"):
        assert torch.equal(getattr(one, key), getattr(ref, key)), key
