"""Where the tags of exchanged words start over (tagged.cuh): the last CTA of a launch clears the words, and the launches after it find
them as those of a new context.  The scorers that exchange: one short layer, CUDA cores, short windows."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu
TAG, LAST = 64 + 2, 0x7f000000            # int of the workspace that holds the last tag; the largest that is passed on


@pytest.mark.parametrize("H,Hkv,d,w,N,dtype", [
    (32, 8, 128, 64, 300, torch.bfloat16), (32, 8, 128, 64, 5003, torch.bfloat16),
    (8, 2, 64, 32, 1000, torch.float32), (32, 8, 128, 8, 5000, torch.bfloat16), (4, 1, 128, 8, 20000, torch.bfloat16),
])
def test_tags_start_over(cuda_device, H, Hkv, d, w, N, dtype):
    from paper_2604_06746_b200 import binding
    g = torch.Generator(device=cuda_device)
    g.manual_seed(N)
    q = [torch.randn((H, w, d), generator=g, device=cuda_device).to(dtype) for _ in range(2)]
    k = [torch.randn((Hkv, N, d), generator=g, device=cuda_device).to(dtype) for _ in range(2)]
    ctx = binding.Context(H, Hkv, d, w, N, dtype, cuda_device)
    word = ctx.workspace[4 * TAG:4 * TAG + 4].view(torch.int32)

    def layer(i):
        s, m, cols = (torch.zeros(x, device=cuda_device) for x in ((N,), (3,), (H, N)))
        ctx.score_layer(q[i], k[i], 1 / math.sqrt(d), s, m, head_cols_out=cols)
        return s, m, cols

    want = [layer(i) for i in range(2)]
    used = word.item() // 2
    assert used >= 1
    word.fill_(LAST - used)
    tags = []
    for i in (0, 1, 0, 1):
        got = layer(i)
        assert ctx.poll_device_status() == binding.OK
        assert all(torch.equal(a, b) for a, b in zip(got, want[i]))
        tags.append(word.item())
    assert tags == [LAST, 0, used, 2 * used]
    ctx.close()
