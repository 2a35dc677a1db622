"""The CUDA-core scorer around its tiles (128 score rows x 64 keys, heads of 8 .. 256 rows, more key tiles
than segments) in fp32 and bf16, against the attention written out in float64; and all layers of a
call against layer after layer."""
import math

import pytest
import torch

from tests.test_gpu_windows import reference

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("H,Hkv,d,w,N", [
    (8, 2, 64, 32, 2048), (8, 2, 64, 32, 63), (8, 2, 128, 32, 65), (2, 2, 64, 1, 129), (6, 2, 128, 5, 700),
    (4, 1, 64, 64, 64), (3, 1, 64, 200, 333), (4, 2, 128, 256, 300), (5, 1, 64, 128, 5000), (4, 4, 128, 16, 4161)])
def test_cuda_core_scorer(cuda_device, H, Hkv, d, w, N, dtype):
    from paper_2604_06746_b200 import binding
    g = torch.Generator(device=cuda_device)
    g.manual_seed(w + N)
    q = torch.randn((H, w, d), generator=g, device=cuda_device).to(dtype)
    k = torch.randn((Hkv, N, d), generator=g, device=cuda_device).to(dtype)
    ctx = binding.Context(H, Hkv, d, w, N, dtype, cuda_device)
    s, m = torch.zeros(N, device=cuda_device), torch.zeros(3, device=cuda_device)
    cols = torch.zeros((H, N), device=cuda_device)
    for scale in (1 / math.sqrt(d), -0.3):
        ctx.score_layer(q, k, scale, s, m, head_cols_out=cols, flags=binding.FLAG_FORCE_SIMT)
        ref_cols, ref_ent = reference(q, k, scale)
        torch.testing.assert_close(cols.double(), ref_cols, rtol=2e-5, atol=1e-7 / N)
        torch.testing.assert_close(s.double(), ref_cols.sum(0), rtol=2e-5, atol=1e-7 * H / N)
        assert abs(m[0].item() - ref_ent.item()) < 1e-5 * abs(ref_ent.item()) + 1e-5
    assert ctx.poll_device_status() == binding.OK
    ctx.close()


def test_fp32_layers_in_one_call_equal_the_layer_by_layer_calls(cuda_device):
    from paper_2604_06746_b200 import binding
    L, H, Hkv, d, w, N = 35, 8, 2, 64, 32, 515
    g = torch.Generator(device=cuda_device)
    g.manual_seed(4)
    qs = [torch.randn((H, w, d), generator=g, device=cuda_device) for _ in range(L)]
    ks = [torch.randn((Hkv, N, d), generator=g, device=cuda_device) for _ in range(L)]
    ctx = binding.Context(H, Hkv, d, w, N, torch.float32, cuda_device)
    s1, s2 = (torch.zeros((L, N), device=cuda_device) for _ in range(2))
    m1, m2 = (torch.zeros((L, 3), device=cuda_device) for _ in range(2))
    h1, h2 = (torch.zeros((L, H, N), device=cuda_device) for _ in range(2))
    c1, c2 = (torch.zeros(N, device=cuda_device) for _ in range(2))
    for l in range(L):
        ctx.score_layer(qs[l], ks[l], 0.125, s1[l], m1[l], c_inout=c1, head_cols_out=h1[l], flags=binding.FLAG_NO_HEAD_STATS)
    ctx.score_layers(qs, ks, [0.125] * L, s2, m2, h2, ctx.layers_workspace(L), c_inout=c2)
    assert torch.equal(s1, s2) and torch.equal(h1, h2) and torch.equal(m1[:, 0], m2[:, 0]) and torch.equal(c1, c2)
    ctx.close()
