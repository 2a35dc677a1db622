"""The CUDA-core scorer's form that multiplies once (up to 64 key tiles of 64, heads of at most 128 rows): the last lengths it
takes and the first it does not, calls of more layers than run at once, repetition and replay on one context."""
import math

import pytest
import torch

from tests.test_gpu_windows import reference

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,H,Hkv,d,w,N", [
    (1, 8, 2, 64, 32, 4096), (1, 8, 2, 64, 32, 4097), (5, 8, 2, 64, 32, 4001), (3, 3, 1, 128, 128, 1000),
    (2, 2, 1, 64, 129, 500), (9, 6, 2, 128, 64, 2049), (2, 16, 1, 64, 16, 77)])
def test_layers_repetition_and_replay(cuda_device, L, H, Hkv, d, w, N):
    from paper_2604_06746_b200 import binding
    g = torch.Generator(device=cuda_device)
    g.manual_seed(N)
    qs = [torch.randn((H, w, d), generator=g, device=cuda_device) for _ in range(L)]
    ks = [torch.randn((Hkv, N, d), generator=g, device=cuda_device) for _ in range(L)]
    ctx = binding.Context(H, Hkv, d, w, N, torch.float32, cuda_device)
    ws = ctx.layers_workspace(L)
    out = [(torch.zeros((L, N), device=cuda_device), torch.zeros((L, 3), device=cuda_device),
            torch.zeros((L, H, N), device=cuda_device)) for _ in range(2)]
    scale = 1 / math.sqrt(d)

    def check():
        for l in range(L):
            ctx.score_layer(qs[l], ks[l], scale, out[0][0][l], out[0][1][l], head_cols_out=out[0][2][l])
            cols, ent = reference(qs[l], ks[l], scale)
            torch.testing.assert_close(out[0][2][l].double(), cols, rtol=2e-5, atol=1e-7 / N)
            assert abs(out[0][1][l, 0].item() - ent.item()) < 1e-5 * abs(ent.item()) + 1e-5
        for a, b in zip(*out):
            assert torch.equal(a[..., :1] if a.shape == (L, 3) else a, b[..., :1] if b.shape == (L, 3) else b)

    for _ in range(2):
        ctx.score_layers(qs, ks, [scale] * L, *(out[1][i] for i in (0, 1, 2)), ws)
        check()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ctx.score_layers(qs, ks, [scale] * L, *(out[1][i] for i in (0, 1, 2)), ws)
    for t in qs + ks:
        t.copy_(torch.randn(t.shape, generator=g, device=cuda_device))
    graph.replay()
    check()
    graph.replay()
    check()
    assert ctx.poll_device_status() == binding.OK
    del graph
    ctx.close()
