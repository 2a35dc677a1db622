"""The scorer of one layer of few keys: its last length and the general scorer's first, one and two pairs of key tiles a
segment, segments by halves and whole, every window's layout, blocks of half the rows; the bits of the same layer among
others, on idle SMs and beside other work."""
import math

import pytest
import torch

from tests.test_gpu_windows import reference

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,Hkv,d,w,N", [
    (32, 8, 128, 64, 64), (32, 8, 128, 64, 129), (32, 8, 128, 64, 2304), (32, 8, 128, 64, 2305),   # by halves; whole
    (32, 8, 128, 64, 4608), (32, 8, 128, 64, 4609), (32, 8, 128, 61, 9216), (32, 8, 128, 64, 9217),   # two pairs; too many
    (8, 8, 64, 100, 1001), (3, 1, 128, 24, 3000), (16, 1, 64, 16, 777), (12, 4, 128, 33, 4097),    # half a block; windows
    (4, 1, 128, 256, 5003), (2, 1, 64, 200, 1300), (16, 2, 64, 128, 2500), (5, 1, 128, 64, 900),   # row blocks; unequal ones
])
def test_bits_of_a_layer_among_others(cuda_device, H, Hkv, d, w, N):
    from paper_2604_06746_b200 import binding
    L = 2
    g = torch.Generator(device=cuda_device)
    g.manual_seed(N + w)
    qs = [torch.randn((H, w, d), generator=g, device=cuda_device).bfloat16() for _ in range(L)]
    ks = [torch.randn((Hkv, N, d), generator=g, device=cuda_device).bfloat16() for _ in range(L)]
    scales = [1 / math.sqrt(d), -0.6 / math.sqrt(d)]
    ctx = binding.Context(H, Hkv, d, w, N, torch.bfloat16, cuda_device)
    ws, bws = ctx.layers_workspace(L), ctx.batch_workspace(1, N)
    s, m, cols = (torch.zeros(x, device=cuda_device) for x in ((L, N), (L, 3), (L, H, N)))
    s1, m1, cols1 = (torch.zeros_like(t) for t in (s, m, cols))
    busy, a = torch.cuda.Stream(), torch.randn((4096, 4096), device=cuda_device)

    def check():
        torch.cuda.synchronize()
        assert ctx.poll_device_status() == binding.OK
        assert torch.equal(s, s1) and torch.equal(cols, cols1) and torch.equal(m[:, 0], m1[:, 0])
        for t in (s1, m1, cols1):
            t.zero_()

    ctx.score_layers(qs, ks, scales, s, m, cols, ws)
    for l in range(L):
        want, ent = reference(qs[l], ks[l], scales[l])
        torch.testing.assert_close(cols[l].double(), want, rtol=2e-4, atol=1e-7 / N)
        assert abs(m[l, 0].item() - ent.item()) < 2e-4 * abs(ent.item()) + 1e-5
    for beside in (False, True):
        for _ in range(3):
            if beside:                                       # the SMs come free one by one: CTAs take several tasks
                with torch.cuda.stream(busy):
                    a @ a
            for l in range(L):
                ctx.score_layer(qs[l], ks[l], scales[l], s1[l], m1[l], head_cols_out=cols1[l], flags=binding.FLAG_NO_HEAD_STATS)
            check()
    for l in range(L):
        ctx.score_layer_batch(qs[l][None], ks[l], [0, N], scales[l], s1[l], m1[l:l + 1], bws, head_cols_out=cols1[l])
    check()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for l in range(L):
            ctx.score_layer(qs[l], ks[l], scales[l], s1[l], m1[l], head_cols_out=cols1[l], flags=binding.FLAG_NO_HEAD_STATS)
    graph.replay()
    check()
    del graph
    ctx.close()
