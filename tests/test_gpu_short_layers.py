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


@pytest.mark.parametrize("H,Hkv,d,w,N", [
    (32, 8, 128, 64, 64), (32, 8, 128, 64, 300), (32, 8, 128, 64, 1900),     # halves, an odd number of tiles: 1, 3, 15
    (32, 8, 128, 64, 256), (32, 8, 128, 64, 2304),                           # an even one
    (32, 8, 128, 64, 2500), (32, 8, 128, 64, 9000),                          # whole segments of one pair and of one or two
    (16, 1, 64, 16, 777), (12, 4, 128, 33, 4097), (3, 1, 128, 24, 3000),     # other windows and head dimensions
    (4, 1, 128, 256, 1300), (2, 1, 64, 200, 5003), (16, 2, 64, 128, 300),    # several row blocks
    (8, 8, 64, 100, 1001),
])
def test_several_tasks_a_cta(cuda_device, H, Hkv, d, w, N):
    """Fewer CTAs than tasks, whatever else runs: the bits of one task a CTA, which are those of a layer among others."""
    from paper_2604_06746_b200 import binding
    g = torch.Generator(device=cuda_device)
    g.manual_seed(N + w)
    q = torch.randn((2, H, w, d), generator=g, device=cuda_device).bfloat16()
    k = torch.randn((2, Hkv, N, d), generator=g, device=cuda_device).bfloat16()
    ctx = binding.Context(H, Hkv, d, w, N, torch.bfloat16, cuda_device)

    def layer(l, ctas):
        s, m, cols = (torch.zeros(x, device=cuda_device) for x in ((N,), (3,), (H, N)))
        ctx.selftest_ctas(ctas)
        ctx.score_layer(q[l], k[l], 1 / math.sqrt(d), s, m, head_cols_out=cols)
        return s, m, cols

    s, m, cols = (torch.zeros(x, device=cuda_device) for x in ((2, N), (2, 3), (2, H, N)))
    ctx.score_layers(list(q), list(k), [1 / math.sqrt(d)] * 2, s, m, cols, ctx.layers_workspace(2))
    whole = [layer(l, 0) for l in range(2)]
    for l in range(2):
        assert torch.equal(whole[l][0], s[l]) and torch.equal(whole[l][1][0], m[l, 0]) and torch.equal(whole[l][2], cols[l])
    for ctas in (1, 2, 3, 5, 11, 0):
        got = [layer(l, ctas) for l in (0, 1, 0)]            # the words of one launch are there in the next
        assert ctx.poll_device_status() == binding.OK, ctas
        for l, r in zip((0, 1, 0), got):
            assert all(torch.equal(a, b) for a, b in zip(r, whole[l])), ctas
    ctx.close()
