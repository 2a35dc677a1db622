"""The scorer of short windows that reads K once (at most 32 score rows per KV group, sequences from 4096 keys on, from 16384
keys of all KV heads on): the edges of its chunks, tiles and teams, both ways its CTAs add up their rows (small teams and large ones),
logits far above the sampled references, repetition on one workspace, and streams side by side."""
import math

import pytest
import torch

from tests.test_gpu_windows import reference, score

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,Hkv,d,w,N", [
    (32, 8, 128, 8, 4095), (32, 8, 128, 8, 4096), (32, 8, 128, 8, 4097),     # the general scorer's last length, this one's first
    (16, 16, 64, 8, 4096), (18, 9, 128, 8, 7001),                            # direct teams of 9 and 16
    (32, 8, 128, 7, 9215), (32, 8, 128, 8, 18433),                           # eight teams of 18, four of 37
    (8, 2, 128, 3, 4161), (8, 2, 64, 8, 20000), (4, 4, 64, 32, 6001),        # teams of 74; of 37; one head of 32 rows
    (4, 1, 128, 8, 4737), (1, 1, 64, 1, 5000), (3, 1, 128, 8, 70001),        # one team of all SMs, its rows summed
    (4, 1, 128, 8, 16383), (4, 1, 128, 8, 16384), (8, 2, 64, 3, 8192),       # few KV heads: the last length, the first ones
    (7, 7, 128, 8, 4100), (24, 6, 128, 8, 4800), (20, 5, 64, 7, 37889),      # teams of 21, 24 and 29, summed
])
def test_edges(cuda_device, H, Hkv, d, w, N):
    score(cuda_device, H, Hkv, d, w, N, 1 / math.sqrt(d))


@pytest.mark.parametrize("H,Hkv,N", [(32, 8, 5000), (4, 1, 5000), (4, 1, 20000), (16, 4, 9000), (32, 16, 5000)])
@pytest.mark.parametrize("scale", [-0.3, 0.0, 1.0, 3.0])
def test_logits_far_above_the_references(cuda_device, H, Hkv, N, scale):
    """Unit-variance keys give logits of 11 |scale| nats' deviation: at 1 a CTA's sums leave the range of the summed
    words, at 3 they overflow against the reference they started from (2^60) and are redone."""
    score(cuda_device, H, Hkv, 128, 8, N, scale)


@pytest.mark.parametrize("Hkv,N", [
    (8, 4200), (1, 4200),
    (4, 4200), (4, 9400),                                                    # teams of 37, one and two tiles a CTA
    (16, 4200), (12, 9400),                                                  # direct teams of 9 and 12
    (7, 4200), (1, 16500),                                                   # teams of 21, seven of them; one of 148
    (1, 70000), (2, 40000),                                                  # summed, four and five tiles a CTA
])
def test_layers_repetition_and_replay(cuda_device, Hkv, N):
    """Layers of one call, the same call again, and a captured call replayed on other inputs: the bits of single
    layers (more layers than a launch holds; the CTAs' tagged words pass from call to call)."""
    from paper_2604_06746_b200 import binding
    L, H, d, w = 34, 4 * Hkv, 64, 8
    g = torch.Generator(device=cuda_device)
    g.manual_seed(11)
    qs = [torch.randn((H, w, d), generator=g, device=cuda_device).bfloat16() for _ in range(L)]
    ks = [torch.randn((Hkv, N, d), generator=g, device=cuda_device).bfloat16() for _ in range(L)]
    ctx = binding.Context(H, Hkv, d, w, N, torch.bfloat16, cuda_device)
    ws = ctx.layers_workspace(L)

    def outputs():
        return torch.zeros((L, N), device=cuda_device), torch.zeros((L, 3), device=cuda_device), torch.zeros((L, H, N), device=cuda_device)

    def one_by_one():
        s, m, h = outputs()
        for l in range(L):
            ctx.score_layer(qs[l], ks[l], 0.125, s[l], m[l], head_cols_out=h[l], flags=binding.FLAG_NO_HEAD_STATS)
        return s, m, h

    s1, m1, h1 = one_by_one()
    s2, m2, h2 = outputs()
    for _ in range(3):
        for t in (s2, m2, h2):
            t.zero_()
        ctx.score_layers(qs, ks, [0.125] * L, s2, m2, h2, ws)
        assert torch.equal(s1, s2) and torch.equal(h1, h2) and torch.equal(m1[:, 0], m2[:, 0])
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ctx.score_layers(qs, ks, [0.125] * L, s2, m2, h2, ws)
    for t in qs + ks:
        t.copy_(torch.randn(t.shape, generator=g, device=cuda_device))
    graph.replay()
    s1, m1, h1 = one_by_one()
    graph.replay()
    torch.cuda.synchronize()
    assert ctx.poll_device_status() == binding.OK
    assert torch.equal(s1, s2) and torch.equal(h1, h2) and torch.equal(m1[:, 0], m2[:, 0])
    del graph
    ctx.close()


def test_two_streams(cuda_device):
    """Contexts of their own on two streams, beside a third stream's copies: every launch's CTAs still all run."""
    from paper_2604_06746_b200 import binding
    H, Hkv, d, w, N = 32, 8, 128, 8, 9000
    g = torch.Generator(device=cuda_device)
    g.manual_seed(5)
    q = [torch.randn((H, w, d), generator=g, device=cuda_device).bfloat16() for _ in range(2)]
    k = [torch.randn((Hkv, N, d), generator=g, device=cuda_device).bfloat16() for _ in range(2)]
    ctx = [binding.Context(H, Hkv, d, w, N, torch.bfloat16, cuda_device) for _ in range(2)]
    s = [torch.zeros((40, N), device=cuda_device) for _ in range(2)]
    m = [torch.zeros((40, 3), device=cuda_device) for _ in range(2)]
    big = torch.zeros((2, 1 << 26), device=cuda_device)
    streams = [torch.cuda.Stream() for _ in range(3)]
    torch.cuda.synchronize()
    for i in range(40):
        for b in range(2):
            with torch.cuda.stream(streams[b]):
                ctx[b].score_layer(q[b], k[b], 0.1, s[b][i], m[b][i])
        if i % 8 == 0:
            with torch.cuda.stream(streams[2]):
                big[0].copy_(big[1])
    torch.cuda.synchronize()
    for b in range(2):
        assert ctx[b].poll_device_status() == binding.OK
        assert torch.equal(s[b], s[b][:1].expand_as(s[b])) and torch.equal(m[b], m[b][:1].expand_as(m[b]))
        cols, ent = reference(q[b], k[b], 0.1)
        torch.testing.assert_close(s[b][0].double(), cols.sum(0), rtol=2e-4, atol=1e-7 * H / N)
        assert abs(m[b][0, 0].item() - ent.item()) < 1e-4 * abs(ent.item()) + 1e-5
        ctx[b].close()


def test_a_layer_takes_two_launches(cuda_device):
    """The scorer and the sums over heads; large teams find their rows' references inside the scorer."""
    from cuda.bindings import runtime as rt

    from paper_2604_06746_b200 import binding
    H, Hkv, d, w, N = 4, 1, 128, 8, 50000
    q = torch.zeros((H, w, d), device=cuda_device, dtype=torch.bfloat16)
    k = torch.zeros((Hkv, N, d), device=cuda_device, dtype=torch.bfloat16)
    s, m = torch.zeros(N, device=cuda_device), torch.zeros(3, device=cuda_device)
    ctx = binding.Context(H, Hkv, d, w, N, torch.bfloat16, cuda_device)
    ctx.score_layer(q, k, 0.1, s, m, flags=binding.FLAG_NO_HEAD_STATS)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        ctx.score_layer(q, k, 0.1, s, m, flags=binding.FLAG_NO_HEAD_STATS)
    err, _, count = rt.cudaGraphGetNodes(rt.cudaGraph_t(init_value=int(graph.raw_cuda_graph())))
    assert err == rt.cudaError_t.cudaSuccess and count == 2
    del graph
    ctx.close()


@pytest.mark.parametrize("H,Hkv,d,w,N", [
    (32, 16, 128, 8, 5000), (9, 9, 64, 32, 4200),                            # small teams
    (32, 8, 128, 8, 5000), (8, 8, 64, 32, 4200),
    (16, 4, 64, 7, 9001), (6, 2, 128, 5, 40000), (4, 1, 128, 8, 20000),      # teams with common references
])
def test_layouts_of_k(cuda_device, H, Hkv, d, w, N):
    """Token-major K, and rows and heads with room between them: the bits of contiguous K, for a layer by itself, for several,
    and on the static scratch."""
    from paper_2604_06746_b200 import binding
    g = torch.Generator(device=cuda_device)
    g.manual_seed(N)
    q = [torch.randn((H, w, d), generator=g, device=cuda_device).bfloat16() for _ in range(2)]
    k = [torch.randn((Hkv, N, d), generator=g, device=cuda_device).bfloat16() for _ in range(2)]
    ctx = binding.Context(H, Hkv, d, w, N, torch.bfloat16, cuda_device)
    ws = ctx.layers_workspace(2)

    def run(ks):
        s, m, h = (torch.zeros(x, device=cuda_device) for x in ((4, N), (4, 3), (4, H, N)))
        ctx.score_layer(q[0], ks[0], 0.1, s[0], m[0], head_cols_out=h[0], flags=binding.FLAG_NO_HEAD_STATS)
        binding.score_layer_static(H, Hkv, d, w, N, q[0], ks[0], 0.1, s[1], m[1], head_cols_out=h[1], flags=binding.FLAG_NO_HEAD_STATS)
        ctx.score_layers(q, ks, [0.1, 0.1], s[2:], m[2:], h[2:], ws)
        assert ctx.poll_device_status() == binding.OK
        return s, m[:, 0], h

    first = run(k)
    for a in first:
        assert torch.equal(a[0], a[1]) and torch.equal(a[0], a[2])
    cols, ent = reference(q[1], k[1], 0.1)
    torch.testing.assert_close(first[2][3].double(), cols, rtol=2e-4, atol=1e-7 / N)
    assert abs(first[1][3].item() - ent.item()) < 1e-4 * ent.item()
    for lay in (lambda x: x.transpose(0, 1).contiguous().transpose(0, 1),                        # [N, H_kv, d]
                lambda x: torch.nn.functional.pad(x, (0, 8, 0, 3))[:, :N, :d]):                  # room after rows and heads
        views = [lay(x) for x in k]
        assert not views[0].is_contiguous() or Hkv == 1
        for a, b in zip(run(views), first):
            assert torch.equal(a, b)
    ctx.close()
