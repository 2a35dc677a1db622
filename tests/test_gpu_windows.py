"""The tensor-core scorer over windows, groupings and logit scales: every layout of the score rows (the
narrow ones of up to 32 and 64 rows per KV group, heads of 8 .. 256 rows in 256-row blocks, windows
that are no power of two), sequences from the window itself to ragged key tiles, against the
attention written out in float64."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


def reference(q, k, scale):
    H, w, _ = q.shape
    Hkv, N, _ = k.shape
    x = torch.einsum("hid,hjd->hij", q.double(), k.double().repeat_interleave(H // Hkv, 0)) * scale
    i, j = torch.arange(w, device=q.device)[:, None], torch.arange(N, device=q.device)[None]
    p = torch.softmax(x.masked_fill((j > N - w + i)[None], -math.inf), -1)
    return p.mean(1), -torch.special.xlogy(p, p).sum(-1).mean()


def score(cuda_device, H, Hkv, d, w, N, scale):
    from paper_2604_06746_b200 import binding
    g = torch.Generator(device=cuda_device)
    g.manual_seed(1000 * w + N)
    q = torch.randn((H, w, d), generator=g, device=cuda_device).bfloat16()
    k = torch.randn((Hkv, N, d), generator=g, device=cuda_device).bfloat16()
    ctx = binding.Context(H, Hkv, d, w, N, torch.bfloat16, cuda_device)
    s, m = torch.zeros(N, device=cuda_device), torch.zeros(3, device=cuda_device)
    cols = torch.zeros((H, N), device=cuda_device)
    ctx.score_layer(q, k, scale, s, m, head_cols_out=cols)
    assert ctx.poll_device_status() == binding.OK
    ref_cols, ref_ent = reference(q, k, scale)
    torch.testing.assert_close(cols.double(), ref_cols, rtol=2e-4, atol=1e-7 / N)
    torch.testing.assert_close(s.double(), ref_cols.sum(0), rtol=2e-4, atol=1e-7 * H / N)
    assert abs(m[0].item() - ref_ent.item()) < 1e-4 * abs(ref_ent.item()) + 1e-5
    ctx.close()


@pytest.mark.parametrize("H,Hkv,d,w,N", [
    (32, 8, 128, 8, 8), (32, 8, 128, 8, 900), (32, 8, 128, 8, 20011),       # 32 rows per group
    (32, 8, 128, 16, 3001), (28, 4, 128, 8, 257), (4, 4, 64, 64, 555),      # 64 rows
    (8, 8, 64, 32, 127), (2, 2, 128, 1, 500), (6, 2, 128, 5, 130),          # narrow, heads that are not full
    (28, 4, 64, 16, 3000), (32, 1, 128, 8, 3000), (32, 2, 64, 16, 3333),    # wide blocks of short heads
    (8, 2, 128, 40, 1000), (4, 1, 128, 100, 1111), (4, 4, 128, 200, 2000),  # padded windows
    (2, 1, 64, 256, 256), (5, 1, 128, 64, 129), (3, 1, 128, 256, 4097),
])
def test_windows_and_groupings(cuda_device, H, Hkv, d, w, N):
    score(cuda_device, H, Hkv, d, w, N, 1 / math.sqrt(d))


@pytest.mark.parametrize("w", [8, 64])
@pytest.mark.parametrize("scale", [-0.1, 0.0, 1.0])
def test_unusual_scales(cuda_device, w, scale):
    """A negative scale flips the logits inside the MMA, a zero one makes the attention uniform, a large
    one makes it so sharp that a chunk's logits rise far above the reference they started from."""
    score(cuda_device, 32, 8, 128, w, 3000, scale)


@pytest.mark.parametrize("L,H,Hkv,d,w,N", [
    (37, 8, 2, 64, 32, 700), (9, 32, 8, 128, 8, 1281), (5, 8, 2, 128, 16, 24577), (40, 6, 2, 64, 5, 513),
    (4, 4, 4, 64, 64, 131), (3, 32, 8, 128, 64, 2000),
])
def test_layers_of_one_launch(cuda_device, L, H, Hkv, d, w, N):
    """structkv_score_layers, also beyond the problems one launch holds and with sequences short enough for
    the first pass to run several layers ahead: the bits of the layer-by-layer calls."""
    from paper_2604_06746_b200 import binding
    g = torch.Generator(device=cuda_device)
    g.manual_seed(3)
    qs = [torch.randn((H, w, d), generator=g, device=cuda_device).bfloat16() for _ in range(L)]
    ks = [torch.randn((Hkv, N, d), generator=g, device=cuda_device).bfloat16() for _ in range(L)]
    ctx = binding.Context(H, Hkv, d, w, N, torch.bfloat16, cuda_device)
    s1, s2 = (torch.zeros((L, N), device=cuda_device) for _ in range(2))
    m1, m2 = (torch.zeros((L, 3), device=cuda_device) for _ in range(2))
    h1, h2 = (torch.zeros((L, H, N), device=cuda_device) for _ in range(2))
    for l in range(L):
        ctx.score_layer(qs[l], ks[l], 0.125, s1[l], m1[l], head_cols_out=h1[l], flags=binding.FLAG_NO_HEAD_STATS)
    ctx.score_layers(qs, ks, [0.125] * L, s2, m2, h2, ctx.layers_workspace(L))
    assert ctx.poll_device_status() == binding.OK
    assert torch.equal(s1, s2) and torch.equal(h1, h2) and torch.equal(m1[:, 0], m2[:, 0])
    ctx.close()
