"""Selection and head statistics at the sizes where their split over CTAs changes, against the oracle.
Selection (one CTA with 4, 8 or 16 entries a thread, clusters of two, four and eight, slices that do not fit the
registers): exact with ties.  Statistics (one CTA of 1024 or 512 threads for a vector, clusters for few long
ones): within the metric tolerance, and the same bits whatever the split."""
import numpy as np
import pytest
import torch

from oracle import structkv_oracle as O
from tests import parity as P

pytestmark = pytest.mark.gpu
EDGES = [1024, 4096, 8192, 16384, 32768, 65536, 131072, 262144]


@pytest.fixture(scope="module")
def ctx(cuda_device):
    from paper_2604_06746_b200 import binding
    c = binding.Context(4, 2, 128, 64, 1 << 19, torch.bfloat16, cuda_device)
    yield c
    c.close()


@pytest.mark.parametrize("batch", [1, 17])
@pytest.mark.parametrize("edge", EDGES)
def test_select_around_the_edges(ctx, edge, batch):
    rng = np.random.default_rng(edge + batch)
    for n in (edge + 63, edge + 64, edge + 65):              # prefix of edge - 1, edge, edge + 1 tokens
        sc = (rng.random((batch, n)) ** 3).astype(np.float32)
        sc[:, ::3] = np.float32(0.125)                       # a third of the tokens tie
        k = 64 + int(0.6 * n) if n % 2 else 64 + n // 50     # the threshold inside the ties, and above them
        out = torch.zeros((batch, k), dtype=torch.int32, device="cuda")
        ctx.select(torch.from_numpy(sc).cuda(), k, 64, out)
        got = out.cpu().numpy()
        for b in {0, batch - 1}:
            assert np.array_equal(got[b], O.select(sc[b], k, 64)), (n, b)


def test_select_beyond_the_registers_of_a_cluster(ctx):
    rng = np.random.default_rng(9)
    n, k = 300001, 40000
    sc = rng.integers(0, 1000, size=n).astype(np.float32)
    out = torch.zeros((1, k), dtype=torch.int32, device="cuda")
    ctx.select(torch.from_numpy(sc).cuda(), k, 64, out)
    assert np.array_equal(out[0].cpu().numpy(), O.select(sc, k, 64))


def test_packed_selection_of_unequal_prompts(ctx):
    rng = np.random.default_rng(10)
    lens, budgets = (70, 5000, 64, 40001, 900), (66, 5000, 64, 3000, 64)
    cu = np.concatenate([[0], np.cumsum(lens)]).tolist()
    sc = rng.integers(-50, 50, size=cu[-1]).astype(np.float32)
    out = torch.zeros((len(lens), 6000), dtype=torch.int32, device="cuda")
    ctx.select_batch(torch.from_numpy(sc).cuda(), cu, budgets, 64, out)
    got = out.cpu().numpy()
    for b, k in enumerate(budgets):
        assert np.array_equal(got[b, :k], O.select(sc[cu[b]:cu[b + 1]], k, 64)), b
        assert np.all(got[b, k:] == -1)


@pytest.mark.parametrize("edge", EDGES[1:])
def test_head_statistics_around_the_edges(ctx, edge):
    rng = np.random.default_rng(edge)
    for n in (edge, edge + 1):
        x = rng.random((1, 4, n)) ** 4
        x[:, :, ::5] = 0.0
        x[:, :2, 1::5] = 0.3                                 # ties across the threshold
        x[:, 3, 7] += 0.1 * n
        x32 = (x / x.sum(axis=2, keepdims=True)).astype(np.float32)
        m = torch.zeros((1, 3), device="cuda")
        ctx.head_stats(torch.from_numpy(x32).cuda(), m)
        rho, var = O.head_statistics(x32[0].astype(np.float64))
        P.assert_metric_close(m[0, 1].item(), rho, f"sparsity at {n}")
        P.assert_metric_close(m[0, 2].item(), var, f"variance at {n}")


@pytest.mark.parametrize("layers", [20, 40])
@pytest.mark.parametrize("n", [7, 601, 2048, 2049, 4097, 8192, 8193, 16385, 50000, 51200, 51201])
def test_head_statistics_of_many_vectors(ctx, layers, n):
    """An SM per vector, and more vectors than SMs: within the tolerance, and the bits of a layer by itself."""
    rng = np.random.default_rng(n + layers)
    buf = torch.zeros((layers, 4, n + 1), device="cuda")     # odd strides: every alignment of a vector
    x = rng.random((layers, 4, n)) ** 4
    x[:, :2, 1::5] = 0.3
    x32 = (x / x.sum(axis=2, keepdims=True)).astype(np.float32)
    buf[:, :, 1:] = torch.from_numpy(x32).cuda()
    m = torch.zeros((layers, 3), device="cuda")
    ctx.head_stats(buf[:, :, 1:], m)
    one = torch.zeros((1, 3), device="cuda")
    for l in {0, 1, layers - 1}:
        ctx.head_stats(buf[l:l + 1, :, 1:], one)
        assert torch.equal(m[l], one[0])
        rho, var = O.head_statistics(x32[l].astype(np.float64))
        P.assert_metric_close(m[l, 1].item(), rho, f"sparsity at {n}")
        P.assert_metric_close(m[l, 2].item(), var, f"variance at {n}")


@pytest.mark.parametrize("n", [32768, 32769, 40001, 131073, 262145, 400001])
def test_head_statistics_of_long_vectors(ctx, n):
    """4, 20, 48, 120 and 160 vectors: clusters of eight, four and two CTAs, one of 1024 threads, one of 512."""
    rng = np.random.default_rng(n)
    x = rng.random((4, 4, n)) ** 4
    x[:, :2, 1::5] = 0.3                                     # ties across the threshold
    x[3, :, ::2] = 0.0
    x[2, 3, 7] += 0.1 * n
    x32 = (x / x.sum(axis=2, keepdims=True)).astype(np.float32)
    four = torch.from_numpy(x32).cuda()
    one = torch.zeros((4, 3), device="cuda")
    for l in range(4):
        ctx.head_stats(four[l:l + 1], one[l:l + 1])
        rho, var = O.head_statistics(x32[l].astype(np.float64))
        P.assert_metric_close(one[l, 1].item(), rho, f"sparsity at {n}")
        P.assert_metric_close(one[l, 2].item(), var, f"variance at {n}")
    for layers in (5, 12, 30, 40):
        m = torch.zeros((layers, 3), device="cuda")
        ctx.head_stats(four[torch.arange(layers, device="cuda") % 4], m)
        assert torch.equal(m, one[torch.arange(layers, device="cuda") % 4]), layers


@pytest.mark.parametrize("H,Hkv,n", [(32, 8, 32769), (32, 8, 33000), (8, 2, 33002), (2, 1, 131076), (60, 4, 40000)])
def test_statistics_and_sums_of_a_long_layer(cuda_device, H, Hkv, n):
    """The launch that takes both (its grid in whole clusters): the bits of the sums without statistics and of the
    statistics without sums."""
    from paper_2604_06746_b200 import binding
    g = torch.Generator(device=cuda_device)
    g.manual_seed(n)
    q = torch.randn((H, 16, 64), generator=g, device=cuda_device).bfloat16()
    k = torch.randn((Hkv, n, 64), generator=g, device=cuda_device).bfloat16()
    c = binding.Context(H, Hkv, 64, 16, n, torch.bfloat16, cuda_device)
    s, acc, m, cols = (torch.zeros(x, device=cuda_device) for x in ((2, n), (2, n), (2, 3), (H, n)))
    for i, flags in enumerate((0, binding.FLAG_NO_HEAD_STATS)):
        for _ in range(2):                                   # the counters are left as they were found
            c.score_layer(q, k, 0.125, s[i], m[i], c_inout=acc[i], head_cols_out=cols, flags=flags)
    stats = torch.zeros((1, 3), device=cuda_device)
    c.head_stats(cols[None], stats)
    assert c.poll_device_status() == binding.OK
    assert torch.equal(s[0], s[1]) and torch.equal(acc[0], acc[1]) and m[0, 0] == m[1, 0]
    assert torch.equal(m[0, 1:], stats[0, 1:])
    c.close()


def test_few_long_vectors_use_the_whole_gpu(ctx):
    """Eight times the keys in no more than 2.5 times the time: 46 against 12 us with one SM per vector, 18 with
    clusters.  Best of many, both sides in turn."""
    x = torch.softmax(2.0 * torch.randn((1, 4, 262144), device="cuda"), dim=2)
    m, best = torch.zeros((1, 3), device="cuda"), {}
    for _ in range(10):
        for n in (32768, 262144):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for _ in range(50):
                ctx.head_stats(x[:, :, :n], m)
            b.record()
            torch.cuda.synchronize()
            best[n] = min(best.get(n, 1e9), a.elapsed_time(b))
    assert best[262144] < 2.5 * best[32768], best
