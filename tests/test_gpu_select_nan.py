"""Selection among NaN scores: they come first, ties to the lower index, and nothing is written
beyond a row of the output, however many of them there are.  Vectors of every form (CTAs, items a thread, slices that do not
fit the registers)."""
import numpy as np
import pytest
import torch

from oracle import structkv_oracle as O

pytestmark = pytest.mark.gpu
GUARD, W = 4096, 16


def expected(sc, k):
    return O.select(np.where(np.isnan(sc), np.inf, sc), k, W)


@pytest.mark.parametrize("batch,n", [(1, 700), (3, 8000), (2, 16000), (40, 16000), (2, 32768), (20, 32000), (40, 32000), (1, 65000),
                                     (9, 60000), (1, 131072), (17, 100000), (1, 300000), (17, 150000)])
@pytest.mark.parametrize("nans", ["all", "one more than kept", "as many as kept", "few"])
def test_nan_scores_stay_in_their_row(cuda_device, batch, n, nans):
    from paper_2604_06746_b200 import binding
    ctx = binding.Context(4, 2, 128, 64, 1024, torch.bfloat16, cuda_device)
    k = W + n // 11
    rng = np.random.default_rng(n + batch)
    sc = rng.random((batch, n), dtype=np.float32)
    count = {"all": n, "one more than kept": k - W + 1, "as many as kept": k - W, "few": 5}[nans]
    for row in sc:                                           # bits and signs of all kinds
        row[rng.permutation(n - W)[:count] if nans != "all" else slice(None)] = np.nan
    bits = sc.view(np.uint32)
    bits[np.isnan(sc)] ^= rng.integers(0, 2, np.isnan(sc).sum(), dtype=np.uint32) << np.uint32(31)
    got = torch.full((GUARD + batch * k + GUARD,), -7, dtype=torch.int32, device=cuda_device)
    scores, cu = torch.from_numpy(sc).cuda(), [n * b for b in range(batch + 1)]
    ctx.select(scores, k, W, got[GUARD:-GUARD].view(batch, k))
    packed = torch.full_like(got, -7)
    many = min(batch, 32)
    ctx.select_batch(scores.view(-1)[:many * n], cu[:many + 1], [k] * many, W, packed[GUARD:GUARD + many * k].view(many, k))
    got, packed = got.cpu().numpy(), packed.cpu().numpy()
    for out, rows in ((got, batch), (packed, many)):
        assert (out[:GUARD] == -7).all() and (out[GUARD + rows * k:] == -7).all()
        for b in range(rows):
            assert np.array_equal(out[GUARD + b * k:GUARD + (b + 1) * k], expected(sc[b], k)), b
    ctx.close()


@pytest.mark.parametrize("n", [700, 8000, 16000, 32768, 65000, 131072, 300000])
@pytest.mark.parametrize("more", [1, 40, None])
def test_the_largest_key_is_the_threshold(cuda_device, n, more):
    """NaN with all of their bits set: no key lies above them."""
    from paper_2604_06746_b200 import binding
    ctx = binding.Context(4, 2, 128, 64, 1024, torch.bfloat16, cuda_device)
    k, rng = W + n // 13, np.random.default_rng(n)
    sc = rng.random((2, n), dtype=np.float32)
    for row in sc.view(np.uint32):
        at = slice(None) if more is None else rng.permutation(n - W)[:k - W + more]
        row[at] = rng.integers(0, 2, len(row[at]), dtype=np.uint32) << np.uint32(31) | np.uint32(0x7fffffff)
    got = torch.full((GUARD + 2 * k + GUARD,), -7, dtype=torch.int32, device=cuda_device)
    ctx.select(torch.from_numpy(sc).cuda(), k, W, got[GUARD:-GUARD].view(2, k))
    got = got.cpu().numpy()
    assert (got[:GUARD] == -7).all() and (got[-GUARD:] == -7).all()
    for b in range(2):
        assert np.array_equal(got[GUARD + b * k:GUARD + (b + 1) * k], expected(sc[b], k)), b
    ctx.close()


@pytest.mark.parametrize("H,Hkv,d,w,N,dtype", [(32, 8, 128, 64, 3000, torch.bfloat16), (8, 2, 64, 32, 1500, torch.float32)])
def test_nan_queries_keep_lists_whole(cuda_device, H, Hkv, d, w, N, dtype):
    """A whole prefill with a head of them: every list is ascending, within the prompt and ends with the window."""
    from paper_2604_06746_b200 import binding, pipeline
    L, budget = 3, N // 10
    g = torch.Generator(device=cuda_device)
    g.manual_seed(N)
    layers = []
    for _ in range(L):
        kv = torch.randn((2, Hkv, N, d), generator=g, device=cuda_device).to(dtype)
        q = torch.randn((H, w, d), generator=g, device=cuda_device).to(dtype)
        layers.append({"q_win": q, "k": kv[0], "v": kv[1], "kv": kv, "scale": d ** -0.5})
    layers[1]["q_win"][H // 2] = float("nan")
    pf = pipeline.Prefill(L, H, Hkv, d, w, N, budget, 2 * budget, dtype, device=cuda_device)
    pf.run(layers)
    assert pf.ctx.poll_device_status() == binding.OK and pf.s_hist[1, :N - w].isnan().all() and not pf.s_hist[0].isnan().any()
    for ids in (*pf.i_kv, pf.i_struct):
        assert ids[0] >= 0 and (ids.diff() > 0).all() and torch.equal(ids[-w:], torch.arange(N - w, N, device=cuda_device, dtype=ids.dtype))
    for l in range(L):
        assert torch.equal(pf.kv_out[l], layers[l]["kv"][:, :, pf.i_kv[l].long()])
