"""Selection of so many vectors that the number of CTAs a vector gets depends on it (up to 8, up to 33, more), at the
last lengths of its forms: exact, with thresholds among equal keys and among keys that all differ."""
import numpy as np
import pytest
import torch

from oracle import structkv_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [8, 9, 33, 34])
@pytest.mark.parametrize("n", [16384, 32768, 32769, 65536, 65537])
@pytest.mark.parametrize("ties", [False, True])
def test_select_many_vectors(cuda_device, batch, n, ties):
    from paper_2604_06746_b200 import binding
    ctx = binding.Context(4, 2, 128, 64, 1024, torch.bfloat16, cuda_device)
    rng = np.random.default_rng(batch + n)
    sc = (rng.random((batch, n + 64)) ** 4).astype(np.float32)
    if ties:
        sc = np.round(sc * 50) / 50
    k = 64 + n // 9
    out = torch.zeros((batch, k), dtype=torch.int32, device="cuda")
    ctx.select(torch.from_numpy(sc).cuda(), k, 64, out)
    got = out.cpu().numpy()
    for b in (0, batch // 2, batch - 1):
        assert np.array_equal(got[b], O.select(sc[b], k, 64)), b
    ctx.close()


@pytest.mark.parametrize("batch,n", [(15, 16385), (15, 65537), (16, 65537), (15, 131072), (16, 131072), (30, 131137), (31, 131137),
                                     (16, 262144), (15, 262209), (16, 262209)])
def test_clusters_of_eight_and_of_four(cuda_device, batch, n):
    from paper_2604_06746_b200 import binding
    ctx = binding.Context(4, 2, 128, 64, 1024, torch.bfloat16, cuda_device)
    rng = np.random.default_rng(batch + n)
    sc = (rng.random((batch, n)) ** 4).astype(np.float32)
    sc[1::2] = np.round(sc[1::2] * 50) / 50                  # ties
    k = 64 + n // 9
    out = torch.zeros((batch, k), dtype=torch.int32, device="cuda")
    ctx.select(torch.from_numpy(sc).cuda(), k, 64, out)
    got = out.cpu().numpy()
    for b in (0, 1, batch // 2, batch - 1):
        assert np.array_equal(got[b], O.select(sc[b], k, 64)), b
    ctx.close()
