"""Row gathers over the shapes where units, rows, slabs and blocks do not divide one another: byte exact against the oracle's
indexing, with an index out of range in every kind of unit."""
import pytest
import torch

@pytest.mark.gpu
@pytest.mark.parametrize("slabs,n,row,k,pad", [
    (1, 40, 1, 40, 0), (3, 100, 7, 33, 0), (2, 300, 12, 299, 4), (5, 513, 16, 512, 0), (16, 700, 48, 511, 16),
    (7, 2000, 80, 1025, 0), (1, 5000, 8192, 1111, 0), (2, 64, 65552, 63, 0), (40000, 9, 16, 5, 0), (3, 1, 4, 1, 0)])
def test_rows(cuda_device, slabs, n, row, k, pad):
    from paper_2604_06746_b200 import binding
    ctx = binding.Context(8, 2, 64, 8, 512, torch.bfloat16, cuda_device)
    src = torch.randint(0, 256, (slabs, n, row + pad), dtype=torch.uint8, device=cuda_device)[..., :row]
    idx = torch.randint(0, n, (k,), device=cuda_device).int()
    out = torch.zeros((slabs, k, row), dtype=torch.uint8, device=cuda_device)
    ctx.compact(src, idx, out)
    assert torch.equal(out, src[:, idx.long()])
    lists = torch.randint(0, n, (min(slabs, 50), k), device=cuda_device).int()
    out = torch.zeros((len(lists), k, row), dtype=torch.uint8, device=cuda_device)
    ctx.compact_per_slab(src[:len(lists)], lists, out)
    assert torch.equal(out, torch.stack([s[i.long()] for s, i in zip(src, lists)]))
    both = torch.zeros((2, slabs, k, row), dtype=torch.uint8, device=cuda_device)
    ctx.compact_layers([src, src], lists[:1].repeat(2, 1), both)
    assert all(torch.equal(b, src[:, lists[0].long()]) for b in both)
    assert ctx.poll_device_status() == binding.OK
    idx[k // 2] = n                                        # nothing is copied for it, and it is recorded
    out = torch.full((slabs, k, row), 99, dtype=torch.uint8, device=cuda_device)
    ctx.compact(src, idx, out)
    ok = torch.arange(k, device=cuda_device) != k // 2
    assert torch.equal(out[:, ok], src[:, idx[ok].long()]) and (out[:, ~ok] == 99).all()
    assert ctx.poll_device_status() == binding.ERR_INVALID_ARG
    ctx.close()


def test_division_by_row_units():
    """The multiplication that stands for u / d, u < 2^31 (the rule of csrc/compact.cu, restated)."""
    import random
    rng = random.Random(1)
    for d in [*range(1, 300), 4095, 4096, 4097, 65537, (1 << 20) + 1, (1 << 30) - 1, 1 << 30, (1 << 30) + 1, (1 << 31) - 1]:
        l = (d - 1).bit_length()
        mul, shift = (0, 0) if d == 1 else ((1 << (31 + l)) // d + 1, l - 1)
        assert mul < 1 << 32
        top = (1 << 31) - 1
        for u in {0, 1, d - 1, d, d + 1, top, top // d * d, top // d * d - 1, *(rng.randrange(1 << 31) for _ in range(50))}:
            if 0 <= u <= top:
                assert (u if mul == 0 else (u * mul >> 32) >> shift) == u // d, (u, d)
