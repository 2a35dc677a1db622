"""What a whole prefill gathers in one launch (K and V of all layers, hidden states, positions) or, where a row is no
multiple of 16 bytes, in two: every row by torch's own indexing, from one block a slab to several."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [8, 12, 13, 96, 4096])
@pytest.mark.parametrize("seq,layers,budget", [(64, 1, 8), (700, 3, 9), (2049, 2, 1000), (5000, 5, 2500)])
def test_gathered_rows(cuda_device, dim, seq, layers, budget):
    from paper_2604_06746_b200 import binding, pipeline
    H, Hkv, d, w = 4, 2, 64, 8
    g = torch.Generator(device=cuda_device)
    g.manual_seed(dim + seq)
    rnd = lambda *s: torch.randn(s, generator=g, device=cuda_device).bfloat16()
    ls = []
    for _ in range(layers):
        kv = rnd(2, Hkv, seq, d)
        ls.append({"q_win": rnd(H, w, d), "k": kv[0], "v": kv[1], "kv": kv, "scale": 0.125})
    struct = min(seq, 2 * budget)
    hidden, pos = rnd(seq, dim), torch.randperm(seq, generator=g, device=cuda_device, dtype=torch.int32)
    pf = pipeline.Prefill(layers, H, Hkv, d, w, seq, budget, struct, torch.bfloat16, hidden_dim=dim, device=cuda_device)
    pf.run(ls, hidden, pos)
    assert pf._plan is not None and pf.ctx.poll_device_status() == binding.OK
    i = pf.i_struct.long()
    assert torch.equal(pf.hidden_out, hidden[i]) and torch.equal(pf.pos_out, pos[i])
    for l in range(layers):
        assert torch.equal(pf.kv_out[l], ls[l]["kv"][:, :, pf.i_kv[l].long()])
