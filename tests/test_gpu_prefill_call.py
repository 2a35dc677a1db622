"""structkv_pivot_select and structkv_prefill against the separate calls they stand for: the same bits, the
same pivot and transition scores, also with a cap, without hidden states, with one layer, and when the
tensors change from call to call."""
import gc
import weakref

import pytest
import torch

from paper_2604_06746_b200 import synth

pytestmark = pytest.mark.gpu
OUT = ("s_hist", "metrics", "c_running", "c_star", "i_kv", "i_struct", "kv_out")


def step_by_step(pf, layers, hidden, positions):
    """The separate entry points, pivot on the host."""
    pf.score_all(layers)
    pf.finish_scores(len(layers))
    pf.pivot, pf.transition = pf.ctx.pivot(pf.metrics, pf.weights, pf.l_limit)
    pf.ctx.accumulate(pf.s_hist, pf.pivot, pf.lam, pf.c_star)
    pf.ctx.select(pf.s_hist, pf.kv_budget, pf.w, pf.i_kv)
    pf.ctx.select(pf.c_star, pf.struct_budget, pf.w, pf.i_struct)
    pf.compact_all_kv(layers)
    if hidden is not None:
        pf.compact_hidden(hidden, positions)


@pytest.mark.parametrize("name,seq,n_layers,budget,l_limit,with_hidden", [
    ("llama32k", 3000 + 1, 6, 300, -1, True), ("llama32k", 20000, 5, 1000, 2, True), ("tiny", 2048, 4, 256, -1, True),
    ("qwen64k", 1500, 3, 200, 1, False), ("llama32k", 900, 1, 100, -1, True)])
def test_one_call_equals_the_separate_calls(cuda_device, name, seq, n_layers, budget, l_limit, with_hidden):
    from paper_2604_06746_b200 import binding, pipeline
    wl = synth.WORKLOADS[name].scaled(seq, n_layers=n_layers, n_hubs=6, budgets=(budget,))
    pl = synth.plan(wl)
    dt = synth.torch_dtype(wl.dtype)
    sets = []
    for shift in (0, 1):                                  # two prompts: a reused context must not mix them up
        ls = [synth.make_layer(wl, pl, (l + shift) % n_layers, device=cuda_device) for l in range(n_layers)]
        hid = torch.randn((seq, 96), device=cuda_device).to(torch.bfloat16) if with_hidden else None
        pos = torch.arange(seq, device=cuda_device, dtype=torch.int32) + shift if with_hidden else None
        sets.append((ls, hid, pos))
    make = lambda: pipeline.Prefill(wl.n_layers, wl.n_q_heads, wl.n_kv_heads, wl.head_dim, wl.window, wl.seq, budget,
                                    wl.struct_budget(), dt, hidden_dim=96 if with_hidden else 0, device=cuda_device,
                                    l_limit=l_limit)
    one, ref = make(), make()
    one.c_running.fill_(7.0)                              # C starts from zero whatever the buffer holds
    for ls, hid, pos in (sets[0], sets[1], sets[1], sets[0]):
        one.run(ls, hid, pos)
        assert one._plan is not None
        step_by_step(ref, ls, hid, pos)
        torch.cuda.synchronize()
        assert one.pivot == ref.pivot and one.transition == ref.transition
        for key in OUT + (("hidden_out", "pos_out") if with_hidden else ()):
            assert torch.equal(getattr(one, key), getattr(ref, key)), key
    assert one.ctx.poll_device_status() == binding.OK


def test_pivot_on_the_device_equals_the_host_rule(cuda_device):
    """Ties, constant columns, NaN columns (head statistics switched off), many layers."""
    from paper_2604_06746_b200 import binding
    n, w = 200, 8
    ctx = binding.Context(8, 2, 64, w, n, torch.float32, cuda_device)
    g = torch.Generator().manual_seed(1)
    for L in (1, 2, 3, 33, 128, 131):                     # 131: beyond the device form
        for kind in range(4):
            m = torch.rand((L, 3), generator=g)
            if kind == 1:
                m[:, 1] = 0.25                            # zero range
            if kind == 2:
                m[:, 1:] = float("nan")
            if kind == 3:
                m = torch.round(m * 2) / 2                # tied transitions: the first maximum wins
            m = m.to(cuda_device)
            s = torch.rand((L, n), device=cuda_device)
            c1, c2 = torch.zeros(n, device=cuda_device), torch.zeros(n, device=cuda_device)
            i_kv = torch.zeros((L, 50), dtype=torch.int32, device=cuda_device)
            i_st = torch.zeros(90, dtype=torch.int32, device=cuda_device)
            for limit in (-1, 1):
                got = ctx.pivot_select(s, m, (0.2, 0.3, 0.5), limit, 0.9, w, 50, i_kv, 90, c1, i_st)
                want = ctx.pivot(m, (0.2, 0.3, 0.5), limit)
                assert got == want, (L, kind, limit)
                ctx.accumulate(s, want[0], 0.9, c2)
                assert torch.equal(c1, c2)
    ctx.close()


def prompt(cuda_device, seq, n_layers, budget, shift=0, **more):
    from paper_2604_06746_b200 import pipeline
    wl = synth.WORKLOADS["llama32k"].scaled(seq, n_layers=n_layers, n_hubs=6, budgets=(budget,))
    pl = synth.plan(wl)
    layers = [synth.make_layer(wl, pl, (l + shift) % n_layers, device=cuda_device) for l in range(n_layers)]
    hidden = torch.randn((seq, 96), device=cuda_device).to(torch.bfloat16)
    positions = torch.arange(seq, device=cuda_device, dtype=torch.int32) + shift
    pf = pipeline.Prefill(wl.n_layers, wl.n_q_heads, wl.n_kv_heads, wl.head_dim, wl.window, wl.seq, budget,
                          wl.struct_budget(), torch.bfloat16, hidden_dim=96, device=cuda_device, **more)
    return pf, (layers, hidden, positions)


def test_every_run_reads_the_attributes(cuda_device):
    """Hyper-parameters, flags and output buffers changed between two runs over the very same tensors count for
    the second one, as they do for a Prefill made with them."""
    from paper_2604_06746_b200 import binding
    pf, args = prompt(cuda_device, 2001, 6, 300)
    pf.run(*args)
    changes = [dict(weights=(0.0, 0.0, 1.0)), dict(weights=(1.0, 0.0, 0.0)), dict(l_limit=1), dict(lam=0.25),
               dict(flags=binding.FLAG_FORCE_SIMT), dict(flags=0, l_limit=-1)]
    now = {}
    for change in changes:
        now.update(change)
        for name, value in change.items():
            setattr(pf, name, value)
        fresh, _ = prompt(cuda_device, 2001, 6, 300, **now)
        pf.run(*args)
        fresh.run(*args)
        assert (pf.pivot, pf.transition) == (fresh.pivot, fresh.transition), change
        for key in OUT + ("hidden_out", "pos_out"):
            assert torch.equal(getattr(pf, key), getattr(fresh, key)), (change, key)
    for key in OUT + ("hidden_out", "pos_out"):
        old = getattr(pf, key)
        was = old.clone()
        old.zero_()
        setattr(pf, key, torch.empty_like(old))
        pf.run(*args)
        assert torch.equal(getattr(pf, key), was) and not old.any(), key
    pf.i_kv = pf.i_kv.long()                              # a buffer that does not fit is refused, not written to
    with pytest.raises(AssertionError):
        pf.run(*args)


def test_a_finished_run_keeps_no_tensor_of_its_prompt(cuda_device):
    pf, args = prompt(cuda_device, 1501, 4, 200)
    pf.run(*args)
    gone = [weakref.ref(t) for d in args[0] for t in d.values() if torch.is_tensor(t)] + [weakref.ref(t) for t in args[1:]]
    torch.cuda.synchronize()
    del args
    gc.collect()
    assert not [r() for r in gone if r() is not None]


def test_the_gather_reads_the_layout_of_every_call(cuda_device):
    """Head-major and token-major K/V at the same addresses, another output buffer, nothing kept afterwards."""
    from paper_2604_06746_b200 import pipeline
    L, Hkv, N, d, budget = 3, 2, 300, 64, 40
    pf = pipeline.Prefill(L, 4, Hkv, d, 8, N, budget, 80, torch.bfloat16, device=cuda_device)
    pf.i_kv.copy_(torch.stack([torch.randperm(N, device=cuda_device)[:budget].sort().values for _ in range(L)]))
    raw = [torch.randn(2 * Hkv * N * d, device=cuda_device).to(torch.bfloat16) for _ in range(L)]
    views = (lambda x: x.view(2, Hkv, N, d), lambda x: x.view(N, 2, Hkv, d).permute(1, 2, 0, 3))
    for view in (*views, views[0]):
        layers = [{"kv": view(x)} for x in raw]
        pf.kv_out = torch.zeros_like(pf.kv_out)
        pf.compact_all_kv(layers)
        for l, t in enumerate(layers):
            assert torch.equal(pf.kv_out[l], t["kv"][:, :, pf.i_kv[l].long()])
    gone = [weakref.ref(x) for x in raw]
    del raw, layers, t, view
    gc.collect()
    assert not [r() for r in gone if r() is not None]
