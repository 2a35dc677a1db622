"""The native module behind the binding, on the CPU: the argument block of a prefill field by field, the forms it
leaves to the step-by-step path, and the checks that refuse a call before it reaches the library."""
import ctypes

import pytest
import torch


@pytest.fixture(scope="module")
def B():
    from paper_2604_06746_b200 import build
    build.build()
    from paper_2604_06746_b200 import binding
    return binding


L, H, HKV, N, D, W, BUDGET, ROWS = 3, 6, 2, 50, 64, 4, 9, 20


class Prompt:
    """CPU tensors in the form of the one-call path."""

    def __init__(self, token_major=False, dtype=torch.bfloat16, hkv=HKV):
        self.hkv, self.dtype = hkv, dtype
        kv = [torch.empty((N, 2, hkv, D), dtype=dtype).permute(1, 2, 0, 3) if token_major else torch.empty((2, hkv, N, D), dtype=dtype)
              for _ in range(L)]
        self.layers = [{"q_win": torch.empty((H, W, D), dtype=dtype), "k": x[0], "v": x[1], "kv": x, "scale": 0.1 * (l + 1)}
                       for l, x in enumerate(kv)]
        self.hidden = torch.empty((N, 24), dtype=torch.bfloat16)[:, :16]
        self.positions = torch.empty(2 * N, dtype=torch.int32)[::2]
        f, i = torch.float32, torch.int32
        self.s_hist, self.head_cols, self.metrics = torch.empty((L, N)), torch.empty((L, H, N)), torch.empty((L, 3))
        self.c_running, self.c_star = torch.empty(N, dtype=f), torch.empty(N, dtype=f)
        self.i_kv, self.i_struct = torch.empty((L, BUDGET), dtype=i), torch.empty(ROWS, dtype=i)
        self.kv_out = torch.empty((L, 2, hkv, BUDGET, D), dtype=dtype)
        self.hidden_out, self.pos_out = torch.empty((ROWS, 16), dtype=torch.bfloat16), torch.empty(ROWS, dtype=i)
        self.ws = torch.empty(1000, dtype=torch.uint8)
        self.weights = (0.2, 0.3, 0.5)

    def fill(self, B, block):
        return B.fill_prefill(block, self.layers, self.hidden, self.positions, self.s_hist, self.head_cols, self.metrics,
                              self.c_running, self.c_star, self.i_kv, self.i_struct, self.kv_out, self.hidden_out, self.pos_out,
                              self.ws, (H, self.hkv, N, D, W, BUDGET, ROWS, -1), self.dtype, 0.9, self.weights)


@pytest.mark.parametrize("token_major", [False, True])
@pytest.mark.parametrize("dtype,hkv", [(torch.bfloat16, 2), (torch.float32, 2), (torch.bfloat16, 1)])
def test_block_of_a_prefill(B, token_major, dtype, hkv):
    p = Prompt(token_major, dtype, hkv)
    block = B.PrefillArgs.for_layers(L)
    assert p.fill(B, block) is True
    kv0, es = p.layers[0]["kv"], p.kv_out.element_size()
    for l, t in enumerate(p.layers):
        assert (block.q_windows[l], block.ks[l], block.kv_srcs[l]) == tuple(t[n].data_ptr() for n in ("q_win", "k", "kv"))
        assert block.scales[l] == ctypes.c_float(t["scale"]).value
    want = dict(n_layers=L, k_stride_head=kv0.stride(1), k_stride_token=kv0.stride(2), n_keys=N, lam=ctypes.c_float(0.9).value,
                s_out=p.s_hist.data_ptr(), s_layer_stride=N, c_out=p.c_running.data_ptr(), head_cols=p.head_cols.data_ptr(),
                head_cols_layer_stride=H * N, metrics=p.metrics.data_ptr(), layers_workspace=p.ws.data_ptr(),
                layers_workspace_bytes=1000, l_limit=-1, window=W, kv_budget=BUDGET, struct_budget=ROWS,
                i_kv=p.i_kv.data_ptr(), i_struct=p.i_struct.data_ptr(), c_star=p.c_star.data_ptr(),
                kv_slab_stride_bytes=kv0.stride(1 if hkv > 1 else 0) * es, kv_row_stride_bytes=kv0.stride(2) * es, kv_row_bytes=D * es,
                kv_slabs=2 * hkv, kv_rows=N, kv_dst=p.kv_out.data_ptr(), kv_dst_layer_stride_bytes=2 * hkv * BUDGET * D * es,
                hidden=p.hidden.data_ptr(), hidden_row_stride_bytes=48, hidden_row_bytes=32, hidden_dst=p.hidden_out.data_ptr(),
                positions=p.positions.data_ptr(), position_row_stride_bytes=8, position_row_bytes=4,
                positions_dst=p.pos_out.data_ptr())
    assert {k: getattr(block, k) for k in want} == want
    assert list(block.weights) == [ctypes.c_float(x).value for x in p.weights]
    p.hidden = p.positions = None
    assert p.fill(B, block) is True
    assert block.hidden is block.hidden_dst is block.positions is block.positions_dst is None


def other(p, name, value):
    setattr(p, name, value)


CHANGES = {
    "too few layers": lambda p: p.layers.pop(),
    "no joint storage": lambda p: p.layers[1].pop("kv"),
    "another mapping": lambda p: p.layers.__setitem__(0, __import__("types").MappingProxyType(p.layers[0])),
    "K of another length": lambda p: p.layers[0].update(k=p.layers[0]["k"][:, :-1]),
    "K of another layout": lambda p: p.layers[2].update(k=p.layers[2]["k"].transpose(1, 2).contiguous().transpose(1, 2)),
    "K/V of another shape": lambda p: p.layers[1].update(kv=p.layers[1]["kv"][:, :, :-1]),
    "K/V of another dtype": lambda p: p.layers[1].update(kv=p.layers[1]["kv"].float()),
    "queries of another dtype": lambda p: p.layers[1].update(q_win=p.layers[1]["q_win"].float()),
    "queries with gaps": lambda p: p.layers[1].update(q_win=torch.empty((H, W, 2 * D), dtype=p.dtype)[..., :D]),
    "slabs without a stride": lambda p: p.layers.__setitem__(slice(None), [
        dict(t, kv=x, k=x[0]) for t in p.layers for x in [torch.empty((2, HKV + 1, N, D), dtype=p.dtype)[:, :HKV]]]),
    "history of another length": lambda p: other(p, "s_hist", torch.empty((L, N + 1))),
    "history with gaps": lambda p: other(p, "s_hist", torch.empty((L, 2 * N))[:, :N]),
    "long indices": lambda p: other(p, "i_kv", p.i_kv.long()),
    "float64 metrics": lambda p: other(p, "metrics", p.metrics.double()),
    "output of another budget": lambda p: other(p, "kv_out", p.kv_out[:, :, :, :-1]),
    "hidden states with gaps": lambda p: other(p, "hidden", torch.empty((N, 32), dtype=torch.bfloat16)[:, ::2]),
    "hidden states of another dtype": lambda p: other(p, "hidden", p.hidden.float()),
    "no place for hidden states": lambda p: other(p, "hidden_out", None),
    "long positions": lambda p: other(p, "positions", p.positions.long()),
}


@pytest.mark.parametrize("change", CHANGES)
def test_forms_left_to_the_step_by_step_path(B, change):
    p = Prompt()
    assert p.fill(B, B.PrefillArgs.for_layers(L)) is True
    CHANGES[change](p)
    assert p.fill(B, B.PrefillArgs.for_layers(L)) is False


def test_checks_before_the_library(B):
    ctx = object.__new__(B.Context)                        # no device: the checks come first
    ctx._h, ctx.cfg, ctx.dtype = ctypes.c_void_p(), B.Config(4, 2, 64, 4, 100, B.BF16), torch.bfloat16
    q, k = torch.empty((4, 4, 64), dtype=torch.bfloat16), torch.empty((2, 100, 64), dtype=torch.bfloat16)
    s, m, i = torch.empty(100), torch.empty(3), torch.empty(10, dtype=torch.int32)
    for bad in (lambda: ctx.score_layer(q[..., :32], k, 1.0, s, m), lambda: ctx.score_layer(q, k.transpose(1, 2), 1.0, s, m),
                lambda: ctx.score_layer(q.float(), k, 1.0, s, m), lambda: ctx.score_layer(q, k.float(), 1.0, s, m),
                lambda: ctx.select(s.double(), 10, 4, i), lambda: ctx.select(s, 10, 4, i.long()), lambda: ctx.select(s, 9, 4, i),
                lambda: ctx.select(torch.empty(200)[::2], 10, 4, i), lambda: ctx.select(s, 5, 4, torch.empty(10, dtype=torch.int32)[::2]),
                lambda: ctx.compact(k, i.long(), torch.empty(2, 10, 64)), lambda: ctx.compact(k, i, torch.empty(2, 10, 128)[..., ::2]),
                lambda: ctx.compact(torch.empty(2, 9, 8, 64)[..., ::2], i, s), lambda: ctx.compact_per_slab(k, i, s),
                lambda: ctx.compact_per_slab(k, torch.empty((3, 5), dtype=torch.int32), s),
                lambda: ctx.group_saliency(torch.empty(4, 100), torch.empty(3, 100)),
                lambda: ctx.group_saliency(torch.empty(5, 100), torch.empty(2, 100)),
                lambda: ctx.group_saliency(torch.empty(4, 100), torch.empty(2, 99)),
                lambda: ctx.block_scores(s, 16, torch.empty(6)), lambda: ctx.block_scores(s.double(), 16, torch.empty(7)),
                lambda: ctx.mass_recovery(s, i.long(), torch.empty(1)), lambda: ctx.mass_recovery(s, i, torch.empty(2))):
        with pytest.raises(AssertionError):
            bad()
    with pytest.raises(TypeError):
        ctx.select([1.0, 2.0], 1, 0, i)
    with pytest.raises(IndexError):
        ctx.compact(k[:0], i, s)
