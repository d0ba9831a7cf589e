"""Sequences of different lengths in shared launches (groups of 16 in one launch per kernel): every
sequence of a ragged call leaves what a call of its own leaves, bit for bit, for every kernel path, with more
sequences than one group, lengths around the row blocks and tiles, and NaN in every cache row past a sequence's end."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

LENS = [1, 700, 8, 9, 63, 64, 65, 127, 128, 129, 255, 256, 257, 31, 300, 1000, 17, 5, 130, 66]


@pytest.mark.parametrize("source,dtype,d,g", [("query", "bf16", 64, 4), ("query", "bf16", 64, 1), ("query", "bf16", 128, 2),
                                              ("key", "bf16", 64, 2), ("key", "bf16", 128, 4), ("key_packed", "bf16", 64, 4),
                                              ("bottom_up", "bf16", 64, 2), ("query", "f32", 64, 2), ("query", "f32", 128, 1)])
@pytest.mark.parametrize("shape", ["block", "sliding"])
def test_ragged_call_equals_single_calls(source, dtype, d, g, shape):
    from paper_2507_19608_b200 import binding as B
    Hk, n = 2, len(LENS)
    H, T_max = g * Hk, max(LENS) + 3
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    src = {"query": B.DELTA_SRC_QUERY, "key": B.DELTA_SRC_KEY, "key_packed": B.DELTA_SRC_KEY,
           "bottom_up": B.DELTA_SRC_QUERY_BOTTOM_UP}[source]
    win = B.DELTA_WIN_BLOCK if shape == "block" else B.DELTA_WIN_SLIDING
    gen = torch.Generator("cuda").manual_seed(11)
    rnd = lambda *s: torch.randn(*s, generator=gen, device="cuda").to(dt)      # noqa: E731
    kc = torch.full((n, Hk, T_max, d), float("nan"), dtype=dt, device="cuda")
    vc, qs, wins = kc.clone(), [], []
    for b, T in enumerate(LENS):
        kc[b, :, :T], vc[b, :, :T] = rnd(Hk, T, d), rnd(Hk, T, d)
        qs.append(rnd(H, T, d))
        wins.append((0, 40, 64, 128, 1000)[b % 5])

    def state(batch):
        st = B.delta_state_init(B.make_config(batch, H, Hk, d, T_max, dtype, source=src, prefill_window=win))
        if source == "key_packed":
            B.delta_state_set_key_cache(st, True)
        return st
    st = state(n)
    packed = torch.cat([x.reshape(-1) for x in qs])
    out = torch.full_like(packed, float("nan"))
    B.delta_attn_prefill_varlen(st, packed, kc, vc, out, LENS, wins, 0.6)
    Hs = Hk if source.startswith("key") else H
    shapes = {B.DELTA_VIEW_DQ: (T_max, d), B.DELTA_VIEW_MASK: (T_max, d // 32), B.DELTA_VIEW_ROW_NNZ: (T_max,),
              B.DELTA_VIEW_IDX: (T_max, d), B.DELTA_VIEW_QHAT: (d,), B.DELTA_VIEW_TILE_NNZ: (-(-T_max // 64),)}
    if source == "query":
        shapes[B.DELTA_VIEW_R] = (T_max,)

    def arrays(s, batch, b, T):
        res = {}
        for what, tail in shapes.items():
            x = B.delta_state_view(s, what).reshape(-1)[:batch * Hs * int(torch.tensor(tail).prod())].view(batch, Hs, *tail)[b]
            res[what] = x if what == B.DELTA_VIEW_QHAT else x[:, :-(-T // 64)] if what == B.DELTA_VIEW_TILE_NNZ else x[:, :T]
        return res
    at, total = 0, None
    for b, T in enumerate(LENS):
        one = state(1)
        o = torch.full_like(qs[b], float("nan"))[None]
        B.delta_attn_prefill(one, qs[b][None], kc[b:b + 1], vc[b:b + 1], o, T, H, Hk, d, 0.6, wins[b])
        mine = out[at:at + o.numel()].view_as(o[0])
        at += o.numel()
        assert torch.isfinite(mine).all()
        assert torch.equal(mine, o[0]), (b, T)
        for what, x in arrays(one, 1, 0, T).items():
            y = arrays(st, n, b, T)[what]
            assert torch.equal(x, y), (b, T, what)
        s = B.delta_sparsity_stats(one)["prefill"]
        c = [s[k] for k in ("nnz", "elements", "macs_done", "macs_dense")]
        total = c if total is None else [a + x for a, x in zip(total, c)]
        assert B.delta_state_sequence_position(st, b) == T
    s = B.delta_sparsity_stats(st)
    assert [s["prefill"][k] for k in ("nnz", "elements", "macs_done", "macs_dense")] == total and s["device_status"] == 0


@pytest.mark.parametrize("source,dtype,H,Hk,lens,kernel", [
    # query tiles: 8 (both forms), 20 (two heads), 3, 15, 5 (one)
    ("query", "bf16", 32, 8, (1024, 2500, 300, 1900, 640), -1),
    ("key", "bf16", 32, 8, (640, 2433, 1100, 90), -1), ("bottom_up", "bf16", 32, 16, (1152, 2500, 513), -1),
    ("query", "f32", 16, 4, (100, 1500, 500, 1000), -1),         # 4, 1 and 2 warps per row group
    # one form forced: one head per CTA, two, both
    ("query", "bf16", 8, 4, (300, 128, 700), 3), ("query", "bf16", 8, 4, (300, 128, 700), 4),
    ("query", "bf16", 8, 4, (300, 128, 700), 5), ("key", "bf16", 8, 4, (300, 128, 700), 5)])
def test_sequences_of_a_ragged_call_keep_the_form_of_their_own_call(source, dtype, H, Hk, lens, kernel):
    """The attention kernels' forms round differently; which one a sequence takes follows its own length and
    heads, so a neighbour never changes its bits (here: each with and without the others)."""
    from paper_2507_19608_b200 import binding as B
    d, n, T_max, dt = 64, len(lens), max(lens), torch.bfloat16 if dtype == "bf16" else torch.float32
    src = {"query": B.DELTA_SRC_QUERY, "key": B.DELTA_SRC_KEY, "bottom_up": B.DELTA_SRC_QUERY_BOTTOM_UP}[source]
    gen = torch.Generator("cuda").manual_seed(5)
    rnd = lambda *s: torch.randn(*s, generator=gen, device="cuda").to(dt)      # noqa: E731
    kc, vc, qs = rnd(n, Hk, T_max, d), rnd(n, Hk, T_max, d), [rnd(H, T, d) for T in lens]
    wins = [(64, 100, 0, 128, 37)[b] for b in range(n)]
    packed = torch.cat([x.reshape(-1) for x in qs])
    out = torch.full_like(packed, float("nan"))
    st = B.delta_state_init(B.make_config(n, H, Hk, d, T_max, dtype, source=src))
    B.delta_state_set_prefill_kernel(st, kernel)
    B.delta_attn_prefill_varlen(st, packed, kc, vc, out, lens, wins, 0.6)
    at = 0
    for b, T in enumerate(lens):
        one = B.delta_state_init(B.make_config(1, H, Hk, d, T_max, dtype, source=src))
        B.delta_state_set_prefill_kernel(one, kernel)
        o = torch.empty_like(qs[b])
        B.delta_attn_prefill(one, qs[b], kc[b], vc[b], o, T, H, Hk, d, 0.6, wins[b])
        assert torch.equal(out[at:at + o.numel()].view_as(o), o), (b, T)
        at += o.numel()
    assert B.delta_sparsity_stats(st)["device_status"] == 0
