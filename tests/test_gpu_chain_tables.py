"""The delta chain from helper-built tables (k1_delta_construct.cu) at the sizes where it can go wrong: ends on and beside
8-row sub-blocks and 64-row stages, the rings of staged rows (8 stages) and of tables (4 stages) filled and wrapped, one
and two CTAs per SM, and the first size that goes row by row.  Bit for bit against the oracle, both orders."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from oracle import delta_oracle as O          # noqa: E402
from paper_2507_19608_b200 import workloads as WL      # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2507_19608_b200 import binding
    return binding


@pytest.mark.parametrize("T", [1, 7, 8, 9, 63, 64, 65, 72, 127, 128, 129, 255, 257, 320, 505, 512, 520, 575, 777])
@pytest.mark.parametrize("order", ["top_down", "bottom_up"])
@pytest.mark.parametrize("H,d,dtype,theta,init", [
    (2, 64, "bf16", 0.25, "basis_exact"), (1, 128, "f32", 0.3, "zero_state"), (1, 128, "bf16", 0.6, "zero_state")])
def test_chain_ends(B, T, order, H, d, dtype, theta, init):
    _check(B, H, T, d, dtype, theta, init, order)


@pytest.mark.parametrize("H,d,dtype", [(74, 64, "bf16"), (75, 64, "bf16"), (148, 64, "bf16"), (149, 64, "bf16"), (37, 128, "f32"),
                                       (38, 128, "f32")])
@pytest.mark.parametrize("order", ["top_down", "bottom_up"])
def test_chain_many_heads(B, H, d, dtype, order):
    _check(B, H, 333, d, dtype, 0.2, "basis_exact", order)


def _check(B, H, T, d, dtype, theta, init, order):
    from tests.gpu_helpers import to_cache, to_dev
    if order == "bottom_up" and dtype == "f32":
        pytest.skip("bottom-up query deltas are bf16")
    q = WL.make_qkv(WL.Workload("t", 1, H, H, T, d, dtype, 0.95, 0.5, 0, (), 31 + T + H))["q"]
    q[0, 0, T // 2, 3] = np.nan
    q[0, 0, T // 3, 4] = np.inf
    k = np.zeros((1, H, T, d), np.float32)
    cfg = B.make_config(1, H, H, d, T, dtype,
                        source=B.DELTA_SRC_QUERY if order == "top_down" else B.DELTA_SRC_QUERY_BOTTOM_UP,
                        init=B.DELTA_INIT_BASIS_EXACT if init == "basis_exact" else B.DELTA_INIT_ZERO_STATE)
    st = B.delta_state_init(cfg)
    dq, kc = to_dev(q, dtype), to_cache(k, T, dtype)
    out = torch.empty_like(dq)
    B.delta_attn_prefill(st, dq, kc, kc, out, T, H, H, d, theta, 8)
    torch.cuda.synchronize()
    got_dq = B.delta_state_view(st, B.DELTA_VIEW_DQ).cpu().numpy()
    got_mask = B.delta_state_view(st, B.DELTA_VIEW_MASK).cpu().numpy().view(np.uint32)
    got_ref = B.delta_state_view(st, B.DELTA_VIEW_QHAT).cpu().numpy()
    got_tile = B.delta_state_view(st, B.DELTA_VIEW_QHAT_TILE).cpu().numpy()
    flip = slice(None, None, -1 if order == "bottom_up" else 1)
    for h in range(H):
        r = O.delta_construct(q[0, h][flip], theta, init)
        assert np.array_equal(got_dq[0, h, :T].view(np.uint32), r["dq"][flip].view(np.uint32)), h
        assert np.array_equal(got_mask[0, h, :T], r["mask"][flip]), h
        assert np.array_equal(got_ref[0, h].view(np.uint32), r["ahat"].view(np.uint32)), h
        if order == "top_down":
            nt = (T + 63) // 64
            assert np.array_equal(got_tile[0, h, :nt].view(np.uint32), r["ahat_tile"].view(np.uint32)), h
    assert B.delta_sparsity_stats(st)["device_status"] == 0


@pytest.mark.parametrize("source", ["query", "key", "bottom_up"])
@pytest.mark.parametrize("d,lens", [(64, (600, 561, 599, 600)), (64, (600, 595, 600, 599, 580)), (64, (777, 8, 513, 64, 1, 505)),
                                    (64, (240, 9, 100)), (64, (239, 9, 100)), (128, (400, 400)), (128, (400, 399, 400)), (64, (100,) * 17 + (600,))])
def test_ragged_groups(B, source, d, lens):
    """Query deltas: 4 and 5, 2 and 3 sequences of a length lie on either side of one line between tables and rows, the longest
    sequence of 240 or 239 tokens among three on either side of the other."""
    H, Hk, T_max = 32, 8, max(lens) + 2
    gen = torch.Generator("cuda").manual_seed(len(lens))
    rnd = lambda *s: (torch.randn(*s, generator=gen, device="cuda").cumsum(-2) * 0.1).bfloat16()      # noqa: E731
    src = {"query": B.DELTA_SRC_QUERY, "key": B.DELTA_SRC_KEY, "bottom_up": B.DELTA_SRC_QUERY_BOTTOM_UP}[source]
    kc = torch.full((len(lens), Hk, T_max, d), float("nan"), dtype=torch.bfloat16, device="cuda")
    qs = [rnd(H, n, d) for n in lens]
    for b, n in enumerate(lens):
        kc[b, :, :n] = rnd(Hk, n, d)
    st = B.delta_state_init(B.make_config(len(lens), H, Hk, d, T_max, "bf16", source=src))
    out = torch.empty(sum(q.numel() for q in qs), dtype=torch.bfloat16, device="cuda")
    B.delta_attn_prefill_varlen(st, torch.cat([q.reshape(-1) for q in qs]), kc, kc, out, list(lens), [16] * len(lens), 0.25)
    Hs = Hk if source == "key" else H
    dq = B.delta_state_view(st, B.DELTA_VIEW_DQ).reshape(-1)[:len(lens) * Hs * T_max * d].view(len(lens), Hs, T_max, d)
    ref = B.delta_state_view(st, B.DELTA_VIEW_QHAT).reshape(-1)[:len(lens) * Hs * d].view(len(lens), Hs, d)
    for b, n in enumerate(lens):
        x = (kc[b, :, :n] if source == "key" else qs[b]).float()
        order = range(n - 1, -1, -1) if source == "bottom_up" else range(n)
        r, want = None, []
        for i in order:                                    # Eq. 2-3 row by row: one subtraction, a strict comparison
            diff = x[:, i] if r is None else x[:, i] - r
            fire = torch.ones_like(diff, dtype=torch.bool) if r is None else diff.abs() > 0.25
            r = torch.where(fire, x[:, i], r if r is not None else diff)
            want.append(torch.where(fire, diff, torch.zeros_like(diff)))
        if source == "bottom_up":
            want.reverse()
        assert torch.equal(dq[b, :, :n], torch.stack(want, 1)) and torch.equal(ref[b], r), b
    assert B.delta_sparsity_stats(st)["device_status"] == 0
