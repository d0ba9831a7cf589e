"""The attention kernel that begins while the delta chain goes on (k2_hybrid_attn_tcq.cu): on either side of every line of
the rule that says when (148 SMs), for lengths around 64-row stages and 128-row query tiles, both orders, and prefill
after prefill of different lengths on one state, it leaves the bits of the kernels run one behind the other (as they
are while per-kernel timing is on)."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


def _inputs(Bn, H, Hk, d, T, seed):
    gen = torch.Generator("cuda").manual_seed(seed)
    rnd = lambda h: (torch.randn(Bn, h, T, d, generator=gen, device="cuda").cumsum(2) * 0.05).bfloat16()      # noqa: E731
    return rnd(H), rnd(Hk), rnd(Hk)


def _state(B, Bn, H, Hk, d, T_max, source, timing):
    st = B.delta_state_init(B.make_config(Bn, H, Hk, d, T_max, "bf16",
                                          source=B.DELTA_SRC_QUERY_BOTTOM_UP if source == "bottom_up" else B.DELTA_SRC_QUERY))
    B.delta_state_enable_profiling(st, timing)
    return st


def _arrays(B, st, T):
    return [B.delta_state_view(st, B.DELTA_VIEW_QHAT).clone(), B.delta_state_view(st, B.DELTA_VIEW_R)[:, :, :T].clone()]


@pytest.mark.parametrize("Bn,H,Hk,d,lens", [
    (1, 32, 8, 64, (1281, 2048, 1300, 1345, 2048)),           # two heads per CTA; the light ones first
    (1, 32, 8, 64, (1024, 1100, 1151, 1153)),                 # both forms in one grid
    (1, 20, 5, 128, (2048, 900, 1985, 1984, 513, 2047)),      # one head per CTA
    (1, 24, 3, 128, (1200, 1217)), (1, 4, 1, 64, (4000, 1)),
    (2, 20, 5, 128, (1531, 700)), (3, 32, 8, 64, (514, 449)),     # the chain's CTAs share SMs
    (2, 32, 8, 64, (1024, 1700)), (1, 16, 4, 64, (1024, 1421))])  # off | on
@pytest.mark.parametrize("source", ["query", "bottom_up"])
def test_beside_equals_behind(Bn, H, Hk, d, lens, source):
    from paper_2507_19608_b200 import binding as B
    T_max = max(lens)
    states = [_state(B, Bn, H, Hk, d, T_max, source, t) for t in (False, True)]
    for i, T in enumerate(lens):
        q, k, v = _inputs(Bn, H, Hk, d, T, 7 * i + T)
        kc, vc = (torch.zeros(Bn, Hk, T_max, d, dtype=torch.bfloat16, device="cuda") for _ in range(2))
        kc[:, :, :T], vc[:, :, :T] = k, v
        outs = []
        for st in states:
            B.delta_state_reset(st)
            out = torch.full_like(q, float("nan"))
            for _ in range(3):                                 # behind one another: what the last one left must not matter
                B.delta_state_reset(st)
                B.delta_attn_prefill(st, q, kc, vc, out, T, H, Hk, d, 0.3, 64 + 36 * (i % 2))
            outs.append([out] + _arrays(B, st, T))
        torch.cuda.synchronize()
        assert torch.isfinite(outs[0][0]).all()
        for x, y in zip(*outs):
            assert torch.equal(x, y), (T, x.shape)
        assert all(B.delta_sparsity_stats(st)["device_status"] == 0 for st in states)
        assert B.delta_sparsity_stats(states[0])["prefill"] == B.delta_sparsity_stats(states[1])["prefill"]


def test_ragged_and_replayed():
    from paper_2507_19608_b200 import binding as B
    lens, H, Hk, d = [1900, 1000, 130, 90, 1500, 64], 32, 8, 64
    T_max = max(lens)
    packed, caches = [], [torch.zeros(len(lens), Hk, T_max, d, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    for b, n in enumerate(lens):
        q, k, v = _inputs(1, H, Hk, d, n, n)
        packed.append(q.reshape(-1))
        caches[0][b, :, :n], caches[1][b, :, :n] = k[0], v[0]
    q = torch.cat(packed)
    outs = []
    for timing in (False, True):
        st = _state(B, len(lens), H, Hk, d, T_max, "query", timing)
        out = torch.full_like(q, float("nan"))
        B.delta_attn_prefill_varlen(st, q, *caches, out, lens, [64] * len(lens), 0.3)
        torch.cuda.synchronize()
        outs.append([out, B.delta_state_view(st, B.DELTA_VIEW_QHAT).clone()])
    for x, y in zip(*outs):
        assert torch.equal(x, y)
    # captured once, replayed with other inputs in the same buffers
    T = 2048
    q, k, v = _inputs(1, H, Hk, d, T, 5)
    st, out = _state(B, 1, H, Hk, d, T, "query", False), torch.empty_like(q)
    run = lambda s, o: (B.delta_state_reset(s), B.delta_attn_prefill(s, q, k, v, o, T, H, Hk, d, 0.3, 64))      # noqa: E731
    run(st, out)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run(st, out)
    for seed in (6, 7):
        for x, y in zip((q, k, v), _inputs(1, H, Hk, d, T, seed)):
            x.copy_(y)
        graph.replay()
        graph.replay()
        ref = torch.empty_like(q)
        run(_state(B, 1, H, Hk, d, T, "query", True), ref)
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
