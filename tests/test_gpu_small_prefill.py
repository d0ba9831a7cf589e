"""Small prefills do the finish kernel's work in the attention kernel's launch (k1_finish.cuh): on either side of the line
(148 SMs) and at the ends of 8-row blocks and 64-row tiles the outputs and every array left behind are those of the
separate launches (as they are while per-kernel timing is on), call after call on one state."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.mark.parametrize("Bn,H,Hk,lens", [
    (1, 1, 1, (128, 1, 7, 8, 9, 63, 64, 65, 130)), (1, 8, 8, (400, 401, 320, 321, 200)), (2, 8, 2, (129, 257, 64)),
    (1, 4, 1, (1, 500, 1000, 333)), (3, 2, 1, (191, 192, 193)), (1, 32, 4, (64, 65, 40))])
@pytest.mark.parametrize("source,dtype,d", [("query", "f32", 64), ("query", "f32", 128), ("query", "bf16", 64), ("query", "bf16", 128),
                                            ("bottom_up", "bf16", 64)])
def test_one_launch_equals_two(Bn, H, Hk, lens, source, dtype, d):
    from paper_2507_19608_b200 import binding as B
    T_max = max(lens) + 3
    src = B.DELTA_SRC_QUERY_BOTTOM_UP if source == "bottom_up" else B.DELTA_SRC_QUERY
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    states = [B.delta_state_init(B.make_config(Bn, H, Hk, d, T_max, dtype, source=src)) for _ in range(2)]
    B.delta_state_enable_profiling(states[1], True)
    gen = torch.Generator("cuda").manual_seed(H + d)
    rnd = lambda h, n: (torch.randn(Bn, h, n, d, generator=gen, device="cuda").cumsum(2) * 0.1).to(dt)      # noqa: E731
    for i, T in enumerate(lens):
        q = rnd(H, T)
        kc, vc = (torch.full((Bn, Hk, T_max, d), float("nan"), dtype=dt, device="cuda") for _ in range(2))
        kc[:, :, :T], vc[:, :, :T] = rnd(Hk, T), rnd(Hk, T)
        got = []
        for st in states:
            out = torch.full_like(q, float("nan"))
            for _ in range(2):
                B.delta_state_reset(st)
                B.delta_attn_prefill(st, q, kc, vc, out, T, H, Hk, d, 0.3, (16, 0, 64, 100)[i % 4])
            torch.cuda.synchronize()
            view = lambda w, *t: B.delta_state_view(st, w).reshape(-1)[:Bn * H * torch.Size(t).numel()].view(Bn, H, *t)      # noqa: E731
            arrays = [view(B.DELTA_VIEW_DQ, T_max, d)[:, :, :T], view(B.DELTA_VIEW_MASK, T_max, d // 32)[:, :, :T],
                      view(B.DELTA_VIEW_ROW_NNZ, T_max)[:, :, :T], view(B.DELTA_VIEW_IDX, T_max, d)[:, :, :T],
                      view(B.DELTA_VIEW_TILE_NNZ, -(-T_max // 64))[:, :, :-(-T // 64)], view(B.DELTA_VIEW_QHAT, d)]
            if source == "query":
                arrays.append(view(B.DELTA_VIEW_R, T_max)[:, :, :T])
            s = B.delta_sparsity_stats(st)
            assert s["device_status"] == 0
            got.append(([out] + [a.clone() for a in arrays], s["prefill"]))
        assert torch.isfinite(got[0][0][0]).all()
        for x, y in zip(got[0][0], got[1][0]):
            assert torch.equal(x, y), (T, x.shape, x.dtype)
        assert got[0][1] == got[1][1]
