"""Which query tiles go one head per CTA and which two (k2_hybrid_attn_tcq.cu) follows the grid: on either side of every line
of that rule (148 SMs) the outputs agree with the one-head form forced."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.mark.parametrize("Bn,H,Hk,T,source,W", [
    (1, 32, 8, 384, "query", 64), (1, 32, 8, 385, "query", 64),          # all one head | half of the query tiles
    (1, 16, 4, 1024, "query", 100), (1, 16, 4, 1025, "query", 100),
    (1, 32, 8, 1000, "key", 64),                                         # as many as fit one wave
    (1, 32, 8, 1024, "query", 64), (1, 32, 8, 1025, "query", 64),        # the last such size | all two heads
    (1, 32, 8, 1153, "key", 100), (3, 16, 8, 800, "query", 0), (2, 32, 8, 640, "query", 0)])
def test_forms_agree(Bn, H, Hk, T, source, W):
    from paper_2507_19608_b200 import binding as B
    gen = torch.Generator(device="cuda").manual_seed(T)
    rnd = lambda h: (torch.randn(Bn, h, T, 64, generator=gen, device="cuda").cumsum(2) * 0.1).bfloat16()      # noqa: E731
    q, k, v = rnd(H), rnd(Hk), rnd(Hk)
    outs = []
    for kernel in (None, 3):
        st = B.delta_state_init(B.make_config(Bn, H, Hk, 64, T, "bf16",
                                              source=B.DELTA_SRC_KEY if source == "key" else B.DELTA_SRC_QUERY))
        if kernel is not None:
            B.delta_state_set_prefill_kernel(st, kernel)
        out = torch.full_like(q, float("nan"))
        B.delta_attn_prefill(st, q, k, v, out, T, H, Hk, 64, 0.2, W)
        torch.cuda.synchronize()
        assert B.delta_sparsity_stats(st)["device_status"] == 0
        outs.append(out.float())
    a, b = outs
    # Both are within half a bf16 step (2^-9) of their own fp32 result; the forms' bf16 probabilities are rounded at
    # different scales, 2^-9 of each addend, independent: a row differs by a few 2^-9 of its largest element at most.
    err = (a - b).abs().amax(-1) / b.abs().amax(-1).clamp_min(1e-30)
    assert torch.isfinite(a).all() and err.max() <= 4 * 2.0 ** -9 * 2


def _reference(q, k, v, theta, W, keys):
    """The method in fp32, block windows: Eq. 2-3 row by row, then dense softmax over the selected scores."""
    x = (k if keys else q).float()
    ref, rows = x[:, :, 0], [x[:, :, 0]]                                     # the first row is the basis
    for i in range(1, x.shape[2]):
        ref = torch.where((x[:, :, i] - ref).abs() > theta, x[:, :, i], ref)
        rows.append(ref)
    hat, g, T = torch.stack(rows, 2), q.shape[1] // k.shape[1], q.shape[2]
    grp = lambda t: t.float().repeat_interleave(g, 1)                        # noqa: E731
    s = q.float() @ grp(k).transpose(2, 3)
    i = torch.arange(T, device=q.device)
    if W < T:
        far = q.float() @ grp(hat).transpose(2, 3) if keys else hat @ grp(k).transpose(2, 3)
        s = torch.where(i[:, None] // W == i[None, :] // W, s, far) if W else far
    s = (s / q.shape[3] ** 0.5).masked_fill(i[:, None] < i[None, :], float("-inf"))
    return s.softmax(-1) @ grp(v)


@pytest.mark.parametrize("H,Hk,d,T,source,W", [
    (32, 8, 64, 1217, "query", 64), (32, 8, 64, 1217, "query", 192), (20, 10, 64, 2000, "query", 320),    # quarters of a tile
    (32, 8, 64, 1217, "query", 100), (32, 8, 64, 1300, "query", 0), (32, 8, 64, 1217, "key", 192),
    (8, 2, 64, 1000, "query", 192), (4, 1, 128, 700, "query", 192), (4, 1, 128, 129, "query", 128)])
def test_forms_meet_the_reference(H, Hk, d, T, source, W):
    from paper_2507_19608_b200 import binding as B
    gen = torch.Generator(device="cuda").manual_seed(T + W)
    rnd = lambda h: (torch.randn(1, h, T, d, generator=gen, device="cuda").cumsum(2) * 0.05).bfloat16()      # noqa: E731
    q, k, v = rnd(H), rnd(Hk), rnd(Hk)
    st = B.delta_state_init(B.make_config(1, H, Hk, d, T, "bf16",
                                          source=B.DELTA_SRC_KEY if source == "key" else B.DELTA_SRC_QUERY))
    out = torch.full_like(q, float("nan"))
    B.delta_attn_prefill(st, q, k, v, out, T, H, Hk, d, 0.2, W)
    torch.cuda.synchronize()
    assert B.delta_sparsity_stats(st)["device_status"] == 0
    ref = _reference(q, k, v, 0.2, W, source == "key")
    # the output's rounding is half a bf16 step (2^-9 of an element), the probabilities' the same of each addend
    err = (out.float() - ref).abs().amax(-1) / ref.abs().amax(-1).clamp_min(1e-30)
    vmax = v.float().abs().amax() / ref.abs().amax(-1).clamp_min(1e-30)
    assert torch.isfinite(out.float()).all() and (err <= 2.0 ** -9 * (1 + vmax)).all()
