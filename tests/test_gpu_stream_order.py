"""A decode step enqueued directly behind a prefill comes behind everything the prefill writes: its output laid over
rows of the prefill's output survives, and the prefill's other rows are whole."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.mark.parametrize("Bn,H,Hk,T,dtype,source", [
    (1, 32, 8, 1024, "bf16", "query"), (4, 32, 8, 2048, "bf16", "query"), (1, 8, 8, 129, "bf16", "query"),
    (2, 32, 8, 1500, "bf16", "key"), (1, 16, 16, 1000, "f32", "query")])
def test_step_output_over_the_prefill_output(Bn, H, Hk, T, dtype, source):
    from paper_2507_19608_b200 import binding as B
    d, dt = 64, torch.bfloat16 if dtype == "bf16" else torch.float32
    cfg = B.make_config(Bn, H, Hk, d, T + 8, dtype, source=B.DELTA_SRC_KEY if source == "key" else B.DELTA_SRC_QUERY)
    gen = torch.Generator(device="cuda").manual_seed(T)
    rnd = lambda *s: torch.randn(*s, generator=gen, device="cuda").to(dt)      # noqa: E731
    q, kc, vc = rnd(Bn, H, T, d), rnd(Bn, Hk, T + 8, d), rnd(Bn, Hk, T + 8, d)
    new = [rnd(Bn, H, d), rnd(Bn, Hk, d), rnd(Bn, Hk, d)]
    st = B.delta_state_init(cfg)
    out, step = torch.empty_like(q), torch.empty(Bn, H, d, dtype=dt, device="cuda")
    B.delta_attn_prefill(st, q, kc, vc, out, T, H, Hk, d, 0.3, 64)
    torch.cuda.synchronize()
    B.delta_attn_decode_step(st, *new, kc, vc, step, 0.3, 64)
    torch.cuda.synchronize()
    want = out.clone().view(-1)
    want[-step.numel():] = step.view(-1)              # (the last rows: the heaviest query tiles)
    want[:step.numel()] = step.view(-1)               # (the first rows: written by the kernel's last CTAs)
    got = torch.empty_like(want)
    for over in (got[:step.numel()], got[-step.numel():]):
        for _ in range(10):
            got.fill_(float("nan"))
            B.delta_state_reset(st)
            B.delta_attn_prefill(st, q, kc, vc, got, T, H, Hk, d, 0.3, 64)
            B.delta_attn_decode_step(st, *new, kc, vc, over, 0.3, 64)
            torch.cuda.synchronize()
            part = slice(None, -step.numel()) if over.data_ptr() == got.data_ptr() else slice(step.numel(), None)
            assert torch.equal(got[part], want[part])
