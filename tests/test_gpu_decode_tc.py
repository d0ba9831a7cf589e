"""The decode steps whose warps work on units of 32 keys (bf16: tensor cores; fp32) against the FP32-pipe step
that walks tiles behind block barriers (itself held to the oracle in test_gpu_parity.py) where its slicing can go wrong: lengths around the 32-key unit, one warp's share and
a slice's end, every head-group size, both head dimensions, clusters of all sizes, the merge through
global memory, window edges inside a unit, and ragged batches beyond one launch's 64 sequences."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.fixture(scope="module")
def B():
    from paper_2507_19608_b200 import binding
    return binding


def _run(B, kernel, source, Bn, H, Hk, d, lens, W_d, steps, seed, ramp=0.0):
    """Prefill (ragged where the lengths differ), then decode steps with the given decode kernel.
    ramp: every key is 2^ramp times as large as the one in front of it."""
    gen = torch.Generator("cuda").manual_seed(seed)
    dt = torch.float32 if source == "f32" else torch.bfloat16
    rnd = lambda *s: torch.randn(*s, generator=gen, device="cuda").to(dt)      # noqa: E731
    T = max(lens)
    T_max = T + steps + 3
    src = B.DELTA_SRC_KEY if source == "key" else B.DELTA_SRC_QUERY
    st = B.delta_state_init(B.make_config(Bn, H, Hk, d, T_max, "f32" if source == "f32" else "bf16", source=src))
    B.delta_state_set_decode_kernel(st, -1 if source == "f32" and kernel else kernel)      # (fp32: the default against 0)
    kc = torch.full((Bn, Hk, T_max, d), float("nan"), dtype=dt, device="cuda")
    vc = kc.clone()
    for b, n in enumerate(lens):
        kc[b, :, :n], vc[b, :, :n] = rnd(Hk, n, d), rnd(Hk, n, d)
        if ramp:
            kc[b, :, :n] *= torch.exp2(ramp * torch.arange(n, device="cuda"))[:, None].to(dt)
    q = torch.cat([rnd(H, n, d).reshape(-1) for n in lens])
    out = torch.empty_like(q)
    B.delta_attn_prefill_varlen(st, q, kc, vc, out, lens, [16] * Bn, 0.7)
    outs = []
    for _ in range(steps):
        o = torch.full((Bn, H, d), float("nan"), dtype=dt, device="cuda")
        B.delta_attn_decode_step(st, rnd(Bn, H, d), rnd(Bn, Hk, d), rnd(Bn, Hk, d), kc, vc, o, 0.7, W_d)
        outs.append(o)
    R = B.delta_state_view(st, B.DELTA_VIEW_R)
    R = [R[b, :, :n + steps].clone() for b, n in enumerate(lens)] if source != "key" else []
    return (torch.stack(outs).float(), kc, vc, B.delta_state_view(st, B.DELTA_VIEW_QHAT).clone(), R,
            B.delta_sparsity_stats(st))


def _compare(B, source, Bn, H, Hk, d, lens, W_d, steps, seed=7, ramp=0.0):
    a = _run(B, 1, source, Bn, H, Hk, d, lens, W_d, steps, seed, ramp)
    r = _run(B, 0, source, Bn, H, Hk, d, lens, W_d, steps, seed, ramp)
    assert torch.isfinite(a[0]).all()
    rms = r[0].pow(2).mean(dim=-1, keepdim=True).sqrt()
    most, rel = (2e-5, 2e-6) if source == "f32" else (2e-2, 3e-3)
    assert ((a[0] - r[0]).abs() / torch.maximum(rms, r[0].abs())).max() <= most
    assert (a[0] - r[0]).norm() / r[0].norm() <= rel
    for x, y in ((a[1], r[1]), (a[2], r[2])):                   # the caches, appended rows included
        assert torch.equal(x.view(torch.int16), y.view(torch.int16))
    assert torch.equal(a[3], r[3])
    for x, y in zip(a[4], r[4]):
        assert (x - y).abs().max() <= 1e-3 * max(1.0, float(y.abs().max()))
    assert a[5] == r[5]                                         # counters and status


@pytest.mark.parametrize("T", [1, 2, 30, 31, 32, 33, 63, 127, 128, 129, 254, 255, 256, 257, 511, 513])
@pytest.mark.parametrize("source,d", [("query", 64), ("query", 128), ("key", 64), ("key", 128), ("f32", 64),
                                      ("f32", 128)])
def test_lengths_around_units_and_slices(B, T, source, d):
    _compare(B, source, 1, 4, 1, d, [T], 8, 4)


@pytest.mark.parametrize("g", [1, 2, 4, 8])
@pytest.mark.parametrize("source", ["query", "key", "f32"])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("W_d", [0, 1, 45, 5000])
def test_head_groups_and_windows(B, g, source, d, W_d):
    _compare(B, source, 2, 3 * g, 3, d, [700, 700], W_d, 3)


@pytest.mark.parametrize("source", ["query", "f32"])
@pytest.mark.parametrize("Bn,Hk,T,d", [
    (1, 1, 3000, 64), (1, 1, 40000, 64), (1, 2, 50000, 128),      # 12 slices; slices merged through global memory
    (5, 1, 2500, 64), (3, 5, 2100, 128), (40, 4, 1100, 64), (80, 4, 300, 128)])
def test_slices(B, source, Bn, Hk, T, d):
    _compare(B, source, Bn, 4 * Hk, Hk, d, [T] * Bn, 64, 2)


@pytest.mark.parametrize("source,Bn,d", [("query", 6, 64), ("key", 6, 64), ("query", 70, 64), ("key", 5, 128),
                                         ("f32", 6, 64), ("f32", 67, 128)])
def test_ragged_batches(B, source, Bn, d):
    lens = [1 + (i * 7919) % 900 for i in range(Bn)]
    _compare(B, source, Bn, 2, 1, d, lens, 40, 3)


@pytest.mark.parametrize("source", ["query", "key"])
@pytest.mark.parametrize("d,ramp", [(64, 0.004), (64, -0.004), (128, 0.006), (128, -0.006)])
def test_scores_that_run_away(B, source, d, ramp):
    # Several units per warp: a row's maximum moves by more than the 2^8 up to which the scale is kept (a warp's units
    # are 256 keys apart, 128 at d = 128: scores grow by 2 and 1.7 from unit to unit, up to hundreds), or only falls.
    # 160 KV heads take one slice each, since clusters of two have no room (320 CTAs, 1.75 per SM at most): 35 units on
    # a CTA's 8 or 4 warps.
    assert 2 * 160 > 1.75 * torch.cuda.get_device_properties(0).multi_processor_count
    _compare(B, source, 40, 16, 4, d, [1100] * 40, 64, 2, ramp=ramp)
