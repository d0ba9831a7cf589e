"""The host-buffer prefill in chunks of KV heads: same output bit for bit, delta arrays and counters as the device call,
for one, two and four chunks (uneven ones included), every source, both cache layouts, pinned and pageable
buffers, and from several host threads at once."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


def _both(B, Bn, H, Hk, d, T, T_max, source, dtype, seed, pinned=True, stream=None):
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    src = {"query": B.DELTA_SRC_QUERY, "key": B.DELTA_SRC_KEY, "key_packed": B.DELTA_SRC_KEY,
           "bottom_up": B.DELTA_SRC_QUERY_BOTTOM_UP}[source]
    cfg = B.make_config(Bn, H, Hk, d, T_max, dtype, source=src)
    gen = torch.Generator().manual_seed(seed)
    host = [torch.randn(Bn, h, T, d, generator=gen).to(dt) for h in (H, Hk, Hk)]
    out_h = torch.empty_like(host[0])
    if pinned:
        host, out_h = [x.pin_memory() for x in host], out_h.pin_memory()
    sts = [B.delta_state_init(cfg) for _ in range(2)]
    if source == "key_packed":
        for st in sts:
            B.delta_state_set_key_cache(st, True)
    staging = torch.empty(B.delta_prefill_staging_bytes(cfg, T), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    B.delta_attn_prefill_host(sts[0], *host, out_h, staging, T, 0.4, 64, stream=stream)
    q = host[0].cuda()
    kc, vc = (torch.zeros(Bn, Hk, T_max, d, dtype=dt, device="cuda") for _ in range(2))
    kc[:, :, :T], vc[:, :, :T] = host[1].cuda(), host[2].cuda()
    out = torch.empty_like(q)
    B.delta_attn_prefill(sts[1], q, kc, vc, out, T, H, Hk, d, 0.4, 64)
    torch.cuda.synchronize()
    assert torch.equal(out_h, out.cpu())
    Hs = Hk if source.startswith("key") else H
    for what, tail in ((B.DELTA_VIEW_DQ, d), (B.DELTA_VIEW_MASK, d // 32), (B.DELTA_VIEW_IDX, d)):
        x, y = (B.delta_state_view(st, what).reshape(-1)[:Bn * Hs * T_max * tail].view(Bn * Hs, T_max, tail)[:, :T] for st in sts)
        assert torch.equal(x, y)
    if source == "query":
        x, y = (B.delta_state_view(st, B.DELTA_VIEW_R)[:, :, :T] for st in sts)
        assert torch.equal(x, y)
    assert B.delta_sparsity_stats(sts[0]) == B.delta_sparsity_stats(sts[1])


@pytest.mark.parametrize("Bn,H,Hk,d,T,T_max,source,dtype", [
    (1, 4, 1, 64, 100, 100, "query", "bf16"), (1, 32, 8, 64, 1024, 1024, "query", "bf16"),
    (1, 20, 5, 128, 900, 950, "query", "bf16"), (3, 6, 3, 64, 1500, 1503, "key", "bf16"),
    (2, 12, 3, 64, 1300, 1310, "key_packed", "bf16"), (1, 14, 7, 64, 1111, 1111, "bottom_up", "bf16"),
    (1, 8, 8, 64, 700, 701, "query", "f32"), (4, 32, 8, 64, 1024, 1030, "query", "bf16"),
    (3, 20, 5, 64, 1024, 1030, "query", "bf16"), (3, 12, 3, 128, 1100, 1100, "key_packed", "bf16")])
def test_host_call_equals_device_call(Bn, H, Hk, d, T, T_max, source, dtype):
    from paper_2507_19608_b200 import binding as B
    _both(B, Bn, H, Hk, d, T, T_max, source, dtype, seed=T)
    _both(B, Bn, H, Hk, d, T, T_max, source, dtype, seed=T + 1, pinned=False)


def test_host_calls_from_several_threads():
    from paper_2507_19608_b200 import binding as B
    errors = []

    def work(i):
        try:
            s = torch.cuda.Stream()
            for k in range(3):
                _both(B, 1, 16, 4, 64, 600 + 50 * i, 700 + 50 * i, "query", "bf16", seed=10 * i + k, stream=s)
        except Exception as ex:      # noqa: BLE001
            errors.append(ex)
    threads = [threading.Thread(target=work, args=(i,)) for i in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def test_host_call_on_a_capturing_stream_is_refused_and_leaves_the_capture_valid():
    from paper_2507_19608_b200 import binding as B
    T, x = 1024, torch.ones(1024, device="cuda")
    cfg = B.make_config(1, 32, 8, 64, T, "bf16")
    host = [torch.zeros(1, h, T, 64, dtype=torch.bfloat16).pin_memory() for h in (32, 8, 8, 32)]
    st = B.delta_state_init(cfg)
    staging = torch.empty(B.delta_prefill_staging_bytes(cfg, T), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        with pytest.raises(B.DeltaError):
            B.delta_attn_prefill_host(st, *host, staging, T, 0.4, 64)
        x += 1
    g.replay()
    B.delta_attn_prefill_host(st, *host, staging, T, 0.4, 64)
    torch.cuda.synchronize()
    assert bool((x == 2).all()) and B.delta_state_position(st) == T
