"""The fp32-arithmetic prefill kernel in its three forms (one, two or four warps per 16 query rows, chosen
by the size of the launch): a small launch is held to the oracle at the edges of its tiles, and the same
sequence inside larger launches, which take the other forms, to the small launch."""
import numpy as np
import pytest
import torch

from oracle import delta_oracle as O
from paper_2507_19608_b200 import workloads as WL

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.mark.parametrize("T", [1, 8, 15, 16, 17, 31, 33, 63, 64, 65, 127, 129, 200])
@pytest.mark.parametrize("d,W,shape", [(64, 20, "sliding"), (64, 48, "block"), (128, 20, "block"), (128, 0, "block")])
def test_forms_agree_with_the_oracle_at_tile_edges(T, d, W, shape):
    from paper_2507_19608_b200 import binding as B
    from tests.gpu_helpers import run_prefill, to_host_f64
    w = WL.Workload("t", 1, 2, 1, T, d, "f32", 0.95, 0.5, W, (), 900 + T)
    t = WL.make_qkv(w)
    _, one, _, _ = run_prefill(B, t["q"], t["k"], t["v"], 0.2, W, "f32", shape=shape)
    ref, _ = O.prefill_mha(t["q"], t["k"], t["v"], 0.2, W, shape)
    assert np.abs(to_host_f64(one) - ref).max() <= 1e-4
    for batch in (24, 96, 200):
        many = {x: np.repeat(t[x], batch, axis=0) for x in ("q", "k", "v")}
        st, out, _, _ = run_prefill(B, many["q"], many["k"], many["v"], 0.2, W, "f32", shape=shape)
        assert (out - one).abs().max() <= 2e-6 * max(1.0, float(one.abs().max()))
        assert B.delta_sparsity_stats(st)["device_status"] == 0


def test_parts_keep_fp32_precision():
    """Against fp64 dense attention (theta = 0), values with a common offset: no worse than fp32 arithmetic."""
    from paper_2507_19608_b200 import binding as B
    T, H, d = 1500, 3, 64
    gen = torch.Generator("cuda").manual_seed(5)
    q, k, v = (torch.randn(1, H, T, d, generator=gen, device="cuda") * 1.5 for _ in range(3))
    v = v + 1.0
    st = B.delta_state_init(B.make_config(1, H, H, d, T, "f32"))
    out = torch.empty_like(q)
    B.delta_attn_prefill(st, q, k, v, out, T, H, H, d, 0.0, 64)
    s = (q.double() @ k.double().transpose(-1, -2)) / d ** 0.5
    s = s.masked_fill(torch.ones(T, T, dtype=torch.bool, device="cuda").triu(1), float("-inf"))
    ref = torch.softmax(s, -1) @ v.double()
    assert (out.double() - ref).norm() / ref.norm() <= 4e-7
