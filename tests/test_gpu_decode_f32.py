"""The fp32 decode step (k3_decode_step_f32.cu) where a unit of 32 keys ends: the row that arrives with the step first or last in
its unit, the cache's last row inside a unit (what lies behind is NaN), one slice and several, groups of 1 to 8 heads.
Outputs within 1e-4 of the oracle (fp32 sums of at most 2 d + L terms), states and caches bit for bit."""
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


@pytest.mark.parametrize("H,Hk,d", [(2, 2, 64), (4, 2, 64), (4, 1, 64), (8, 1, 64), (1, 1, 128), (4, 1, 128), (8, 1, 128)])
@pytest.mark.parametrize("T,slack", [(1, 0), (30, 0), (31, 40), (63, 0), (255, 0), (257, 31), (700, 3)])
def test_step_at_unit_ends(B, H, Hk, d, T, slack):
    from tests.gpu_helpers import run_prefill, to_dev, to_host_f64
    steps, theta, W = 4, 0.2, 40
    t = WL.make_qkv(WL.Workload("t", 2, H, Hk, T, d, "f32", 0.95, 0.5, W, (), 5 + T + d, n_decode=steps))
    st, _, kc, vc = run_prefill(B, t["q"], t["k"], t["v"], theta, W, "f32", shape="sliding", T_max=T + steps + slack)
    _, heads = O.prefill_mha(t["q"], t["k"], t["v"], theta, W, "sliding")
    states = {key: r["state"] for key, r in heads.items()}
    for s in range(steps):
        new = [t[x][:, :, s] for x in ("q_dec", "k_dec", "v_dec")]
        dev = [to_dev(x, "f32") for x in new]
        o = torch.full_like(dev[0], float("nan"))
        B.delta_attn_decode_step(st, *dev, kc, vc, o, theta, W)
        torch.cuda.synchronize()
        ref, _ = O.decode_mha(states, *new, theta, W)
        assert np.abs(to_host_f64(o) - ref).max() <= 1e-4
        assert torch.equal(kc[:, :, T + s], dev[1]) and torch.equal(vc[:, :, T + s], dev[2])
        R = B.delta_state_view(st, B.DELTA_VIEW_R).cpu().numpy()
        qh = B.delta_state_view(st, B.DELTA_VIEW_QHAT).cpu().numpy()
        for (b, h), x in states.items():
            assert np.abs(R[b, h, :T + s + 1] - x["R"]).max() <= 1e-4 * max(1.0, np.abs(x["R"]).max())
            assert np.array_equal(qh[b, h].view(np.uint32), x["qhat"].view(np.uint32))
    assert torch.isnan(kc[:, :, T + steps:]).all() and torch.isnan(vc[:, :, T + steps:]).all()
    assert B.delta_sparsity_stats(st)["device_status"] == 0
