"""Key tiles that lie partly inside the window, several in a row, in every form of the tensor-core
attention kernel's grid: the window's edge inside a tile and on its borders, rows of a tile in up to
eight window blocks, the diagonal tile mixed or not."""
import numpy as np
import pytest
import torch

from oracle import delta_oracle as O
from paper_2507_19608_b200 import workloads as WL

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.mark.parametrize("W,shape", [(1, "sliding"), (17, "block"), (65, "sliding"), (128, "sliding"), (150, "block"),
                                     (200, "sliding"), (320, "block"), (450, "sliding")])
@pytest.mark.parametrize("source,d", [("query", 64), ("key", 64), ("bottom_up", 64), ("query", 128), ("key", 128)])
def test_partly_exact_tiles(source, d, W, shape):
    from paper_2507_19608_b200 import binding as B
    from tests.gpu_helpers import to_cache, to_dev, to_host_f64
    H, Hk, T = 4, 2, 650
    t = WL.make_qkv(WL.Workload("t", 1, H, Hk, T, d, "bf16", 0.95, 0.5, W, (), 700 + W))
    src = {"query": B.DELTA_SRC_QUERY, "key": B.DELTA_SRC_KEY, "bottom_up": B.DELTA_SRC_QUERY_BOTTOM_UP}[source]
    cfg = B.make_config(1, H, Hk, d, T, "bf16", source=src,
                        prefill_window=B.DELTA_WIN_BLOCK if shape == "block" else B.DELTA_WIN_SLIDING)
    args = dict(source="key") if source == "key" else dict(order="bottom_up") if source == "bottom_up" else {}
    ref, _ = O.prefill_mha(t["q"], t["k"], t["v"], 0.2, W, shape, **args)
    q, kc, vc = to_dev(t["q"], "bf16"), to_cache(t["k"], T, "bf16"), to_cache(t["v"], T, "bf16")
    for form in (3,) if d == 128 else (3, 4, 5):          # one head per CTA, two, both
        st = B.delta_state_init(cfg)
        B.delta_state_set_prefill_kernel(st, form)
        out = torch.full_like(q, float("nan"))
        B.delta_attn_prefill(st, q, kc, vc, out, T, H, Hk, d, 0.2, W)
        got = to_host_f64(out)
        assert np.isfinite(got).all()
        row = np.abs(ref).max(-1)
        assert (np.abs(got - ref).max(-1) <= 2e-2 * row).all()
        assert np.sqrt(((got - ref) ** 2).mean() / (ref ** 2).mean()) <= 5e-3
        assert B.delta_sparsity_stats(st)["device_status"] == 0
