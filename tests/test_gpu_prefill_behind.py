"""A prefill is launched while the kernel in front of it still runs: that kernel's writes to the inputs, its reads of the
outputs and of the state's arrays come first all the same, eagerly and in a captured graph."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

# table chain, row-by-row chain (320 CTAs), key deltas, bottom-up, fp32
CASES = [(1, 32, 8, 1024, 64, "bf16", "query"), (5, 32, 8, 200, 64, "bf16", "query"), (2, 32, 8, 900, 64, "bf16", "key"),
         (1, 8, 8, 333, 128, "bf16", "bottom_up"), (1, 16, 4, 500, 64, "f32", "query")]


def _setup(case):
    from paper_2507_19608_b200 import binding as B
    Bn, H, Hk, T, d, dtype, source = case
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    src = {"query": B.DELTA_SRC_QUERY, "key": B.DELTA_SRC_KEY, "bottom_up": B.DELTA_SRC_QUERY_BOTTOM_UP}[source]
    st = B.delta_state_init(B.make_config(Bn, H, Hk, d, T, dtype, source=src))
    gen = torch.Generator(device="cuda").manual_seed(T)
    inputs = [[torch.randn(Bn, h, T, d, generator=gen, device="cuda").to(dt) for h in (H, Hk, Hk)] for _ in range(3)]
    buf = [torch.empty_like(x) for x in inputs[0]]
    out = torch.empty_like(buf[0])

    def call():
        B.delta_state_reset(st)
        B.delta_attn_prefill(st, *buf, out, T, H, Hk, d, 0.3, 64)

    return B, st, inputs, buf, out, call


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(map(str, c)))
@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("front", ["kernel", "copy"])
def test_prefill_behind_writes_of_its_inputs(case, captured, front):
    B, st, inputs, buf, out, call = _setup(case)
    want = []
    for x in inputs:
        for a, b in zip(buf, x):
            a.copy_(b)
        torch.cuda.synchronize()
        call()
        torch.cuda.synchronize()
        want.append((out.clone(), B.delta_state_view(st, B.DELTA_VIEW_MASK).clone()))
    step, stage = call, [torch.empty_like(x) for x in buf]

    def whole():      # kernels (or copies) write the inputs, the call, a kernel reads its results
        for a, b in zip(buf, stage):
            torch.mul(b, 1, out=a) if front == "kernel" else a.copy_(b)
        step()
        return out * 1, B.delta_state_view(st, B.DELTA_VIEW_MASK).clone()

    if captured:
        side = torch.cuda.Stream()
        with torch.cuda.stream(side):
            whole()
        side.synchronize()
        graph = torch.cuda.CUDAGraph()
        B.delta_state_reset(st)
        with torch.cuda.graph(graph, stream=side):
            got = whole()
    for i in [0, 1, 2, 0, 2, 1] * 5:
        for a, b in zip(stage, inputs[i]):
            a.copy_(b)
        if captured:
            graph.replay()
        else:
            got = whole()
        torch.cuda.synchronize()
        assert torch.equal(got[0], want[i][0]) and torch.equal(got[1], want[i][1])
