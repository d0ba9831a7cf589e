"""Steps from the compressed key-delta cache fetch and rebuild what earlier steps left ahead of their wait for the kernel in
front: with steps of several states in turn on one stream, and prefills between them, every state's results are the
bits it has by itself."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

STEPS = 40                                   # over a segment's end, whatever the length


class _Layer:
    def __init__(self, B, seed, Bn, d, T):
        gen = torch.Generator("cuda").manual_seed(seed)
        rnd = lambda *s: torch.randn(*s, generator=gen, device="cuda").bfloat16()      # noqa: E731
        self.B, self.T, self.d, self.T_max, self.i = B, T, d, T + STEPS + 3, 0
        self.st = B.delta_state_init(B.make_config(Bn, 8, 2, d, self.T_max, "bf16", source=B.DELTA_SRC_KEY))
        B.delta_state_set_key_cache(self.st, True)
        self.k0 = torch.full((Bn, 2, self.T_max, d), float("nan"), device="cuda").bfloat16()
        self.v0 = self.k0.clone()
        self.k0[:, :, :T], self.v0[:, :, :T] = rnd(Bn, 2, T, d), rnd(Bn, 2, T, d)
        self.q = rnd(Bn, 8, T, d)
        self.new = [(rnd(Bn, 8, d), rnd(Bn, 2, d), rnd(Bn, 2, d)) for _ in range(STEPS)]
        self.out = torch.empty_like(self.q)

    def prefill(self):
        self.k, self.v, self.outs, self.i = self.k0.clone(), self.v0.clone(), [], 0
        self.B.delta_state_reset(self.st)
        self.B.delta_attn_prefill(self.st, self.q, self.k, self.v, self.out, self.T, 8, 2, self.d, 0.5, 64)

    def step(self):
        q, k, v = self.new[self.i]
        o = torch.full_like(q, float("nan"))
        self.B.delta_attn_decode_step(self.st, q, k, v, self.k, self.v, o, 0.5, 20)
        self.outs.append(o)
        self.i += 1

    def result(self):
        torch.cuda.synchronize()
        assert self.B.delta_sparsity_stats(self.st)["device_status"] == 0
        return torch.stack(self.outs).view(torch.int16).clone()


@pytest.mark.parametrize("Bn,d,T", [(1, 64, 31), (1, 64, 320), (2, 64, 1000), (1, 128, 700), (24, 64, 900)])
def test_states_in_turn(Bn, d, T):
    from paper_2507_19608_b200 import binding as B
    layers = [_Layer(B, s, Bn, d, T + 7 * s) for s in range(3)]
    alone = []
    for x in layers:
        x.prefill()
        for _ in range(STEPS):
            x.step()
        alone.append(x.result())
        assert torch.isfinite(alone[-1].view(torch.bfloat16).float()).all()
    for x in layers[:2]:
        x.prefill()
    for i in range(STEPS):
        layers[0].step()
        layers[1].step()
        if i == STEPS // 2:                  # the third joins in the middle, its prefill between two steps
            layers[2].prefill()
        if i >= STEPS // 2:
            layers[2].step()
    for _ in range(STEPS - layers[2].i):
        layers[2].step()
    for x, a in zip(layers, alone):
        assert torch.equal(x.result(), a)
