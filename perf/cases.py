"""Performance cases of the delta-attention library: what a program that uses it has it do.

A case is one attention layer's work for one request batch, through the public binding:
the state is reset, a prompt is prefilled and, where the case has steps, that many tokens are
generated one by one against the growing cache.  listed() gives the configurations the package is
quoted on (workloads.py, bench.py) and the options it offers beside them; draw() gives more cases
over the same ranges.

Fields of a case:
  api       "device": prompt in device memory; "host": prompt and result in pinned host memory
            (delta_attn_prefill_host); "ragged": one call over sequences of different lengths
            (delta_attn_prefill_varlen), each with its own Eq. 5 window
  source    "query" (strategy 1), "key" (strategy 3), "key_packed" (strategy 3 decoding from the
            compressed key-delta cache), "bottom_up" (strategy 2, prefill only)
  dtype, B, H, H_kv, d, T     layer shape and prompt length ("ragged": the longest prompt)
  theta, W, shape             delta threshold, prefill window and its shape
  steps, W_d                  generated tokens and the decode window
  slack                       cache rows kept free behind the last token
  T_lo, gamma                 "ragged" only: shortest prompt, scaling factor of Eq. 5
"""
import math
import random

import torch

from paper_2507_19608_b200 import binding as B

RHO = 0.95            # AR(1) coefficient along tokens (the benchmark's generator)
CHANNEL_SIGMA = 0.5   # log-normal spread of the channel scales
W_MAX = 256           # upper end of Eq. 5's window in the benchmark's grid

SOURCES = {"query": B.DELTA_SRC_QUERY, "key": B.DELTA_SRC_KEY, "key_packed": B.DELTA_SRC_KEY,
           "bottom_up": B.DELTA_SRC_QUERY_BOTTOM_UP}
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


def _case(name, B, H, H_kv, d, T, theta, W, *, dtype="bf16", api="device", source="query", shape="block", steps=0,
          W_d=0, slack=0, T_lo=0, gamma=0.0):
    return dict(name=name, api=api, source=source, dtype=dtype, B=B, H=H, H_kv=H_kv, d=d, T=T, theta=theta, W=W,
                shape=shape, steps=steps, W_d=W_d, slack=slack, T_lo=T_lo, gamma=gamma)


def listed():
    return [
        # the smallest configuration: one short fp32 head; a call is launches and latency
        _case("single_head_fp32", 1, 1, 1, 64, 128, 0.1, 16, dtype="f32"),
        # the headline: one Llama-3.2-1B layer reads a 1024-token prompt
        _case("llama_layer_1k", 1, 32, 8, 64, 1024, 0.1, 64),
        # the same call for a caller whose tensors are in host memory
        _case("llama_layer_1k_host", 1, 32, 8, 64, 1024, 0.1, 64, api="host"),
        # one BitNet-b1.58-2B-4T layer (head dimension 128) reads a 2048-token prompt
        _case("bitnet_layer_2k", 1, 20, 5, 128, 2048, 0.29, 128),
        # the BitNet layer answers a prompt of ordinary, ragged length for two users
        _case("bitnet_generate", 2, 20, 5, 128, 1531, 0.29, 100, shape="sliding", steps=64, W_d=128, slack=5),
        # decoding for one user: 256 tokens behind a 2048-token prompt, latency per step counts
        _case("llama_decode_b1", 1, 32, 8, 64, 2048, 0.1, 64, steps=256, W_d=64),
        # decoding for sixteen users
        _case("llama_decode_b16", 16, 32, 8, 64, 2048, 0.1, 64, steps=256, W_d=64),
        # the largest configuration: one layer of the 16-layer stack, long prompts, then 128 tokens
        _case("stack_layer", 8, 32, 8, 64, 4096, 0.2, 256, steps=128, W_d=256),
        # key deltas (the strategy the paper adopts), odd prompt length, sliding window
        _case("key_generate", 4, 32, 8, 64, 1777, 0.3, 100, source="key", shape="sliding", steps=64, W_d=64),
        # key deltas decoded from the compressed key-delta cache (memory-limited deployment)
        _case("key_packed_generate", 4, 32, 8, 64, 1024, 0.3, 64, source="key_packed", steps=64, W_d=64),
        # prompts of different lengths in one call, Eq. 5 windows, the paper's decode window of 4
        _case("ragged_batch", 6, 32, 8, 64, 1900, 0.2, 0, api="ragged", steps=24, W_d=4, T_lo=90, gamma=0.05),
        # a full-precision layer: fp32 prompt and decode
        _case("fp32_layer", 1, 16, 4, 64, 1000, 0.1, 64, dtype="f32", shape="sliding", steps=32, W_d=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    api = rng.choice(["device"] * 7 + ["host", "ragged", "ragged"])
    source = rng.choice(["query"] * 5 + ["key"] * 3 + ["key_packed", "bottom_up"])
    dtype = rng.choice(["bf16", "bf16", "bf16", "f32"]) if source == "query" else "bf16"
    d = rng.choice([64, 64, 128])
    H, H_kv = rng.choice([(32, 8), (32, 8), (20, 5), (16, 4), (24, 3), (16, 8), (8, 8), (4, 1), (1, 1)])
    batch = _log_int(rng, 2, 8) if api == "ragged" else _log_int(rng, 1, 16)
    T = _log_int(rng, 48, 4096)
    steps = 0 if source == "bottom_up" or api == "host" or rng.random() < 0.4 else _log_int(rng, 4, 256)
    # Fit the pass under the largest listed one: fp32 arithmetic, the compressed cache, copies
    # over PCIe and the one-by-one calls of a ragged batch cost more per unit of work.
    if api == "ragged":
        steps = min(steps, 192 // batch)
    if source == "key_packed":
        steps = min(steps, 48)
    if dtype == "f32":
        steps = min(steps, 64)
    flops_cap = 1.0e10 if dtype == "f32" else 2.0e11
    bytes_cap = 4.0e7 if api == "host" else 4.0e9
    c = dict(api=api, source=source, dtype=dtype, B=batch, H=H, H_kv=H_kv, d=d, T=T, theta=round(rng.uniform(0.05, 0.4), 3),
             W=0, shape=rng.choice(["block", "sliding"]), steps=steps, W_d=rng.choice([4, 16, 64, 128, _log_int(rng, 1, 512)]),
             slack=rng.choice([0, rng.randrange(1, 100)]), T_lo=0, gamma=0.0)
    if api == "ragged":
        c["T_lo"], c["gamma"] = max(1, T // rng.choice([2, 8, 20])), rng.choice([0.02, 0.05, 0.1])
    while _prefill_flops(c) > flops_cap or work(c)["bytes"] > bytes_cap:
        if c["B"] > (2 if api == "ragged" else 1):
            c["B"] -= 1
        else:
            c["T"] = c["T"] * 3 // 4
            c["T_lo"] = min(c["T_lo"], c["T"])
    c["W"] = rng.choice([0, 64, 128, 256, _log_int(rng, 1, c["T"]), _log_int(rng, 1, c["T"])])
    return c


def _lengths(case):
    """Prompt lengths of the batch; "ragged": spread over the logarithm from T_lo to T, the longest first."""
    if case["api"] != "ragged":
        return [case["T"]] * case["B"]
    r = random.Random(case["B"] * 100003 + case["T"])
    lo, hi = math.log(case["T_lo"]), math.log(case["T"])
    return [case["T"]] + [int(round(math.exp(r.uniform(lo, hi)))) for _ in range(case["B"] - 1)]


def _prefill_flops(case):
    return sum(4.0 * case["d"] * case["H"] * n * (n + 1) / 2 for n in _lengths(case))


def work(case):
    """Bytes: the prompt's q, k, v and output, the delta arrays the prefill leaves (values, mask,
    counts, indices, tile references, score row), and per generated token the cached keys and values
    read once per KV head, the score row written (query deltas) and the new rows.  Flops: a score and
    a P.V multiply-add per causal pair and channel (the telescoped form of Eq. 4 is dense)."""
    es = 4 if case["dtype"] == "f32" else 2
    H, H_kv, d = case["H"], case["H_kv"], case["d"]
    key = case["source"].startswith("key")
    Hs = H_kv if key else H                                    # heads of the delta stream
    nbytes = flops = 0.0
    for n in _lengths(case):
        nbytes += n * (2 * H + 2 * H_kv) * d * es              # q, out, k, v
        nbytes += n * Hs * (4 * d + d / 8 + 2 + d) + Hs * (n / 64) * (4 + 4 * d)
        nbytes += 0 if key else 4 * H * n                      # R
        flops += 4.0 * d * H * n * (n + 1) / 2
        for s in range(case["steps"]):
            L = n + s
            nbytes += 2 * H_kv * L * d * es + (0 if key else 4 * H * L) + (2 * H + 4 * H_kv) * d * es + 8 * Hs * d
            flops += 4.0 * d * H * (L + 1)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Masks, counts and indices are whole numbers and exact.  fp32: sums of up to 128 products and a
    softmax row in another order.  bf16: the output's rounding and the bf16 probabilities of P.V."""
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.0}
    return {"rel": 5e-3, "max": 3e-2, "differ": 0.0}


def _streams(gen, batch, heads, rows, d, dtype):
    """[batch, heads, rows, d] AR(1) chains along the rows, unit variance times a channel scale."""
    x = torch.randn(batch, heads, rows, d, generator=gen, device="cuda")
    x[:, :, 1:] *= math.sqrt(1.0 - RHO * RHO)
    k = 1
    while k < rows and RHO ** k > 1e-9:                        # x_t = sum of RHO^s e_(t-s), by doubling
        y = x.clone()
        y[:, :, k:].add_(x[:, :, :-k], alpha=RHO ** k)
        x, k = y, 2 * k
    scale = torch.exp(CHANNEL_SIGMA * torch.randn(1, heads, 1, d, generator=gen, device="cuda"))
    return (x * scale).to(DTYPES[dtype])


def prepare(case, seed):
    c, gen = case, torch.Generator("cuda").manual_seed(seed)
    nb, H, H_kv, d, T, steps, dt = c["B"], c["H"], c["H_kv"], c["d"], c["T"], c["steps"], c["dtype"]
    lens = _lengths(c)
    T_max = T + steps + c["slack"]
    cfg = B.make_config(nb, H, H_kv, d, T_max, dt, source=SOURCES[c["source"]],
                        prefill_window=B.DELTA_WIN_BLOCK if c["shape"] == "block" else B.DELTA_WIN_SLIDING)
    st = B.delta_state_init(cfg)
    if c["source"] == "key_packed":
        B.delta_state_set_key_cache(st, True)
    q = _streams(gen, nb, H, T + steps, d, dt)
    k = _streams(gen, nb, H_kv, T + steps, d, dt)
    v = _streams(gen, nb, H_kv, T + steps, d, dt)
    s = dict(case=c, st=st, lens=lens)

    if c["api"] == "host":
        host = lambda x: x[:, :, :T].contiguous().cpu().pin_memory()       # noqa: E731
        s["q"], s["k"], s["v"] = host(q), host(k), host(v)
        s["out"] = torch.empty_like(s["q"]).pin_memory()
        s["staging"] = torch.empty(B.delta_prefill_staging_bytes(cfg, T), dtype=torch.uint8, device="cuda")
    else:
        if c["api"] == "ragged":
            s["q"] = torch.cat([q[b, :, :n].reshape(-1) for b, n in enumerate(lens)])
            s["windows"] = [B.delta_window_from_gamma(n, c["gamma"], W_MAX) for n in lens]
        else:
            s["q"] = q[:, :, :T].contiguous()
        s["out"] = torch.empty_like(s["q"])
        s["k"] = torch.zeros(nb, H_kv, T_max, d, dtype=k.dtype, device="cuda")   # the layer's KV cache
        s["v"] = torch.zeros_like(s["k"])
        s["k"][:, :, :T], s["v"][:, :, :T] = k[:, :, :T], v[:, :, :T]
        # the generated tokens' rows, as a model's projections would hand them over one by one
        rows = lambda x: x[:, :, T:].permute(2, 0, 1, 3).contiguous()      # noqa: E731
        s["dec_out"] = torch.empty(steps, nb, H, d, dtype=q.dtype, device="cuda")
        s["tokens"] = list(zip(rows(q).unbind(0), rows(k).unbind(0), rows(v).unbind(0), s["dec_out"].unbind(0)))

    # the delta arrays the prefill leaves in the state (key deltas: one set per KV head)
    Hs = H_kv if c["source"].startswith("key") else H

    def view(what, heads, *tail):
        x = B.delta_state_view(st, what)
        return x.reshape(-1)[:nb * heads * math.prod(tail)].view(nb, heads, *tail)

    tiles = -(-T_max // B.DELTA_TILE_ROWS)
    s["arrays"] = arrays = {}
    for b, n in enumerate(lens if c["api"] == "ragged" else [T]):
        at = slice(b, b + 1) if c["api"] == "ragged" else slice(None)
        arrays["dq%d" % b] = view(B.DELTA_VIEW_DQ, Hs, T_max, d)[at, :, :n]
        arrays["mask%d" % b] = view(B.DELTA_VIEW_MASK, Hs, T_max, d // 32)[at, :, :n]
        arrays["row_nnz%d" % b] = view(B.DELTA_VIEW_ROW_NNZ, Hs, T_max)[at, :, :n]
        arrays["idx%d" % b] = view(B.DELTA_VIEW_IDX, Hs, T_max, d)[at, :, :n]
        arrays["tile_nnz%d" % b] = view(B.DELTA_VIEW_TILE_NNZ, Hs, tiles)[at, :, :-(-n // 64)]
        if c["source"] == "query":
            arrays["R%d" % b] = view(B.DELTA_VIEW_R, H, T_max)[at, :, :n + steps]
    return s


def run(s):
    c, st = s["case"], s["st"]
    B.delta_state_reset(st)
    if c["api"] == "host":
        B.delta_attn_prefill_host(st, s["q"], s["k"], s["v"], s["out"], s["staging"], c["T"], c["theta"], c["W"])
        return dict(s["arrays"], out=s["out"])
    if c["api"] == "ragged":
        B.delta_attn_prefill_varlen(st, s["q"], s["k"], s["v"], s["out"], s["lens"], s["windows"], c["theta"])
    else:
        B.delta_attn_prefill(st, s["q"], s["k"], s["v"], s["out"], c["T"], c["H"], c["H_kv"], c["d"], c["theta"], c["W"])
    for q_new, k_new, v_new, out in s["tokens"]:
        B.delta_attn_decode_step(st, q_new, k_new, v_new, s["k"], s["v"], out, c["theta"], c["W_d"])
    return dict(s["arrays"], out=s["out"], generated=s["dec_out"], k_cache=s["k"], v_cache=s["v"],
                reference=B.delta_state_view(st, B.DELTA_VIEW_QHAT).reshape(-1)[:c["B"] * _ref_heads(c) * c["d"]])


def _ref_heads(case):
    return case["H_kv"] if case["source"].startswith("key") else case["H"]
