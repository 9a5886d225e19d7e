"""What the performance of this framework is measured on.

Every case is one request as a serving or scoring program runs it: the prompt's keys and values are compressed into the
cache (corm_compress_prompt for every layer), then tokens are decoded through one of the step entry points, and at the
end the program reads the cache's totals and live lengths, as a scheduler that accounts KV memory does. A pass starts
with the prompt pass, which replaces whatever the cache held, so passes are independent of one another.

Inputs follow the recipe of paper_2404_15949_b200/workload, formed on the GPU: keys and queries are AR(1) chains
(rho 0.9, sigma 0.44), a few planted "heavy-hitter" keys are four times as large, values are N(0, 1), and the query
heads of a group share 0.7 of their variance.
"""
import math

import torch

from paper_2404_15949_b200.binding import CormCache

DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}
# how the tokens are decoded: one call per layer and token (a sampling loop over a model's layers), one call per token
# for all layers, all tokens in one call (scoring a given text), the same from pinned host memory
APIS = ("step", "layers", "steps", "steps_host")


def case(name, **kw):
    c = dict(name=name, layers=1, batch=1, kv_heads=8, group=1, head_dim=128, dtype="bf16", prompt_min=512,
             prompt_max=512, steps=32, window=8, recent=256, alpha=1.0, heavy=32, pool_pages=0, api="step")
    c.update(kw)
    return c


def listed():
    return [
        # the smallest request: one layer, one short sequence, fp32 cache; launches and round trips are all of it
        case("tiny_f32", dtype="f32", prompt_min=512, prompt_max=512, steps=64, recent=32, heavy=4),
        # one chat sequence through a 32-layer model, a call per layer and token: latency and host time per call
        case("single_sequence_32_layers", layers=32, kv_heads=32, prompt_min=4096, prompt_max=4096, steps=16),
        # batched serving, one query head per KV head, ragged prompts, sampling loop
        case("batch32_sampling", batch=32, kv_heads=32, prompt_min=2048, prompt_max=4096, steps=96),
        # the same model scoring given texts from host memory: all tokens of a layer in one call
        case("batch32_scoring_host", batch=32, kv_heads=32, prompt_min=1500, prompt_max=3001, steps=128,
             api="steps_host"),
        # grouped heads, 8k prompts, sampling loop
        case("grouped_sampling", batch=16, kv_heads=8, group=4, prompt_min=8192, prompt_max=8192, steps=96),
        # grouped heads scoring with a paged cache, ragged prompts
        case("grouped_scoring_paged", batch=16, kv_heads=8, group=4, prompt_min=3001, prompt_max=8192, steps=128,
             pool_pages=32768, api="steps"),
        # long context, few sequences, wider window and protected tail
        case("long_context_grouped", batch=4, kv_heads=8, group=4, prompt_min=32768, prompt_max=32768, steps=96,
             window=16, recent=512, heavy=16),
        # the paper's own setting, 256 recent queries and 256 protected tokens: wide prompt window, long live units
        case("window256", batch=4, kv_heads=32, prompt_min=2048, prompt_max=4096, steps=48, window=256),
        # the paper's 128 + 128 with grouped heads
        case("window128_grouped", batch=4, kv_heads=8, group=4, prompt_min=8192, prompt_max=8192, steps=48, window=128,
             recent=128),
        # groups of eight query heads
        case("group8", batch=8, kv_heads=8, group=8, prompt_min=1024, prompt_max=3000, steps=48),
        # 64-channel heads in groups of four
        case("head64_grouped", batch=16, kv_heads=8, group=4, head_dim=64, prompt_min=1024, prompt_max=3000, steps=48,
             window=16),
        # an fp32 cache of ordinary size, grouped heads, odd batch
        case("f32_grouped", batch=5, kv_heads=4, group=2, dtype="f32", prompt_min=700, prompt_max=2001, steps=48,
             recent=128, window=8),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: batch 1-32, 1-32 KV heads, groups of 1-8, prompts of 48-32768 tokens (ragged
    ones half of the time), windows of 4-256 queries, 16-512 protected tokens, both dtypes and head sizes, every way of
    decoding."""
    while True:
        c = dict(layers=1, batch=_log_uniform(rng, 1, 32), kv_heads=rng.choice([1, 2, 3, 4, 8, 8, 16, 32]),
                 group=rng.choice([1, 1, 2, 4, 4, 8]), head_dim=rng.choice([128, 128, 128, 64]),
                 dtype=rng.choice(["bf16", "bf16", "bf16", "f32"]), prompt_max=_log_uniform(rng, 48, 32768),
                 steps=_log_uniform(rng, 8, 128), window=_log_uniform(rng, 4, 256) if rng.random() < 0.5 else 8,
                 recent=_log_uniform(rng, 16, 512), alpha=rng.choice([1.0, 1.0, 1.0, 0.5, 0.0]),
                 heavy=rng.randint(4, 64), pool_pages=0, api=rng.choice(APIS + ("step",)))
        c["prompt_min"] = c["prompt_max"] if rng.random() < 0.5 else max(1, c["prompt_max"] // 2 - rng.randint(0, 9))
        if c["api"] == "layers" or rng.random() < 0.15:
            c["layers"] = rng.randint(2, 8)
        units = c["batch"] * c["kv_heads"]
        if rng.random() < 0.25:                       # a page pool with room for every key
            c["pool_pages"] = -(-units * ((c["prompt_max"] + c["steps"]) // 32 + 2) // 32) * 32
        keys = c["layers"] * units * c["prompt_max"]
        row_keys = keys * c["window"] * c["group"]    # prompt rows x keys
        if c["dtype"] == "bf16" and c["head_dim"] == 128 and c["group"] < 8:
            most, most_unit = 1.3e8, 4e6
        else:                                         # used with small windows and models
            most, most_unit = 1.5e7, 1.5e5
            c["steps"] = min(c["steps"], 256 // c["layers"])
        if keys * c["head_dim"] * (2 if c["dtype"] == "bf16" else 4) <= 6e8 and row_keys <= most \
                and c["layers"] * c["prompt_max"] * c["window"] * c["group"] <= most_unit and work(c)["bytes"] <= 1.2e10:
            return c


def _ar1(gen, shape, device):
    """AR(1) chains along the second to last axis (rho 0.9, sigma 0.44, started at N(0, 1)), by repeated doubling."""
    x = torch.randn(shape, generator=gen, device=device)
    x[..., 1:, :] *= 0.44
    step, rho = 1, 0.9
    while step < shape[-2] and step <= 128:           # 0.9^256 is below the last bit
        x[..., step:, :] += rho * x[..., :-step, :].clone()
        step, rho = 2 * step, rho * rho
    return x


def prepare(case, seed):
    dev = torch.device("cuda", 0)
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    host = torch.Generator()
    host.manual_seed(seed)
    L, B, H, G, d = case["layers"], case["batch"], case["kv_heads"], case["group"], case["head_dim"]
    w, r, n, dt = case["window"], case["recent"], case["steps"], DTYPES[case["dtype"]]
    lo, hi = case["prompt_min"], case["prompt_max"]
    lens = torch.randint(lo, hi + 1, (B,), generator=host).to(torch.int32).numpy()
    p_max = int(lens.max())
    cache = CormCache(L, B, H * G, H, d, hi + n, w, r, case["alpha"], case["dtype"], 0, pool_pages=case["pool_pages"])
    q = torch.empty((n, L, B, H * G, d), dtype=dt, device=dev)
    k_new = torch.empty((n, L, B, H, d), dtype=dt, device=dev)
    v_new = torch.randn((n, L, B, H, d), generator=gen, device=dev).to(dt)
    prompts = []
    for layer in range(L):
        k = torch.empty((B, H, p_max, d), dtype=dt, device=dev)
        v = torch.empty((B, H, p_max, d), dtype=dt, device=dev)
        q_last = torch.zeros((B, H * G, w, d), dtype=dt, device=dev)
        for b in range(B):
            P = int(lens[b])
            keys = _ar1(gen, (H, P + n, d), dev)
            if P > r:
                at = torch.randint(0, P - r, (H, case["heavy"]), generator=gen, device=dev)
                planted = 4.0 * torch.randn((H, case["heavy"], d), generator=gen, device=dev)
                for i in range(case["heavy"]):        # one at a time: positions may repeat, the last one stays
                    keys.scatter_(1, at[:, i:i + 1, None].expand(H, 1, d), planted[:, i:i + 1])
            k[b, :, :P] = keys[:, :P].to(dt)
            k_new[:, layer, b] = keys[:, P:].transpose(0, 1).to(dt)
            v[b, :, :P] = torch.randn((H, P, d), generator=gen, device=dev).to(dt)
            wp = min(P, w)
            qs = _ar1(gen, (H, G, wp + n, d), dev)
            if G > 1:
                qs = math.sqrt(0.7) * _ar1(gen, (H, 1, wp + n, d), dev) + math.sqrt(0.3) * qs
            qs = qs.reshape(H * G, wp + n, d)
            q_last[b, :, w - wp:] = qs[:, :wp].to(dt)
            q[:, layer, b] = qs[:, wp:].transpose(0, 1).to(dt)
        for b in range(B):                            # rows past a sequence's length are never read
            k[b, :, int(lens[b]):] = 0
            v[b, :, int(lens[b]):] = 0
        prompts.append((k, v, q_last))
    if case["api"] == "steps_host":
        q, k_new, v_new = (t.cpu().pin_memory() for t in (q, k_new, v_new))
        out = torch.empty_like(q).pin_memory()
    else:
        out = torch.empty_like(q)
    s = dict(api=case["api"], L=L, n=n, cache=cache, prompts=prompts, lens=lens, q=q, k_new=k_new, v_new=v_new, out=out)
    # a model hands the cache one tensor per token (and layer): views made here once, not indexing inside the loop
    if case["api"] == "step":
        s["calls"] = [(l, q[i, l], k_new[i, l], v_new[i, l], out[i, l]) for i in range(n) for l in range(L)]
    elif case["api"] == "layers":
        s["calls"] = [tuple([t[i, l] for l in range(L)] for t in (q, k_new, v_new, out)) for i in range(n)]
    return s


def run(state):
    cache = state["cache"]
    for layer, (k, v, q_last) in enumerate(state["prompts"]):
        cache.corm_compress_prompt(layer, k, v, q_last, state["lens"])
    if state["api"] == "step":
        for layer, q, k, v, out in state["calls"]:
            cache.corm_decode_step(layer, q, k, v, out)
    elif state["api"] == "layers":
        for q, k, v, out in state["calls"]:
            cache.corm_decode_step_layers(0, q, k, v, out)
    elif state["api"] == "steps":
        cache.corm_decode_steps(0, state["L"], state["q"], state["k_new"], state["v_new"], state["out"])
    else:
        cache.corm_decode_steps_host(0, state["L"], state["q"], state["k_new"], state["v_new"], state["out"])
    stats = cache.corm_cache_stats()
    totals = [int(stats[k]) for k in ("live_keys", "appended_keys", "evicted_keys", "attended_keys", "important_keys",
                                      "device_status")]
    live = [cache.corm_cache_live_lens(layer) for layer in {0, state["L"] - 1}]
    return {"out": state["out"], "totals": totals, "live": live}


def live_keys(case):
    """(keys of a unit that survive the prompt pass, mean live keys over the decode steps), as these inputs show them: a
    fit to measured totals over prompts of 256-32768 tokens, windows of 4-256 and groups of 1-8, within about a fifth."""
    P, w, r, G, n = (case["prompt_min"] + case["prompt_max"]) / 2, case["window"], case["recent"], case["group"], case["steps"]
    if P <= r or P < w or case["alpha"] == 0.0:
        return P, P + (n + 1) / 2
    x = -0.48 + 0.474 * math.log(P / 4096) + 0.779 * math.log(w / 8) + 0.4 * (w - 8) / 64 + 0.618 * math.log(G)
    kept = r + (P - r) / (1 + math.exp(-x))
    decay = n / (20 * math.exp(w / 24) * G ** 0.35)
    return kept, r + (kept - r) * -math.expm1(-decay) / decay + n / 4


def work(case):
    """What a pass cannot do without. Prompt: every key once and the last queries; the survivors' values in, their keys,
    values, registers and positions out; a product per recorded row and key. A step: the live keys and values once,
    their registers and positions in and the registers out, the token's rows in and out; two products per head and key."""
    L, G, d, w, n = case["layers"], case["group"], case["head_dim"], case["window"], case["steps"]
    units, e = case["batch"] * case["kv_heads"], 2 if case["dtype"] == "bf16" else 4
    P = (case["prompt_min"] + case["prompt_max"]) / 2
    kept, live = live_keys(case)
    prompt = P * d * e + min(P, w) * G * d * e + kept * (3 * d * e + 8)
    step = live * (2 * d * e + 12) + 2 * G * d * e + 4 * d * e
    flops = 2 * min(P, w) * G * P * d + n * live * 4 * G * d
    return {"bytes": L * units * (prompt + n * step), "flops": L * units * flops}


def tolerance(case):
    """Outputs: sums of at most 32768 terms in fp32, rounded to the cache's type. The same path with its splits cut
    elsewhere or on the simplest kernels differs by 1e-4 (bf16: roundings that fall the other way, one bit at most) and
    1.4e-7 (fp32) in the norm, 7.8e-3 and 1e-6 at the worst value. Totals and live lengths are whole numbers and stay
    the same: verdicts compare fp64 logits."""
    return {"rel": 4e-4, "max": 3.2e-2} if case["dtype"] == "bf16" else {"rel": 6e-7, "max": 4e-6}
