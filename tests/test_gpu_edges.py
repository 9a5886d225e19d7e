"""Corners of the decode and prompt kernels: precision of the outputs, long units, magnitudes far outside the usual range,
length reports. Against the CPU oracle unless a test says otherwise."""
import numpy as np
import pytest
import torch

from paper_2404_15949_b200.workload import CONFIGS, generate
from parity_util import OUT_TOL, assert_states_equal, make_gpu_cache, make_oracle, sorted_state, stamps_to_ages, to_dev

pytestmark = pytest.mark.gpu


def _cfg(dtype, d, G, nkv, B, prange, steps, w, r, seed=50, **kw):
    return CONFIGS[1].with_(name="edges", batch=B, n_q_heads=nkv * G, n_kv_heads=nkv, head_dim=d, dtype=dtype,
                            prompt_min=prange[0], prompt_max=prange[1], steps=steps, window_w=w, recent_r=r,
                            gqa_rho=0.7 if G > 1 else 0.0, hh_min=2, hh_max=6, seed=seed, **kw)


@pytest.mark.parametrize("d,G", [(128, 1), (128, 2), (128, 4), (128, 8), (64, 1), (64, 4), (64, 8)])
def test_bf16_outputs_are_the_exact_ones_rounded(d, G):
    """Probabilities and products of fp32 precision leave an output off by about 2^-22 of its scale, so it rounds to
    another bf16 than the exact one about once in 2^-22 / 2^-8 = 6 10^-5 (and a little more where outputs are small);
    probabilities cut to two bf16 parts make that 10^-3. Bound: 3 10^-4, four standard deviations above 10^-4 for the
    smallest number of outputs here (2 10^4)."""
    nkv, B, steps = max(1, 8 // G), 4, 20
    cfg = _cfg("bf16", d, G, nkv, B, (900, 1100), steps, 64, 256, alpha=1.0)
    data = generate(cfg)
    gpu, orc = make_gpu_cache(cfg, B, nkv), make_oracle(cfg, B, nkv)
    gpu.corm_compress_prompt(0, to_dev(data.k_prompt, "bf16"), to_dev(data.v_prompt, "bf16"), to_dev(data.q_last, "bf16"),
                             data.prompt_lens)
    orc.compress_prompt(0, data.k_prompt, data.v_prompt, data.q_last, data.prompt_lens)
    q, k, v = (to_dev(x, "bf16") for x in (data.q, data.k_new, data.v_new))
    wrong = total = 0
    for s in range(steps):
        ref = torch.from_numpy(orc.decode_step(0, data.q[s], data.k_new[s], data.v_new[s])).to(torch.bfloat16)
        out = gpu.corm_decode_step(0, q[s], k[s], v[s]).cpu()
        wrong += int((out != ref).sum())
        total += out.numel()
    assert_states_equal(gpu, orc, 0, B, nkv, "end")
    assert total >= 20000 and wrong <= 3e-4 * total, (wrong, total)


# one block per unit as long as its list space allows (a split length beyond the unit), so a block owns about as many 32-slot
# words as it can keep track of (3583 for fp32 / 64 channels, 4096 otherwise; EVICTED below has exactly as many and one more), or
# two blocks where a unit may have more than that
LONG_UNITS = [
    # dtype, head_dim, group, live keys, max_tokens, paged
    ("f32", 64, 1, 98250, 3071 * 32, False),
    ("f32", 64, 8, 98270, 3071 * 32, True),
    ("f32", 64, 2, 98290, 3072 * 32, False),
    ("bf16", 64, 1, 100000, 4096 * 32, False),
    ("bf16", 128, 4, 70000, 4097 * 32, True),
]


@pytest.mark.parametrize("case", LONG_UNITS, ids=lambda c: "-".join(str(x) for x in c))
def test_long_unit_loses_thousands_of_keys_in_one_step(case):
    """An imported unit whose keys are all up for eviction (window of one query): the first step removes thousands
    of them, so the moves are listed in scratch, by blocks that own as many words as they may."""
    dtype, d, G, n, C, paged = case
    cfg = _cfg(dtype, d, G, 1, 1, (1, 1), 3, 1, 64)
    rng = np.random.default_rng(17 + d + G)
    to = (lambda x: to_dev(x, dtype).float().cpu().numpy())
    k, v = (to(rng.standard_normal((n, d), dtype=np.float32)) for _ in range(2))
    q = to(rng.standard_normal((3, 1, G, d), dtype=np.float32))
    kn, vn = (to(rng.standard_normal((3, 1, 1, d), dtype=np.float32)) for _ in range(2))
    word, pos = np.ones(n, np.uint32), np.arange(1, n + 1, dtype=np.int32)
    gpu = make_gpu_cache(cfg, 1, 1, max_tokens=C, pool_pages=(C // 1024 + 2) * 32 if paged else 0)
    orc = make_oracle(cfg, 1, 1, max_tokens=C)
    orc.set_near_band(1e-10)           # 10^5 keys a step put one within the usual 10^-6; sums of fp64 terms differ by 10^-13
    gpu.corm_cache_set_tuning(1 << 18, True)
    gpu.corm_cache_import_state(0, 0, 0, k, v, word, pos, n, 1)
    orc.import_unit(0, 0, 0, k, v, word, pos, n, 1)
    for s in range(3):
        out = gpu.corm_decode_step(0, to_dev(q[s], dtype), to_dev(kn[s], dtype), to_dev(vn[s], dtype))
        ref = orc.decode_step(0, q[s], kn[s], vn[s])
        assert np.abs(out.float().cpu().numpy() - ref).max() <= OUT_TOL[dtype]
        assert_states_equal(gpu, orc, 0, 1, 1, f"step {s}")
    assert orc.counters()["near_threshold"] == 0
    st = gpu.corm_cache_stats()
    assert st["device_status"] == 0 and st["evicted_keys"] > 8000


def test_a_key_appended_next_to_an_overflowed_query_counts():
    """Two steps whose queries leave the range of the exact pieces (an element of 2^60) append the largest keys a unit has
    seen, 2^20 against 1, one bit of one channel apart. Later ordinary queries find their probabilities next to the
    threshold often enough (128 units, 30 steps) to show logits formed on a grid that does not know these keys."""
    B, nkv, d, steps = 8, 16, 128, 32
    cfg = _cfg("bf16", d, 1, nkv, B, (40, 40), steps, 32, 256)
    data = generate(cfg)
    rng = np.random.default_rng(5)
    big = (rng.standard_normal((B, nkv, d)) * 2.0 ** 20).astype(np.float32)
    big = torch.from_numpy(big).to(torch.bfloat16).float().numpy()
    big[..., 0] = 2.0 ** 12
    q, kn, vn = data.q.copy(), data.k_new.copy(), data.v_new.copy()
    kn[0], kn[1] = big, big
    kn[1][..., 0] += 32.0                              # a bit of 2^12 in bf16: logits 2.8 q_0 apart
    q[:2, ..., 1] = 2.0 ** 60
    gpu, orc = make_gpu_cache(cfg, B, nkv), make_oracle(cfg, B, nkv)
    gpu.corm_cache_set_tuning(0, 4)                    # the cluster kernel
    orc.set_near_band(1e-10)
    gpu.corm_compress_prompt(0, to_dev(data.k_prompt, "bf16"), to_dev(data.v_prompt, "bf16"), to_dev(data.q_last, "bf16"),
                             data.prompt_lens)
    orc.compress_prompt(0, data.k_prompt, data.v_prompt, data.q_last, data.prompt_lens)
    for s in range(steps):
        gpu.corm_decode_step(0, to_dev(q[s], "bf16"), to_dev(kn[s], "bf16"), to_dev(vn[s], "bf16"))
        orc.decode_step(0, q[s], kn[s], vn[s])
        assert_states_equal(gpu, orc, 0, B, nkv, f"step {s}")
    assert gpu.corm_cache_stats()["device_status"] == 0


def test_destroy_waits_for_launches_that_report_even_after_a_reset():
    """Kernels write lengths to pinned host memory of the cache. A reset forgets the reports that are on their way, but the
    launches behind them still run: the cache's memory must outlive them."""
    cfg = _cfg("bf16", 128, 4, 8, 4, (2000, 2000), 64, 8, 64)
    data = generate(cfg)
    gpu = make_gpu_cache(cfg, 4, 8)
    p = [to_dev(x, "bf16") for x in (data.k_prompt, data.v_prompt, data.q_last)]
    q, k, v = (to_dev(x, "bf16") for x in (data.q, data.k_new, data.v_new))
    out = torch.empty_like(q)
    torch.cuda.synchronize()
    for _ in range(8):
        gpu.corm_compress_prompt(0, *p, data.prompt_lens)
        for s in range(64):
            gpu.corm_decode_step(0, q[s], k[s], v[s], out[s])
    done = torch.cuda.Event()
    done.record()
    gpu.corm_cache_reset()
    gpu.close()
    assert done.query()


def test_layers_of_different_history_stepped_together_still_report_their_lengths():
    """One layer has had a prompt pass more than the other. Launches over both must go on reporting lengths: the grids of
    the block-per-split kernel follow them, and once the units are known to fit one split (1024 keys) a step is one launch
    instead of two."""
    cfg = _cfg("bf16", 128, 1, 4, 2, (3000, 3000), 40, 8, 64)                    # 1900 keys of a unit survive the prompt, 900 the steps
    data = [generate(cfg, layer=l) for l in range(2)]
    gpu = make_gpu_cache(cfg, 2, 4, n_layers=2)
    gpu.corm_cache_set_tuning(1024, 3)
    for l in (0, 0, 1):
        gpu.corm_compress_prompt(l, *(to_dev(getattr(data[l], n), "bf16") for n in ("k_prompt", "v_prompt", "q_last")),
                                 data[l].prompt_lens)
    q, k, v = (torch.stack([to_dev(getattr(x, n), "bf16") for x in data], dim=1).contiguous() for n in ("q", "k_new", "v_new"))
    out = torch.empty_like(q)
    for s in range(40):
        torch.cuda.synchronize()                       # whatever was asked for has been reported
        before = gpu.corm_cache_kernel_launches()
        gpu.corm_decode_step_layers(0, *([t[s, l] for l in range(2)] for t in (q, k, v, out)))
    assert max(int(gpu.corm_cache_live_lens(l).max()) for l in range(2)) < 1000
    assert gpu.corm_cache_kernel_launches() - before == 1


# magnitudes that the pieces of the tensor-core logits do not hold (2^56 and more), and logits beyond fp32
OUT_OF_RANGE = [
    # dtype, head_dim, group, kv heads, batch, prompt range, steps, paged, what
    ("bf16", 128, 1, 2, 2, (300, 420), 12, False, "keys"),
    ("bf16", 128, 2, 2, 1, (31, 33), 40, True, "late key"),
    ("bf16", 128, 4, 2, 2, (700, 900), 12, True, "queries"),
    ("bf16", 128, 8, 1, 2, (500, 600), 12, False, "late key"),
    ("bf16", 64, 1, 3, 1, (1, 17), 40, True, "late key"),
    ("bf16", 64, 4, 2, 1, (900, 1000), 12, False, "keys"),
    ("bf16", 64, 8, 1, 1, (600, 600), 12, False, "both"),
    ("bf16", 128, 4, 1, 1, (3000, 3000), 6, False, "both"),
    ("f32", 128, 2, 2, 1, (400, 500), 12, False, "both"),
    ("f32", 64, 1, 1, 2, (100, 130), 24, True, "late key"),
]


@pytest.mark.parametrize("case", OUT_OF_RANGE, ids=lambda c: "-".join(str(x) for x in c))
def test_decode_of_magnitudes_out_of_the_pieces_range(case):
    """Prompts of ordinary keys, then keys and queries scaled by powers of two (so that logits are spread over 2^60 and
    the top key has all the weight, or, between one key and its double, exactly known weights): the oracle's registers,
    rows and outputs through per-step and chained calls."""
    dtype, d, G, nkv, B, prange, steps, paged, what = case
    cfg = _cfg(dtype, d, G, nkv, B, prange, steps, 8, 16)
    data = generate(cfg)
    q, kn = data.q.copy(), data.k_new.copy()
    big = 2.0 ** 60 if dtype == "bf16" else 2.0 ** 70
    if what == "keys":
        kn[2:] *= big
    elif what == "late key":
        kn[steps // 2] *= big
    elif what == "queries":
        q[3:6] *= big
    else:
        kn[1] *= big
        q[2:] *= big if dtype == "bf16" else 2.0 ** 60
    pages = -(-B * nkv * (cfg.max_tokens // 32 + 2) // 32) * 32 if paged else 0
    one, many = (make_gpu_cache(cfg, B, nkv, pool_pages=pages) for _ in range(2))
    orc = make_oracle(cfg, B, nkv)
    orc.set_near_band(1e-12)
    p = [to_dev(x, dtype) for x in (data.k_prompt, data.v_prompt, data.q_last)]
    for g in (one, many):
        g.corm_cache_set_tuning(0, 4)                  # the cluster kernel for every shape
        g.corm_compress_prompt(0, *p, data.prompt_lens)
    orc.compress_prompt(0, data.k_prompt, data.v_prompt, data.q_last, data.prompt_lens)
    qd, kd, vd = (to_dev(x, dtype) for x in (q, kn, data.v_new))
    outs = many.corm_decode_steps(0, 1, qd[:, None], kd[:, None], vd[:, None])
    for s in range(steps):
        ref = orc.decode_step(0, q[s], kn[s], data.v_new[s])
        out = one.corm_decode_step(0, qd[s], kd[s], vd[s])
        assert np.abs(out.float().cpu().numpy() - ref).max() <= OUT_TOL[dtype], s
        assert np.abs(outs[s, 0].float().cpu().numpy() - ref).max() <= OUT_TOL[dtype], s
        assert_states_equal(one, orc, 0, B, nkv, f"step {s}")
    assert_states_equal(many, orc, 0, B, nkv, "multi-step")
    assert one.corm_cache_stats()["device_status"] == many.corm_cache_stats()["device_status"] == 0


@pytest.mark.parametrize("dtype,d,G", [("bf16", 128, 8), ("bf16", 64, 2), ("f32", 128, 1), ("f32", 64, 4)])
@pytest.mark.parametrize("what", ["nan", "inf"])
def test_a_key_that_is_not_a_number(dtype, d, G, what):
    """One NaN or infinite channel of one key, against the generic kernel (tuning value 0): the same outputs are NaN, the
    others agree, and so do the registers."""
    cfg = _cfg(dtype, d, G, 2, 1, (200, 260), 12, 8, 16)
    data = generate(cfg)
    kn = data.k_new.copy()
    kn[3, 0, 1, 7] = np.nan if what == "nan" else np.inf
    caches = [make_gpu_cache(cfg, 1, 2) for _ in range(2)]
    caches[1].corm_cache_set_tuning(0, False)
    p = [to_dev(x, dtype) for x in (data.k_prompt, data.v_prompt, data.q_last)]
    for g in caches:
        g.corm_compress_prompt(0, *p, data.prompt_lens)
    for s in range(12):
        a, b = (g.corm_decode_step(0, to_dev(data.q[s], dtype), to_dev(kn[s], dtype), to_dev(data.v_new[s], dtype)).float().cpu()
                for g in caches)
        assert torch.equal(torch.isnan(a), torch.isnan(b)), s
        assert (a - b).nan_to_num().abs().max() <= OUT_TOL[dtype], s
        for h in range(2):
            x, y = (g.corm_cache_export_state(0, 0, h) for g in caches)
            i, j = np.argsort(x["pos"]), np.argsort(y["pos"])
            assert np.array_equal(x["pos"][i], y["pos"][j]) and np.array_equal(x["word"][i], y["word"][j]), (s, h)


# one key channel f times the others, its query channel 1 / f: logits stay as they are, bounds on the tensor cores grow by f.
# f = 64 is on this side of the switch to the fp64 loop for groups and beyond it for single heads, 4096 beyond it for all
@pytest.mark.parametrize("f", [64.0, 4096.0])
@pytest.mark.parametrize("d,G", [(128, 1), (128, 2), (128, 4), (128, 8), (64, 1), (64, 4)])
def test_one_large_key_channel(d, G, f):
    """Outputs stay the exact ones rounded (the bound of the test of that name) and registers the oracle's, also where some
    of a unit's keys, from the middle of the run on, are the first large ones."""
    nkv, B, steps = max(1, 8 // G), 2, 24
    cfg = _cfg("bf16", d, G, nkv, B, (900, 1100), steps, 8, 64)
    data = generate(cfg)
    rnd = (lambda a: torch.from_numpy(a).to(torch.bfloat16).float().numpy())
    q, kn, kp, ql = (rnd(x.copy()) for x in (data.q, data.k_new, data.k_prompt, data.q_last))
    q[..., 3] /= f
    kn[..., 3] *= f
    kp[0, ..., 3] *= f                                 # the second sequence meets its first large key in a decode step
    ql[0, ..., 3] /= f
    gpu, orc = make_gpu_cache(cfg, B, nkv), make_oracle(cfg, B, nkv)
    orc.set_near_band(1e-11)
    gpu.corm_compress_prompt(0, to_dev(kp, "bf16"), to_dev(data.v_prompt, "bf16"), to_dev(ql, "bf16"), data.prompt_lens)
    orc.compress_prompt(0, kp, data.v_prompt, ql, data.prompt_lens)
    wrong = total = 0
    for s in range(steps):
        ref = torch.from_numpy(orc.decode_step(0, q[s], kn[s], data.v_new[s])).to(torch.bfloat16)
        out = gpu.corm_decode_step(0, to_dev(q[s], "bf16"), to_dev(kn[s], "bf16"), to_dev(data.v_new[s], "bf16")).cpu()
        wrong += int((out != ref).sum())
        total += out.numel()
        assert_states_equal(gpu, orc, 0, B, nkv, f"step {s}")
    assert wrong <= 3e-4 * total + 6, (wrong, total)


def _prompt_time(cfg, data, dtype):
    """median time of five prompt passes (ms), after two"""
    gpu = make_gpu_cache(cfg, len(data.seqs), len(data.kv_heads))
    p = [to_dev(x, dtype) for x in (data.k_prompt, data.v_prompt, data.q_last)]
    times = []
    for _ in range(7):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        torch.cuda.synchronize()
        a.record()
        gpu.corm_compress_prompt(0, *p, data.prompt_lens)
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    return sorted(times[2:])[2], gpu


@pytest.mark.parametrize("d,G", [(128, 1), (64, 4)])
def test_fp32_prompt_without_eviction_leaves_nothing_open(d, G):
    """alpha = 0 puts every threshold at minus infinity: no verdict is near it, so the pass takes no longer than with
    thresholds that evict (it took ten times as long while every key went through the exact rows)."""
    t, cache = {}, None
    for alpha in (1.0, 0.0):
        cfg = _cfg("f32", d, G, 8, 8, (300, 300), 1, 8, 16, alpha=alpha)
        t[alpha], cache = _prompt_time(cfg, generate(cfg), "f32")
    assert (cache.corm_cache_live_lens(0) == 300).all()
    word = cache.corm_cache_export_state(0, 0, 0)["word"]
    assert (word[:293] == 0xff).all()
    assert t[0.0] < 3 * t[1.0], t


@pytest.mark.parametrize("C", [150000, 176000])
def test_verdict_launch_next_to_the_default_shared_memory_limit(C):
    """The verdict launch of long slabs takes 38-46 KB of dynamic shared memory next to its static lists: together they are
    beyond what a kernel gets unasked."""
    cfg = _cfg("bf16", 128, 1, 1, 1, (3000, 3000), 3, 8, 64)
    data = generate(cfg)
    gpu, orc = make_gpu_cache(cfg, 1, 1, max_tokens=C), make_oracle(cfg, 1, 1, max_tokens=C)
    gpu.corm_cache_set_tuning(512, 3)
    gpu.corm_compress_prompt(0, to_dev(data.k_prompt, "bf16"), to_dev(data.v_prompt, "bf16"), to_dev(data.q_last, "bf16"),
                             data.prompt_lens)
    orc.compress_prompt(0, data.k_prompt, data.v_prompt, data.q_last, data.prompt_lens)
    for s in range(3):
        gpu.corm_decode_step(0, to_dev(data.q[s], "bf16"), to_dev(data.k_new[s], "bf16"), to_dev(data.v_new[s], "bf16"))
        orc.decode_step(0, data.q[s], data.k_new[s], data.v_new[s])
    assert gpu.corm_cache_kernel_launches() == 2 + 6           # prompt pass; streaming and verdict launch per step
    assert_states_equal(gpu, orc, 0, 1, 1, "end")


# the lines between the cluster and the block-per-split kernel: few long units that keep their keys take the latter and the
# verdict launch (two launches a step), on either side of the length at which they do; short units of single heads it alone
FEW_UNITS = [
    # group, kv heads, batch, prompt, steps, w, alpha, paged, launches per step
    (1, 1, 1, 3600, 6, 8, 0.0, False, 2),
    (1, 2, 3, 3600, 6, 100, 1.0, True, 2),
    (1, 1, 1, 3000, 6, 8, 0.0, False, 1),
    (2, 1, 2, 6200, 4, 8, 0.0, True, 2),
    (4, 2, 1, 6300, 4, 40, 1.0, False, 2),
    (4, 2, 1, 6000, 4, 8, 0.0, True, 1),
    (4, 1, 1, 12500, 3, 8, 0.25, False, 2),
    (1, 2, 2, 240, 40, 8, 0.0, False, 1),               # 256 keys are reached on the way
    (1, 2, 2, 120, 40, 4, 1.0, True, 1),
]


@pytest.mark.parametrize("case", FEW_UNITS, ids=lambda c: "-".join(str(x) for x in c))
def test_few_units_on_either_side_of_the_kernels_lines(case):
    G, nkv, B, P, steps, w, alpha, paged, launches = case
    cfg = _cfg("bf16", 128, G, nkv, B, (P, P), steps, w, 32, alpha=alpha)
    data = generate(cfg)
    pages = -(-B * nkv * (cfg.max_tokens // 32 + 2) // 32) * 32 if paged else 0
    one, many = (make_gpu_cache(cfg, B, nkv, pool_pages=pages) for _ in range(2))
    orc = make_oracle(cfg, B, nkv)
    orc.set_near_band(1e-11)
    for g in (one, many):
        g.corm_compress_prompt(0, to_dev(data.k_prompt, "bf16"), to_dev(data.v_prompt, "bf16"), to_dev(data.q_last, "bf16"),
                               data.prompt_lens)
    orc.compress_prompt(0, data.k_prompt, data.v_prompt, data.q_last, data.prompt_lens)
    q, k, v = (to_dev(x, "bf16") for x in (data.q, data.k_new, data.v_new))
    outs = many.corm_decode_steps(0, 1, q[:, None], k[:, None], v[:, None])
    before = one.corm_cache_kernel_launches()
    for s in range(steps):
        ref = orc.decode_step(0, data.q[s], data.k_new[s], data.v_new[s])
        out = one.corm_decode_step(0, q[s], k[s], v[s])
        assert np.abs(out.float().cpu().numpy() - ref).max() <= OUT_TOL["bf16"], s
        assert np.abs(outs[s, 0].float().cpu().numpy() - ref).max() <= OUT_TOL["bf16"], s
    assert_states_equal(one, orc, 0, B, nkv, "per step")
    assert_states_equal(many, orc, 0, B, nkv, "multi-step")
    assert one.corm_cache_stats()["device_status"] == many.corm_cache_stats()["device_status"] == 0
    assert one.corm_cache_kernel_launches() - before == launches * steps


# prompts whose logits overflow plain sums of exponentials, whose elements leave the pieces' range, or whose bounds are too
# wide to be of use: row counts below, at and beyond one unit of four rows per warp, windows below and beyond a register
WIDE_PROMPTS = [
    # dtype, head_dim, group, prompt range, w, what
    ("bf16", 128, 1, (300, 340), 3, "large logits"),
    ("bf16", 128, 4, (1000, 1100), 8, "large logits"),
    ("bf16", 128, 8, (250, 420), 33, "one channel"),
    ("bf16", 64, 1, (600, 700), 256, "one channel"),
    ("bf16", 64, 2, (2040, 2060), 16, "out of range"),
    ("bf16", 128, 1, (1, 40), 5, "out of range"),
    # (from 96 rows on: on tcgen05; logits of 640 and 662 lie on either side of the largest that plain sums may hold)
    ("bf16", 128, 4, (1000, 1100), 40, "large logits"),
    ("bf16", 64, 1, (600, 700), 128, "large logits"),
    ("bf16", 128, 8, (300, 420), 16, "out of range"),
    ("bf16", 64, 4, (500, 560), 128, "out of range"),
    ("bf16", 128, 2, (700, 700), 100, "640"),
    ("bf16", 128, 1, (256, 330), 128, "662"),
    ("bf16", 64, 1, (900, 1000), 96, "640"),
    ("bf16", 64, 8, (400, 450), 32, "662"),
    ("bf16", 128, 4, (500, 600), 128, "one channel"),
    ("f32", 128, 2, (900, 1000), 40, "large logits"),
    ("f32", 64, 8, (255, 300), 64, "large logits"),
]


def _widen(data, what, dtype):
    rnd = (lambda a: torch.from_numpy(a).to(torch.bfloat16).float().numpy()) if dtype == "bf16" else (lambda a: a)
    kp, ql = rnd(data.k_prompt.copy()), rnd(data.q_last.copy())
    if what == "large logits":
        kp *= 128.0
    elif what == "out of range":
        kp *= 2.0 ** 58
    elif what in ("640", "662"):                       # the logit of every query with the sixth key, but for 3 of other channels
        kp[..., 0], ql[..., 0] = 0.0, 8.0
        kp[..., 5, 0] = float(what) * np.sqrt(kp.shape[-1]) / 8.0
        kp = rnd(kp)
    else:
        kp[..., 3] *= 4096.0
        ql[..., 3] /= 4096.0
    return kp, ql


@pytest.mark.parametrize("case", WIDE_PROMPTS, ids=lambda c: "-".join(str(x) for x in c))
def test_prompts_of_wide_range(case):
    dtype, d, G, prange, w, what = case
    cfg = _cfg(dtype, d, G, 2, 3, prange, 2, w, 16)
    data = generate(cfg)
    kp, ql = _widen(data, what, dtype)
    orc = make_oracle(cfg, 3, 2)
    orc.set_near_band(1e-11)
    orc.compress_prompt(0, kp, data.v_prompt, ql, data.prompt_lens)
    for pool in (0, -(-6 * (cfg.max_tokens // 32 + 2) // 32) * 32):
        gpu = make_gpu_cache(cfg, 3, 2, pool_pages=pool)
        gpu.corm_compress_prompt(0, to_dev(kp, dtype), to_dev(data.v_prompt, dtype), to_dev(ql, dtype), data.prompt_lens)
        assert_states_equal(gpu, orc, 0, 3, 2, f"pool {pool}")
        assert gpu.corm_cache_stats()["device_status"] == 0


@pytest.mark.parametrize("what", ["large logits", "one channel"])
def test_prompts_of_wide_range_take_fp64_time_not_a_pass_per_row(what):
    """256 rows of 32 units: both phases in fp64 take about five times the ordinary pass on tcgen05 (184 and 954 us); forming
    each row apart, with two passes over its keys, took more than ten times."""
    cfg = _cfg("bf16", 128, 1, 8, 4, (2000, 2000), 1, 256, 64)
    data = generate(cfg)
    plain, _ = _prompt_time(cfg, data, "bf16")
    data.k_prompt, data.q_last = _widen(data, what, "bf16")
    wide, _ = _prompt_time(cfg, data, "bf16")
    assert wide < 7 * plain, (plain, wide)


# a step lists its row moves on chip up to 992 evicted slots (what moves lies in the unit's last 32 words then), and in scratch
# beyond; holes spread out, all at the front, all in the last words; the most words a block of fp32 / 64 channels may own
EVICTED = [
    # dtype, head_dim, group, live keys, max_tokens, evicted, where, one block
    ("bf16", 128, 4, 3000, 3100, 1, "anywhere", False),
    ("bf16", 128, 1, 3000, 3100, 991, "anywhere", False),
    ("bf16", 128, 4, 3007, 3100, 992, "front", False),
    ("bf16", 64, 8, 3040, 3100, 992, "back", False),
    ("f32", 128, 2, 2999, 3100, 993, "anywhere", False),
    ("f32", 64, 1, 1500, 1600, 992, "anywhere", True),
    ("bf16", 128, 2, 1055, 1100, 992, "front", True),
    ("f32", 64, 1, 114000, 3583 * 32, 1500, "anywhere", True),
    ("f32", 64, 2, 114600, 3584 * 32, 700, "back", True),
]


@pytest.mark.parametrize("case", EVICTED, ids=lambda c: "-".join(str(x) for x in c))
def test_steps_around_the_lists_of_row_moves(case):
    dtype, d, G, n, C, evicted, where, one_block = case
    cfg = _cfg(dtype, d, G, 1, 1, (1, 1), 2, 4, 8, alpha=1e9)         # no key is important: what goes is what has no bit set
    rng = np.random.default_rng(evicted + d)
    to = (lambda x: to_dev(x, dtype).float().cpu().numpy())
    k, v = (to(rng.standard_normal((n, d), dtype=np.float32)) for _ in range(2))
    q = to(rng.standard_normal((2, 1, G, d), dtype=np.float32))
    kn, vn = (to(rng.standard_normal((2, 1, 1, d), dtype=np.float32)) for _ in range(2))
    word, pos = np.ones(n, np.uint32), np.arange(1, n + 1, dtype=np.int32)
    old = n - 16                                                      # (the last eight tokens stay in any case)
    word[{"anywhere": rng.choice(old, evicted, replace=False), "front": np.arange(evicted), "back": np.arange(old - evicted, old)}[where]] = 0
    gpu, orc = make_gpu_cache(cfg, 1, 1, max_tokens=C), make_oracle(cfg, 1, 1, max_tokens=C)
    gpu.corm_cache_set_tuning(1 << 18 if one_block else 0, 4)
    gpu.corm_cache_import_state(0, 0, 0, k, v, word, pos, n, 4)
    orc.import_unit(0, 0, 0, k, v, word, pos, n, 4)
    for s in range(2):
        out = gpu.corm_decode_step(0, to_dev(q[s], dtype), to_dev(kn[s], dtype), to_dev(vn[s], dtype))
        ref = orc.decode_step(0, q[s], kn[s], vn[s])
        assert np.abs(out.float().cpu().numpy() - ref).max() <= OUT_TOL[dtype]
        assert_states_equal(gpu, orc, 0, 1, 1, f"step {s}")
        if s == 0:
            assert gpu.corm_cache_stats()["evicted_keys"] == evicted
    assert gpu.corm_cache_stats()["device_status"] == 0


# windows and groups of 96 to 1024 rows on prompts from 256 keys on go through tcgen05, 128 rows and 64 keys at a time: the
# rows just enough, a full and a nearly empty last group, the most; tiles full, one key over, one short; ragged prompts
# shorter than the window and than a tile
MANY_ROWS = [
    # head_dim, group, kv heads, batch, prompt range, w
    (128, 1, 2, 3, (256, 256), 96),
    (128, 8, 1, 3, (257, 330), 12),
    (128, 8, 1, 2, (1000, 1100), 16),
    (128, 1, 2, 3, (319, 321), 128),
    (128, 1, 3, 4, (3, 700), 129),
    (128, 2, 2, 2, (640, 640), 100),
    (128, 4, 2, 2, (500, 2100), 256),
    (64, 1, 2, 3, (40, 600), 97),
    (64, 4, 1, 3, (255, 449), 32),
    (64, 8, 1, 2, (1023, 1025), 128),
    (64, 1, 8, 12, (256, 320), 192),                    # more blocks of 64 channels than SMs
]


@pytest.mark.parametrize("scale", [1.0, 1e6], ids=["", "all-open"])
@pytest.mark.parametrize("case", MANY_ROWS, ids=lambda c: "-".join(str(x) for x in c))
def test_prompts_of_many_rows(case, scale):
    """Verdicts are the oracle's; with the bounds a million times as wide every one is left open and formed again."""
    d, G, nkv, B, prange, w = case
    if scale > 1.0 and w * G * prange[1] > 150000:
        pytest.skip("a pass per row: long")
    cfg = _cfg("bf16", d, G, nkv, B, prange, 2, w, 16)
    data = generate(cfg)
    orc = make_oracle(cfg, B, nkv)
    orc.set_near_band(1e-11)
    orc.compress_prompt(0, data.k_prompt, data.v_prompt, data.q_last, data.prompt_lens)
    for pool in (0, -(-B * nkv * (cfg.max_tokens // 32 + 2) // 32) * 32):
        gpu = make_gpu_cache(cfg, B, nkv, pool_pages=pool)
        gpu.corm_cache_set_bound_scale(scale)
        gpu.corm_compress_prompt(0, to_dev(data.k_prompt, "bf16"), to_dev(data.v_prompt, "bf16"), to_dev(data.q_last, "bf16"),
                                 data.prompt_lens)
        assert_states_equal(gpu, orc, 0, B, nkv, f"pool {pool}")
        assert gpu.corm_cache_stats()["device_status"] == 0


# logits that the causal mask hides, where 2^(logit / ln 2) leaves the exponents of fp64 for infinity and NaN: 709.8..710.4 and
# -709.8..-709.1, every 1419.6 from there on
HIDDEN_LOGITS = (710.1, -709.45, 2129.7, -2129.0)


@pytest.mark.parametrize("target", HIDDEN_LOGITS)
@pytest.mark.parametrize("d,G,w", [(128, 1, 128), (64, 1, 128), (128, 4, 32), (64, 2, 64)])
def test_hidden_logits_of_any_size(d, G, w, target):
    """Every query but the last has the target logit with the prompt's last key, which none of them sees; the last query,
    which does, is orthogonal to it. All visible logits are ordinary. Elements are multiples of 1/16, so that the unit's
    bounds stay narrow next to so large a key."""
    cfg = _cfg("bf16", d, G, 2, 3, (256, 330), 2, w, 16)
    data = generate(cfg)
    kp, ql = (np.round(x * 16.0) / 16.0 for x in (data.k_prompt, data.q_last))
    grid = torch.arange(64, 160) / 16.0                                         # the query's channel; the key's follows from it
    key = (abs(target) * np.sqrt(d) / grid).to(torch.bfloat16).float()
    best = (grid * key / np.sqrt(d) - abs(target)).abs().argmin()
    assert abs(float(grid[best] * key[best]) / np.sqrt(d) - abs(target)) < 0.3
    kp[..., 0] = 0.0
    ql[:, :, :w - 1, 0], ql[:, :, w - 1, 0] = float(grid[best]), 0.0
    for b, P in enumerate(data.prompt_lens):
        kp[b, :, P - 1, 0] = float(key[best]) * np.sign(target)
    kp, ql = kp.astype(np.float32), ql.astype(np.float32)
    orc, gpu = make_oracle(cfg, 3, 2), make_gpu_cache(cfg, 3, 2)
    orc.set_near_band(1e-11)
    orc.compress_prompt(0, kp, data.v_prompt, ql, data.prompt_lens)
    gpu.corm_compress_prompt(0, to_dev(kp, "bf16"), to_dev(data.v_prompt, "bf16"), to_dev(ql, "bf16"), data.prompt_lens)
    assert_states_equal(gpu, orc, 0, 3, 2, "")
    assert gpu.corm_cache_stats()["device_status"] == 0


@pytest.mark.parametrize("dtype,d,G", [("bf16", 128, 1), ("bf16", 128, 4), ("bf16", 64, 8), ("f32", 64, 1), ("f32", 128, 2)])
def test_rows_that_move_in_the_step_that_wrote_them(dtype, d, G):
    """Every step evicts, so the row it appends, and the registers it has just updated in the unit's last words, move into
    holes that other blocks of the unit fill (blocks of two words each): newest bits, rows and positions travel."""
    nkv, B, steps = 8, 8, 72
    cfg = _cfg(dtype, d, G, nkv, B, (600, 700), steps, 4, 2)
    data = generate(cfg)
    orc = make_oracle(cfg, B, nkv)
    orc.set_near_band(1e-11)
    one, many = (make_gpu_cache(cfg, B, nkv) for _ in range(2))
    for g in (one, many):
        g.corm_cache_set_tuning(64, 4)
        g.corm_compress_prompt(0, to_dev(data.k_prompt, dtype), to_dev(data.v_prompt, dtype), to_dev(data.q_last, dtype),
                               data.prompt_lens)
    orc.compress_prompt(0, data.k_prompt, data.v_prompt, data.q_last, data.prompt_lens)
    q, k, v = (to_dev(x, dtype) for x in (data.q, data.k_new, data.v_new))
    for s0 in range(0, steps, 12):
        many.corm_decode_steps(0, 1, *(x[s0:s0 + 12, None] for x in (q, k, v)))
        for s in range(s0, s0 + 12):
            one.corm_decode_step(0, q[s], k[s], v[s])
            orc.decode_step(0, data.q[s], data.k_new[s], data.v_new[s])
        assert_states_equal(one, orc, 0, B, nkv, f"per step, {s0 + 12}")
        assert_states_equal(many, orc, 0, B, nkv, f"chained, {s0 + 12}")
    st = one.corm_cache_stats()
    assert st["device_status"] == 0 and st["moved_rows"] > steps * B * nkv // 4, st


# many units, or long ones: clusters of one, two and four blocks of 1024 to 2048 keys (16 to 32 tiles), several waves of them
LONG_BLOCKS = [
    # head_dim, group, kv heads, batch, prompt range, w, sampled sequences, sampled kv heads
    (128, 1, 29, 10, (1024, 1024), 192, [0, 9], [3, 28]),
    (128, 1, 32, 4, (2048, 4096), 256, [1, 3], [0, 17]),
    (128, 4, 8, 4, (8192, 8192), 128, [2], [5]),
    (64, 2, 16, 12, (1500, 3000), 128, [4, 11], [7]),
]


@pytest.mark.parametrize("case", LONG_BLOCKS, ids=lambda c: "-".join(str(x) for x in c))
def test_prompts_of_many_rows_in_long_blocks(case):
    """Sampled units against the oracle, as they come from a pass over all of them."""
    d, G, nkv, B, prange, w, seqs, heads = case
    cfg = _cfg("bf16", d, G, nkv, B, prange, 2, w, 64)
    data, sub = generate(cfg), generate(cfg, seqs=seqs, kv_heads=heads)
    orc = make_oracle(cfg, len(seqs), len(heads))
    orc.set_near_band(1e-11)
    orc.compress_prompt(0, sub.k_prompt, sub.v_prompt, sub.q_last, sub.prompt_lens)
    gpu = make_gpu_cache(cfg, B, nkv)
    gpu.corm_compress_prompt(0, to_dev(data.k_prompt, "bf16"), to_dev(data.v_prompt, "bf16"), to_dev(data.q_last, "bf16"),
                             data.prompt_lens)
    for i, b in enumerate(seqs):
        for j, h in enumerate(heads):
            g, o = sorted_state(gpu.corm_cache_export_state(0, b, h)), orc.export_unit(0, i, j)
            assert g["live_len"] == o["live_len"] and np.array_equal(g["pos"], o["pos"]), (b, h)
            assert np.array_equal(stamps_to_ages(g["word"], g["n_tokens"], w), o["age"]), (b, h)
            assert np.array_equal(g["k"].astype(np.float64), o["k"]) and np.array_equal(g["v"].astype(np.float64), o["v"]), (b, h)
    assert gpu.corm_cache_stats()["device_status"] == 0
