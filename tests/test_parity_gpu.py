"""GPU parity: the CUDA path, called through the C ABI, against the fp64 oracle in lock-step on the same
seeded inputs.  Kept sets bit-exact outside a 1e-4 relative band around the cut, outputs within 2e-2 (bf16) /
1e-4 (fp32) max-abs, cached rows bit-exact."""
import numpy as np
import pytest
import torch

import paper_2412_05693_b200 as bm
from paper_2412_05693_b200.workloads import CFG5_SWEEP, WORKLOADS, Inputs, Workload, schedule
from tests.lockstep import make_config, run_lockstep

pytestmark = pytest.mark.gpu


def all_units(wl, samples=None):
    samples = range(wl.b) if samples is None else samples
    return [(s, h) for s in samples for h in range(wl.Hkv)]


def tiny(name, **kw):
    base = dict(b=2, Hq=4, Hkv=2, d=64, dtype="f32", s=200, B=48, K=40, steps=6, seed=123, heavy_count=4)
    base.update(kw)
    return Workload(name, **base)


# ------------------------------------------------------------------ configs of the benchmark table
def test_cfg1_everything():
    wl = WORKLOADS["cfg1"]
    st = run_lockstep(wl, all_units(wl), check_rows_every=1)
    assert st["evictions"] >= (6 + 16) * 8
    assert st["max_out_err"] <= 1e-4


@pytest.mark.parametrize("compaction", ["stable", "fill"])
def test_cfg2_full_size_sampled_units(compaction):
    wl = WORKLOADS["cfg2"]
    st = run_lockstep(wl, [(0, 0), (7, 3), (15, 7)], check_rows_every=16, compaction=compaction)
    assert st["evictions"] > 0 and st["max_out_err"] <= 2e-2


@pytest.mark.parametrize("compaction", ["stable", "fill"])
def test_cfg3_full_size_sampled_units(compaction):
    wl = WORKLOADS["cfg3"].with_(steps=8)
    run_lockstep(wl, [(3, 1), (12, 6)], check_rows_every=8, compaction=compaction)


def test_cfg3_decode_only_compression_arm():
    # whole prompt cached (cap = s + 1), one compression to K after the prompt, then decode (Sec. 1)
    wl = WORKLOADS["cfg3"].with_(b=2, s=2048, steps=4)
    calls = [("prefill", p, wl.B, -1) for p in range(0, wl.s, wl.B)] + [("evict", 0, 0, wl.K)]
    calls += [("decode", wl.s + t, 1, wl.K) for t in range(wl.steps)]
    run_lockstep(wl, [(0, 0), (1, 5)], calls=calls, growth=wl.s + 1 - wl.K)


def test_cfg4_layers_are_independent():
    wl = WORKLOADS["cfg4"].with_(b=2, L=3, s=2048, steps=3)
    for layer in (0, 2):
        run_lockstep(wl, [(1, 2)], layer=layer, check_rows_every=4)


@pytest.mark.parametrize("B,K", CFG5_SWEEP)      # all six (block, kv_max) pairs of the configuration
def test_cfg5_large_candidate_sets(B, K):
    wl = WORKLOADS["cfg5"].with_(b=2, B=B, K=K, s=8192, steps=4)
    run_lockstep(wl, [(1, 17)], check_rows_every=4)
    run_lockstep(wl, [(0, 30)], check_rows_every=4, compaction="fill")


def test_cfg5_full_length_prompt():
    # the largest candidate set of the table (2048 cached + 2048 new) at the full prompt length
    wl = WORKLOADS["cfg5"].with_(b=2, B=2048, K=2048, steps=2)
    run_lockstep(wl, [(0, 5)], check_rows_every=4)


def test_cfg4_all_32_layers_share_one_handle():
    wl = WORKLOADS["cfg4"].with_(b=2, s=1024, steps=2)
    for layer in (0, 17, 31):
        run_lockstep(wl, [(0, 0), (1, 7)], layer=layer, check_rows_every=2)


def random_workloads(n, seed=2024):
    rng = np.random.default_rng(seed)
    out = []
    for i in range(n):
        g = int(rng.choice([1, 2, 4, 8]))
        hkv = int(rng.integers(1, 4))
        d = int(rng.choice([64, 128]))
        dtype = str(rng.choice(["bf16", "f32"]))
        B = int(rng.integers(1, 200))
        K = int(rng.integers(1, 300))
        s = int(rng.integers(1, 700))
        out.append(Workload(f"rand{i}_{dtype}_g{g}_d{d}_B{B}_K{K}_s{s}", b=int(rng.integers(1, 4)), Hq=g * hkv, Hkv=hkv,
                            d=d, dtype=dtype, s=s, B=B, K=K, steps=int(rng.integers(0, 12)), seed=1000 + i,
                            heavy_count=int(rng.integers(1, 9)), p_dec=int(rng.choice([1, 1, 3, 16]))))
    return out


@pytest.mark.parametrize("wl", random_workloads(10), ids=lambda w: w.name)
def test_random_shapes(wl):
    units = [(int(s), int(h)) for s in range(wl.b) for h in range(wl.Hkv)][:4]
    st = run_lockstep(wl, units, check_rows_every=2)
    assert st["calls"] == len(schedule(wl))


def random_cadence(wl, rng):
    """The workload's schedule with evictions switched off at random, explicit bm_evict / bm_keep_most_recent calls
    (targets from 0 up) thrown in, and an eviction forced wherever the cache would overflow."""
    growth = wl.B + 5
    calls, n = [], 0
    for kind, pos0, I, ev in schedule(wl):
        if n + I > wl.K + growth - 1 or rng.random() < 0.3:
            tgt = int(rng.integers(0, wl.K + 1))
            calls.append(("recent" if rng.random() < 0.3 else "evict", 0, 0, tgt))
            n = min(n, tgt)
        use_ev = ev if rng.random() < 0.5 else -1
        if use_ev < 0 and n + I > wl.K + growth:
            use_ev = wl.K
        calls.append((kind, pos0, I, use_ev))
        n = n + I if use_ev < 0 else min(n + I, use_ev)
    return calls, growth


@pytest.mark.parametrize("seed", range(8))
def test_random_cadences_rules_and_padding(seed):
    # seeded samples of the randomised sweep this suite was hardened with: any cadence of the four calls, any rule,
    # left padding, evictions down to an empty cache
    rng = np.random.default_rng(4200 + seed)
    g, hkv, d = int(rng.choice([1, 2, 4, 8])), int(rng.integers(1, 4)), int(rng.choice([64, 128]))
    wl = Workload(f"cad{seed}", b=int(rng.integers(1, 4)), Hq=g * hkv, Hkv=hkv, d=d, dtype=str(rng.choice(["bf16", "f32"])),
                  s=int(rng.integers(50, 900)), B=int(rng.integers(1, 300)), K=int(rng.integers(1, 400)),
                  steps=int(rng.integers(0, 16)), seed=4200 + seed, heavy_count=3, p_dec=int(rng.choice([1, 3])))
    rule = str(rng.choice(["average", "sum_recent", "current_query"]))
    if seed % 2 == 0:
        calls, growth = random_cadence(wl, rng)
        run_lockstep(wl, all_units(wl)[:3], calls=calls, growth=growth, rule=rule, check_rows_every=3)
    else:
        pads = [int(rng.integers(0, wl.s + 1)) for _ in range(wl.b)]
        run_lockstep(wl, all_units(wl)[:3], pads=pads, rule=rule, check_rows_every=3)


@pytest.mark.parametrize("seed", range(6))
def test_random_cadences_of_the_pooled_window_and_deviation_rules(seed):
    # the two rules with parameters of their own (Sec. 2: SnapKV, RoCo) under any cadence of the four calls
    rng = np.random.default_rng(5200 + seed)
    g, hkv, d = int(rng.choice([1, 2, 4])), int(rng.integers(1, 4)), int(rng.choice([64, 128]))
    wl = Workload(f"cad2_{seed}", b=int(rng.integers(1, 4)), Hq=g * hkv, Hkv=hkv, d=d, dtype=str(rng.choice(["bf16", "f32"])),
                  s=int(rng.integers(50, 700)), B=int(rng.integers(1, 250)), K=int(rng.integers(1, 300)),
                  steps=int(rng.integers(0, 12)), seed=5200 + seed, heavy_count=3, p_dec=int(rng.choice([1, 3])))
    calls, growth = random_cadence(wl, rng)
    if seed % 2 == 0:
        params = dict(window=int(rng.integers(1, 80)), pool=int(rng.choice([1, 3, 5, 9])))
        run_lockstep(wl, all_units(wl)[:3], calls=calls, growth=growth, rule="window_pooled", rule_params=params,
                     check_rows_every=3)
    else:
        params = dict(std_share=float(rng.choice([0.1, 0.333, 0.5, 0.9])))
        run_lockstep(wl, all_units(wl)[:3], calls=calls, growth=growth, rule="average_std", rule_params=params,
                     check_rows_every=3)


# ------------------------------------------------------------------ shapes, tails and degenerate cases
@pytest.mark.parametrize("wl", [
    tiny("ragged_f32"),                                               # I = 48, tail of 8, g = 2
    tiny("gqa8_bf16", Hq=16, Hkv=2, dtype="bf16", d=128, B=50, K=70, s=333),
    tiny("mha_bf16_d64", Hq=3 * 1, Hkv=3, dtype="bf16", d=64, B=64, K=64, s=256),
    tiny("block_gt_cache", B=96, K=16, s=300),                        # B > K: no Algorithm-1 counterpart
    tiny("short_prompt", s=30, B=16, K=64, steps=40),                 # s < K: eviction starts in decode
    tiny("one_token_blocks", s=40, B=1, K=8, steps=3),
    tiny("keep_one", s=64, B=16, K=1, steps=5),
    tiny("f32_d128_g4", Hq=8, Hkv=2, d=128, B=40, K=100, s=260),
    tiny("decode_growth", p_dec=8, s=96, B=32, K=32, steps=30),       # evict every 8th step
], ids=lambda w: w.name)
def test_small_shapes(wl):
    st = run_lockstep(wl, all_units(wl), check_rows_every=1)
    assert st["calls"] == len(schedule(wl))


@pytest.mark.parametrize("d,g,B,K,s", [
    (128, 2, 64, 320, 900),      # Algorithm 1's p = 64 on a short cache: 3 cached + 1 new key tile, 128 query rows
    (128, 1, 64, 300, 700),      # half a tile of query rows, ragged cached tile
    (128, 4, 32, 384, 600),      # grouped heads: 32 inputs x 4 heads
    (64, 1, 128, 256, 640),      # d = 64, a whole tile of inputs, causal part spans the tile
    (64, 8, 16, 100, 333),       # g = 8, ragged everything
    (128, 4, 20, 50, 171),       # rows past the block's end (80 of 128) must add nothing to the column sums
])
def test_short_blocks_take_forward_and_column_sums_in_one_kernel(d, g, B, K, s):
    # one exponential per pair, logits resident in tensor memory (the single-pass variant for short caches)
    wl = tiny(f"onepass_d{d}_g{g}_B{B}_K{K}", dtype="bf16", d=d, Hq=2 * g, Hkv=2, B=B, K=K, s=s, steps=3, b=3)
    st = run_lockstep(wl, all_units(wl), check_rows_every=2)
    assert st["onepass_calls"] == len([c for c in schedule(wl) if c[0] == "prefill"])
    # the same rule with evictions made by explicit calls before each block (Algorithm 1's order), limit K + B
    calls = []
    n = 0
    for kind, pos0, I, ev in schedule(wl):
        if n + I > K + B:                     # (a decode step is a block of one input)
            calls.append(("evict", 0, 0, K))
            n = K
        calls.append((kind, pos0, I, -1 if kind == "prefill" else ev))
        n = n + I if kind == "prefill" else min(n + 1, K)
    st = run_lockstep(wl, all_units(wl)[:3], calls=calls, growth=B, check_rows_every=2)
    assert st["onepass_calls"] > 0


def test_algorithm1_cadence_on_gpu():
    # Algorithm 1 as printed: limit kv_bar, remove p before each block / when full during decoding
    kv_bar, p, s, gen = 96, 32, 288, 70
    wl = tiny("alg1", s=s, B=p, K=kv_bar - p, steps=gen, p_dec=p, dtype="bf16", d=128, Hq=8, Hkv=2)
    calls = [("prefill", t, p, -1) for t in range(0, kv_bar, p)]
    t1 = kv_bar
    while t1 < s:
        calls.append(("evict", 0, 0, kv_bar - p))
        calls.append(("prefill", t1, min(p, s - t1), -1))
        t1 += p
    n = kv_bar
    for t in range(gen):
        if n == kv_bar:
            calls.append(("evict", 0, 0, kv_bar - p))
            n -= p
        calls.append(("decode", s + t, 1, -1))
        n += 1
    run_lockstep(wl, all_units(wl), calls=calls, growth=p, check_rows_every=3)


@pytest.mark.parametrize("dtype,d,kv_bar", [("bf16", 128, 2), ("bf16", 128, 65), ("f32", 64, 5)])
def test_extreme_decoding_arm_on_gpu(dtype, d, kv_bar):
    # Algorithm 3: full cache during the prompt, then only the most recent pair survives each cut
    s, gen = 200, 70
    wl = tiny("ed", s=s, B=48, K=s, steps=gen, dtype=dtype, d=d, Hq=8, Hkv=2)
    calls = [("prefill", t, min(48, s - t), -1) for t in range(0, s, 48)] + [("recent", 0, 0, 1)]
    n = 1
    for t in range(gen):
        calls.append(("decode", s + t, 1, -1))
        n += 1
        if n == kv_bar:
            calls.append(("recent", 0, 0, 1))
            n = 1
    st = run_lockstep(wl, all_units(wl), calls=calls, growth=kv_bar, check_rows_every=5)
    assert st["calls"] == len(calls)


@pytest.mark.parametrize("g", [1, 4])
def test_decode_with_more_caches_than_two_ctas_per_sm(g):
    # 320 caches: the decode kernel takes its 128-thread shape (four CTAs per SM); fewer caches take the 256-thread one
    wl = tiny("many_units", b=40, Hq=8 * g, Hkv=8, s=160, B=64, K=72, steps=10, dtype="bf16", d=128)
    units = [(0, 0), (13, 5), (39, 7), (27, 2)]
    st = run_lockstep(wl, units, check_rows_every=2)
    assert st["evictions"] >= len(units) * 10


@pytest.mark.parametrize("b,Hkv,g,d,K,kw", [
    (24, 8, 4, 128, 100, {}),                             # 192 caches: up to two per SM, the stream from 48 KB a cache on
    (24, 8, 2, 64, 33, dict(rule="sum_recent")),          # ... and below, on the other kernel
    (37, 8, 1, 128, 128, dict(compaction="fill")),        # 296: the most that two per SM make
    (40, 8, 2, 128, 200, {}),                             # 320: from 96 KB a cache on
    (40, 8, 2, 128, 190, {}),                             # ... and below, on the other kernel
    (64, 8, 1, 128, 300, dict(rule="current_query")),     # 512: from 150 KB on under this rule, not under the average
    (64, 8, 1, 128, 300, {}),
])
def test_decode_kernel_by_number_and_length_of_caches(b, Hkv, g, d, K, kw):
    wl = tiny("by_grid", b=b, Hq=g * Hkv, Hkv=Hkv, s=K + 21, B=K, K=K, steps=4, dtype="bf16", d=d)
    st = run_lockstep(wl, [(0, 0), (b // 2, 3), (b - 1, Hkv - 1)], check_rows_every=1, **kw)
    assert st["evictions"] >= 3 * 4


@pytest.mark.parametrize("b,Hkv,g,d,K,kw,path", [
    (18, 8, 1, 64, 60, {}, 4),                             # up to one per SM: the stream
    (25, 4, 4, 128, 400, dict(rule="current_query"), 3),   # ... but under this rule, 380 to 640 pairs, K in registers
    (25, 4, 1, 128, 639, dict(rule="current_query"), 3),
    (25, 4, 1, 128, 640, dict(rule="current_query"), 4),
    (25, 4, 8, 128, 500, dict(rule="current_query"), 4),
    (25, 4, 4, 128, 500, dict(rule="current_query", compaction="fill"), 4),
    (24, 8, 4, 128, 60, {}, 4),                            # 192 caches: from 24 KB on in groups of four,
    (24, 8, 2, 128, 200, {}, 2), (24, 8, 2, 128, 270, {}, 4),   # 128 KB in groups of two,
    (24, 8, 1, 128, 390, {}, 2), (24, 8, 1, 128, 420, {}, 4),   # 200 KB without
    (24, 8, 1, 128, 300, dict(L=4), 4),                    # ... where all layers do not stay in L2
    (24, 8, 1, 64, 200, dict(rule="sum_recent"), 2), (24, 8, 1, 64, 300, dict(rule="sum_recent"), 4),
    (48, 8, 1, 128, 270, {}, 2), (48, 8, 1, 128, 300, {}, 4),   # 384
    (60, 8, 4, 128, 360, {}, 2), (60, 8, 4, 128, 390, {}, 4),   # 480
    (80, 8, 4, 64, 390, {}, 2), (80, 8, 4, 64, 410, {}, 4),     # 640
    (150, 8, 4, 64, 230, dict(L=2), 2), (150, 8, 4, 64, 340, dict(L=2), 4),   # 1200, out of HBM
])
def test_decode_kernel_that_the_rule_chooses(b, Hkv, g, d, K, kw, path):
    kw = dict(kw)
    wl = tiny("chosen", b=b, Hq=g * Hkv, Hkv=Hkv, s=K, B=K, K=K, steps=3, dtype="bf16", d=d, L=kw.pop("L", 1))
    run_lockstep(wl, [(0, 0), (b // 2, Hkv // 2), (b - 1, Hkv - 1)], check_rows_every=1, **kw)
    assert bm.last_decode_path() == path


@pytest.mark.parametrize("K,kw", [(380, {}), (300, dict(rule="average_std")), (639, dict(rule="window_pooled")),
                                  (380, dict(p_dec=2))])
def test_decode_with_k_in_registers(K, kw):
    # a handle's caches that two SMs would share, in ranges of at most one per SM, and cuts by several values: the instance that
    # keeps K in registers, stages V by TMA and moves rows as TMA tiles, against the oracle
    kw = dict(kw)
    wl = tiny("k_in_registers", b=24, Hq=8, Hkv=8, s=K + 100, B=K, K=K, steps=5, dtype="bf16", d=128, p_dec=kw.pop("p_dec", 1))
    run_lockstep(wl, [(0, 0), (5, 3), (6, 0), (23, 7)], check_rows_every=1, micro=6, micro_dec=6, **kw)
    assert bm.last_decode_path() == 3
    if not kw:                                             # the whole batch, two CTAs per SM: the same bits
        assert_same_run(run_free(wl), run_free(wl, micro=6))


@pytest.mark.parametrize("K,g", [(511, 4), (512, 1), (600, 4), (639, 2), (640, 4)])
def test_decode_with_one_cache_per_sm(K, g):
    # six caches around whole numbers of tiles: the stream over clusters
    wl = tiny("one_per_sm", b=3, Hq=2 * g, Hkv=2, s=K + 140, B=128, K=K, steps=14, dtype="bf16", d=128)
    st = run_lockstep(wl, all_units(wl), check_rows_every=1)
    assert st["evictions"] >= 6 * 14


@pytest.mark.parametrize("b,Hkv,g,d,K,dtype,kw", [
    (8, 8, 4, 128, 200, "bf16", {}),                            # the stream, one cache per SM
    (25, 4, 4, 128, 400, "bf16", dict(rule="current_query")),   # K in registers, moves by TMA
    (40, 8, 2, 64, 60, "bf16", {}),                             # small CTAs
    (40, 8, 2, 64, 60, "bf16", dict(compaction="fill")),
    (40, 8, 2, 64, 60, "bf16", dict(rule="sum_recent")),
    (1, 4, 2, 128, 900, "bf16", {}),                            # the stream, a cache over a cluster
    (20, 8, 1, 128, 700, "bf16", {}),                           # ... several caches per CTA
    (3, 2, 2, 64, 100, "f32", {}),
])
def test_evicting_decode_step_with_a_nan_query(b, Hkv, g, d, K, dtype, kw):
    # every ranking value of a cache is NaN: still exactly one of its pairs leaves (the highest position), and no other
    # cache changes
    wl = tiny("nan_query", b=b, Hq=g * Hkv, Hkv=Hkv, s=K, B=K, K=K, steps=2, dtype=dtype, d=d)
    inp = Inputs(wl, "cuda")
    prompt, steps = inp.block(0, 0, K), [tuple(x[:, 0].contiguous() for x in inp.block(0, K + t, 1)) for t in range(2)]
    smp, kh = b // 2, Hkv - 1
    states = []
    for nan in (False, True):
        cache = bm.BatchMaxCache(make_config(wl, **kw))
        cache.prefill_block(*prompt, 0)
        before = cache.export(0, smp, kh, rows=True)
        for q, k, v in steps:
            q = q.clone()
            if nan:
                q[smp, kh * g, 3] = float("nan")
            cache.decode_step(q, k, v, evict_to=K)
        assert cache.status() == 0
        states.append({u: cache.export(0, *u, rows=True) for u in all_units(wl, {0, max(0, smp - 1), smp, min(b - 1, smp + 1), b - 1})})
        cache.close()
    for u, want in states[0].items():
        if u != (smp, kh):
            assert all(torch.equal(x, y) for x, y in zip(states[1][u], want))
    ids, sums, k_rows, v_rows = states[1][(smp, kh)]
    assert torch.isnan(sums).all()
    assert torch.equal(ids, before[0]) and torch.equal(k_rows, before[2]) and torch.equal(v_rows, before[3])


@pytest.mark.parametrize("b,Hkv,g,d,K,dtype", [
    (1, 3, 2, 64, 40, "f32"),            # shared by four CTAs, ten rows each
    (2, 4, 4, 128, 300, "f32"),          # by eight
    (1, 4, 2, 128, 1024, "bf16"),        # the stream over a cluster of eight
    (4, 8, 4, 128, 1024, "bf16"),        # ... of four
])
def test_evicting_decode_step_with_nan_keys_in_one_part_of_a_shared_cache(b, Hkv, g, d, K, dtype):
    # the first half of one cache's keys is NaN (whole shares of some of the CTAs): every weight of the cache is NaN, its
    # highest position leaves, and no other cache changes
    wl = tiny("nan_keys", b=b, Hq=g * Hkv, Hkv=Hkv, s=K, B=K, K=K, steps=1, dtype=dtype, d=d)
    inp = Inputs(wl, "cuda")
    prompt, (q, k, v) = inp.block(0, 0, K), (x[:, 0].contiguous() for x in inp.block(0, K, 1))
    smp, kh = b // 2, Hkv - 1
    states, outs = [], []
    for nan in (False, True):
        cache = bm.BatchMaxCache(make_config(wl))
        cache.prefill_block(*prompt, 0)
        ids, sums, k_rows, v_rows = cache.export(0, smp, kh, rows=True)
        if nan:
            k_rows = k_rows.clone()
            k_rows[:K // 2] = float("nan")
            cache.import_(ids, sums, k_rows, v_rows, 0, smp, kh)
        outs.append(cache.decode_step(q, k, v, evict_to=K).view(b, Hkv, g * d))
        assert cache.status() == 0
        states.append({u: cache.export(0, *u, rows=True) for u in all_units(wl)})
        cache.close()
    for u, want in states[0].items():
        if u != (smp, kh):
            assert all(torch.equal(x, y) for x, y in zip(states[1][u], want)) and torch.equal(outs[0][u], outs[1][u])
    assert torch.isnan(outs[1][smp, kh]).all()
    got = states[1][(smp, kh)]
    assert torch.isnan(got[1]).all()
    assert torch.equal(got[0], ids) and torch.equal(got[2].nan_to_num(), k_rows.nan_to_num()) and torch.equal(got[3], v_rows)


# the forward kernel with two row tiles per CTA: the handle's batch makes 1024 pairs of tiles
PAIR_GRIDS = [(64, 16, 1, 64, 200, 150),     # the second tile ragged, and it sees one key tile more than the first
              (64, 16, 1, 128, 300, 129),    # three tiles: the last CTA's second tile has no rows
              (64, 8, 4, 128, 130, 140),     # five tiles of which the last holds 8 rows
              (32, 8, 8, 64, 200, 260)]


@pytest.mark.parametrize("b,Hkv,g,d,B,K", PAIR_GRIDS)
def test_forward_on_pairs_of_row_tiles(b, Hkv, g, d, B, K):
    wl = tiny("pair", b=b, Hq=g * Hkv, Hkv=Hkv, s=2 * B + 5, B=B, K=K, steps=1, dtype="bf16", d=d)
    run_lockstep(wl, [(0, 0), (b - 1, Hkv - 1)], check_rows_every=2)


@pytest.mark.parametrize("b,Hkv,g,d,B,K", PAIR_GRIDS[1:3])
def test_forward_on_pairs_of_row_tiles_when_the_maximum_grows(b, Hkv, g, d, B, K):
    # later keys with ever larger logits: the accumulator is rescaled at every key tile
    import torch
    from paper_2412_05693_b200 import BatchMaxCache, Config
    gen = torch.Generator(device="cuda").manual_seed(3)
    f = lambda *s: torch.randn(*s, device="cuda", generator=gen)
    q, k, v = (x.bfloat16() for x in (f(b, B, g * Hkv, d), f(b, B, Hkv, d), f(b, B, Hkv, d)))
    grow = torch.linspace(1, 12, B, device="cuda")
    k = (k * grow[None, :, None, None]).bfloat16()
    cache = BatchMaxCache(Config(batch=b, n_q_heads=g * Hkv, n_kv_heads=Hkv, head_dim=d, kv_max=B, block_max=B))
    out = cache.prefill_block(q, k, v, 0)
    assert cache.status() == 0
    for s, h in ((0, 0), (b - 1, Hkv - 1)):
        logits = torch.einsum("igd,jd->gij", q[s, :, h * g:(h + 1) * g].float(), k[s, :, h].float()) / d ** 0.5
        logits.masked_fill_(torch.ones(B, B, device="cuda", dtype=torch.bool).triu(1), -float("inf"))
        want = torch.einsum("gij,jd->igd", logits.softmax(-1), v[s, :, h].float())
        assert (out[s, :, h * g:(h + 1) * g].float() - want).abs().max() < 2e-2


@pytest.mark.parametrize("b,Hkv,g,d,B,K", PAIR_GRIDS)
def test_forward_on_pairs_of_row_tiles_is_bitwise_independent_of_sample_ranges(b, Hkv, g, d, B, K):
    # a single sample's tiles have an SM each: one tile per CTA.  With one padded sample: no range takes another kernel
    # (short blocks do, so there is none)
    for tail, pads in ((5, None), (0, [0] * (b - 1) + [B + 7])):
        wl = tiny("pair_ranges", b=b, Hq=g * Hkv, Hkv=Hkv, s=2 * B + tail, B=B, K=K, steps=0, dtype="bf16", d=d)
        base = run_free(wl, pads=pads)
        assert_same_run(base, run_free(wl, micro=b // 2, pads=pads))
        assert_same_run(base, run_free(wl, micro=1, pads=pads))


# row tiles of any caches in a work item: one each where a call's have an SM each, two where caches with an odd number of them
# would leave many items with a single one
ANY_GRIDS = [(25, 7, 2, 128, 60, 600, {}),                     # a ragged tile per cache, 175 of them: the last item has one
             (16, 5, 1, 64, 300, 200, dict(pads=True)),        # three tiles of 80 caches, padding
             (10, 8, 4, 128, 77, 200, {}),                     # three tiles per cache, 240: an item's tiles see different numbers of keys
             (16, 11, 8, 64, 41, 0, dict(compaction="fill")),  # 528 of them, two rounds; no cached pairs at first
             (60, 8, 2, 128, 64, 260, dict(rule="current_query"))]   # 480 caches with a tile each


@pytest.mark.parametrize("b,Hkv,g,d,B,K,kw", ANY_GRIDS)
def test_forward_on_row_tiles_of_any_caches(b, Hkv, g, d, B, K, kw):
    # whole calls against the oracle; a row's arithmetic does not depend on the tile beside it, so that single samples' calls, whose
    # items have one tile each, give the same bits
    kw = dict(kw)
    pads = [(37 * s) % (B + K) for s in range(b)] if kw.pop("pads", False) else None
    wl = tiny("any", b=b, Hq=g * Hkv, Hkv=Hkv, s=K + 2 * B if K else 3 * B, B=B, K=max(K, B), steps=0, dtype="bf16", d=d)
    run_lockstep(wl, [(0, 0), (b // 2, Hkv // 2), (b - 1, Hkv - 1)], check_rows_every=2, pads=pads, **kw)
    base = run_free(wl, pads=pads)
    assert_same_run(base, run_free(wl, micro=1, pads=pads))


# few row tiles: the two softmax groups of a CTA take the key tiles of one row tile in turn
SPLIT_GRIDS = [(1, 1, 1, 128, 131, 0),    # two row tiles: one key tile (the second group has none), then two
               (2, 2, 4, 64, 200, 129),   # cached tiles end in a single key; up to four key tiles
               (1, 4, 8, 128, 70, 640),   # a row tile of 16 inputs, the last one ragged
               (2, 1, 2, 64, 385, 257)]


@pytest.mark.parametrize("b,Hkv,g,d,B,K", SPLIT_GRIDS)
def test_forward_with_key_tiles_taken_in_turn(b, Hkv, g, d, B, K):
    # plain keys, then one NaN, inf or -inf in a key of every cache; the logits of the first query are all -inf in the last
    gen = torch.Generator(device="cuda").manual_seed(11)
    f = lambda *s: torch.randn(*s, device="cuda", generator=gen).bfloat16()
    n = K + B
    q, k, v = f(b, n, g * Hkv, d), f(b, n, Hkv, d), f(b, n, Hkv, d)
    q[..., 3] = q[..., 3].abs() + 0.1                      # (an infinite element of a key gives logits of one sign)
    hidden = torch.ones(n, n, device="cuda", dtype=torch.bool).triu(1)
    for value in (None, float("nan"), float("inf"), -float("inf")):
        if value is not None:
            for u in range(b * Hkv):
                k[u // Hkv, n // 2, u % Hkv, 3] = value
        if value == -float("inf"):
            k[:, 0, :, 3] = value
        cache = bm.BatchMaxCache(bm.Config(batch=b, n_q_heads=g * Hkv, n_kv_heads=Hkv, head_dim=d, kv_max=n, block_max=max(B, K)))
        parts = [cache.prefill_block(*(x[:, :K].contiguous() for x in (q, k, v)), 0)] if K else []
        parts.append(cache.prefill_block(*(x[:, K:].contiguous() for x in (q, k, v)), K))
        assert cache.status() == 0
        out = torch.cat(parts, 1).float()
        cache.close()
        for s in range(b):
            logits = torch.einsum("ihgd,jhd->hgij", q[s].float().view(n, Hkv, g, d), k[s].float()) / d ** 0.5
            want = torch.einsum("hgij,jhd->ihgd", logits.masked_fill_(hidden, -float("inf")).softmax(-1), v[s].float())
            want = want.reshape(n, g * Hkv, d)
            assert torch.equal(torch.isnan(out[s]), torch.isnan(want))
            assert (out[s] - want).nan_to_num_(0.0).abs().max() < 2e-2


@pytest.mark.parametrize("d,pads", [(64, None), (128, None), (128, [0, 130, 37, 0])])
def test_forward_with_key_tiles_taken_in_turn_on_few_free_sms(d, pads):
    # another stream's kernels hold 140 SMs, so that the CTAs that start on the others take several work items each: exchange
    # columns, output stage and barriers are used again, and nothing changes
    gen = torch.Generator(device="cuda").manual_seed(13)
    f = lambda *s: torch.randn(*s, device="cuda", generator=gen).bfloat16()
    long = [f(35, 4096, 4, 128) for _ in range(3)]
    holder = bm.BatchMaxCache(bm.Config(batch=35, n_q_heads=4, n_kv_heads=4, head_dim=128, kv_max=8192, block_max=4096))
    holder.prefill_block(*long, 0)
    long = [x[:, :128].contiguous() for x in long]
    blocks = [[f(4, I, h, d) for h in (32, 16, 16)] for I in (300, 128)]

    def run():
        cache = bm.BatchMaxCache(bm.Config(batch=4, n_q_heads=32, n_kv_heads=16, head_dim=d, kv_max=500, block_max=300))
        if pads is not None:
            cache.set_left_pad(pads)
        cache.prefill_block(*blocks[0], 0)
        torch.cuda.synchronize()
        held = torch.empty_like(long[0])
        for t in range(6 if others else 0):
            with torch.cuda.stream(side):
                holder.prefill_block(*long, 4096 + at[0], out=held, evict_to=4096)
                at[0] += 128
        out = cache.prefill_block(*blocks[1], 300)         # 128 row tiles
        torch.cuda.synchronize()
        assert cache.status() == 0 and holder.status() == 0
        sums = [cache.export(0, s, h)[1] for s in range(4) for h in range(16)]
        cache.close()
        return out, torch.cat(sums)

    side, at = torch.cuda.Stream(), [0]
    torch.cuda.synchronize()
    others = False
    want = run()
    others = True
    for _ in range(4):
        got = run()
        assert all(torch.equal(x, y) for x, y in zip(got, want))
    holder.close()


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("nan_at,large_at", [(5, 3 * 128 + 7), (128 + 9, 4 * 128 + 1), (2 * 128, 128)])
def test_forward_with_key_tiles_taken_in_turn_keeps_a_nan_far_below_the_maximum(d, nan_at, large_at):
    # the key tiles with the NaN go to one group, a logit 250 (log2) above everything else to the other: the first group's weight
    # is too small for fp32, and every row is NaN all the same, as softmax has it
    gen = torch.Generator(device="cuda").manual_seed(12)
    f = lambda *s: torch.randn(*s, device="cuda", generator=gen).bfloat16()
    K, B = 640, 64
    q, k, v = f(1, K + B, 1, d), f(1, K + B, 1, d), f(1, K + B, 1, d)
    q[..., 3] = q[..., 3].abs() + 1.0
    cache = bm.BatchMaxCache(bm.Config(batch=1, n_q_heads=1, n_kv_heads=1, head_dim=d, kv_max=K + B, block_max=K))
    k[0, large_at, 0, 3] = 2000.0
    k[0, nan_at, 0, 3] = float("nan")
    cache.prefill_block(*(x[:, :K].contiguous() for x in (q, k, v)), 0)
    out = cache.prefill_block(*(x[:, K:].contiguous() for x in (q, k, v)), K)
    assert torch.isnan(out).all() and cache.status() == 0
    cache.close()


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("b,Hkv,g,d,B,K", PAIR_GRIDS[1:3])
def test_forward_on_pairs_of_row_tiles_with_nan_and_inf_keys(b, Hkv, g, d, B, K, value):
    # one such element in one key of every cache, at every position of a block: a row is NaN where fp32 attention says
    # so, and as without that key where its weight is 0 or the row does not see it
    gen = torch.Generator(device="cuda").manual_seed(5)
    f = lambda *s: torch.randn(*s, device="cuda", generator=gen).bfloat16()
    q, k, v = f(b, B, g * Hkv, d), f(b, B, Hkv, d), f(b, B, Hkv, d)
    for u in range(b * Hkv):
        k[u // Hkv, u % B, u % Hkv, 3] = value
    cache = bm.BatchMaxCache(bm.Config(batch=b, n_q_heads=g * Hkv, n_kv_heads=Hkv, head_dim=d, kv_max=B, block_max=B))
    out = cache.prefill_block(q, k, v, 0).float()
    assert cache.status() == 0
    hidden = torch.ones(B, B, device="cuda", dtype=torch.bool).triu(1)
    for s in range(b):
        logits = torch.einsum("ihgd,jhd->hgij", q[s].float().view(B, Hkv, g, d), k[s].float()) / d ** 0.5
        want = torch.einsum("hgij,jhd->ihgd", logits.masked_fill_(hidden, -float("inf")).softmax(-1), v[s].float())
        assert torch.equal(torch.isnan(out[s]), torch.isnan(want).reshape(B, g * Hkv, d))
        assert (out[s] - want.reshape(B, g * Hkv, d)).nan_to_num_(0.0).abs().max() < 2e-2


@pytest.mark.parametrize("b,Hkv,g,d,B,K,kw", [
    (1, 2, 1, 128, 64, 700, {}),                            # one query tile, a key tile per CTA
    (40, 8, 1, 64, 33, 530, {}),                            # ... all key tiles of a cache in one CTA, a chunk past the last row
    (10, 8, 4, 128, 32, 640, {}),                           # ... exactly 128 rows, several key tiles per CTA
    (2, 2, 8, 128, 16, 777, dict(rule="average_std")),
    (2, 2, 2, 64, 50, 601, dict(rule="window_pooled", rule_params=dict(window=16, pool=5))),
    (2, 2, 1, 128, 150, 600, {}),                           # two query tiles, the last with a single chunk of rows
])
def test_score_pass_of_short_blocks_against_long_caches(b, Hkv, g, d, B, K, kw):
    wl = tiny("short_score", b=b, Hq=g * Hkv, Hkv=Hkv, s=K + 3 * B, B=B, K=K, steps=1, dtype="bf16", d=d)
    calls = [("prefill", p, min(300, K - p), -1) for p in range(0, K, 300)]
    calls += [("prefill", K + i * B, B, K) for i in range(3)]
    run_lockstep(wl.with_(B=300), [(0, 0), (b - 1, Hkv - 1)], calls=calls, check_rows_every=2, **kw)


@pytest.mark.parametrize("b,Hkv,d,dtype,K,kw", [
    (1, 2, 128, "bf16", 1100, {}),                          # clusters of 8, a ragged last chunk
    (2, 8, 64, "bf16", 900, {}),                            # too little to move for a cluster
    (3, 8, 64, "f32", 700, {}),                             # clusters of 4
    (1, 4, 128, "f32", 513, dict(compaction="fill")),       # unordered rows
    (1, 4, 128, "bf16", 600, dict(rule="average_std")),     # the second accumulator is read after the first select
    (1, 4, 128, "bf16", 1100, dict(rule="average_std")),    # ... in a cluster of 8
    (1, 8, 128, "bf16", 1030, dict(rule="window_pooled", rule_params=dict(window=16, pool=5))),
    (1, 8, 128, "bf16", 1024, {}),                          # exactly enough rows for clusters of 8
    (2, 8, 128, "bf16", 512, {}),                           # ... of 4
    (5, 8, 128, "bf16", 512, {}),                           # ... of 2
    (8, 8, 64, "f32", 600, {}),                             # clusters of 2
    (1, 4, 128, "bf16", 600, dict(rule="window_pooled", rule_params=dict(window=16, pool=5))),
    (20, 8, 128, "bf16", 130, {}),                          # more caches than SMs: small chunks
])
def test_evictions_by_grid_size(b, Hkv, d, dtype, K, kw):
    wl = tiny("evict_grid", b=b, Hq=Hkv, Hkv=Hkv, s=K + 150, B=120, K=K, steps=2, dtype=dtype, d=d)
    run_lockstep(wl, [(0, 0), (b - 1, Hkv - 1)], check_rows_every=2, **kw)


def test_largest_cut_of_a_call():
    # the largest candidate set: the cut's work arrays fit a CTA's shared memory up to 10460 pairs kept
    f = lambda h: torch.zeros(1, 12288, h, 64, device="cuda", dtype=torch.bfloat16)
    for keep in (10461, 10460):
        cache = bm.BatchMaxCache(bm.Config(batch=1, n_q_heads=1, n_kv_heads=1, head_dim=64, kv_max=keep, block_max=12288))
        if keep > 10460:
            with pytest.raises(bm.BMError) as err:
                cache.prefill_block(f(1), f(1), f(1), 0, evict_to=keep)
            assert err.value.code == 3 and cache.length()[0] == 0
        else:
            cache.prefill_block(f(1), f(1), f(1), 0, evict_to=keep)
            assert cache.status() == 0 and cache.length()[0] == keep
        cache.close()


@pytest.mark.parametrize("b,Hkv,g,d,K", [(1, 4, 2, 128, 1024), (2, 8, 1, 64, 900), (20, 8, 4, 128, 700), (40, 8, 2, 64, 60)])
def test_decode_step_with_logits_that_are_all_minus_infinity(b, Hkv, g, d, K):
    # softmax of such a row is NaN whatever the kernel and the cluster, and stays in its own cache
    f = lambda *s: torch.rand(*s, device="cuda").bfloat16() + 0.5
    k = f(b, K, Hkv, d)
    k[b // 2, :, 1] = -float("inf")
    cache = bm.BatchMaxCache(bm.Config(batch=b, n_q_heads=g * Hkv, n_kv_heads=Hkv, head_dim=d, kv_max=K, block_max=K))
    cache.prefill_block(f(b, K, g * Hkv, d), k, f(b, K, Hkv, d), 0)
    out = cache.decode_step(f(b, g * Hkv, d), k[:, 0].contiguous(), f(b, Hkv, d)).view(b, Hkv, g, d)
    assert cache.status() == 0
    nan = torch.zeros(b, Hkv, dtype=torch.bool, device="cuda")
    nan[b // 2, 1] = True
    assert torch.equal(torch.isnan(out).all(-1).all(-1), nan) and torch.equal(torch.isnan(out).any(-1).any(-1), nan)


@pytest.mark.parametrize("b,Hkv,d,K", [(2, 4, 128, 1024), (4, 8, 64, 1500), (24, 8, 128, 700)])
def test_decode_stream_is_bitwise_independent_of_sample_ranges(b, Hkv, d, K):
    import torch
    from paper_2412_05693_b200 import BatchMaxCache, Config
    gen = torch.Generator(device="cuda").manual_seed(7)
    f = lambda *s: torch.randn(*s, device="cuda", generator=gen).bfloat16()
    prompt = (f(b, K, 2 * Hkv, d), f(b, K, Hkv, d), f(b, K, Hkv, d))
    steps = [(f(b, 2 * Hkv, d), f(b, Hkv, d), f(b, Hkv, d)) for _ in range(3)]
    runs = []
    for parts in (1, 2, b):
        cache = BatchMaxCache(Config(batch=b, n_q_heads=2 * Hkv, n_kv_heads=Hkv, head_dim=d, kv_max=K, block_max=K))
        cache.prefill_block(*prompt, 0)
        ns, outs = b // parts, []
        for q, k, v in steps:
            outs.append(torch.cat([cache.decode_step(q[s:s + ns], k[s:s + ns], v[s:s + ns], evict_to=K, sample0=s)
                                   for s in range(0, b, ns)]))
        assert cache.status() == 0
        runs.append((outs, cache.export(0, b - 1, Hkv - 1, rows=True)))
        cache.close()
    for outs, state in runs[1:]:
        assert all(torch.equal(x, y) for x, y in zip(outs, runs[0][0]))
        assert all(torch.equal(x, y) for x, y in zip(state, runs[0][1]))


@pytest.mark.parametrize("b,Hkv,g,d,B,K", [
    (1, 1, 1, 64, 7, 30),       # one tile of 8 rows, keys past the end
    (2, 4, 2, 128, 65, 64),     # tiles of 8 rows; key tiles of 16 in the score pass
    (3, 6, 4, 64, 77, 50),      # tiles of 16 rows; a cluster shares the query tiles of a key tile
    (2, 3, 8, 128, 130, 70),    # ... a cluster of 8 with a ragged last query tile
    (5, 8, 4, 128, 100, 129),   # tiles of 64 rows
])
def test_f32_kernels_by_grid_size(b, Hkv, g, d, B, K):
    wl = tiny("f32_grid", b=b, Hq=g * Hkv, Hkv=Hkv, s=2 * B + 9, B=B, K=K, steps=2, dtype="f32", d=d)
    run_lockstep(wl, [(0, 0), (b - 1, Hkv - 1)], check_rows_every=1)


@pytest.mark.parametrize("b,Hkv,g,d,K,kw", [
    (2, 4, 1, 64, 31, {}),                                # 32 pairs with the step's own: 8 rows for each CTA of four
    (1, 3, 8, 128, 203, {}),                              # shared by eight, uneven pieces
    (3, 2, 2, 64, 191, dict(compaction="fill")),          # a cut that follows as a launch of its own
    (5, 4, 4, 128, 150, dict(rule="sum_recent")),
    (5, 4, 4, 64, 97, dict(rule="current_query")),
    (2, 4, 4, 128, 130, dict(rule="average_std")),
    (4, 4, 4, 128, 790, {}),                              # the most that four hold: 198 rows each
    (4, 4, 4, 128, 791, {}),                              # 199: shared by eight
    (20, 4, 1, 64, 40, {}),                               # 80 caches: not shared
])
def test_f32_decode_with_caches_shared_by_clusters(b, Hkv, g, d, K, kw):
    wl = tiny("f32_shared", b=b, Hq=g * Hkv, Hkv=Hkv, s=K + 40, B=K, K=K, steps=6, dtype="f32", d=d)
    run_lockstep(wl, [(0, 0), (b - 1, Hkv - 1)], check_rows_every=1, **kw)
    if not kw:
        assert_same_run(run_free(wl), run_free(wl, micro=1))


@pytest.mark.parametrize("b,Hkv,g,d,K,path", [
    (4, 4, 4, 128, 1583, 1),                              # 198 rows for each of eight
    (4, 4, 4, 128, 1584, 0),                              # more than eight hold: a CTA per cache
    (2, 4, 1, 64, 30, 0), (2, 4, 1, 64, 31, 1),           # from 32 pairs on
    (18, 4, 2, 64, 50, 1), (19, 4, 2, 64, 50, 0),         # up to half as many caches as SMs
])
def test_f32_decode_kernel_by_number_and_length_of_caches(b, Hkv, g, d, K, path):
    wl = tiny("f32_by_grid", b=b, Hq=g * Hkv, Hkv=Hkv, s=K, B=min(K, 800), K=K, steps=2, dtype="f32", d=d)
    run_lockstep(wl, [(0, 0), (b - 1, Hkv - 1)], check_rows_every=1)
    assert bm.last_decode_path() == path


@pytest.mark.parametrize("b,Hkv,g,d,K,bound", [
    (1, 8, 1, 128, 900, 2.5e-7),      # shared by eight
    (4, 4, 4, 128, 512, 2.15e-7),     # by eight, 64 rows each
    (1, 8, 1, 128, 100, 2.0e-7),      # by four
    (1, 1, 8, 64, 300, 1.8e-7),
])
def test_f32_decode_weights_of_shared_caches_against_64_bits(b, Hkv, g, d, K, bound):
    # 2-norm of a step's weights (the rule keeps the last step's alone) from 64 bits, relative.  The bounds are what a CTA with a
    # cache of its own leaves on these inputs (2.26e-7, 1.94e-7, 1.81e-7, 1.62e-7) and a tenth; clusters that summed 32
    # products in one chain and multiplied two approximate exponentials were at 3.07e-7, 2.47e-7, 2.34e-7 and 1.73e-7
    num = den = 0.0
    for seed in range(6):
        gen = torch.Generator("cuda").manual_seed(seed)
        draw = lambda *n: [torch.randn(b, *n, h, d, device="cuda", generator=gen) * s
                           for h, s in ((g * Hkv, 1.5), (Hkv, 1.0), (Hkv, 1.0))]
        cache = bm.BatchMaxCache(bm.Config(batch=b, n_q_heads=g * Hkv, n_kv_heads=Hkv, head_dim=d, kv_max=K + 4, block_max=K,
                                           dtype="f32", rule="current_query"))
        prompt = draw(K)
        cache.prefill_block(*prompt, 0)
        keys = prompt[1].double()
        for _ in range(4):
            q, k, v = draw()
            cache.decode_step(q, k, v)
            keys = torch.cat([keys, k[:, None].double()], 1)
            logits = torch.einsum("bhgd,bnhd->bhgn", q.double().view(b, Hkv, g, d), keys) / d ** 0.5
            want = torch.softmax(logits, -1).sum(2)
            for smp, kh in [(x, h) for x in range(b) for h in range(Hkv)]:
                got = cache.export(0, smp, kh)[1].double().to("cuda")
                num += (got - want[smp, kh]).square().sum().item()
                den += want[smp, kh].square().sum().item()
        cache.close()
    assert (num / den) ** 0.5 < bound


@pytest.mark.parametrize("b,Hkv,g,d,B,K", [
    (4, 4, 4, 128, 256, 1280),   # the whole batch would share a key tile among 2 CTAs, a single sample among 8
    (4, 4, 4, 128, 256, 512),    # ... 4 and 8
    (6, 2, 2, 64, 130, 300),     # key tiles of 16 for a single sample
])
def test_f32_blocks_are_bitwise_independent_of_sample_ranges(b, Hkv, g, d, B, K):
    wl = tiny("f32_ranges", b=b, Hq=g * Hkv, Hkv=Hkv, s=K + 2 * B, B=B, K=K, steps=0, dtype="f32", d=d)
    base = run_free(wl)
    assert_same_run(base, run_free(wl, micro=b // 2))
    assert_same_run(base, run_free(wl, micro=1))


@pytest.mark.parametrize("b,Hkv,g,d,K,kw", [
    (1, 3, 1, 64, 40, {}),                                  # less than one tile of rows
    (1, 2, 4, 128, 1023, {}),                               # a cluster of 8 CTAs per cache; the step's row ends a tile
    (1, 8, 2, 128, 1024, {}),                               # ... or starts one
    (4, 8, 8, 64, 1100, {}),                                # 32 caches: clusters of 4
    (6, 8, 1, 128, 1300, {}),                               # 48 caches: clusters of 2, K tiles behind the V tiles in the ring
    (20, 8, 1, 128, 641, {}),                               # more caches than SMs: a second cache per CTA
    (40, 8, 4, 64, 1090, {}),                               # three caches per CTA
    (20, 8, 4, 128, 700, dict(p_dec=3)),                    # the cut follows as a launch of its own
    (1, 4, 2, 64, 1100, dict(rule="average_std")),
    (9, 8, 2, 128, 660, {}),                                # 72 caches in L2: the other kernel, beyond its rows in registers
    (9, 8, 2, 128, 660, dict(compaction="fill")),
    (20, 8, 4, 128, 700, dict(compaction="fill")),
    (1, 4, 2, 128, 1024, dict(compaction="fill")),
    (1, 4, 2, 128, 900, dict(rule="sum_recent")),
    (20, 8, 1, 128, 660, dict(rule="current_query")),
    (3, 4, 2, 128, 700, dict(pads=[1500, 0, 700])),         # padding still cached when decoding starts
])
def test_decode_as_a_stream(b, Hkv, g, d, K, kw):
    kw = dict(kw)
    wl = tiny("stream", b=b, Hq=g * Hkv, Hkv=Hkv, s=K + 90, B=512, K=K, steps=7, dtype="bf16", d=d, p_dec=kw.pop("p_dec", 1))
    units = [(0, 0), (b // 2, Hkv - 1), (b - 1, Hkv // 2)] if b * Hkv > 16 else all_units(wl)
    if "pads" in kw:
        wl = wl.with_(s=1600)
    run_lockstep(wl, units, check_rows_every=3, **kw)


# ------------------------------------------------------------------ unordered caches (BM_COMPACT_FILL)
@pytest.mark.parametrize("name,kw", [
    ("f32_simt", dict(dtype="f32", d=64, Hq=4, Hkv=4, s=300, B=48, K=80, steps=12)),
    ("bf16_one_per_sm", dict(dtype="bf16", d=128, Hq=8, Hkv=2, s=700, B=128, K=512, steps=14)),
    ("bf16_ragged_tail", dict(dtype="bf16", d=128, Hq=4, Hkv=4, s=333, B=100, K=77, steps=9)),
    ("bf16_block_larger_than_cache", dict(dtype="bf16", d=64, Hq=2, Hkv=2, s=400, B=160, K=48, steps=6)),
    ("bf16_decode_cuts_of_8", dict(dtype="bf16", d=128, Hq=8, Hkv=2, s=256, B=64, K=64, steps=20, p_dec=8)),
])
def test_unordered_cache_lockstep(name, kw):
    # same kept sets, sums and outputs as the ordered cache; rows compared after sorting the export by position
    wl = tiny("fill_" + name, **kw)
    st = run_lockstep(wl, all_units(wl), compaction="fill", check_rows_every=1)
    assert st["evictions"] > 0


def test_unordered_cache_many_units_decode():
    wl = tiny("fill_many", b=40, Hq=32, Hkv=8, s=160, B=64, K=72, steps=10, dtype="bf16", d=128)
    run_lockstep(wl, [(0, 0), (13, 5), (39, 7), (27, 2)], compaction="fill", check_rows_every=2)


@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("f32", 64)])
def test_unordered_cache_breaks_ties_by_position(dtype, d):
    # A crafted state: rows in shuffled order, every sum_weights zero, one key (position 0) whose logit exceeds all
    # others by more than 1000, so that every other weight underflows to exactly 0 in fp32 and in fp64 alike.  All
    # those pairs tie at the cut; the lower positions must stay (select on kv_ids in the block eviction, arg-min on
    # kv_ids in the decode step), pairs that stay must not move, and every row must keep its own position.
    import torch
    from paper_2412_05693_b200 import BatchMaxCache
    from paper_2412_05693_b200.binding import Config
    td = torch.bfloat16 if dtype == "bf16" else torch.float32
    g, Hkv, K, n0 = 2, 2, 24, 32
    cfg = Config(batch=1, n_q_heads=g * Hkv, n_kv_heads=Hkv, head_dim=d, kv_max=K, block_max=32, growth=40,
                 dtype=dtype, compaction="fill")
    cache = BatchMaxCache(cfg)
    dev = torch.device("cuda", 0)
    gen = torch.Generator().manual_seed(5)
    rnd = lambda *shape: torch.randn(*shape, generator=gen).to(td).to(dev)
    cache.prefill_block(rnd(1, n0, g * Hkv, d), rnd(1, n0, Hkv, d), rnd(1, n0, Hkv, d), 0, evict_to=-1)
    perm = {}
    for h in range(Hkv):
        ids = torch.randperm(n0, generator=gen).to(torch.int32)
        perm[h] = ids.tolist()
        kr = torch.zeros(n0, d, dtype=td)
        kr[ids == 0] = 10.0
        vr = ids.to(td)[:, None].expand(n0, d).contiguous()      # a row's value is its position
        cache.import_(ids, torch.zeros(n0), kr, vr, sample=0, kv_head=h)

    def check(expect, before):
        for h in range(Hkv):
            ids, sw, kr, vr = cache.export(0, 0, h, rows=True)
            ids = ids.tolist()
            assert sorted(ids) == sorted(expect), f"head {h}: kept {sorted(ids)}, expected {sorted(expect)}"
            assert torch.equal(vr[:, 0].float(), torch.tensor(ids, dtype=torch.float32)), "a row lost its position"
            assert all(float(kr[r].float().abs().max()) == (10.0 if i in hot else 0.0) for r, i in enumerate(ids))
            for r, i in enumerate(before[h][:len(ids)]):
                if i in expect:
                    assert ids[r] == i, f"head {h}: pair {i} stayed but moved from row {r}"
            before[h] = ids

    hot = {0}
    q10 = lambda n: torch.full((1, n, g * Hkv, d), 10.0, dtype=td, device=dev)
    vpos = lambda p0, n: torch.arange(p0, p0 + n, dtype=torch.float32)[None, :, None, None].expand(1, n, Hkv, d).to(td).to(dev)
    # a block of 16: every pair but position 0 ties at zero -> positions 0..23 stay, the block's pairs all leave
    cache.prefill_block(q10(16), torch.zeros(1, 16, Hkv, d, dtype=td, device=dev), vpos(n0, 16).contiguous(), n0, evict_to=K)
    expect = list(range(K))
    check(expect, perm)
    # decode steps whose own key matches the query as well as position 0 does: the step's pair stays, and of the pairs
    # tied at zero the highest position leaves
    for t in range(6):
        pos = n0 + 16 + t
        cache.decode_step(q10(1)[:, 0].contiguous(), torch.full((1, Hkv, d), 10.0, dtype=td, device=dev),
                          vpos(pos, 1)[:, 0].contiguous(), evict_to=K)
        hot.add(pos)
        expect.remove(max(i for i in expect if i not in hot))
        expect.append(pos)
        check(expect, perm)
    assert cache.status() == 0
    cache.close()


@pytest.mark.parametrize("dtype,d,s,B,K,pads", [
    ("f32", 64, 200, 48, 40, [0, 37, 150]),
    ("bf16", 128, 600, 128, 160, [0, 301, 77]),     # cached padding scattered over the rows of several key tiles
    ("bf16", 128, 333, 100, 77, [5, 250, 0]),
    ("bf16", 64, 256, 64, 300, [0, 200, 64]),       # nothing leaves during the prompt: padding stays cached in decoding
])
def test_unordered_cache_left_padding(dtype, d, s, B, K, pads):
    # padding pairs are masked by their kv_ids wherever their rows are, and leave first
    wl = tiny("fill_pad", b=3, s=s, B=B, K=K, steps=8, dtype=dtype, d=d, Hq=8 if d == 128 else 4, Hkv=2)
    run_lockstep(wl, all_units(wl), pads=pads, compaction="fill", check_rows_every=2)
    run_lockstep(wl, all_units(wl), pads=pads, compaction="fill", rule="sum_recent", check_rows_every=4)


@pytest.mark.parametrize("rule", ["sum_recent", "current_query"])
@pytest.mark.parametrize("dtype,d,Hq,Hkv,p_dec", [("bf16", 128, 8, 2, 1), ("f32", 64, 4, 4, 1), ("bf16", 128, 8, 2, 8)])
def test_unordered_cache_alternative_rules(rule, dtype, d, Hq, Hkv, p_dec):
    # the window of recent pairs is a select on kv_ids here, in the block eviction and in the decode step alike
    wl = tiny("fill_rules", s=400, B=128, K=96, steps=12, dtype=dtype, d=d, Hq=Hq, Hkv=Hkv, p_dec=p_dec)
    run_lockstep(wl, all_units(wl), rule=rule, compaction="fill", check_rows_every=2)


@pytest.mark.parametrize("kv_bar", [2, 33])
def test_unordered_cache_extreme_decoding_arm(kv_bar):
    # Algorithm 3's cut keeps the highest positions, wherever their rows are
    s, gen = 200, 70
    wl = tiny("fill_ed", s=s, B=48, K=s, steps=gen, dtype="bf16", d=128, Hq=8, Hkv=2)
    calls = [("prefill", t, min(48, s - t), -1) for t in range(0, s, 48)] + [("recent", 0, 0, 1)]
    n = 1
    for t in range(gen):
        calls.append(("decode", s + t, 1, -1))
        n += 1
        if n == kv_bar:
            calls.append(("recent", 0, 0, 1))
            n = 1
    run_lockstep(wl, all_units(wl), calls=calls, growth=kv_bar, compaction="fill", check_rows_every=5)


@pytest.mark.parametrize("seed", range(6))
def test_unordered_cache_random_cadences(seed):
    rng = np.random.default_rng(9100 + seed)
    g, hkv, d = int(rng.choice([1, 2, 4, 8])), int(rng.integers(1, 4)), int(rng.choice([64, 128]))
    wl = Workload(f"fillcad{seed}", b=int(rng.integers(1, 4)), Hq=g * hkv, Hkv=hkv, d=d, dtype=str(rng.choice(["bf16", "f32"])),
                  s=int(rng.integers(50, 900)), B=int(rng.integers(1, 300)), K=int(rng.integers(1, 400)),
                  steps=int(rng.integers(0, 16)), seed=9100 + seed, heavy_count=3, p_dec=int(rng.choice([1, 3])))
    rule = str(rng.choice(["average", "sum_recent", "current_query"]))
    if seed % 2 == 0:
        calls, growth = random_cadence(wl, rng)     # prefill / decode / evict / recency cuts in any order
        run_lockstep(wl, all_units(wl)[:3], calls=calls, growth=growth, rule=rule, compaction="fill", check_rows_every=3)
    else:
        pads = [int(rng.integers(0, wl.s + 1)) for _ in range(wl.b)]
        run_lockstep(wl, all_units(wl)[:3], pads=pads, rule=rule, compaction="fill", check_rows_every=3)


# ------------------------------------------------------------------ the rules of Sec. 2 on the same kernels
@pytest.mark.parametrize("rule", ["sum_recent", "current_query"])
@pytest.mark.parametrize("dtype,d,Hq,Hkv", [("bf16", 128, 8, 2), ("f32", 64, 4, 4)])
def test_alternative_eviction_rules_lockstep(rule, dtype, d, Hq, Hkv):
    wl = tiny("rules", s=400, B=128, K=96, steps=12, dtype=dtype, d=d, Hq=Hq, Hkv=Hkv)
    st = run_lockstep(wl, all_units(wl), rule=rule, check_rows_every=2)
    assert st["evictions"] >= 2 * Hkv * (3 + 12)


@pytest.mark.parametrize("window,pool", [(1, 1), (8, 3), (16, 7), (64, 5)])
@pytest.mark.parametrize("dtype,d,Hq,Hkv,B,K", [("bf16", 128, 8, 2, 48, 40), ("f32", 64, 4, 4, 20, 33), ("bf16", 128, 4, 4, 160, 150)])
def test_window_pooled_rule_lockstep(window, pool, dtype, d, Hq, Hkv, B, K):
    # Sec. 2, SnapKV: sums over the last `window` queries of the pass, max-pooled over neighbours, recent window kept
    wl = tiny(f"snap_{dtype}_w{window}_p{pool}", dtype=dtype, d=d, Hq=Hq, Hkv=Hkv, s=3 * B + 7, B=B, K=K, steps=5)
    st = run_lockstep(wl, all_units(wl), rule="window_pooled", rule_params=dict(window=window, pool=pool),
                      check_rows_every=2)
    assert st["evictions"] > 0


def test_window_pooled_rule_one_compression_after_the_prompt():
    # the rule's own cadence (Sec. 2): nothing leaves during prefilling, one compression after the prompt
    wl = tiny("snap_once", dtype="bf16", d=128, Hq=8, Hkv=2, s=300, B=64, K=96, steps=4)
    calls = [("prefill", p, min(wl.B, wl.s - p), -1) for p in range(0, wl.s, wl.B)] + [("evict", 0, 0, wl.K)]
    calls += [("decode", wl.s + t, 1, -1) for t in range(wl.steps)]
    st = run_lockstep(wl, all_units(wl), calls=calls, growth=wl.s + wl.steps - wl.K, rule="window_pooled",
                      rule_params=dict(window=32, pool=7), check_rows_every=2)
    assert st["evictions"] == len(all_units(wl))


def test_window_pooled_rule_with_left_padding():
    wl = tiny("snap_pad", dtype="bf16", d=128, Hq=8, Hkv=2, s=200, B=40, K=48, steps=6)
    run_lockstep(wl, all_units(wl), pads=[0, 57], rule="window_pooled", rule_params=dict(window=8, pool=3),
                 check_rows_every=2)


@pytest.mark.parametrize("share", [0.0, 0.25, 0.5, 1.0])
@pytest.mark.parametrize("dtype,d,Hq,Hkv,B,K,p_dec", [("bf16", 128, 8, 2, 48, 40, 1), ("f32", 64, 4, 4, 20, 33, 1),
                                                       ("bf16", 128, 4, 4, 160, 150, 4)])
def test_average_std_rule_lockstep(share, dtype, d, Hq, Hkv, B, K, p_dec):
    # Sec. 2 / Sec. 3.2 last paragraph, RoCo: part of the kept pairs by the standard deviation of their weights
    wl = tiny(f"roco_{dtype}_{share}", dtype=dtype, d=d, Hq=Hq, Hkv=Hkv, s=3 * B + 7, B=B, K=K, steps=9, p_dec=p_dec)
    st = run_lockstep(wl, all_units(wl), rule="average_std", rule_params=dict(std_share=share), check_rows_every=2)
    assert st["evictions"] > 0


def test_rules_that_need_ordered_rows_refuse_unordered_caches_and_padding():
    wl = tiny("refuse", dtype="bf16", d=128)
    for rule in ("window_pooled", "average_std"):
        with pytest.raises(bm.BMError):
            bm.arena_bytes(make_config(wl, rule=rule, compaction="fill"))
    cache = bm.BatchMaxCache(make_config(wl, rule="average_std"))
    with pytest.raises(bm.BMError):
        cache.set_left_pad([0, 3])
    # the memory model charges the second accumulator: 4 more bytes per row
    a = bm.cache_bytes_per_sample(make_config(wl, rule="average_std"))
    b = bm.cache_bytes_per_sample(make_config(wl, rule="average"))
    assert a - b == 4 * wl.Hkv * (wl.K + 1)


def test_alternative_rule_with_left_padding():
    # first blocks entirely padding: the recent window holds padding, which still ranks last
    wl = tiny("rules_pad", b=3, s=320, B=64, K=40, steps=6, dtype="bf16", d=128, Hq=8, Hkv=2)
    run_lockstep(wl, all_units(wl), rule="sum_recent", pads=[0, 100, 300], check_rows_every=2)
    run_lockstep(wl, all_units(wl), rule="current_query", pads=[5, 64, 250], check_rows_every=2)


def test_alternative_rule_with_growth_falls_back_to_the_general_select():
    # decode evicts 8 pairs at a time: the fused arg-min does not apply, the select kernel ranks by the rule
    wl = tiny("rules_g", s=256, B=64, K=64, steps=20, p_dec=8, dtype="bf16", d=128, Hq=8, Hkv=2)
    run_lockstep(wl, all_units(wl), rule="sum_recent", check_rows_every=4)


# ------------------------------------------------------------------ left-padded samples (Sec. 3)
@pytest.mark.parametrize("dtype,d,s,B,K,pads", [
    ("f32", 64, 200, 48, 40, [0, 37, 150]),         # SIMT path; padding inside a block and over whole blocks
    ("bf16", 128, 640, 128, 160, [0, 70, 300]),     # tensor-core path; a whole 128-key tile of cached padding
    ("bf16", 128, 640, 256, 96, [5, 255, 256]),     # padding ending at / just before a block boundary
    ("bf16", 64, 300, 64, 64, [299, 1, 128]),       # one sample almost entirely padding
])
def test_left_padded_samples_lockstep(dtype, d, s, B, K, pads):
    wl = tiny("leftpad", b=3, s=s, B=B, K=K, steps=6, dtype=dtype, d=d, Hq=8, Hkv=2)
    st = run_lockstep(wl, all_units(wl), pads=pads, check_rows_every=2)
    assert st["evictions"] > 0
    if dtype == "bf16":
        assert st["tc_calls"] == -(-s // B)          # every prefill call took the tensor-core kernels


@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("f32", 64)])
def test_left_padding_still_cached_during_decoding(dtype, d):
    # prompt shorter than the limit: the padding is still cached when decoding starts, is masked there, and is
    # what the first evicting decode steps remove (highest padding position first)
    wl = tiny("leftpad_dec", b=3, s=50, B=32, K=60, steps=24, dtype=dtype, d=d, Hq=8, Hkv=2)
    st = run_lockstep(wl, all_units(wl), pads=[0, 7, 30], check_rows_every=3)
    assert st["evictions"] >= 3 * 2 * 10


def test_left_pad_setter_errors():
    wl = tiny("leftpad_err", dtype="bf16", d=128)
    cache = bm.BatchMaxCache(make_config(wl))
    with pytest.raises(bm.BMError) as e:
        cache.set_left_pad([0, -1])
    assert e.value.code == 1
    cache.set_left_pad([3, 0])
    cache.set_left_pad(None)
    q, k, v = Inputs(wl, "cuda").block(0, 0, 48)
    cache.prefill_block(q, k, v, 0, evict_to=wl.K)
    with pytest.raises(bm.BMError) as e:
        cache.set_left_pad([1, 1])                                       # only while every cache is empty
    assert e.value.code == 4
    cache.close()


def test_moved_row_counters_match_the_kept_sets():
    # rows a compaction moves = rows from the first one whose content changes to the end of the kept set
    wl = tiny("moved", b=2, s=192, B=64, K=40, steps=10, dtype="bf16", d=128, Hq=8, Hkv=2)
    cache = bm.BatchMaxCache(make_config(wl))
    cache.count_moved_rows(True)
    inp = Inputs(wl, "cuda")
    units = all_units(wl)
    before = {u: [] for u in units}
    expected = 0
    for kind, pos0, I, ev in schedule(wl):
        q, k, v = inp.block(0, pos0, I)
        if kind == "prefill":
            cache.prefill_block(q, k, v, pos0, evict_to=ev)
        else:
            cache.decode_step(q[:, 0].contiguous(), k[:, 0].contiguous(), v[:, 0].contiguous(), evict_to=ev)
        for u in units:
            ids = cache.export(0, u[0], u[1])[0].tolist()
            n_old = len(before[u])
            cand = before[u] + list(range(pos0, pos0 + I))
            evicted = len(ids) < len(cand)
            if kind == "prefill" or evicted:      # a decode step that only appends moves nothing
                first = next((r for r in range(len(ids)) if ids[r] != cand[r] or r >= n_old), len(ids))
                expected += len(ids) - first
            before[u] = ids
    assert cache.moved_rows() == expected
    assert cache.moved_rows(reset=True) == expected
    assert cache.moved_rows() == 0
    cache.close()


# ------------------------------------------------------------------ API behaviour on the device
def test_error_codes_and_state_tracking():
    wl = tiny("errors", dtype="bf16", d=128)
    cfg = make_config(wl)
    cache = bm.BatchMaxCache(cfg)
    inp = Inputs(wl, "cuda")
    q, k, v = inp.block(0, 0, 48)
    with pytest.raises(bm.BMError) as e:
        cache.prefill_block(q, k, v, 5)                                  # pos0 must follow curr_id
    assert e.value.code == 4
    q2 = torch.randn(2, 49, wl.Hq, wl.d, device="cuda").to(wl.torch_dtype)
    with pytest.raises(bm.BMError) as e:
        cache.prefill_block(q2, q2[:, :, :wl.Hkv].contiguous(), q2[:, :, :wl.Hkv].contiguous(), 0)
    assert e.value.code == 1                                             # I > block_max
    with pytest.raises(bm.BMError) as e:
        cache.evict(-3)
    assert e.value.code == 1
    cache.close()
    # capacity: appending without eviction beyond cap
    cache = bm.BatchMaxCache(cfg)
    cache.prefill_block(q, k, v, 0, evict_to=wl.K)
    q, k, v = inp.block(0, 48, 48)
    with pytest.raises(bm.BMError) as e:
        cache.prefill_block(q, k, v, 48, evict_to=-1)
    assert e.value.code == 3
    assert cache.length() == (wl.K, 47)                                  # failed call left the mirror alone
    # sample ranges with unequal n cannot share a call
    cache.prefill_block(q[:1], k[:1], v[:1], 48, evict_to=wl.K, sample0=0)
    with pytest.raises(bm.BMError) as e:
        cache.prefill_block(q, k, v, 48, evict_to=wl.K)
    assert e.value.code == 4
    cache.prefill_block(q[1:], k[1:], v[1:], 48, evict_to=wl.K, sample0=1)
    assert cache.length(sample=0) == cache.length(sample=1) == (wl.K, 95)
    assert cache.status() == 0
    cache.close()
    # more caches in one prefill call than the launch grid can index: refused before anything is enqueued
    big = bm.BatchMaxCache(bm.Config(batch=8200, n_q_heads=8, n_kv_heads=8, head_dim=64, kv_max=4, block_max=2, dtype="bf16"))
    qb = torch.zeros(8200, 1, 8, 64, device="cuda", dtype=torch.bfloat16)
    with pytest.raises(bm.BMError) as e:
        big.prefill_block(qb, qb, qb, 0)
    assert e.value.code == 3
    big.prefill_block(qb[:4096], qb[:4096], qb[:4096], 0, sample0=0)
    big.prefill_block(qb[4096:], qb[4096:], qb[4096:], 0, sample0=4096)
    assert big.length(sample=8199) == (1, 0) and big.status() == 0
    big.close()


def test_bounded_wait_times_out_and_context_survives():
    # failure detection without a GPU fault: a wait that nothing satisfies gives up, the status word says so,
    # and the same handle keeps working afterwards
    wl = tiny("timeout", dtype="bf16", d=128, Hq=8, Hkv=2, s=96, B=48, K=40, steps=0)
    cache = bm.BatchMaxCache(make_config(wl))
    assert cache.status() == 0
    cache.selftest_wait_timeout()
    assert cache.status() == 6                     # BM_ERR_TIMEOUT
    cache.clear_status()
    assert cache.status() == 0
    cache.close()
    st = run_lockstep(wl, all_units(wl), check_rows_every=1)
    assert st["calls"] == 2


def run_free(wl, host=False, micro=None, pads=None):
    """Whole schedule on the GPU only; returns final state and all outputs (for determinism / variants)."""
    cfg = make_config(wl)
    cache = bm.BatchMaxCache(cfg)
    if pads is not None:
        cache.set_left_pad(pads)
    inp = Inputs(wl, "cuda")
    outs, keep = [], []
    for kind, pos0, I, ev in schedule(wl):
        q, k, v = inp.block(0, pos0, I)
        if kind == "decode":
            q, k, v = q[:, 0].contiguous(), k[:, 0].contiguous(), v[:, 0].contiguous()
        if host and not (host == "mixed" and len(outs) % 2 == 1):
            qh, kh, vh = (t.cpu().pin_memory() for t in (q, k, v))
            oh = torch.empty_like(qh).pin_memory()
            if kind == "prefill":
                cache.prefill_block_host(qh, kh, vh, pos0, oh, evict_to=ev)
            else:
                cache.decode_step_host(qh, kh, vh, oh, evict_to=ev)
            if host is True:
                torch.cuda.synchronize()
                outs.append(oh.clone())
            else:               # calls stay in flight; only the caller's stream is synchronised at the end
                outs.append(oh)
                keep.append((qh, kh, vh))
        elif micro and kind == "prefill":
            o = torch.empty_like(q)
            for s0 in range(0, wl.b, micro):
                cache.prefill_block(q[s0:s0 + micro], k[s0:s0 + micro], v[s0:s0 + micro], pos0, out=o[s0:s0 + micro],
                                    evict_to=ev, sample0=s0)
            outs.append(o.cpu())
        elif micro:
            o = torch.empty_like(q)
            for s0 in range(0, wl.b, micro):
                cache.decode_step(q[s0:s0 + micro], k[s0:s0 + micro], v[s0:s0 + micro], out=o[s0:s0 + micro],
                                  evict_to=ev, sample0=s0)
            outs.append(o.cpu())
        else:
            o = cache.prefill_block(q, k, v, pos0, evict_to=ev) if kind == "prefill" else \
                cache.decode_step(q, k, v, evict_to=ev)
            outs.append(o if host else o.cpu())
    torch.cuda.current_stream().synchronize()
    outs = [o.cpu().clone() for o in outs]
    state = [cache.export(0, s, h, rows=True) for s in range(wl.b) for h in range(wl.Hkv)]
    cache.close()
    return outs, state


def assert_same_run(a, b):
    for x, y in zip(a[0], b[0]):
        assert torch.equal(x, y)
    for sa, sb in zip(a[1], b[1]):
        for x, y in zip(sa, sb):
            assert torch.equal(x, y)


@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("f32", 64)])
def test_bitwise_reproducible_and_variants_agree(dtype, d):
    wl = tiny("repro", b=4, dtype=dtype, d=d, Hq=8, Hkv=2, s=256, B=64, K=64, steps=5)
    base = run_free(wl)
    assert_same_run(base, run_free(wl))                 # run-to-run determinism (no float atomics)
    assert_same_run(base, run_free(wl, host=True))      # host-fed entry points
    assert_same_run(base, run_free(wl, host="pipelined"))   # ... with every call left in flight
    assert_same_run(base, run_free(wl, host="mixed"))       # ... alternating with device-fed calls, no syncs
    assert_same_run(base, run_free(wl, micro=1))        # sample ranges: micro-batched calls


@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("f32", 64)])
def test_handles_without_the_native_step_give_the_same_results(dtype, d, monkeypatch):
    wl = tiny("general_way", dtype=dtype, d=d, steps=12)
    base = run_free(wl)
    monkeypatch.setattr(bm.binding, "_fastcall", False)
    assert bm.binding.fastcall() is None
    assert_same_run(base, run_free(wl))


@pytest.mark.parametrize("which", ["tiny", "cfg2"])
def test_cuda_graph_replay_matches_eager_launches(which):
    # the benchmark replays one CUDA graph per step; a captured schedule must leave the same bits as eager launches
    # (which the lock-step tests hold against the oracle) -- also at the benchmark's own full size
    wl = tiny("graph", b=4, dtype="bf16", d=128, Hq=8, Hkv=2, s=256, B=64, K=64, steps=6) if which == "tiny" \
        else WORKLOADS["cfg2"]
    eager_outs, eager_state = run_free(wl)
    cfg = make_config(wl)
    inp = Inputs(wl, "cuda")
    calls = schedule(wl)
    ins, outs = [], []
    for kind, pos0, I, ev in calls:
        q, k, v = inp.block(0, pos0, I)
        if kind == "decode":
            q, k, v = q[:, 0].contiguous(), k[:, 0].contiguous(), v[:, 0].contiguous()
        ins.append((q, k, v))
        outs.append(torch.empty_like(q))
    arena = torch.empty(bm.arena_bytes(cfg), dtype=torch.uint8, device="cuda")
    workspace = torch.empty(max(bm.workspace_bytes(cfg), 256), dtype=torch.uint8, device="cuda")

    def step():
        cache = bm.BatchMaxCache(cfg, arena=arena, workspace=workspace)
        for (kind, pos0, I, ev), (q, k, v), o in zip(calls, ins, outs):
            if kind == "prefill":
                cache.prefill_block(q, k, v, pos0, out=o, evict_to=ev)
            else:
                cache.decode_step(q, k, v, out=o, evict_to=ev)
        return cache

    step().close()                       # first use of every kernel outside the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        captured = step()
    for _ in range(2):                   # a replay starts from the re-created (zeroed) cache
        graph.replay()
    torch.cuda.synchronize()
    for o, ref in zip(outs, eager_outs):
        assert torch.equal(o.cpu(), ref)
    state = [captured.export(0, s_, h, rows=True) for s_ in range(wl.b) for h in range(wl.Hkv)]
    for sa, sb in zip(state, eager_state):
        for x, y in zip(sa, sb):
            assert torch.equal(x, y)
    assert captured.status() == 0
    captured.close()


@pytest.mark.parametrize("compaction", ["stable", "fill"])
def test_sample_ranges_on_concurrent_streams_match_whole_batch_calls(compaction):
    # the launch configuration of the benchmark: the batch split into sample ranges, each range's calls on a stream of
    # its own, all in flight together; every cache must end up bit-identical to the whole-batch run
    import torch
    from paper_2412_05693_b200 import BatchMaxCache
    from paper_2412_05693_b200.workloads import Inputs, schedule
    from tests.lockstep import make_config
    wl = WORKLOADS["cfg2"].with_(b=8, s=1536, steps=12)
    dev = torch.device("cuda", 0)
    inp = Inputs(wl, dev)
    ins = [(kind, pos0, I, ev, inp.block(0, pos0, I)) for kind, pos0, I, ev in schedule(wl)]

    def run(R):
        cache = BatchMaxCache(make_config(wl, compaction=compaction))
        outs = [torch.zeros(wl.b, I, wl.Hq, wl.d, dtype=torch.bfloat16, device=dev) for _, _, I, _, _ in ins]
        streams = [torch.cuda.Stream() for _ in range(R)]
        nb = wl.b // R
        torch.cuda.synchronize()
        for r in range(R):
            with torch.cuda.stream(streams[r]):
                for (kind, pos0, I, ev, (q, k, v)), o in zip(ins, outs):
                    sl = slice(r * nb, (r + 1) * nb)
                    if kind == "prefill":
                        cache.prefill_block(q[sl], k[sl], v[sl], pos0, out=o[sl], evict_to=ev, sample0=r * nb)
                    else:
                        cache.decode_step(q[sl, 0].contiguous(), k[sl, 0].contiguous(), v[sl, 0].contiguous(),
                                          out=o[sl, 0], evict_to=ev, sample0=r * nb)
        torch.cuda.synchronize()
        assert cache.status() == 0
        state = [cache.export(0, s_, h, rows=True) for s_ in range(wl.b) for h in (0, wl.Hkv - 1)]
        cache.close()
        return outs, state

    ref_out, ref_state = run(1)
    for R in (2, 4):
        outs, state = run(R)
        assert all(torch.equal(a, b) for a, b in zip(outs, ref_out)), f"{R} ranges: outputs differ"
        for got, want in zip(state, ref_state):
            assert all(torch.equal(a, b) for a, b in zip(got, want)), f"{R} ranges: cache state differs"


@pytest.mark.parametrize("rule", ["average", "average_std"])
def test_export_import_roundtrip_resumes_identically(rule):
    wl = tiny("ckpt", dtype="bf16", d=128, Hq=8, Hkv=2, s=192, B=64, K=48, steps=0)
    cfg = make_config(wl, rule=rule)
    inp = Inputs(wl, "cuda")
    a = bm.BatchMaxCache(cfg)
    for kind, pos0, I, ev in schedule(wl)[:2]:
        a.prefill_block(*inp.block(0, pos0, I), pos0, evict_to=ev)
    b = bm.BatchMaxCache(cfg)
    for s in range(wl.b):
        n, cur = a.length(sample=s)
        b.set_len(n, cur, sample=s)
        for h in range(wl.Hkv):
            b.import_(*a.export(0, s, h, rows=True), sample=s, kv_head=h)
            if rule == "average_std":       # the rule's second accumulator travels on its own pair of calls
                b.import_sum_sq(a.export_sum_sq(0, s, h), sample=s, kv_head=h)
    kind, pos0, I, ev = schedule(wl)[2]
    q, k, v = inp.block(0, pos0, I)
    oa, ob = a.prefill_block(q, k, v, pos0, evict_to=ev), b.prefill_block(q, k, v, pos0, evict_to=ev)
    assert torch.equal(oa, ob)
    for s in range(wl.b):
        for h in range(wl.Hkv):
            for x, y in zip(a.export(0, s, h, rows=True), b.export(0, s, h, rows=True)):
                assert torch.equal(x, y)
            if rule == "average_std":
                assert torch.equal(a.export_sum_sq(0, s, h), b.export_sum_sq(0, s, h))


def test_batch_sized_by_the_allocator_fits_its_arena():
    # allocator: batch = max fitting a budget; both arms (P&D, decode-only compression) live in arenas of that size
    wl = WORKLOADS["cfg3"].with_(s=1024, B=256, K=128, steps=2)
    budget = 64 * 2 ** 20
    pd_cfg = make_config(wl, batch=1)
    do_cfg = make_config(wl, batch=1, growth=wl.s + 1 - wl.K)
    b_pd, b_do = bm.max_batch(pd_cfg, budget), bm.max_batch(do_cfg, budget)
    assert b_pd / b_do == pytest.approx((wl.s + 1) / (wl.K + 1), rel=0.08)
    for b, growth in ((b_pd, None), (b_do, wl.s + 1 - wl.K)):
        w = wl.with_(b=b)
        cfg = make_config(w, growth=growth, max_call_samples=16)
        assert bm.arena_bytes(cfg) <= budget
        arena = torch.empty(budget + 512, dtype=torch.uint8, device="cuda")
        arena[budget:] = 0xA5                                            # canary behind the arena
        cache = bm.BatchMaxCache(cfg, arena=arena[:budget])
        inp = Inputs(w, "cuda")
        for pos0 in range(0, w.s, w.B):
            for s0 in range(0, b, 16):
                ns = min(16, b - s0)
                q, k, v = inp.block(0, pos0, w.B, s0, ns)
                cache.prefill_block(q, k, v, pos0, evict_to=(w.K if growth is None else -1), sample0=s0)
        if growth is not None:
            for s0 in range(0, b, 16):
                cache.evict(w.K, sample0=s0, nsamples=min(16, b - s0))
        torch.cuda.synchronize()
        assert cache.status() == 0
        assert cache.length(sample=b - 1)[0] == w.K
        assert bool((arena[budget:] == 0xA5).all())
        ids, sw, _, _ = cache.export(0, b - 1, w.Hkv - 1)
        assert np.all(np.diff(ids.numpy()) > 0) and float(sw.min()) >= 0
        cache.close()
