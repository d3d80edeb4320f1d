"""The data path at the sizes where its kernels change over: decode steps around 16 and 128 rows, units of the decode
attention that are cut or not, token passes, rows of logits around chunk and split limits."""
import numpy as np
import pytest
import torch

import att_plan
from gpu_util import compare_with_oracle, gpu_run_forced
from oracle import sampler as S
from paper_2604_07609_b200 import binding as B
from synth import make_weights
from synth.weights import TENSOR_NAMES, weight_layout
from synth.configs import ModelCfg, SchedCfg
from synth.workload import Request

pytestmark = pytest.mark.gpu
PH_ROPE, PH_FNORM = 2, 9   # places in a step's phase times

# four query heads per kv head: the shape that runs its GEMMs on CTA pairs
MODELS = {1024: ModelCfg(2, 1024, 8, 2, 128, 1024, 4096), 2048: ModelCfg(1, 2048, 16, 4, 64, 768, 4096),
          4096: ModelCfg(1, 4096, 8, 2, 128, 640, 1024)}


def _requests(prompts, new, vocab, seed=11, **how):
    rng = np.random.default_rng(seed)
    return [Request(ticket=t, arrival_s=0.0, prompt=rng.integers(0, vocab, size=p, dtype=np.int64).astype(np.int32), max_new=new,
                    seed=seed + t, user_tag=t, **how) for t, p in enumerate(prompts)]


def _check(model, prompts, new, chunk, layout=B.WEIGHTS_ROW_MAJOR, relative=True):
    """The bound of the large shapes: two correct evaluations that round at different places are N apart on these inputs.
    Without `relative` the absolute bound of the small shapes alone."""
    sched = SchedCfg(max_batch=len(prompts), prefill_chunk_tokens=chunk, n_slots=256, max_prompt=max(prompts), max_new=new,
                     n_blocks=sum((p + new + 15) // 16 for p in prompts))
    return compare_with_oracle(model, sched, _requests(prompts, new, model.vocab), make_weights(model, 5, "cpu", random_gains=True),
                               2e-2, noise_relative=relative, oracle_dtype=np.float32, weights_layout=layout)


@pytest.mark.parametrize("d", [1024, 2048, 4096])
@pytest.mark.parametrize("rows", [1, 2, 3, 15, 16, 17])
def test_small_decode_steps(rows, d):
    r = _check(MODELS[d], [3 + (7 * i) % 30 for i in range(rows)], 4, 512,
               B.WEIGHTS_STREAMING if d != 1024 else B.WEIGHTS_ROW_MAJOR)
    assert any(int(n) == rows for n in r["its"]["n_decode"])


@pytest.mark.parametrize("rows", [127, 128, 129])
def test_decode_steps_around_128_rows(rows):
    r = _check(MODELS[1024], [2 + i % 5 for i in range(rows)], 3, 512)
    assert any(int(n) == rows for n in r["its"]["n_decode"])


@pytest.mark.parametrize("prompts", [[15], [16], [383], [384, 1], [1500, 17, 800], [401] * 5], ids=str)
def test_decode_attention_units_whole_and_cut(prompts):
    _check(MODELS[2048], prompts, 3, 512, B.WEIGHTS_STREAMING)


@pytest.mark.parametrize("d, rows", [(2048, 38), (2048, 73), (1024, 75)])   # 152, 292 and 150 units: half CTAs take them
def test_decode_attention_units_of_half_ctas(d, rows):
    r = _check(MODELS[d], [100 + (37 * i) % 120 for i in range(rows)], 3, 16384, B.WEIGHTS_STREAMING if d == 2048 else B.WEIGHTS_ROW_MAJOR)
    assert any(int(n) == rows for n in r["its"]["n_decode"])


def _decode_keys(prompts, new):
    """Contexts of the first step in which every request decodes (they are all there from the first step on)."""
    return [p + 1 for p in prompts], [p + new - 1 for p in prompts]


@pytest.mark.parametrize("heads", [(16, 16, 64), (32, 16, 64), (64, 16, 64), (128, 16, 64), (32, 8, 128), (64, 8, 128)], ids=str)
def test_decode_attention_of_half_ctas_with_any_head_group(heads):
    """One, two, four and eight query heads per kv head; the rule is asked that half CTAs take the decode steps."""
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    rows, new = n_sm // heads[1] + 3, 3
    prompts = [100 + (37 * i) % 120 for i in range(rows)]
    for keys in _decode_keys(prompts, new):
        assert rows > 16 or heads[1] > 8
        assert att_plan.decode_way(keys, heads[1], n_sm) == "half"
    # The prompts' rows see up to 220 keys, whose probabilities the prefill kernel rounds (as below: rms 3 % above the oracles'
    # distance); logits of d = 512, sigma 0.45, and the absolute bound of the small shapes
    r = _check(ModelCfg(1, 512, *heads, 256, 1024), prompts, new, 8192, relative=False)
    assert r["err_plain"] <= 2e-2
    assert any(int(n) == rows for n in r["its"]["n_decode"])


@pytest.mark.parametrize("heads", [(16, 16, 64), (32, 16, 64), (64, 16, 64), (128, 16, 64)], ids=str)
@pytest.mark.parametrize("rows", [10, 16])
def test_half_ctas_that_also_rotate_and_write_keys_and_values(rows, heads):
    """Steps of at most 16 rows with more units than CTAs: RoPE and the K/V write run in the groups (no RoPE phase in those steps)."""
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    assert n_sm < rows * heads[1] <= 2 * n_sm
    # CTA pairs (four query heads) at d = 1024; else d = 256, whose logits (sigma 0.32) the absolute bound was made for
    pair = heads[0] == 4 * heads[1]
    r = _check(ModelCfg(2, 1024 if pair else 256, *heads, 256, 1024), [3 + (37 * i) % 70 for i in range(rows)], 4, 4096, relative=pair)
    assert r["err_plain"] <= 2e-2
    steps = [it for it in r["its"] if int(it["n_tokens"]) == int(it["n_decode"]) == rows]
    assert steps and all(int(it["phase_ns"][PH_ROPE]) == 0 for it in steps)


@pytest.mark.parametrize("tokens", [257, 300, 512, 513])
def test_prefill_steps_of_several_token_passes(tokens):
    # 6144 QKV rows: 24 pairs of weight tiles, which three token passes divide evenly over 74 pairs of CTAs
    model = ModelCfg(1, 512, 32, 8, 128, 256, 1024)
    # Every sampled row attends to hundreds of keys whose probabilities the prefill kernel rounds to bf16, a rounding
    # point that neither oracle has: relative error 2^-9 / sqrt(3) per key on top of the others, which puts the rms 2 %
    # above the distance between the oracles (1.70e-3 | 1.66e-3, max 6.6e-3).  d = 512 makes logits of sigma 0.45, for
    # which the absolute bound of the small shapes, 2e-2, holds.
    r = _check(model, [tokens], 2, 1024, B.WEIGHTS_STREAMING, relative=False)
    assert r["err_plain"] <= 2e-2
    assert int(r["its"]["n_tokens"][0]) == tokens


@pytest.mark.parametrize("heads", [(4, 2, 64), (2, 2, 128)], ids=str)
@pytest.mark.parametrize("rows", [1, 7, 9, 190, 191])   # 191 x 256 x 2048 products are above the limit of the folded phases
def test_fp32_steps_with_and_without_element_wise_phases(rows, heads):
    model = ModelCfg(2, 256, *heads, 1024, 1004, dtype="fp32")
    sched = SchedCfg(max_batch=1, prefill_chunk_tokens=512, n_slots=16, max_prompt=rows, max_new=3, n_blocks=(rows + 18) // 16)
    r = compare_with_oracle(model, sched, _requests([rows], 3, model.vocab), make_weights(model, 5, "cpu", random_gains=True), 1e-4)
    assert int(r["its"]["n_tokens"][0]) == rows


@pytest.mark.parametrize("rows, folded", [(24, True), (25, False)])   # 24 x 256 x 32400 products are the last below the limit
def test_fp32_steps_with_and_without_the_final_norm_inside_the_lm_head(rows, folded):
    model = ModelCfg(1, 256, 4, 2, 64, 512, 32400, dtype="fp32")
    sched = SchedCfg(max_batch=rows, prefill_chunk_tokens=512, n_slots=32, max_prompt=8, max_new=3, n_blocks=rows)
    r = compare_with_oracle(model, sched, _requests([3 + i % 5 for i in range(rows)], 3, model.vocab), make_weights(model, 5, "cpu", random_gains=True), 1e-4)
    steps = [it for it in r["its"] if int(it["n_sample_rows"]) == rows]
    assert steps and all((int(it["phase_ns"][PH_FNORM]) == 0) == folded for it in steps)


# more than 256 keys: prompt attention on CTA pairs, in units of 64 rows and tiles of 128 keys
@pytest.mark.parametrize("prompts, chunk", [([256], 512), ([257], 512), ([383, 385], 512), ([1026], 512), ([600, 40, 300], 256),
                                            ([1500, 17, 800], 700)], ids=str)
def test_prompt_attention_around_units_and_tiles(prompts, chunk):
    # (the probabilities' rounding of the test above; logits of d = 512)
    r = _check(ModelCfg(1, 512, 8, 2, 128, 256, 1024), prompts, 2, chunk, B.WEIGHTS_STREAMING, relative=False)
    assert r["err_plain"] <= 2e-2


def test_prompt_attention_of_more_units_than_pairs():
    # 8 prompts x 5 units x 2 kv heads on 74 pairs, two layers: some pairs have a second unit in every layer
    _check(ModelCfg(2, 512, 8, 2, 128, 256, 1024), [290, 300, 310, 320, 257, 319, 288, 305], 2, 4096, B.WEIGHTS_STREAMING, relative=False)


@pytest.mark.parametrize("heads, prompts", [((32, 8, 128), [270, 288]), ((8, 2, 128), [260, 20, 270, 288, 257, 30, 280, 265, 272, 288])], ids=str)
def test_prompt_attention_that_would_take_the_pairs_a_second_round(heads, prompts):
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    assert att_plan.prompts_on_pairs([(0, p) for p in prompts], heads[1], n_sm) == 0
    assert att_plan.prompts_on_pairs([(0, p) for p in prompts + [290]], heads[1], n_sm) > 0
    _check(ModelCfg(1, 512, *heads, 256, 1024), prompts, 2, 4096, B.WEIGHTS_STREAMING, relative=False)


def test_prompt_attention_leaves_the_pools_old_contents_alone():
    """Keys and values beyond a request's last token are whatever the pool held, NaN here."""
    model = ModelCfg(1, 512, 8, 2, 128, 256, 1024)
    sched = SchedCfg(max_batch=2, prefill_chunk_tokens=512, n_slots=16, max_prompt=512, max_new=2, n_blocks=80)
    weights = make_weights(model, 5, "cuda")
    out = []
    for fill in (0, 0xFF):
        kv = torch.full((sched.n_blocks * B.kv_bytes_per_block(model, 16),), fill, dtype=torch.uint8, device="cuda")
        logits = torch.zeros(4, model.vocab, device="cuda")
        torch.cuda.synchronize()
        eng = B.Blink(model, sched, weights, kv, exec_mode=B.EXEC_MANUAL, logits_capture=logits)
        for r in _requests([270, 491], 2, model.vocab):
            eng.submit_request(r, forced_tokens=np.zeros(2, np.int32))
        eng.blink_run(4)
        eng.drain(4)
        eng.blink_destroy()
        out.append(logits)
    assert torch.isfinite(out[1]).all()
    # split-K sums in another order move a 16-bit rounding here and there: 2^-8 of a value of up to sigma 0.45 x 4
    assert (out[0] - out[1]).abs().max() <= 2 ** -8 * 1.8


@pytest.mark.parametrize("V", [2, 5, 1023, 4099, 32768, 32772, 65540, (1 << 20) + 4])
def test_sampler_rows_around_chunk_limits(V):
    rng = np.random.default_rng(V)
    rows = 9
    logits = (rng.normal(size=(rows, V)) * 1.3).astype(np.float32)
    logits[3, V // 2:] = logits[3].max() + 1.0   # a plateau that ends with the row
    logits[4] = 0.5
    top_k = np.array([0, min(50, V), 0, 7, 0, 0, 1, 64, 0], dtype=np.int32)
    top_p = np.array([0, 0, 0.9, 0.5, 0.7, 0.999, 0, 0.3, 0.05], dtype=np.float32)
    temp, ticket = np.full(rows, 0.8, np.float32), np.arange(rows, dtype=np.uint64)
    gen, seed = np.arange(rows, dtype=np.int32), np.full(rows, 99, np.uint64)
    got = B.blink_sample_top_p(torch.from_numpy(logits).cuda(), top_k, temp, top_p, ticket, gen, seed)
    for r in range(rows):
        assert int(got[r]) == S.sample(logits[r], int(top_k[r]), 0.8, r, r, 99, float(top_p[r])), (V, r)


@pytest.mark.parametrize("V", [32768, 36864, 40004])
def test_sampling_inside_the_loop_equals_the_oracle_on_the_loops_own_logits(V):
    """Rows of more than 24576 entries are prepared by all CTAs (maxima, nucleus weights): greedy, top-k, nucleus and both
    together in one batch; the oracle's sampler on the captured rows gives the tokens, bit for bit."""
    model = ModelCfg(1, 256, 4, 4, 64, 256, V, dtype="fp32")
    sched = SchedCfg(max_batch=8, prefill_chunk_tokens=64, n_slots=16, max_prompt=16, max_new=6, n_blocks=32)
    reqs = _requests([4, 5, 6, 7, 8, 9], 6, V)
    how = [(0, 0.0), (50, 0.0), (0, 0.9), (0, 0.5), (40, 0.8), (0, 0.99)]
    for r, (k, p) in zip(reqs, how):
        r.top_k, r.top_p, r.temperature = k, p, 0.8
    trace, toks, logits, _ = gpu_run_forced(model, sched, reqs, make_weights(model, 5, "cpu"), None)
    slot_ticket, row, n = {}, 0, {t: 0 for t in range(len(reqs))}
    for rec in trace:   # row r of the capture is the r-th sampled row since the start
        slot_ticket.update({b: t for t, b in rec["admitted"]})
        for b, tok in rec["sampled"]:
            q = reqs[slot_ticket[b]]
            want = S.sample(logits[row], q.top_k, q.temperature, q.ticket, n[q.ticket], q.seed, q.top_p)
            assert tok == want == toks[q.ticket][n[q.ticket]], (q.ticket, n[q.ticket])
            n[q.ticket] += 1
            row += 1
    assert row == 36


def _sample(logits, top_k, top_p, temp=0.8):
    """The sampler on rows that lie inside a larger buffer of -inf."""
    rows, V = logits.shape
    buf = torch.full((1024 + rows * V + 1024,), float("-inf"), device="cuda")
    buf[1024:1024 + rows * V] = torch.from_numpy(logits).cuda().reshape(-1)
    x = buf[1024:1024 + rows * V].view(rows, V)
    return [int(t) for t in B.blink_sample_top_p(x, np.full(rows, top_k, np.int32), np.full(rows, temp, np.float32),
                                                 np.full(rows, top_p, np.float32), np.arange(rows, dtype=np.uint64),
                                                 np.zeros(rows, np.int32), np.full(rows, 3, np.uint64))]


@pytest.mark.parametrize("V", [5, 4096, 40004, 140000])
def test_greedy_rows_with_nan_and_infinities(V):
    rng = np.random.default_rng(V)
    x = rng.normal(size=(6, V)).astype(np.float32)
    x[0] = np.nan                      # nothing to choose from: token 0
    x[1] = -np.inf
    x[2, 1:] = np.nan                  # one number
    x[3, V // 2] = x[3, V - 1] = np.inf
    x[4, ::2] = np.nan                 # NaN is never the largest
    x[5] = np.nan
    x[5, V - 1] = -np.inf              # -inf is larger than no number at all
    want = [0, 0, 0, V // 2, int(np.nanargmax(x[4])), V - 1]
    assert _sample(x, 0, 0.0) == want


@pytest.mark.parametrize("V", [5, 4096, 40004, 140000])
def test_nucleus_rows_without_a_finite_largest_value(V):
    """exp(z - z0) has no value there: the first of the largest is the nucleus, token 0 when there is no number."""
    rng = np.random.default_rng(V)
    x = rng.normal(size=(5, V)).astype(np.float32)
    x[0] = np.nan
    x[1] = -np.inf
    x[2, V - 2] = np.inf
    x[3, V // 2] = x[3, V // 2 + 1] = np.inf
    x[4] = np.nan
    x[4, V - 1] = -np.inf
    assert _sample(x, 0, 0.9) == [0, 0, V - 2, V // 2, V - 1]
    y = np.abs(rng.normal(size=(1, V))).astype(np.float32) + 1   # a temperature so small that every z overflows
    assert _sample(y, 0, 0.9, temp=1e-39) == [0]
    y[0, 0] = -1
    assert _sample(y, 0, 0.9, temp=1e-39) == [1]


@pytest.mark.parametrize("top_p", [0.0, 0.9])
@pytest.mark.parametrize("V", [5, 4096, 40004])
def test_top_k_rows_with_nan_answer_the_same_member_of_the_row_each_time(V, top_p):
    x = np.full((3, V), np.nan, np.float32)
    x[1, 1:3] = [0.5, -0.5]
    x[2, : V // 2] = 0.25
    first = _sample(x, min(50, V), top_p)
    assert all(0 <= t < V for t in first)
    assert all(_sample(x, min(50, V), top_p) == first for _ in range(3))


@pytest.mark.parametrize("V", [1 << 18, (1 << 18) + 4, (1 << 21) + 36, 2300001])
def test_nucleus_of_very_long_rows_adds_up_every_weight(V):
    """Weights are added in limbs of a few bits: a row of equal weights with all limbs nearly full carries the sums as far
    as they go.  Two values, so the order and the cut have a closed form."""
    d = np.arange(1, 40001, dtype=np.float32) / 4096          # the drop whose weight has the fullest lower limbs
    q = np.floor(np.exp(-d.astype(np.float64)) * 2.0 ** 40).astype(np.int64)
    fill = np.min([(q >> s) & 2047 for s in (0, 11, 22)], axis=0)
    drop, w = float(d[fill.argmax()]), int(q[fill.argmax()])
    assert int(fill.max()) > 1900
    x = np.full((4, V), -drop, np.float32)
    top = np.array([V - 1, 0, V // 2, 7])
    x[np.arange(4), top] = 0.0                                # z0, weight 2^40
    Q = (V - 1) * w + (1 << 40)
    p24 = int(np.rint(np.float64(np.float32(0.9)) * (1 << 24)))
    need = -(-p24 * Q // (1 << 24))
    n = -(-(need - (1 << 40)) // w)                           # entries of the nucleus beside the top one
    got = _sample(x, 0, 0.9, temp=1.0)
    for r in range(4):
        target = ((S.philox_word(r, 0, 3) >> 8) * ((1 << 40) + n * w)) >> 24
        j = max(0, -(-(target + 1 - (1 << 40)) // w))         # place in the order: 0 is the top entry
        want = int(top[r]) if j == 0 else int(np.delete(np.arange(V), top[r])[j - 1])
        assert got[r] == want, (r, got[r], want)


@pytest.mark.parametrize("broken", [2, 4])   # behind two others: with two choices never the first still open
def test_an_expert_whose_router_logit_is_nan_is_as_good_as_absent(broken):
    """NaN is larger than nothing: unless it is the first still open, such an expert is never chosen, and the model
    answers as the one without it."""
    model = ModelCfg(2, 256, 4, 4, 64, 256, 512, n_experts=5, top_k_experts=2, dtype="fp32")
    less = model.with_(n_experts=4)
    w = make_weights(model, 17, "cpu")
    (lay, _), (lay_less, total) = weight_layout(model), weight_layout(less)
    w_less = torch.zeros(total, dtype=torch.uint8)
    keep = [e for e in range(5) if e != broken]
    for name in TENSOR_NAMES:
        (o, shape, dt), (ol, shape_l, _) = lay[name], lay_less[name]
        t = w[o:o + int(np.prod(shape)) * 4].view(dt).view(shape)
        t_less = w_less[ol:ol + int(np.prod(shape_l)) * 4].view(dt).view(shape_l)
        t_less.copy_(t[:, keep] if name in ("wgu", "wd", "wr") else t)
        if name == "wr":
            t[:, broken] = float("nan")
    sched = SchedCfg(max_batch=4, prefill_chunk_tokens=32, n_slots=16, max_prompt=16, max_new=6, n_blocks=32)
    reqs = _requests([4, 9, 16, 7], 6, model.vocab)
    forced = {r.ticket: list(range(10 * r.ticket, 10 * r.ticket + 6)) for r in reqs}
    a = gpu_run_forced(model, sched, reqs, w, forced)
    b = gpu_run_forced(less, sched, reqs, w_less, forced)
    assert np.isfinite(b[2]).all() and float(np.abs(b[2]).max()) > 0.1
    assert float(np.abs(a[2] - b[2]).max()) <= 1e-4    # the bound of the fp32 mode; the experts' sums are added in any order


@pytest.mark.parametrize("V", [1025, 4099, 32000])
def test_nucleus_of_rows_whose_first_entries_do_not_show_their_spread(V):
    """The buckets take the spread of a row from its first entries; whatever those are, the answer is the oracle's."""
    rng = np.random.default_rng(V)
    x = rng.normal(size=(7, V)).astype(np.float32)
    x[0] = 3.0 + 1e-4 * x[0]           # nearly equal
    x[1, :1024] = -np.inf              # the first entries masked
    x[2, :1024] = 9.0                  # the first entries equal and the largest
    x[3, :1024] = -9.0                 # the first entries equal and the smallest
    x[4] = 60.0 * x[4]                 # most entries without a weight
    x[5, :1024] = 9.0 + 1e-3 * x[5, :1024]
    x[6] = 2.5                         # all equal
    for p in (0.05, 0.6, 0.999):
        got = _sample(x, 0, p)
        for r in range(len(x)):
            assert got[r] == S.sample(x[r], 0, 0.8, r, 0, 3, p), (r, p)


@pytest.mark.parametrize("V", [24576, 24580, 32000])
def test_sampling_inside_the_loop_around_the_limit_of_shared_rows(V):
    test_sampling_inside_the_loop_equals_the_oracle_on_the_loops_own_logits(V)


@pytest.mark.parametrize("rows", [37, 38, 60, 75])
def test_decode_attention_of_short_units_in_one_round_and_two(rows):
    # four kv heads: 148 units fill the CTAs once, more take two rounds by CTAs or one by warps; beyond 296 warps only
    _check(MODELS[2048], [20 + i % 7 for i in range(rows)], 3, 2048, B.WEIGHTS_STREAMING)
