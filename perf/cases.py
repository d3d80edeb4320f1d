"""Workloads by which the speed of the serving loop is judged.

A case is one job for the framework: a number of prompts, each with its number of new tokens, on one of the
model shapes of `synth.configs`.  `prepare` does what a server does once (weights in place, KV pool carved out,
context created) and draws the prompts; `run` hands the prompts in, lets the loop work and collects every token:

  mode "stream"  the persistent loop, one request, tokens read with blink_poll as they come: somebody waits for
                 each of them.  The loop is told to leave the GPU at the end of the pass.
  mode "batch"   all requests are handed in first, then one launch of the loop kernel runs the steps they need
                 (blink_run), then the tokens are collected: an offline job, many requests at once.

What comes back is every token and the KV cache that the pass has filled: keys and values of all layers at all
positions.  The schedule of a pass is the same every time (all requests are known before the first step), so the
cache blocks are too.
"""
import math
import random

import numpy as np
import torch

from paper_2604_07609_b200 import binding as B
from synth import model_cfg, sched_cfg

CONFIG = {"tiny": 1, "1b": 2, "8b": 3, "moe": 5}


def _case(name, model, mode, requests, prompt, new, dtype="bf16", layout="streaming", policy="chunked", sampling="greedy",
          layers=0):
    c = dict(model=model, mode=mode, requests=requests, prompt_lo=prompt[0], prompt_hi=prompt[1], new_lo=new[0],
             new_hi=new[1], dtype=dtype, layout=layout, policy=policy, sampling=sampling, layers=layers)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest call: a short answer from the small configuration; launches and latency are all there is
        _case("tiny one short request", "tiny", "stream", 1, (16, 16), (8, 8), layout="row-major"),
        # the small configuration's own workload in the fp32 reference mode (prompts 16-64, 32 new tokens, batch of 8)
        _case("tiny fp32 batch of 8", "tiny", "batch", 8, (16, 64), (32, 32), dtype="fp32", layout="row-major"),
        # a single user of the 1B shape with weights left in the exchange layout, the API's default
        _case("1b one request", "1b", "stream", 1, (201, 201), (32, 32), layout="row-major"),
        # the 1B shape with a nearly full batch of short prompts: decode steps of about a hundred rows
        _case("1b batch of 100", "1b", "batch", 100, (17, 130), (24, 24)),
        # a single user of the 8B shape, top-k sampling: prompt, then one decode row per step
        _case("8b one request", "8b", "stream", 1, (300, 300), (24, 24), sampling="top_k"),
        # a long document and a short answer: chunked prefill over a growing context
        _case("8b long prompt", "8b", "stream", 1, (3999, 3999), (3, 3)),
        # 64 conversations: decode steps of 64 rows
        _case("8b batch of 64", "8b", "batch", 64, (20, 60), (24, 24), sampling="top_k"),
        # the largest batch of the 8B configuration: prefill beside decode, then decode steps of 256 rows
        _case("8b batch of 256", "8b", "batch", 256, (16, 48), (12, 20), sampling="top_k"),
        # the stream of the 8B configuration in small: prompts and answers of very different lengths together
        _case("8b mixed lengths", "8b", "batch", 24, (24, 1500), (4, 40), sampling="top_k"),
        # the paper's own policy and sampler: whole prompts in steps of their own, nucleus sampling
        _case("8b pause and resume", "8b", "batch", 20, (64, 300), (16, 16), policy="pause-resume", sampling="top_p"),
        # a few long conversations: decode over contexts of thousands of tokens
        _case("8b long contexts", "8b", "batch", 4, (1200, 1800), (48, 48), sampling="top_k"),
        # routed experts, four layers of the 32-layer shape (a state has to fit several times): prefill, then decode
        _case("moe batch of 24", "moe", "batch", 24, (40, 260), (20, 20), layers=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more job: a model shape, a mode, and sizes anywhere in the ranges of the listed jobs."""
    model = rng.choice(["tiny", "tiny", "1b", "1b", "8b", "8b", "8b", "8b", "moe"])
    mode = rng.choice(["stream", "batch"])
    sampling = rng.choice(["greedy", "top_k", "top_p"])
    layout = rng.choice(["streaming", "streaming", "row-major"])
    most = {"tiny": 8, "1b": 128, "8b": 256, "moe": 64}[model]
    n = 1 if mode == "stream" else _log_int(rng, 2, most)
    longest = {"tiny": 64, "1b": 1000, "8b": 4000, "moe": 2000}[model]
    # about 9000 prompt tokens at most, and answers so that a job of many long prompts has short ones
    hi = max(5, min(longest, _log_int(rng, 16, 9000) // n))
    lo = rng.randint(max(4, hi // 8), hi)
    new_hi = rng.randint(4, 32)
    new_lo = rng.randint(max(2, new_hi // 2), new_hi)
    dtype = rng.choice(["bf16", "fp32"]) if model == "tiny" else "bf16"
    policy = rng.choice(["chunked", "chunked", "pause-resume"]) if model in ("1b", "8b") and mode == "batch" else "chunked"
    return _case(None, model, mode, n, (lo, hi), (new_lo, new_hi), dtype, "row-major" if dtype == "fp32" else layout,
                 policy, sampling, 4 if model == "moe" else 0)


# ---- sizes and schedule of a case: they follow from the case alone, not from the seed --------------------------
def _model(case):
    m = model_cfg(CONFIG[case["model"]], dtype=case["dtype"])
    return m.with_(n_layers=case["layers"]) if case["layers"] else m


def _lengths(case):
    """Prompt and answer lengths: spread evenly over the logarithm of their ranges, in a fixed mixed order."""
    n = case["requests"]

    def spread(lo, hi, key):
        v = [int(round(lo * (hi / lo) ** ((i + 0.5) / n))) for i in range(n)]
        random.Random(key).shuffle(v)
        return v
    return spread(case["prompt_lo"], case["prompt_hi"], 1), spread(case["new_lo"], case["new_hi"], 2)


def _sched(case):
    s = sched_cfg(CONFIG[case["model"]])
    P, N = _lengths(case)
    blocks = sum((p + n - 1 + s.block_size - 1) // s.block_size for p, n in zip(P, N))
    if case["policy"] == "pause-resume":   # whole prompts have to fit into a step
        s = s.with_(prefill_chunk_tokens=max(s.prefill_chunk_tokens, s.max_prompt))
    return s.with_(n_blocks=blocks)


def _steps(case):
    """The steps of a pass: for each a list of (first position, rows, samples a token) over the requests in it."""
    P, N = _lengths(case)
    s = _sched(case)
    done, gen = [0] * len(P), [0] * len(P)
    was_prefill, out = False, []
    while any(g < n for g, n in zip(gen, N)):
        step, left = [], s.prefill_chunk_tokens
        prefill = [i for i in range(len(P)) if done[i] < P[i]]
        decode = [i for i in range(len(P)) if done[i] == P[i] and gen[i] < N[i]]
        if case["policy"] == "pause-resume":
            was_prefill = bool(prefill) and (not was_prefill or not decode)
            decode = [] if was_prefill else decode
            prefill = prefill if was_prefill else []
        for i in decode:
            step.append((P[i] + gen[i] - 1, 1, True))
            gen[i] += 1
        for i in prefill:
            take = min(P[i] - done[i], left)
            if case["policy"] == "pause-resume" and take < P[i]:
                break
            if take > 0:
                step.append((done[i], take, done[i] + take == P[i]))
                done[i] += take
                left -= take
                gen[i] += done[i] == P[i]
        out.append(step)
    return out


def work(case):
    """Every step reads the weights it needs once and, of each request in it, the keys and values of the steps before;
    it writes those of its own rows.  A step's operations are the dense contractions, the experts chosen, attention
    over the keys each row sees, and the output projection of the rows that sample."""
    m = _model(case)
    e = 2 if m.dtype == "bf16" else 4
    attn = m.qkv_dim * m.d_model + m.d_model * m.q_dim
    ffn = 3 * m.d_ff * m.d_model
    kv = m.n_layers * 2 * m.kv_dim * e
    nbytes = flops = 0.0
    for step in _steps(case):
        T = sum(r for _, r, _ in step)
        rows = sum(1 for _, _, s in step if s)
        keys = sum(r * p + r * (r + 1) // 2 for p, r, _ in step)
        k, E = (m.top_k_experts, m.n_experts) if m.n_experts else (1, 1)
        touched = E * (1 - (1 - k / E) ** T) if E > 1 else 1   # experts that some row of the step is sent to
        nbytes += m.n_layers * (attn + touched * ffn) * e + (m.vocab * m.d_model * e if rows else 0)
        nbytes += sum(p for p, _, _ in step) * kv + T * (kv + m.d_model * e)
        flops += 2.0 * T * m.n_layers * (attn + k * ffn) + 2.0 * rows * m.vocab * m.d_model
        flops += 4.0 * keys * m.q_dim * m.n_layers
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # Keys and values of the last layers carry the 16-bit roundings of all layers before them; the tokens are
    # far apart (see _weights), so that they change at a tie of two probabilities only.
    if case["dtype"] == "fp32":
        return {"rel": 2e-5, "max": 2e-3, "differ": 0.0}
    return {"rel": 1e-2, "max": 0.4, "differ": 0.005}


# ---- the pass ---------------------------------------------------------------------------------------------------
def _weights(m, seed, layout):
    """Random weights: N(0, 0.02), projections back into the residual stream narrower by the square root of their
    number, so that the stream grows over the layers as in a model that is in use; a token's successor is its likeliest
    continuation by a wide margin, as in text, so that a pass makes the same tokens whatever the order of its sums."""
    w = torch.zeros(B.blink_weights_bytes(m), dtype=torch.uint8, device="cuda")
    dt = torch.bfloat16 if m.dtype == "bf16" else torch.float32
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)

    def view(tensor, rows, cols, kind):
        off = B.blink_weight_offset(m, tensor)
        return w[off:off + rows * cols * kind.itemsize].view(kind).view(rows, cols)
    L, E1, d = m.n_layers, max(1, m.n_experts), m.d_model
    back = 0.02 / math.sqrt(2 * L)
    embed = view(0, m.vocab, d, dt).normal_(0, 1, generator=g)
    if m.n_experts:   # decisive routing, as a trained router's: a token carries the marks of the two experts it goes to
        E = m.n_experts
        mark = torch.randint(0, 2, (E, d), device="cuda", generator=g).mul_(2).sub_(1).to(dt)
        v = torch.arange(m.vocab, device="cuda")
        embed.add_(mark[v % E]).add_(mark[(v + 1 + v // E % (E - 1)) % E], alpha=0.6)
    view(1, L * m.qkv_dim, d, dt).normal_(0, 0.02, generator=g)
    view(2, L * d, m.q_dim, dt).normal_(0, back, generator=g)
    view(3, L * E1 * 2 * m.d_ff, d, dt).normal_(0, 0.02, generator=g)
    view(4, L * E1 * d, m.d_ff, dt).normal_(0, back, generator=g)
    if m.n_experts:
        view(5, L * E, d, torch.float32).normal_(0, 0.002, generator=g).view(L, E, d).add_(mark, alpha=0.005)
    for norm, rows in ((6, L), (7, L), (8, 1)):
        view(norm, rows, d, torch.float32).normal_(1, 0.1, generator=g)
    head = view(9, m.vocab, d, dt).normal_(0, 0.02, generator=g)
    head.add_(torch.roll(embed, 1, 0), alpha=0.04 if d < 1024 else 0.01)
    if layout == "streaming":
        B.blink_convert_weights(m, w, B.WEIGHTS_ROW_MAJOR, B.WEIGHTS_STREAMING)
        return w, B.WEIGHTS_STREAMING
    return w, B.WEIGHTS_ROW_MAJOR


def prepare(case, seed):
    m, s = _model(case), _sched(case)
    weights, layout = _weights(m, seed, case["layout"])
    kv = torch.zeros(s.n_blocks * B.kv_bytes_per_block(m, s.block_size), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    stream = case["mode"] == "stream"
    engine = B.Blink(m, s, weights, kv, exec_mode=B.EXEC_PERSISTENT if stream else B.EXEC_MANUAL, weights_layout=layout,
                     policy=B.POLICY_PAUSE_RESUME if case["policy"] == "pause-resume" else B.POLICY_CHUNKED)
    if stream:
        engine.blink_stop()   # off the GPU until a request comes
    P, N = _lengths(case)
    rng = np.random.default_rng(seed)
    how = {"greedy": {}, "top_k": dict(top_k=50, temperature=0.8), "top_p": dict(temperature=0.8, top_p=0.9)}[case["sampling"]]
    requests = [dict(prompt=rng.integers(0, m.vocab, size=p, dtype=np.int32), max_new_tokens=n,
                     seed=int(rng.integers(1 << 62)), **how) for p, n in zip(P, N)]
    first = np.concatenate([[0], np.cumsum(N)])
    return dict(engine=engine, stream=stream, requests=requests, first=first, steps=len(_steps(case)),
                kv=kv.view(torch.bfloat16 if m.dtype == "bf16" else torch.float32))


def run(state):
    engine, first = state["engine"], state["first"]
    total = int(first[-1])
    tickets = [engine.blink_submit(**r) for r in state["requests"]]
    if not state["stream"]:
        engine.blink_run(state["steps"])
    events = engine.drain(total)
    if state["stream"]:
        engine.blink_stop()
    tokens = np.empty(total, dtype=np.int32)
    tokens[first[events["ticket"].astype(np.int64) - tickets[0]] + events["index"]] = events["token"]
    return {"tokens": tokens, "kv": state["kv"]}
