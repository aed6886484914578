"""What a user has this library do, as cases that can be timed one by one.

A case is a dict of plain values.  `prepare` makes what a program holds before the call (weights, the context, prompts),
`run` is one call or one request through the public binding, `work` says what that pass cannot do without, `tolerance`
how far another correct implementation may be off.

Kinds of case:
  request     a whole response: prompt pass, then Tandem + SPEED decoding of `new` tokens, natural acceptance
  samples     `samples` sampled responses to each prompt (one prompt pass per prompt), sampled acceptance
  adaptive    a response with router-chosen block lengths
  prompt      the prompt pass alone (time to the first token of a long document)
  evaluate    teacher-forced scoring of given sequences (accuracy / cross-entropy evaluation)
  attention   the stand-alone decode attention over a mixed context
  project     the stand-alone FF_Tandem projection with the small layer's key / value maps

The weights are random-init, except that both models predict confidently, as trained ones do: a token's embedding stands
out of the residual stream, and the output head holds, for every token, one successor's row aligned with that embedding.
The two models agree on the successor of about AGREE of the tokens, which gives accept lengths a spread that trained
pairs show; a token id therefore does not hang on the last bits of two nearly equal logits.
"""
from dataclasses import replace
from math import exp, log

import torch

from paper_2402_08644_b200 import binding, synth

AGREE = 0.7          # share of the tokens after which the two models predict the same successor
EMB_STD = 2.0        # embeddings' standard deviation: they stand out of what the layers add to the residual stream
ROUTER_K, ROUTER_HIDDEN, ROUTER_TAU = 4, 64, 0.5
DRAW_POS = 8960      # position tables of the bf16 pairs (the benchmark's largest context)


def listed():
    return [
        # the fp32 pair of the exact-arithmetic mode, the smallest request there is: launches and latency only
        {"name": "request_tiny_fp32", "kind": "request", "pair": "tiny", "batch": 1, "prompt": 32, "ragged": 0.0, "gamma": 4, "new": 64, "kv_large": 0, "kv_small": 0},
        # one interactive user, small pair: a chain of short kernels
        {"name": "request_small", "kind": "request", "pair": "small", "batch": 1, "prompt": 512, "ragged": 0.0, "gamma": 3, "new": 64, "kv_large": 0, "kv_small": 0},
        # eight users served together, prompts of unequal length
        {"name": "request_medium_b8", "kind": "request", "pair": "medium", "batch": 8, "prompt": 2048, "ragged": 0.5, "gamma": 3, "new": 32, "kv_large": 0, "kv_small": 0},
        # a 7B-class pair with grouped-query attention, two users with long prompts
        {"name": "request_large_gqa_b2", "kind": "request", "pair": "large", "batch": 2, "prompt": 4000, "ragged": 0.25, "gamma": 5, "new": 32, "kv_large": 8, "kv_small": 4},
        # four sampled responses to one prompt, ranked afterwards by the caller
        {"name": "samples_small_4", "kind": "samples", "pair": "small", "batch": 1, "samples": 4, "prompt": 300, "gamma": 3, "new": 48},
        # the adaptive block length: the host follows the router after every draft
        {"name": "adaptive_small", "kind": "adaptive", "pair": "small", "batch": 1, "prompt": 512, "gamma": 6, "new": 48},
        # time to the first token: a chat-sized prompt, and a long document on the largest pair
        {"name": "prompt_small", "kind": "prompt", "pair": "small", "batch": 1, "prompt": 512, "ragged": 0.0, "kv_large": 0, "kv_small": 0},
        {"name": "prompt_large_8k", "kind": "prompt", "pair": "large", "batch": 1, "prompt": 8192, "ragged": 0.0, "kv_large": 0, "kv_small": 0},
        # scoring held-out text of unequal length under the block-structured context
        {"name": "evaluate_small", "kind": "evaluate", "pair": "small", "batch": 4, "length": 257, "ragged": 0.5, "gamma": 4},
        # the small model's attention of one draft step: one short context, and a large batch of long ones
        {"name": "attention_1x1k", "kind": "attention", "batch": 1, "heads": 16, "d_head": 64, "derived": 1024, "own": 4},
        {"name": "attention_32x8k", "kind": "attention", "batch": 32, "heads": 16, "d_head": 64, "derived": 8191, "own": 3},
        # one block's rows of a 4096-wide model through FF_Tandem into a 1024-wide one's keys and values
        {"name": "project_4096_1024", "kind": "project", "rows": 4, "d_large": 4096, "d_small": 1024},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(exp(rng.uniform(log(lo), log(hi)))))))


def draw(rng):
    kind = rng.choice(["request", "request", "request", "samples", "adaptive", "prompt", "prompt", "evaluate", "attention", "attention", "project"])
    if kind in ("request", "prompt"):
        pair = rng.choice(["tiny", "small", "small", "medium", "large"] if kind == "request" else ["small", "medium", "large"])
        batch = _log_int(rng, 1, {"tiny": 4, "small": 8, "medium": 8, "large": 2}[pair])
        most = {"tiny": 60, "small": 8000, "medium": 16000 // batch, "large": 6000 // batch}[pair]
        case = {"kind": kind, "pair": pair, "batch": batch, "prompt": _log_int(rng, 2 if kind == "request" else 64, min(most, 8000)),
                "ragged": rng.choice([0.0, 0.25, 0.5]), "kv_large": 0, "kv_small": 0}
        if pair == "large" and rng.random() < 0.5:
            case.update(kv_large=8, kv_small=4)
        if kind == "request":
            case.update(gamma=rng.randint(2, 4 if pair == "tiny" else 7), new=_log_int(rng, 8, 24 if pair == "large" else 48))
        return case
    if kind == "samples":
        return {"kind": kind, "pair": "small", "batch": rng.randint(1, 2), "samples": rng.randint(2, 8), "prompt": _log_int(rng, 16, 2000),
                "gamma": rng.randint(2, 5), "new": _log_int(rng, 8, 48)}
    if kind == "adaptive":
        return {"kind": kind, "pair": "small", "batch": rng.randint(1, 4), "prompt": _log_int(rng, 16, 2000), "gamma": rng.randint(4, 8),
                "new": _log_int(rng, 8, 48)}
    if kind == "evaluate":
        return {"kind": kind, "pair": "small", "batch": rng.randint(1, 8), "length": _log_int(rng, 32, 400), "ragged": rng.choice([0.0, 0.5]),
                "gamma": rng.randint(2, 8)}
    if kind == "attention":
        heads, d_head = rng.choice([(8, 64), (12, 64), (16, 64), (16, 128), (32, 128)])
        batch = _log_int(rng, 1, 32)
        return {"kind": kind, "batch": batch, "heads": heads, "d_head": d_head,
                "derived": _log_int(rng, 64, min(32768, 32 * 8192 * 16 * 64 // (batch * heads * d_head))), "own": rng.randint(1, 8)}
    d_large, d_small = rng.choice([(1024, 512), (2048, 768), (4096, 1024)])
    return {"kind": kind, "rows": _log_int(rng, 1, 128), "d_large": d_large, "d_small": d_small}


# ---- inputs ------------------------------------------------------------------------------------------------------

def _shape(case):
    shape = synth.named_config(case["pair"], None if case["pair"] == "tiny" else DRAW_POS)
    if case.get("kv_large"):
        shape = replace(shape, large=replace(shape.large, n_kv_heads=case["kv_large"]), small=replace(shape.small, n_kv_heads=case["kv_small"]))
    return shape


def _weights(shape, seed, device):
    if shape.dtype == synth.DTYPE_FP32:
        weights = binding.upload_weights(shape, synth.make_weights(shape, seed), device)
    else:
        weights = synth.device_weights(shape, seed, device)
    g = torch.Generator(device=device).manual_seed(seed + 1)
    vocab = shape.large.vocab
    successor = torch.randperm(vocab, generator=g, device=device)           # the large model's successor of every token
    other = successor.clone()                                               # the small model's: another one for 1 - AGREE of them
    moved = torch.randperm(vocab, generator=g, device=device)[: int(vocab * (1 - AGREE))]
    other[moved] = successor[moved.roll(1)]
    for tag, nxt in (("L", successor), ("S", other)):
        emb = weights[tag + ".emb"]
        weights[tag + ".emb"] = torch.randn(emb.shape, generator=g, device=device).mul_(EMB_STD).to(emb.dtype)
        weights[tag + ".w_out"] = weights[tag + ".emb"][torch.argsort(nxt)] * (0.02 / EMB_STD)
    return weights


def _lengths(case, key):
    """Sequence b gets up to `ragged` of the length less than the first one, in even steps."""
    n, b = case[key], case["batch"]
    return [max(2, n - int(n * case.get("ragged", 0.0) * i / max(1, b - 1))) for i in range(b)]


def _caches(t, lens):
    """The keys and values that a pass leaves for each sequence's first len positions: the state that the next call starts
    from.  Both models' caches lie at the start of the context's arena, [layer][K | V][sequence][head][position][element]."""
    out, off = [], 0
    for d in (t.shape.large, t.shape.small):
        dims = (d.n_layers, 2, t.max_batch, d.kv_heads, t.max_seq, d.d_head)
        store = torch.bfloat16 if t.shape.dtype == synth.DTYPE_BF16 else torch.float32
        size = store.itemsize
        for n in dims:
            size *= n
        cache = t.arena[off:off + size].view(store).view(dims)
        out += [cache[:, :, b, :, :n] for b, n in enumerate(lens)]
        off += (size + 255) // 256 * 256
    return out


def prepare(case, seed):
    kind, device = case["kind"], torch.device("cuda", torch.cuda.current_device())
    s = {"kind": kind, "case": case}
    if kind in ("attention", "project"):
        g = torch.Generator(device=device).manual_seed(seed)
        rn = lambda *n: torch.randn(n, generator=g, device=device).to(torch.bfloat16)  # noqa: E731
        if kind == "attention":
            b, h, dh = case["batch"], case["heads"], case["d_head"]
            s["args"] = [rn(b, h, dh)] + [rn(b, h, n, dh) for n in (case["derived"], case["derived"], case["own"], case["own"])]
            s["out"] = torch.empty_like(s["args"][0])
            s["scratch"] = torch.empty(binding.load_library().tandem_decode_attention_scratch_bytes(b, h, dh, case["derived"], case["own"]),
                                       dtype=torch.uint8, device=device)
        else:
            d_l, d_s, rows = case["d_large"], case["d_small"], case["rows"]
            w_t, wk, wv = (rn(d_s, k) * 0.02 for k in (d_l, d_s, d_s))
            s["args"] = [rn(rows, d_l), w_t, torch.ones(d_s, device=device), torch.zeros(d_s, device=device), wk, wv]
            s["scratch"] = torch.empty(binding.load_library().tandem_ff_tandem_project_scratch_bytes(rows, d_s), dtype=torch.uint8, device=device)
        return s
    shape = _shape(case)
    lens = _lengths(case, "length" if kind == "evaluate" else "prompt")
    new, samples = case.get("new", 0), case.get("samples", 1)
    gamma = case.get("gamma", 1)
    t = binding.Tandem(shape, _weights(shape, seed, device), max_batch=case["batch"] * samples, max_seq=max(lens) + new + gamma + 1,
                       gamma_max=gamma, max_prefill_rows=sum(lens))
    s["t"] = t
    s["prompts"] = synth.make_prompts(case["batch"], lens, shape.large.vocab, seed)
    s["seed"] = seed
    if kind == "samples":
        t.tandem_set_sampling(0.25, 0.25)     # cold enough for ranked answers
    if kind == "adaptive":
        t.tandem_set_router(synth.make_router(shape, ROUTER_K, ROUTER_HIDDEN, seed), ROUTER_TAU)
    if kind != "evaluate":
        s["caches"] = _caches(t, [n + new - 1 for n in lens for _ in range(samples)])
    return s


def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "attention":
        return binding.tandem_decode_attention(*s["args"], s["out"], s["scratch"])
    if kind == "project":
        return binding.tandem_ff_tandem_project(*s["args"], s["scratch"])
    t = s["t"]
    if kind == "evaluate":
        return t.tandem_teacher_forced_forward(s["prompts"], case["gamma"])
    if kind == "samples":
        t.tandem_prefill_samples(s["prompts"], case["samples"])
        ids, lens, _ = t.tandem_speculative_generate(case["gamma"], case["new"], binding.ACCEPT_SAMPLE, s["seed"])
        return {"ids": ids, "lens": lens, "caches": s["caches"]}
    t.tandem_prefill(s["prompts"])
    if kind == "prompt":
        return {"caches": s["caches"]}
    if kind == "adaptive":
        ids, lens, _ = t.tandem_adaptive_generate(case["gamma"], case["new"])
    else:
        ids, lens, _ = t.tandem_speculative_generate(case["gamma"], case["new"])
    return {"ids": ids, "lens": lens, "caches": s["caches"]}


# ---- what a pass cannot do without -------------------------------------------------------------------------------

def _params(d, head):
    return d.n_layers * (2 * d.d_model ** 2 + 2 * d.d_model * d.d_kv + 2 * d.d_model * d.d_ff) + (d.d_model * d.vocab if head else 0)


def _proj_params(shape):
    L, S = shape.large, shape.small
    hid = shape.hidden
    one = S.d_model * L.d_model if shape.ff_tandem_kind == synth.FF_TANDEM_LINEAR else hid * L.d_model + S.d_model * hid
    return S.n_layers * (one + 2 * S.d_model * S.d_kv)


def _prompt_work(shape, lens, copies=1):
    """Weights once, the rows through them, causal attention, both caches written (`copies` times)."""
    L, S, size = shape.large, shape.small, 2 if shape.dtype == synth.DTYPE_BF16 else 4
    rows = sum(n - 1 for n in lens)
    params = _params(L, False) + _proj_params(shape)
    kv = rows * 2 * (L.n_layers * L.d_kv + S.n_layers * S.d_kv)
    flops = 2.0 * params * rows + L.n_layers * 2.0 * L.d_model * sum(float(n - 1) ** 2 for n in lens)
    return size * (params + rows * L.d_model + copies * kv), flops


def _round_work(shape, gamma, contexts, head=True):
    """gamma draft steps and one block pass: every weight once per pass, both caches read once per pass."""
    L, S, size = shape.large, shape.small, 2 if shape.dtype == synth.DTYPE_BF16 else 4
    ctx, b = float(sum(contexts)), len(contexts)
    byt = size * (_params(L, head) + gamma * _params(S, True) + _proj_params(shape) + ctx * 2 * (L.n_layers * L.d_kv + gamma * S.n_layers * S.d_kv))
    rows = b * (gamma + (1 if head else 0))
    flops = 2.0 * (rows * (_params(L, head) + _proj_params(shape)) + b * gamma * _params(S, True))
    flops += 4.0 * ctx * ((gamma + 1) * L.n_layers * L.d_model + gamma * S.n_layers * S.d_model)
    return byt, flops


def work(case):
    kind = case["kind"]
    if kind == "attention":
        b, h, dh, n = case["batch"], case["heads"], case["d_head"], case["derived"] + case["own"]
        return {"bytes": 2 * (2 * b * h * n * dh + 2 * b * h * dh), "flops": 4.0 * b * h * n * dh}
    if kind == "project":
        r, d_l, d_s = case["rows"], case["d_large"], case["d_small"]
        return {"bytes": 2 * (d_s * d_l + 2 * d_s * d_s + r * (d_l + 2 * d_s)), "flops": 2.0 * r * (d_s * d_l + 2 * d_s * d_s)}
    shape = _shape(case)
    lens = _lengths(case, "length" if kind == "evaluate" else "prompt")
    if kind == "evaluate":
        rounds = -(-(max(lens) - 1) // case["gamma"])
        byt, flops = _round_work(shape, case["gamma"], [n / 2 for n in lens], head=False)
        return {"bytes": rounds * byt, "flops": rounds * flops}
    samples = case.get("samples", 1)
    byt, flops = _prompt_work(shape, lens, samples)
    if kind != "prompt":
        # tokens that a round keeps: the drafts up to the first disagreement and the large model's own; the router lets
        # about two drafts through
        gamma = 2 if kind == "adaptive" else case["gamma"]
        rounds = case["new"] / ((1 - AGREE ** (gamma + 1)) / (1 - AGREE))
        b, f = _round_work(shape, gamma, [n + case["new"] / 2 for n in lens for _ in range(samples)])
        byt, flops = byt + rounds * b, flops + rounds * f
    return {"bytes": byt, "flops": flops}


def tolerance(case):
    if case["kind"] in ("attention", "project"):
        return {"rel": 5e-3}                  # bf16 results
    if case.get("pair") == "tiny":
        return {"rel": 2e-5}                  # fp32 sums in another order; token ids the same
    if case["kind"] == "evaluate":
        return {"rel": 2e-3, "differ": 2e-3}  # fp32 scores of bf16 keys and values; a near tie may flip a rank-1 token
    return {"rel": 1e-2}                      # bf16 keys and values; token ids the same
