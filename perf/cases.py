"""What this library is timed on: the calls that a program serving task-routed speculative decoding makes.

A case is one of six kinds of work:

  iterate   one iteration of the decoding loop in steady state: the routed drafts propose gamma tokens for every sequence, the target
            scores them in one pass, the accept rule runs.  The commit (three integers per sequence) is left out so that a pass can be
            repeated on the same context; `request` and `first` include it.
  first     a request up to its first tokens: prompts in, routing, prefill of target and drafts, one full iteration, tokens out.
  request   a whole request: as `first`, then iterations until the wanted number of tokens is there, each iteration's count of
            accepted tokens read back as a program that streams its answer does.
  decode    plain autoregressive decoding of the target, the baseline that the method is compared with.
  classify  the Mamba prompt classifier over a batch of prompts.
  cluster   one K-means step of the offline task partitioning.

Model shapes are those of `synth.CONFIGS`.  Weights are random, with the residual stream balanced between the token's embedding and the
layers, and with an output matrix that makes one next token stand out at every position, as a trained model's does on text that it
knows; the draft names another token than the target for one token in five, so iterations accept some and reject some.  Sharp
distributions also make the tokens comparable between two correct implementations: with near-flat ones any rounding moves the draw.
"""
import math

import numpy as np
import torch

from paper_2505_08600_b200 import binding, synth

DEV = "cuda:0"
LORA = dict(adapters=4, rank=16, scale=2.0)
DISAGREE = 0.2                       # share of tokens after which draft and target name different successors
MAX_CTX = {"tiny": 128, "1b": 512, "7b": 2048, "13b": 8192}


def listed():
    return [
        # the smallest call: launch latency of the fp32 path
        dict(name="tiny_f32_iterate", kind="iterate", model="tiny", batch=1, ctx_lo=32, ctx_hi=32, gamma=4, temperature=1.0, adapters=False),
        # one chat with the small target: latency of many small kernels
        dict(name="1b_iterate", kind="iterate", model="1b", batch=1, ctx_lo=128, ctx_hi=128, gamma=5, temperature=0.7, adapters=False),
        # the headline configuration: one sequence on the 7B target
        dict(name="7b_iterate", kind="iterate", model="7b", batch=1, ctx_lo=512, ctx_hi=512, gamma=5, temperature=1.0, adapters=False),
        # a loaded server: ragged contexts, four task-specific drafts at once
        dict(name="7b_batch16_iterate", kind="iterate", model="7b", batch=16, ctx_lo=256, ctx_hi=1024, gamma=5, temperature=1.0, adapters=False),
        # drafts as adapters of one base model, an odd batch, greedy
        dict(name="7b_lora_iterate", kind="iterate", model="7b", batch=5, ctx_lo=131, ctx_hi=777, gamma=3, temperature=0.0, adapters=True),
        # the largest: long documents on the 13B target, deep drafts
        dict(name="13b_long_iterate", kind="iterate", model="13b", batch=2, ctx_lo=7601, ctx_hi=8100, gamma=8, temperature=1.0, adapters=False),
        # time to the first tokens of a 512-token prompt
        dict(name="7b_first", kind="first", model="7b", batch=1, ctx_lo=512, ctx_hi=512, gamma=5, temperature=1.0, classifier=False),
        # several short ragged prompts at once, routed by the library's own classifier
        dict(name="1b_first_batch5", kind="first", model="1b", batch=5, ctx_lo=37, ctx_hi=480, gamma=5, temperature=0.7, classifier=True),
        # a whole short answer
        dict(name="1b_request", kind="request", model="1b", batch=1, ctx_lo=128, ctx_hi=128, gamma=5, temperature=0.7, classifier=True, new_tokens=128),
        # plain decoding of three sequences
        dict(name="7b_decode3", kind="decode", model="7b", batch=3, ctx_lo=200, ctx_hi=900, temperature=1.0),
        # routing a day's queue of prompts
        dict(name="classify_400", kind="classify", prompts=400, len_lo=32, len_hi=512, classes=4),
        # partitioning a corpus of sentence vectors
        dict(name="cluster_2m", kind="cluster", n=2_000_003, dim=384, k=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["iterate", "iterate", "iterate", "first", "request", "decode", "classify", "cluster"])
    if kind == "classify":
        lo = _log(rng, 4, 200)
        return dict(kind=kind, prompts=_log(rng, 1, 400), len_lo=lo, len_hi=lo + rng.randint(0, 300), classes=rng.randint(2, 6))
    if kind == "cluster":
        return dict(kind=kind, n=_log(rng, 3000, 2_000_000), dim=rng.choice([128, 256, 384, 384, 512]), k=rng.randint(2, 8))
    if kind == "request":
        p = _log(rng, 16, 256)
        return dict(kind=kind, model="1b", batch=1, ctx_lo=p, ctx_hi=p, gamma=rng.randint(2, 7), temperature=rng.choice([0.0, 0.7, 1.0]),
                    classifier=bool(rng.randint(0, 1)), new_tokens=_log(rng, 12, 100))
    model = rng.choice(["1b", "7b"] if kind == "first" else ["tiny", "1b", "1b", "7b", "7b", "13b"] if kind == "iterate" else ["1b", "7b"])
    top = {"tiny": 64, "1b": 460, "7b": 1500, "13b": 8000}[model]
    batch = 1 if model == "tiny" else _log(rng, 1, {"first": 4, "iterate": 2 if model == "13b" else 16, "decode": 16}[kind])
    hi = _log(rng, 20, top)
    if kind == "first" and model == "7b":
        hi = max(20, min(hi, 1000 // batch))
    case = dict(kind=kind, model=model, batch=batch, ctx_lo=rng.randint(max(8, hi // 2), hi), ctx_hi=hi, temperature=rng.choice([0.0, 0.7, 1.0]))
    if kind != "decode":
        case["gamma"] = rng.randint(1, 4) if model == "tiny" else rng.randint(1, 9)
    if kind == "iterate":
        case["adapters"] = model == "7b" and rng.random() < 0.3
    elif kind == "first":
        case["classifier"] = bool(rng.randint(0, 1))
    return case


# ------------------------------------------------------------------------------------------- inputs
def _lengths(case):
    """Context (or prompt) lengths: spread evenly over the case's range, in a mixed order."""
    n, lo, hi = case["batch"], case["ctx_lo"], case["ctx_hi"]
    order = list(range(0, n, 2)) + list(range(1, n, 2))[::-1]
    return [hi] if n == 1 else [lo + (hi - lo) * j // (n - 1) for j in order]


def _models(case):
    cfg = synth.CONFIGS[case["model"]]
    return cfg["dtype"], cfg["target"], cfg["drafts"][:1] if case.get("adapters") else cfg["drafts"], cfg["classifier"]


def _task(case, i):
    return i % (LORA["adapters"] if case.get("adapters") else len(_models(case)[2]))


def _load_model(ctx, model_id, dims, dtype, g, successor):
    td = torch.bfloat16 if dtype == "bf16" else torch.float32

    def normal(shape, std):
        return torch.randn(shape, generator=g, device=DEV, dtype=td).mul_(std)

    embed = normal((dims["vocab"], dims["d_model"]), 1.0)
    lm_head = torch.empty_like(embed)
    lm_head[successor] = embed * max(0.02, 40.0 / dims["d_model"])
    ones = torch.ones(dims["d_model"], device=DEV, dtype=torch.float32)
    ctx.sd_load_tensor(model_id, binding.T_EMBED, 0, embed)
    ctx.sd_load_tensor(model_id, binding.T_LM_HEAD, 0, lm_head)
    ctx.sd_load_tensor(model_id, binding.T_FINAL_NORM, 0, ones)
    out_std = 0.02 / math.sqrt(2 * dims["n_layers"])
    shapes = synth.mat_shapes(dims)
    for l in range(dims["n_layers"]):
        for name in synth.LAYER_MATS:
            ctx.sd_load_tensor(model_id, binding.TENSOR_KIND[name], l, normal(shapes[name], out_std if name in ("wo", "wd") else 0.02))
        ctx.sd_load_tensor(model_id, binding.T_NORM1, l, ones)
        ctx.sd_load_tensor(model_id, binding.T_NORM2, l, ones)


def _load_adapters(ctx, dims, g):
    d, F, r = dims["d_model"], dims["d_ffn"], LORA["rank"]
    dq, dkv = dims["n_heads"] * dims["head_dim"], dims["n_kv_heads"] * dims["head_dim"]
    shapes = [(dq + 2 * dkv, d), (d, dq), (2 * F, d), (d, F)]
    for a in range(LORA["adapters"]):
        for l in range(dims["n_layers"]):
            for mat, (n_out, n_in) in enumerate(shapes):
                ab = [torch.randn(s, generator=g, device=DEV, dtype=torch.bfloat16).mul_(0.05) for s in ((r, n_in), (n_out, r))]
                ctx.sd_load_lora(a, l, mat, *ab)


def _context(case, seed, g):
    dtype, target, drafts, clf = _models(case)
    lora = dict(lora_adapters=LORA["adapters"], lora_rank=LORA["rank"], lora_scale=LORA["scale"]) if case.get("adapters") else {}
    gamma = case.get("gamma", 1)
    ctx = binding.Context(target, drafts, dtype, case["batch"], MAX_CTX[case["model"]], gamma, case["temperature"], seed,
                          clf_d_hidden=clf[1] if case.get("classifier") else 0, device=DEV, **lora)
    V = target["vocab"]
    successor = torch.randperm(V, generator=g, device=DEV)
    _load_model(ctx, 0, target, dtype, g, successor)
    for k, dims in enumerate(drafts):
        other = torch.randperm(V, generator=g, device=DEV)[: int(DISAGREE * V)]
        s = successor.clone()
        s[other] = successor[other.roll(1)]
        _load_model(ctx, 1 + k, dims, dtype, g, s)
    if case.get("adapters"):
        _load_adapters(ctx, drafts[0], g)
    if case.get("classifier"):
        c = synth.make_classifier(*clf, seed=seed)
        ctx.sd_load_classifier(c["w1"], c["b1"], c["w2"], c["b2"])
    return ctx, V


_streams = []


def _stream():
    """The one stream of the serving process: the library replays captured graphs, which the default stream does not allow."""
    if not _streams:
        _streams.append(torch.cuda.Stream())
    return _streams[0]


def prepare(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    if case["kind"] == "classify":
        rng = np.random.default_rng(seed)
        vocab = 21128
        lens = rng.integers(case["len_lo"], case["len_hi"] + 1, size=case["prompts"]).astype(np.int32)
        starts = np.concatenate([[0], np.cumsum(lens)[:-1]]).astype(np.int64)
        tokens = torch.randint(0, vocab, (int(lens.sum()),), generator=g, device=DEV, dtype=torch.int32)
        clf = binding.MambaClassifier(synth.make_mamba_classifier(vocab, n_classes=case["classes"], seed=seed), DEV)
        return dict(case=case, clf=clf, tokens=tokens, starts=starts, lens=lens)
    if case["kind"] == "cluster":
        n, dim, k = case["n"], case["dim"], case["k"]
        centers = torch.nn.functional.normalize(torch.randn((k, dim), generator=g, device=DEV), dim=1)
        x = torch.randn((n, dim), generator=g, device=DEV).mul_(0.6 / math.sqrt(dim))
        x += centers[torch.randint(0, k, (n,), generator=g, device=DEV)]
        x /= x.norm(dim=1, keepdim=True)
        start = centers + 0.2 / math.sqrt(dim) * torch.randn((k, dim), generator=g, device=DEV)      # an iteration on the way
        return dict(case=case, points=x, centroids=start.contiguous(), labels=torch.empty(n, dtype=torch.int32, device=DEV),
                    out=torch.empty((k, dim), device=DEV), counts=torch.empty(k, dtype=torch.int64, device=DEV),
                    inertia=torch.empty(1, dtype=torch.float64, device=DEV))
    with torch.cuda.stream(_stream()):
        ctx, V = _context(case, seed, g)
        n, gamma = case["batch"], case.get("gamma", 0)
        prompts = [torch.randint(0, V, (m,), generator=g, device=DEV, dtype=torch.int32).cpu().numpy() for m in _lengths(case)]
        s = dict(case=case, ctx=ctx, seqs=list(range(n)), prompts=prompts, tasks=[_task(case, i) for i in range(n)],
                 logits=torch.empty((n, gamma + 1, V), device=DEV))
        if case["kind"] != "decode":
            s.update(x=torch.empty((n, gamma), dtype=torch.int32, device=DEV), q=torch.empty((n, gamma, V), device=DEV),
                     n_acc=torch.empty(n, dtype=torch.int32, device=DEV), out_tok=torch.empty((n, gamma + 1), dtype=torch.int32, device=DEV))
        if case["kind"] in ("iterate", "decode"):
            _begin(s)
    torch.cuda.synchronize()
    return s


# ------------------------------------------------------------------------------------------- one pass
def _begin(s):
    ctx, seqs = s["ctx"], s["seqs"]
    for i, p in zip(seqs, s["prompts"]):
        ctx.sd_seq_begin(i, p)
    ctx.sd_route_prompt(seqs, None if s["case"].get("classifier") else s["tasks"])
    ctx.sd_prefill(seqs)


def _step(s):
    ctx, seqs, gamma = s["ctx"], s["seqs"], s["case"]["gamma"]
    ctx.sd_draft_steps(seqs, gamma, s["x"], s["q"])
    ctx.sd_verify_accept(seqs, gamma, s["x"], s["q"], s["logits"], s["n_acc"], s["out_tok"])


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "classify":
        return s["clf"].classify(s["tokens"], s["starts"], s["lens"])
    if kind == "cluster":
        binding.sd_kmeans_step(s["points"], s["centroids"], s["labels"], s["out"], s["counts"], s["inertia"])
        return s["labels"], s["out"], s["counts"], s["inertia"]
    ctx, seqs = s["ctx"], s["seqs"]
    with torch.cuda.stream(_stream()):
        if kind == "decode":
            ctx.sd_target_step(seqs, s["logits"])
            return s["logits"]
        if kind == "iterate":
            gamma = case["gamma"]
            ctx.sd_draft_steps(seqs, gamma, s["x"], s["q"])
            ctx.sd_verify(seqs, gamma, s["x"], s["logits"])
            ctx.sd_accept_seqs(seqs, gamma, s["logits"], s["q"], s["x"], s["n_acc"], s["out_tok"])
            return s["x"], s["q"], s["logits"], s["n_acc"], s["out_tok"]
        _begin(s)
        _step(s)
        if kind == "first":
            return s["x"], s["q"], s["logits"], s["n_acc"], s["out_tok"]
        have = int(s["n_acc"].cpu()[0]) + 1
        while have < case["new_tokens"]:
            _step(s)
            have += int(s["n_acc"].cpu()[0]) + 1
        tokens, _ = ctx.sd_seq_read(0)
        return tokens[: case["ctx_hi"] + case["new_tokens"]], s["x"], s["q"], s["logits"], s["n_acc"], s["out_tok"]


# ------------------------------------------------------------------------------------------- what a pass cannot do without
def _params(d, lm_head=True):
    per_layer = sum(a * b for a, b in synth.mat_shapes(d).values())
    return d["n_layers"] * per_layer + (d["vocab"] * d["d_model"] if lm_head else 0)


def _kv(d):                                              # values of one cached position
    return 2 * d["n_layers"] * d["n_kv_heads"] * d["head_dim"]


def _scored(d):                                          # multiply-adds of one query row against one cached position
    return 2 * d["n_layers"] * d["n_heads"] * d["head_dim"]


def work(case):
    if case["kind"] == "cluster":
        n, dim, k = case["n"], case["dim"], case["k"]
        return dict(bytes=4.0 * n * (dim + 1) + 8.0 * k * dim, flops=n * dim * (3.0 * k + 1))
    if case["kind"] == "classify":
        D, Di, N, R = 128, 256, 16, 8
        T = case["prompts"] * (case["len_lo"] + case["len_hi"]) / 2
        per_token = 2 * (2 * Di * D + 4 * Di + (R + 2 * N) * Di + Di * R) + 6 * Di * N
        return dict(bytes=4.0 * (T + min(T, 21128) * D + 2 * Di * D + (R + 2 * N) * Di + 2 * Di * (N + R) + Di * D), flops=T * per_token)
    dtype, target, drafts, _ = _models(case)
    esz = 2 if dtype == "bf16" else 4
    lens, n, gamma, V = _lengths(case), case["batch"], case.get("gamma", 0), target["vocab"]

    def passes(d, rows, ctxs, lm_head=True):             # one pass of a model: its weights once, the caches once
        return (esz * (_params(d, lm_head) + _kv(d) * sum(ctxs)), 2.0 * (_params(d, lm_head) * rows * len(ctxs) + _scored(d) * rows * sum(ctxs)))

    def step():
        b, f = passes(target, gamma + 1, lens)
        groups = {}
        for i in range(n):
            groups.setdefault(0 if case.get("adapters") else _task(case, i), []).append(lens[i])
        for k, ctxs in groups.items() if gamma else ():
            db, df = passes(drafts[k], 1, ctxs)
            b, f = b + gamma * db, f + gamma * df
        return b + 4.0 * n * V * (2 * gamma + 1), f

    b, f = step()
    if case["kind"] == "first":
        groups = {0: (target, lens)}
        for i in range(n):
            groups.setdefault(1 + _task(case, i), (drafts[_task(case, i)], []))[1].append(lens[i])
        for d, ctxs in groups.values():
            b += esz * (_params(d, False) + _kv(d) * sum(ctxs))
            f += 2.0 * _params(d, False) * sum(ctxs) + _scored(d) * sum(m * m for m in ctxs)
    if case["kind"] == "request":
        steps = case["new_tokens"] / (1 + gamma * 0.6)
        b, f = b * steps, f * steps
    return dict(bytes=b, flops=f)


def tolerance(case):
    # Logits of the tensor-core kernels against the plain CUDA-core ones on the same weights (other order of sums, activations
    # rounded at other places): rel 0.0024 (1b) ... 0.0067 (7b, batch 16); tokens, accepted counts and labels are the same.
    if case["kind"] == "cluster":
        return dict(rel=1e-5, differ=1e-5)
    if case["kind"] == "classify":
        return dict(rel=2e-5)
    return dict(rel=2e-5) if case["model"] == "tiny" else dict(rel=2e-2)
