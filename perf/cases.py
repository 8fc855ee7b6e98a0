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
MAMBA_VOCAB = 21128
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


def _load_model(ctx, model_id, dims, dtype, g, successor):         # ctx: a context, or whatever else takes tensors (exact)
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


def _fill(ctx, case, g):
    """Random weights of the case's models (and adapters) into ctx, drawn from g in a fixed order; the vocabulary's size."""
    dtype, target, drafts, _ = _models(case)
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
    return V


def _context(case, seed, g):
    dtype, target, drafts, clf = _models(case)
    lora = dict(lora_adapters=LORA["adapters"], lora_rank=LORA["rank"], lora_scale=LORA["scale"]) if case.get("adapters") else {}
    gamma = case.get("gamma", 1)
    ctx = binding.Context(target, drafts, dtype, case["batch"], MAX_CTX[case["model"]], gamma, case["temperature"], seed,
                          clf_d_hidden=clf[1] if case.get("classifier") else 0, device=DEV, **lora)
    V = _fill(ctx, case, g)
    if case.get("classifier"):
        c = synth.make_classifier(*clf, seed=seed)
        ctx.sd_load_classifier(c["w1"], c["b1"], c["w2"], c["b2"])
    return ctx, V


def _prompts(case, V, g):
    return [torch.randint(0, V, (m,), generator=g, device=DEV, dtype=torch.int32).cpu().numpy() for m in _lengths(case)]


def _queue(case, seed, g):
    """The classifier's prompts: token ids one prompt after the other, and where each begins and how long it is."""
    lens = np.random.default_rng(seed).integers(case["len_lo"], case["len_hi"] + 1, size=case["prompts"]).astype(np.int32)
    starts = np.concatenate([[0], np.cumsum(lens)[:-1]]).astype(np.int64)
    return torch.randint(0, MAMBA_VOCAB, (int(lens.sum()),), generator=g, device=DEV, dtype=torch.int32), starts, lens


def _corpus(case, g):
    """Sentence vectors in overlapping groups, and centroids as an iteration on the way has them."""
    n, dim, k = case["n"], case["dim"], case["k"]
    centers = torch.nn.functional.normalize(torch.randn((k, dim), generator=g, device=DEV), dim=1)
    x = torch.randn((n, dim), generator=g, device=DEV).mul_(0.6 / math.sqrt(dim))
    x += centers[torch.randint(0, k, (n,), generator=g, device=DEV)]
    x /= x.norm(dim=1, keepdim=True)
    return x, (centers + 0.2 / math.sqrt(dim) * torch.randn((k, dim), generator=g, device=DEV)).contiguous()


def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    return g


_streams = []


def _stream():
    """The one stream of the serving process: the library replays captured graphs, which the default stream does not allow."""
    if not _streams:
        _streams.append(torch.cuda.Stream())
    return _streams[0]


def prepare(case, seed):
    g = _generator(seed)
    if case["kind"] == "classify":
        tokens, starts, lens = _queue(case, seed, g)
        clf = binding.MambaClassifier(synth.make_mamba_classifier(MAMBA_VOCAB, n_classes=case["classes"], seed=seed), DEV)
        return dict(case=case, clf=clf, tokens=tokens, starts=starts, lens=lens)
    if case["kind"] == "cluster":
        x, centroids = _corpus(case, g)
        n, dim, k = case["n"], case["dim"], case["k"]
        return dict(case=case, points=x, centroids=centroids, labels=torch.empty(n, dtype=torch.int32, device=DEV),
                    out=torch.empty((k, dim), device=DEV), counts=torch.empty(k, dtype=torch.int64, device=DEV),
                    inertia=torch.empty(1, dtype=torch.float64, device=DEV))
    with torch.cuda.stream(_stream()):
        ctx, V = _context(case, seed, g)
        n, gamma = case["batch"], case.get("gamma", 0)
        s = dict(case=case, ctx=ctx, seqs=list(range(n)), prompts=_prompts(case, V, g), tasks=[_task(case, i) for i in range(n)],
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
        return dict(bytes=4.0 * (T + min(T, MAMBA_VOCAB) * D + 2 * Di * D + (R + 2 * N) * Di + 2 * Di * (N + R) + Di * D), flops=T * per_token)
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


# ------------------------------------------------------------------------------------------- the same in 64 bits
class _Weights:
    """Takes the tensors that a context would, and keeps them."""

    def __init__(self):
        self.tensors, self.lora = {}, {}

    def sd_load_tensor(self, model, kind, layer, tensor):
        self.tensors[model, kind, layer] = tensor

    def sd_load_lora(self, adapter, layer, mat, a, b):
        self.lora[adapter, layer, mat] = (a, b)


def _norm(h):                                            # all norm gains are 1
    return h * torch.rsqrt((h * h).mean(-1, keepdim=True) + 1e-5)


class _Model64:
    """One sequence's view of a model: weights as given, arithmetic and cache in 64 bits."""

    def __init__(self, w, model, dims, adapter=None):
        self.w, self.model, self.d, self.adapter, self.n = w, model, dims, adapter, 0
        self.k, self.v = ([None] * dims["n_layers"] for _ in range(2))

    def _mats(self, layer, names, mat):
        m = torch.cat([self.w.tensors[self.model, binding.TENSOR_KIND[name], layer].double() for name in names])
        if self.adapter is not None:
            a, b = self.w.lora[self.adapter, layer, mat]
            m += LORA["scale"] * (b.double() @ a.double())
        return m

    def __call__(self, tokens, lm_head=True):
        """Logits of the rows (or None) after `tokens` are appended to the first self.n positions."""
        d, n0, rows = self.d, self.n, len(tokens)
        H, Hkv, hd, F = d["n_heads"], d["n_kv_heads"], d["head_dim"], d["d_ffn"]
        h = self.w.tensors[self.model, binding.T_EMBED, 0][torch.as_tensor(tokens, device=DEV).long()].double()
        pos = torch.arange(n0, n0 + rows, device=DEV, dtype=torch.float64)
        ang = pos[:, None] * 10000.0 ** (-torch.arange(0, hd, 2, device=DEV, dtype=torch.float64) / hd)
        cos, sin = ang.cos()[:, None], ang.sin()[:, None]

        def rope(x):
            a, b = x[..., : hd // 2], x[..., hd // 2:]
            return torch.cat([a * cos - b * sin, a * sin + b * cos], -1)

        mask = torch.arange(n0 + rows, device=DEV)[None] > torch.arange(n0, n0 + rows, device=DEV)[:, None]
        for l in range(d["n_layers"]):
            qkv = (_norm(h) @ self._mats(l, ("wq", "wk", "wv"), 0).T).view(rows, H + 2 * Hkv, hd)
            q, k, v = rope(qkv[:, :H]), rope(qkv[:, H: H + Hkv]), qkv[:, H + Hkv:]
            if self.k[l] is not None:
                k, v = torch.cat([self.k[l][:n0], k]), torch.cat([self.v[l][:n0], v])
            self.k[l], self.v[l] = k, v
            att = torch.empty_like(q)
            for j in range(Hkv):
                mine = slice(j * (H // Hkv), (j + 1) * (H // Hkv))
                s = (q[:, mine].transpose(0, 1) @ k[:, j].T / math.sqrt(hd)).masked_fill(mask, -math.inf)
                att[:, mine] = (s.softmax(-1) @ v[:, j]).transpose(0, 1)
            h = h + att.reshape(rows, H * hd) @ self._mats(l, ("wo",), 1).T
            gu = _norm(h) @ self._mats(l, ("wg", "wu"), 2).T
            h = h + (torch.nn.functional.silu(gu[:, :F]) * gu[:, F:]) @ self._mats(l, ("wd",), 3).T
        self.n = n0 + rows
        return _norm(h) @ self.w.tensors[self.model, binding.T_LM_HEAD, 0].double().T if lm_head else None


def _exact_cluster(case, g):
    x, c = (t.double() for t in _corpus(case, g))
    d2 = torch.stack([((x - ck) ** 2).sum(1) for ck in c], 1)
    near, labels = d2.min(1)
    counts = torch.bincount(labels, minlength=len(c))
    out = torch.stack([x[labels == k].mean(0) if counts[k] else c[k] for k in range(len(c))])
    return labels.int(), out, counts, near.sum()[None]


def _exact_classify(case, seed, g):
    tokens, starts, lens = _queue(case, seed, g)
    w = {k: torch.from_numpy(a).to(DEV).double() for k, a in
         synth.make_mamba_classifier(MAMBA_VOCAB, n_classes=case["classes"], seed=seed).items()}
    n, top, (Di, R), N, taps = len(lens), int(lens.max()), w["w_dt"].shape, w["a_log"].shape[1], w["w_conv"].shape[1]
    ids = torch.zeros((n, top), dtype=torch.long, device=DEV)
    for i, (a, m) in enumerate(zip(starts, lens)):
        ids[i, :m] = tokens[a: a + m]
    last = torch.from_numpy(lens).to(DEV)
    before = torch.zeros((n, taps, Di), dtype=torch.float64, device=DEV)
    state, total = torch.zeros((n, Di, N), dtype=torch.float64, device=DEV), torch.zeros((n, Di), dtype=torch.float64, device=DEV)
    A, silu = -w["a_log"].exp(), torch.nn.functional.silu
    for t in range(top):
        u, z = (w["embed"][ids[:, t]] @ w["w_in"].T).split(Di, 1)
        before = torch.cat([before[:, 1:], u[:, None]], 1)
        v = silu(w["b_conv"] + (before * w["w_conv"].T).sum(1))
        r, B, C = (v @ w["w_x"].T).split([R, N, N], 1)
        dt = torch.nn.functional.softplus(r @ w["w_dt"].T + w["b_dt"])
        state = (dt[:, :, None] * A).exp() * state + (dt * v)[:, :, None] * B[:, None]
        total += (((state * C[:, None]).sum(2) + w["d_skip"] * v) * silu(z)) * (t < last)[:, None]
    scores = (total @ w["w_out"].T / last[:, None]) @ w["w_fc"].T + w["b_fc"]
    return scores, scores.argmax(1).int()


def exact(case, seed):
    """What run() returns, in 64 bits.  One token stands out at every position, so every draw is the most probable one."""
    g = _generator(seed)
    if case["kind"] == "cluster":
        return _exact_cluster(case, g)
    if case["kind"] == "classify":
        return _exact_classify(case, seed, g)
    _, target, drafts, clf = _models(case)
    lens, n, T = _lengths(case), case["batch"], case["temperature"]
    if 2.0 * _params(target, False) * sum(lens) > 1.5e14:                 # too long at the rate of 64-bit sums
        return None
    w = _Weights()
    with torch.cuda.stream(_stream()):
        V = _fill(w, case, g)
        texts = [list(map(int, p)) for p in _prompts(case, V, g)]
    torch.cuda.synchronize()
    classifier = {k: torch.from_numpy(a).to(DEV).double() for k, a in synth.make_classifier(*clf, seed=seed).items()}
    gamma = case.get("gamma", 0)
    logits = torch.empty((n, gamma + 1, V), dtype=torch.float64, device=DEV)
    q = torch.empty((n, gamma, V), dtype=torch.float64, device=DEV)
    x = torch.empty((n, gamma), dtype=torch.int32)
    n_acc, out_tok = torch.empty(n, dtype=torch.int32), torch.full((n, gamma + 1), -1, dtype=torch.int32)
    for i, text in enumerate(texts):
        task = _task(case, i)
        if case.get("classifier"):
            mean = w.tensors[0, binding.T_EMBED, 0][torch.tensor(text, device=DEV)].double().mean(0)
            task = int((classifier["w2"] @ torch.relu(classifier["w1"] @ mean + classifier["b1"]) + classifier["b2"]).argmax())
        model = _Model64(w, 0, target)
        model(text[:-1], lm_head=False)
        if case["kind"] == "decode":
            logits[i] = model(text[-1:])
            continue
        draft = _Model64(w, 1, drafts[0], task) if case.get("adapters") else _Model64(w, 1 + task, drafts[task])
        wanted, have = case.get("new_tokens", 1), 0
        while have < wanted:
            drawn = []
            for s in range(gamma):
                row = draft((text + drawn)[draft.n:])[-1]
                drawn.append(int(row.argmax()))
                q[i, s] = (row / T).softmax(0) if T > 0 else torch.nn.functional.one_hot(row.argmax(), V)
            logits[i] = model(text[-1:] + drawn)
            says = logits[i].argmax(1).tolist()
            kept = next((s for s in range(gamma) if drawn[s] != says[s]), gamma)
            x[i], n_acc[i] = torch.tensor(drawn), kept
            out_tok[i] = torch.tensor(drawn[:kept] + [says[kept]] + [-1] * (gamma - kept))
            text += drawn[:kept] + [says[kept]]
            have += kept + 1
            model.n, draft.n = len(text) - 1, min(len(text) - 1, draft.n)
    if case["kind"] == "decode":
        return logits
    out = (x.to(DEV), q, logits, n_acc.to(DEV), out_tok.to(DEV))
    return (np.array(texts[0][: case["ctx_hi"] + case["new_tokens"]], dtype=np.int32), *out) if case["kind"] == "request" else out
