"""Draft passes whose layers run in two kernels (a cluster per head, a cluster per 128 or 192 features) against the CPU oracle: widths that do not
fill the kernels' k blocks and tiles, 1...8 sequences (one or two rows each; the first pass of more than four is beyond these kernels), and
contexts that end at the edges of a warp's tiles of 16 keys or go around its ring of two."""
import numpy as np
import pytest
import torch

import oracle
from paper_2505_08600_b200 import synth
from gpu_util import DEV

pytestmark = pytest.mark.gpu

V = 509
LOG_TOL = 1e-1               # log q = logit - log sum exp: two numbers that are each within the logits' 5e-2 of the oracle's


def _m(L, d, H, F):
    return dict(n_layers=L, d_model=d, n_heads=H, n_kv_heads=H, head_dim=64, d_ffn=F, vocab=V)


DRAFTS = {
    "d64": _m(2, 64, 1, 128),            # one tile of output features per CTA, one piece
    "d448": _m(2, 448, 3, 384),          # 14 k blocks for 16 warps, 7 tiles
    "d768": _m(2, 768, 12, 3072),
    "d832": _m(1, 832, 5, 640),          # 26 k blocks, 13 tiles
    "d1024": _m(2, 1024, 16, 4096),      # as large as it goes
}


def _run(draft, lens, gamma, streams=True, seqs=None):
    from paper_2505_08600_b200 import binding
    target = _m(1, 64, 1, 64)
    wt, wd = synth.make_weights(target, seed=3, model_index=0, dtype="bf16"), synth.make_weights(draft, seed=3, model_index=1, dtype="bf16")
    n = len(lens)
    ctx = binding.Context(target, [draft], "bf16", n, max(lens) + 64, gamma, 1.0, 7)
    ctx.load_weights(0, wt); ctx.load_weights(1, wd)
    toks = [synth.make_prompt(V, m, seed=9, seq=i) for i, m in enumerate(lens)]
    for s in range(n):
        ctx.sd_seq_begin(s, toks[s], s)
    ctx.sd_route_prompt(list(range(n)), forced_task=[0] * n)
    ctx.sd_prefill(list(range(n)))
    seqs = list(range(n)) if seqs is None else seqs
    x, q = torch.zeros((len(seqs), gamma), dtype=torch.int32, device=DEV), torch.zeros((len(seqs), gamma, V), dtype=torch.float32, device=DEV)
    ctx.sd_draft_steps(seqs, gamma, x, q)
    again_x, again_q = torch.zeros_like(x), torch.zeros_like(q)
    ctx.sd_draft_steps(seqs, gamma, again_x, again_q)
    assert torch.equal(x, again_x) and torch.equal(q, again_q)          # pieces are added in a fixed order
    assert ctx.sd_device_status() == 0
    ctx.close()
    return wd, toks, x.cpu().numpy(), q.cpu().numpy().astype(np.float64)


def _compare(draft, lens, gamma, seqs=None):
    wd, toks, xg, qg = _run(draft, lens, gamma, seqs=seqs)
    om = oracle.OracleModel(draft, wd)
    for i, s in enumerate(range(len(lens)) if seqs is None else seqs):
        logits = om.new_cache(lens[s] + gamma + 1).forward(np.concatenate([toks[s], xg[i, :-1]]), 0)[-gamma:]
        top = logits.max(axis=1, keepdims=True)
        want = logits - top - np.log(np.exp(logits - top).sum(axis=1, keepdims=True))
        assert np.abs(np.log(qg[i]) - want).max() <= LOG_TOL, s


@pytest.mark.parametrize("n_seq", [1, 2, 3, 4, 5, 8])
@pytest.mark.parametrize("name", sorted(DRAFTS))
def test_draft_passes_follow_the_oracle(name, n_seq):
    _compare(DRAFTS[name], [7 + 9 * i for i in range(n_seq)], 3)


@pytest.mark.parametrize("lens", [[2], [15], [16], [17], [33], [513], [2049], [400, 15, 16, 17, 31, 333, 64, 2]], ids=str)
def test_contexts_at_the_edges_of_tiles(lens):
    _compare(_m(1, 128, 2, 128), lens, 4)


def test_slots_and_order_of_the_call():
    _compare(_m(2, 256, 2, 256), [40, 9, 70, 25, 130], 3, seqs=[4, 0, 2])


def test_an_iteration_after_full_and_partial_acceptance():
    """The first pass of an iteration has two rows per sequence, of which the first is active only after a fully accepted iteration."""
    from paper_2505_08600_b200 import binding
    draft, target, gamma = _m(2, 256, 4, 256), _m(1, 64, 1, 64), 3
    wt, wd = synth.make_weights(target, seed=3, model_index=0, dtype="bf16"), synth.make_weights(draft, seed=3, model_index=1, dtype="bf16")
    ctx = binding.Context(target, [draft], "bf16", 2, 128, gamma, 1.0, 7)
    ctx.load_weights(0, wt); ctx.load_weights(1, wd)
    toks = [list(map(int, synth.make_prompt(V, m, seed=9, seq=i))) for i, m in enumerate((20, 31))]
    for s in range(2):
        ctx.sd_seq_begin(s, np.array(toks[s], dtype=np.int32), s)
    ctx.sd_route_prompt([0, 1], forced_task=[0, 0])
    ctx.sd_prefill([0, 1])
    x, q = torch.zeros((2, gamma), dtype=torch.int32, device=DEV), torch.zeros((2, gamma, V), device=DEV)
    om = oracle.OracleModel(draft, wd)
    for it, accepted in enumerate([(3, 1), (0, 3), (3, 3), (2, 0)]):
        ctx.sd_draft_steps([0, 1], gamma, x, q)
        xg, qg = x.cpu().numpy(), q.cpu().numpy().astype(np.float64)
        for s in range(2):
            logits = om.new_cache(128).forward(np.array(toks[s] + xg[s, :-1].tolist()), 0)[-gamma:]
            top = logits.max(axis=1, keepdims=True)
            want = logits - top - np.log(np.exp(logits - top).sum(axis=1, keepdims=True))
            assert np.abs(np.log(qg[s]) - want).max() <= LOG_TOL, (it, s)
        out = np.full((2, gamma + 1), -1, dtype=np.int32)
        for s in range(2):
            new = xg[s, :accepted[s]].tolist() + [(it * 7 + s) % V]
            out[s, :len(new)] = new
            toks[s] += new
        ctx.sd_kv_rollback([0, 1], gamma, torch.tensor(accepted, dtype=torch.int32, device=DEV), torch.from_numpy(out).to(DEV))
    assert ctx.sd_device_status() == 0
    ctx.close()


# ---- what the tests above cannot see: their weights give nearly even attention and logits of a few hundredths, some of their shapes are beyond these
#      kernels, and none asks which kernels ran

CLUSTER_LAYER, FEW_ROWS_LAYER = [2, 3 | 3 << 8], [3 | 1 << 8, 2, 3 | 2 << 8, 3 | 3 << 8, 3 | 2 << 8]      # records of a layer: attention, matrix (QKV 1, residual 2, SwiGLU 3)
DEEP = {                                            # and up to how many sequences they take
    "d448": (_m(6, 448, 3, 384), 6),                # 14 k blocks for 16 warps, 7 tiles, 128 features
    "d512_f576": (_m(6, 512, 8, 576), 6),           # clusters of 192 features, the form for up to 512 columns
    "d768": (_m(3, 768, 12, 3072), 4),              # ... 768
    "d1024_f3072": (_m(4, 1024, 16, 3072), 4),      # ... 1,024: as large as it goes
    "d1024_f2048": (_m(4, 1024, 16, 2048), 4),      # 128 features, 1,024 columns, 32 clusters
    "d1024_f4096": (_m(4, 1024, 16, 4096), 0),      # 48 clusters: one kernel per matrix
}


@pytest.mark.parametrize("n_seq", [1, 2, 4, 5, 6])
@pytest.mark.parametrize("name", sorted(DEEP))
def test_the_kernels_that_are_meant_run_and_follow_the_oracle(name, n_seq):
    """Weights that keep every activation near one; which records a pass leaves tells the kernels apart."""
    from paper_2505_08600_b200 import binding
    (draft, most), target, gamma = DEEP[name], _m(1, 64, 1, 64), 2
    wt = synth.make_weights(target, seed=3, model_index=0, dtype="bf16")
    wd = synth.make_weights(draft, seed=3, model_index=1, dtype="bf16", std=draft["d_model"] ** -0.5)
    seqs = list(range(n_seq))
    ctx = binding.Context(target, [draft], "bf16", n_seq, 96, gamma, 1.0, 7, stream=torch.cuda.Stream())
    ctx.load_weights(0, wt); ctx.load_weights(1, wd)
    toks = [synth.make_prompt(V, 7 + 9 * i, seed=9, seq=i) for i in seqs]
    for s in seqs:
        ctx.sd_seq_begin(s, toks[s], s)
    ctx.sd_route_prompt(seqs, forced_task=[0] * n_seq)
    ctx.sd_prefill(seqs)
    x, q = torch.zeros((n_seq, gamma), dtype=torch.int32, device=DEV), torch.zeros((n_seq, gamma, V), device=DEV)
    torch.cuda.synchronize()
    ctx.sd_launch_stamps(1)
    for _ in range(2):                                                     # captured, replayed
        ctx.sd_draft_steps(seqs, gamma, x, q)
        stamps, kinds = ctx.sd_launch_stamps_read()
        assert kinds.tolist() == draft["n_layers"] * (CLUSTER_LAYER if n_seq <= most else FEW_ROWS_LAYER) + [3]
        t = stamps.astype(np.int64)
        assert (t[:, [0, 1, 5]] > 0).all() and (t[:, 0] <= t[:, 1]).all() and (t[:, 1] <= t[:, 5]).all()
    assert ctx.sd_device_status() == 0
    xg, qg = x.cpu().numpy(), q.cpu().numpy().astype(np.float64)
    ctx.close()
    om = oracle.OracleModel(draft, wd)
    for s in seqs:
        logits = om.new_cache(128).forward(np.concatenate([toks[s], xg[s, :-1]]), 0)[-gamma:]
        top = logits.max(axis=1, keepdims=True)
        want = logits - top - np.log(np.exp(logits - top).sum(axis=1, keepdims=True))
        assert np.abs(np.log(np.maximum(qg[s], 1e-30)) - want).max() <= LOG_TOL, s


NEEDLE = 5


def _needle_model(n_layers):
    """Every query scores the token NEEDLE 14 (in the softmax's exponent) above all others, wherever it stands: feature 0 marks it, feature 1 is one for
    every token, and both meet in the head's slowest rotary pair.  Its value is nearly the whole of the first layer's output; the other layers add nothing."""
    dims = _m(n_layers, 128, 2, 128)
    rng = np.random.default_rng(77)
    w = synth.make_weights(dims, seed=3, model_index=1, dtype="f32")
    w["embed"] = rng.standard_normal((V, 128), dtype=np.float32)
    w["embed"][:, 0], w["embed"][:, 1] = 0.0, 1.0
    w["embed"][NEEDLE, 0] = 8.0
    w["lm_head"] = rng.standard_normal((V, 128), dtype=np.float32) * 0.2
    for l in range(n_layers):
        for name in ("wq", "wk", "wd", "wo"):
            w[name][l] = np.zeros_like(w[name][l])
    for h in range(2):
        w["wq"][0][64 * h + 31, 1] = 4.2
        w["wk"][0][64 * h + 31, 0] = 4.2
    w["wv"][0] = rng.standard_normal(w["wv"][0].shape, dtype=np.float32) * 0.1
    w["wo"][0] = rng.standard_normal(w["wo"][0].shape, dtype=np.float32) * 0.1
    f32 = ("final_norm", "norm1", "norm2")
    return dims, {k: v if k in f32 else [synth.f32_to_bf16_bits(a) for a in v] if isinstance(v, list) else synth.f32_to_bf16_bits(v) for k, v in w.items()}


def _log_q(om, tokens, n):
    logits = om.new_cache(len(tokens) + 1).forward(np.asarray(tokens, dtype=np.int32), 0)[-n:]
    top = logits.max(axis=1, keepdims=True)
    return logits - top - np.log(np.exp(logits - top).sum(axis=1, keepdims=True))


# one position of every 16-key tile (of every eighth in the longest context); four contexts at once: every warp's share
@pytest.mark.parametrize("lens", [[17], [33], [333], [513], [2049], [400, 15, 31, 333]], ids=str)
def test_no_tile_of_the_cache_is_lost(lens):
    from paper_2505_08600_b200 import binding
    dims, wd = _needle_model(2)
    target, gamma, n = _m(1, 64, 1, 64), 2, len(lens)
    om = oracle.OracleModel(dims, wd)
    stride = 128 if max(lens) > 1024 else 16
    seqs = list(range(n))
    ctx = binding.Context(target, [dims], "bf16", n, max(lens) + 8, gamma, 1.0, 7, stream=torch.cuda.Stream())
    ctx.load_weights(0, synth.make_weights(target, seed=3, model_index=0, dtype="bf16")); ctx.load_weights(1, wd)
    x, q = torch.zeros((n, gamma), dtype=torch.int32, device=DEV), torch.zeros((n, gamma, V), device=DEV)
    torch.cuda.synchronize()
    ctx.sd_launch_stamps(1)
    rng = np.random.default_rng(3)
    for k in range((max(lens) + stride - 1) // stride):
        toks = []
        for m in lens:
            t = synth.make_prompt(V, m, seed=9, seq=k)
            t[t == NEEDLE] = NEEDLE + 1
            t[(k * stride + int(rng.integers(0, 16))) % m] = NEEDLE
            toks.append(t)
        for s in seqs:
            ctx.sd_seq_begin(s, toks[s], s)
        ctx.sd_route_prompt(seqs, forced_task=[0] * n)
        ctx.sd_prefill(seqs)
        ctx.sd_draft_steps(seqs, gamma, x, q)
        torch.cuda.synchronize()
        xg, got = x.cpu().numpy(), np.log(np.maximum(q.cpu().numpy().astype(np.float64), 1e-30))
        for s in seqs:
            whole = np.concatenate([toks[s], xg[s, :-1]])
            assert np.abs(got[s] - _log_q(om, whole, gamma)).max() <= LOG_TOL, (k, s)
    assert ctx.sd_launch_stamps_read()[1].tolist() == dims["n_layers"] * CLUSTER_LAYER + [3]
    assert ctx.sd_device_status() == 0
    ctx.close()


def test_the_needle_is_seen_by_the_oracle():
    """Without it the result is elsewhere by far more than the tolerance."""
    dims, wd = _needle_model(1)
    om = oracle.OracleModel(dims, wd)
    for m in (17, 513):
        t = synth.make_prompt(V, m, seed=9, seq=0)
        t[t == NEEDLE] = NEEDLE + 1
        with_it = t.copy()
        with_it[m // 3] = NEEDLE
        assert np.abs(_log_q(om, t, 1) - _log_q(om, with_it, 1)).max() > 10 * LOG_TOL
