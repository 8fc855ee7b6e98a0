"""Draft passes whose layers run in two kernels (a cluster per head, a cluster per 128 features) against the CPU oracle: widths that do not
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
DEEP = {
    "d448": (_m(6, 448, 3, 384), True),             # 14 k blocks for 16 warps, 7 tiles, 128 features
    "d512_f576": (_m(6, 512, 8, 576), True),        # clusters of 192 features, the form for up to 512 columns
    "d768": (_m(3, 768, 12, 3072), True),           # ... 768
    "d1024_f3072": (_m(3, 1024, 16, 3072), True),   # ... 1,024: as large as it goes
    "d1024_f2048": (_m(3, 1024, 16, 2048), True),   # 128 features, 1,024 columns, 32 clusters
    "d1024_f4096": (_m(3, 1024, 16, 4096), False),  # 48 clusters: one kernel per matrix
}


@pytest.mark.parametrize("n_seq", [1, 2, 4, 5, 6])
@pytest.mark.parametrize("name", sorted(DEEP))
def test_the_kernels_that_are_meant_run_and_follow_the_oracle(name, n_seq):
    """Weights that keep every activation near one; which records a pass leaves tells the kernels apart (six layers: up to six sequences)."""
    from paper_2505_08600_b200 import binding
    (draft, fits), target, gamma = DEEP[name], _m(1, 64, 1, 64), 2
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
    clusters = fits and (n_seq <= 4 or draft["n_layers"] >= 6)
    for _ in range(2):                                                     # captured, replayed
        ctx.sd_draft_steps(seqs, gamma, x, q)
        stamps, kinds = ctx.sd_launch_stamps_read()
        assert kinds.tolist() == draft["n_layers"] * (CLUSTER_LAYER if clusters else FEW_ROWS_LAYER) + [3]
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
