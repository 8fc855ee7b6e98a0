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
