"""The few-rows kernels of the draft passes against the CPU oracle: reductions that do not fill the kernel's form, a vocabulary
that does not fill its tiles, heads of 64 and 128, 1...16 rows in one and two groups of eight, and one call beyond them."""
import numpy as np
import pytest
import torch

import oracle
from paper_2505_08600_b200 import synth
from gpu_util import DEV

pytestmark = pytest.mark.gpu

# log q = logit - log sum exp: two numbers that are each within the logits' 5e-2 of the oracle's
LOG_TOL = 1e-1


def _m(L, d, H, hd, F, V):
    return dict(n_layers=L, d_model=d, n_heads=H, n_kv_heads=H, head_dim=hd, d_ffn=F, vocab=V)


DRAFTS = {
    "d288": _m(2, 288, 3, 64, 320, 509),           # 9 k blocks of 32, F = 10; odd vocabulary
    "hd128_f2112": _m(2, 256, 2, 128, 2112, 509),   # the form for up to 3072
    "d1056": _m(1, 1056, 4, 64, 4096, 509),         # the forms for up to 2048 and 4096
    "mixed": _m(1, 1152, 4, 64, 7680, 509),         # gate/up and down stream; QKV as well with one or two rows
    "two_waves": _m(1, 512, 4, 64, 2432, 509),      # gate/up is 304 CTAs: it streams from nine rows on
}


@pytest.mark.parametrize("n_seq", [1, 3, 4, 5, 8, 9])    # first pass of an iteration: 2 n rows, later ones n
@pytest.mark.parametrize("name", sorted(DRAFTS))
def test_draft_passes_follow_the_oracle(name, n_seq):
    from paper_2505_08600_b200 import binding
    draft, target, gamma = DRAFTS[name], _m(1, 64, 1, 64, 64, 509), 3
    wt, wd = synth.make_weights(target, seed=3, model_index=0, dtype="bf16"), synth.make_weights(draft, seed=3, model_index=1, dtype="bf16")
    ctx = binding.Context(target, [draft], "bf16", n_seq, 96, gamma, 1.0, 7)
    ctx.load_weights(0, wt); ctx.load_weights(1, wd)
    toks = [synth.make_prompt(509, 7 + 9 * i, seed=9, seq=i) for i in range(n_seq)]
    seqs = list(range(n_seq))
    for s in seqs:
        ctx.sd_seq_begin(s, toks[s], s)
    ctx.sd_route_prompt(seqs, forced_task=[0] * n_seq)
    ctx.sd_prefill(seqs)
    x, q = torch.zeros((n_seq, gamma), dtype=torch.int32, device=DEV), torch.zeros((n_seq, gamma, 509), dtype=torch.float32, device=DEV)
    ctx.sd_draft_steps(seqs, gamma, x, q)
    xg, qg = x.cpu().numpy(), q.cpu().numpy().astype(np.float64)
    assert ctx.sd_device_status() == 0
    ctx.close()
    om = oracle.OracleModel(draft, wd)
    for s in seqs:
        logits = om.new_cache(128).forward(np.concatenate([toks[s], xg[s, :-1]]), 0)[-gamma:]
        top = logits.max(axis=1, keepdims=True)
        want = logits - top - np.log(np.exp(logits - top).sum(axis=1, keepdims=True))
        assert np.abs(np.log(qg[s]) - want).max() <= LOG_TOL, s


@pytest.mark.parametrize("n_seq", [1, 5])                           # 2, then 1 row; 10, then 5
def test_mixed_passes_with_adapters_follow_the_merged_models(n_seq):
    from oracle import lora
    from paper_2505_08600_b200 import binding
    draft, target, gamma, rank = _m(1, 1152, 4, 64, 7680, 512), _m(1, 64, 1, 64, 64, 512), 2, 8
    wt, wd = synth.make_weights(target, seed=3, model_index=0, dtype="bf16"), synth.make_weights(draft, seed=3, model_index=1, dtype="bf16")
    ctx = binding.Context(target, [draft], "bf16", n_seq, 96, gamma, 1.0, 7, lora_adapters=2, lora_rank=rank, lora_scale=1.0)
    ctx.load_weights(0, wt); ctx.load_weights(1, wd)
    merged = []
    for task in range(2):
        ad = synth.make_lora(draft, rank, task, seed=0)
        for mat, name in enumerate(("qkv", "wo", "gu", "wd")):
            for l, (a, b) in enumerate(ad[name]):
                ctx.sd_load_lora(task, l, mat, a, b)
        merged.append(oracle.OracleModel(draft, lora.merged_weights(draft, wd, ad, 1.0)))
    toks = [synth.make_prompt(512, 7 + 9 * i, seed=9, seq=i) for i in range(n_seq)]
    seqs = list(range(n_seq))
    for s in seqs:
        ctx.sd_seq_begin(s, toks[s], s)
    ctx.sd_route_prompt(seqs, forced_task=[s % 2 for s in seqs])
    ctx.sd_prefill(seqs)
    x, q = torch.zeros((n_seq, gamma), dtype=torch.int32, device=DEV), torch.zeros((n_seq, gamma, 512), dtype=torch.float32, device=DEV)
    ctx.sd_draft_steps(seqs, gamma, x, q)
    xg, qg = x.cpu().numpy(), q.cpu().numpy().astype(np.float64)
    assert ctx.sd_device_status() == 0
    ctx.close()
    for s in seqs:
        logits = merged[s % 2].new_cache(128).forward(np.concatenate([toks[s], xg[s, :-1]]), 0)[-gamma:]
        top = logits.max(axis=1, keepdims=True)
        want = logits - top - np.log(np.exp(logits - top).sum(axis=1, keepdims=True))
        assert np.abs(np.log(qg[s]) - want).max() <= LOG_TOL, s


@pytest.mark.parametrize("two_part", [0, 1])
@pytest.mark.parametrize("n_seq,gamma", [(1, 7), (1, 8), (1, 15), (3, 3)])     # 8, 9, 16 and 12 rows
@pytest.mark.parametrize("d", [1024, 1152, 2048])                              # Wo leaves 64, 72 and 128 pieces of a row's sum of squares
def test_mixed_passes_add_all_pieces_of_the_sum_of_squares(d, n_seq, gamma, two_part):
    """A target whose Wo takes the few-rows kernel while gate/up and the lm_head stream, with the rows in one and in two bf16 parts."""
    from paper_2505_08600_b200 import binding
    target, draft = _m(1, d, 4, 64, 4608, 4096), _m(1, 64, 1, 64, 64, 4096)
    wt, wd = synth.make_weights(target, seed=3, model_index=0, dtype="bf16"), synth.make_weights(draft, seed=3, model_index=1, dtype="bf16")
    ctx = binding.Context(target, [draft], "bf16", n_seq, 96, gamma, 1.0, 7)
    ctx.load_weights(0, wt); ctx.load_weights(1, wd)
    ctx.sd_use_two_part_activations(two_part)
    toks = [synth.make_prompt(4096, 20 + 9 * i, seed=9, seq=i) for i in range(n_seq)]
    seqs = list(range(n_seq))
    for s in seqs:
        ctx.sd_seq_begin(s, toks[s], s)
    ctx.sd_route_prompt(seqs, forced_task=[0] * n_seq)
    ctx.sd_prefill(seqs)
    x = np.stack([synth.make_prompt(4096, gamma, seed=5, seq=s) for s in seqs])
    logits = torch.zeros((n_seq, gamma + 1, 4096), dtype=torch.float32, device=DEV)
    ctx.sd_verify(seqs, gamma, torch.from_numpy(x).to(DEV), logits)
    got = logits.cpu().numpy().astype(np.float64)
    assert ctx.sd_device_status() == 0
    ctx.close()
    om = oracle.OracleModel(target, wt)
    for s in seqs:
        want = om.new_cache(128).forward(np.concatenate([toks[s], x[s]]), 0)[-(gamma + 1):]
        assert np.abs(got[s] - want).max() <= 5e-2, s          # bf16 against the fp64 oracle, as for the verify rows elsewhere


def test_passes_use_their_own_row_plan():
    """Draft passes of sequences with other slots and positions in turn, each first matrix kernel right behind the kernel that writes
    the row plan: what a call returns does not depend on the call before it."""
    from paper_2505_08600_b200 import binding
    draft, target, gamma = DRAFTS["d288"], _m(1, 64, 1, 64, 64, 509), 3
    ctx = binding.Context(target, [draft], "bf16", 3, 160, gamma, 1.0, 7)
    ctx.load_weights(0, synth.make_weights(target, seed=3, model_index=0, dtype="bf16"))
    ctx.load_weights(1, synth.make_weights(draft, seed=3, model_index=1, dtype="bf16"))
    for s, m in enumerate((9, 70, 150)):
        ctx.sd_seq_begin(s, synth.make_prompt(509, m, seed=9, seq=s), s)
    ctx.sd_route_prompt([0, 1, 2], forced_task=[0, 0, 0])
    ctx.sd_prefill([0, 1, 2])
    calls, first = [[0], [1], [2], [2, 0], [1, 2, 0]], {}
    x, q = torch.zeros((3, gamma), dtype=torch.int32, device=DEV), torch.zeros((3, gamma, 509), dtype=torch.float32, device=DEV)
    for graphs in (1, 0):
        ctx.sd_use_graphs(graphs)
        for i in range(40):
            seqs = calls[i * 3 % len(calls)]
            n = len(seqs)
            ctx.sd_draft_steps(seqs, gamma, x[:n], q[:n])
            for j, s in enumerate(seqs):
                got = (x[j].cpu().numpy(), q[j].cpu().numpy())
                want = first.setdefault((s, n), got)               # (with another number of rows other forms may be taken)
                assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1]), (i, seqs, s)
    assert ctx.sd_device_status() == 0
    ctx.close()
