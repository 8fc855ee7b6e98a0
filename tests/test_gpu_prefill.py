"""Prefill passes (many prompt rows of several sequences packed into one pass) against the CPU oracle: the caches that a
prefill leaves are judged by the next token's logits, which read every cached position of every layer."""
import numpy as np
import pytest
import torch

import oracle
from paper_2505_08600_b200 import synth
from gpu_util import DEV

pytestmark = pytest.mark.gpu

LOGITS_TOL = 5e-2                # bf16 activations and KV cache against the fp64 oracle, as for the verify rows


def _m(L, d, H, Hkv, hd, F, V):
    return dict(n_layers=L, d_model=d, n_heads=H, n_kv_heads=Hkv, head_dim=hd, d_ffn=F, vocab=V)


# matrices that do not fill a 256-feature tile, grouped heads of 64, heads of 128, one layer (keys and values only); widths of
# eight columns, and of eight columns beyond a multiple of the 512 that a warp of the row kernels covers
MODELS = {
    "gqa64": _m(3, 320, 6, 2, 64, 448, 512),
    "mha128": _m(2, 384, 3, 3, 128, 1024, 512),
    "one_layer": _m(1, 128, 2, 1, 64, 192, 512),
    "d8": _m(2, 8, 1, 1, 64, 64, 512),
    "d520": _m(2, 520, 8, 8, 64, 576, 512),
    "d1032": _m(2, 1032, 4, 2, 128, 576, 512),
}
# prompt lengths (rows = length - 1): around attention blocks of 64 and around 256, remainders of 3...16 rows (two-part
# activations), fewer rows than a pass takes, more rows than a pass takes
PROMPTS = {
    "fewest": [18],
    "block_edges": [64, 65, 66, 130],
    "row_256_edges": [256, 257, 258, 259],
    "two_part_rests": [2, 5, 17, 18, 260, 273, 274],
    "several_passes": [1001, 37, 1100, 3],
}


@pytest.mark.parametrize("model,prompts", [("gqa64", k) for k in PROMPTS] + [("mha128", "block_edges"), ("mha128", "two_part_rests"), ("one_layer", "row_256_edges"), ("d8", "fewest"), ("d520", "block_edges"), ("d1032", "fewest")])
def test_prefill_leaves_the_oracles_caches(model, prompts):
    from paper_2505_08600_b200 import binding
    dims, lens = MODELS[model], PROMPTS[prompts]
    draft = _m(2, 128, 2, 2, 64, 192, 512)
    w, wd = synth.make_weights(dims, seed=3, model_index=0, dtype="bf16"), synth.make_weights(draft, seed=3, model_index=1, dtype="bf16")
    n, V, gamma = len(lens), dims["vocab"], 1
    ctx = binding.Context(dims, [draft, draft], "bf16", n, 1200, gamma, 1.0, 7)
    ctx.load_weights(0, w); ctx.load_weights(1, wd); ctx.load_weights(2, wd)
    toks = [synth.make_prompt(V, m, seed=9, seq=i) for i, m in enumerate(lens)]
    seqs = list(range(n))
    for s in seqs:
        ctx.sd_seq_begin(s, toks[s], s)
    ctx.sd_route_prompt(seqs, forced_task=[s % 2 for s in seqs])
    ctx.sd_prefill(seqs)
    logits = torch.zeros((n, V), dtype=torch.float32, device=DEV)
    ctx.sd_target_step(seqs, logits)
    x, q = torch.zeros((n, gamma), dtype=torch.int32, device=DEV), torch.zeros((n, gamma, V), dtype=torch.float32, device=DEV)
    ctx.sd_draft_steps(seqs, gamma, x, q)
    got, gq = logits.cpu().numpy().astype(np.float64), q.cpu().numpy().astype(np.float64)
    assert ctx.sd_device_status() == 0
    ctx.close()
    om, od = oracle.OracleModel(dims, w), oracle.OracleModel(draft, wd)
    for s in seqs:
        want = om.new_cache(1200).forward(toks[s], 0)[-1]
        assert np.abs(got[s] - want).max() <= LOGITS_TOL, (s, lens[s])
        e = np.exp((lq := od.new_cache(1200).forward(toks[s], 0)[-1]) - lq.max())
        assert np.abs(gq[s, 0] - e / e.sum()).max() <= 1e-3, (s, lens[s])
