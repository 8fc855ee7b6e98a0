"""fp32 models over a few rows (norm, matrix and step in one kernel) against the CPU oracle: reductions of more than one round of
weights, odd vocabularies, grouped heads, heads of 16 and 256, 1...8 rows and one call beyond them."""
import numpy as np
import pytest
import torch

import oracle
from paper_2505_08600_b200 import synth
from gpu_util import DEV

pytestmark = pytest.mark.gpu

MODELS = {
    "gqa16": dict(n_layers=2, d_model=104, n_heads=6, n_kv_heads=2, head_dim=16, d_ffn=72, vocab=333),
    "hd256": dict(n_layers=1, d_model=256, n_heads=2, n_kv_heads=1, head_dim=256, d_ffn=1544, vocab=1001),     # three rounds of weights
    "mb8": dict(n_layers=2, d_model=512, n_heads=4, n_kv_heads=2, head_dim=64, d_ffn=2048, vocab=333),         # gate/up of 8 MB: 6...8 rows as well
}


@pytest.mark.parametrize("name", sorted(MODELS))
@pytest.mark.parametrize("n_seq,gamma", [(1, 0), (1, 1), (1, 4), (1, 5), (2, 3), (3, 2)])      # 1, 2, 5, 6, 8 and 9 verify rows
def test_verify_rows_follow_the_oracle(name, n_seq, gamma):
    from paper_2505_08600_b200 import binding
    dims = MODELS[name]
    V = dims["vocab"]
    w = synth.make_weights(dims, seed=3, model_index=0, dtype="f32")
    ctx = binding.Context(dims, [dims], "f32", n_seq, 96, max(gamma, 1), 1.0, 7)
    ctx.load_weights(0, w); ctx.load_weights(1, w)
    toks = [synth.make_prompt(V, (3, 70, 33)[s], seed=9, seq=s) for s in range(n_seq)]
    seqs = list(range(n_seq))
    for s in seqs:
        ctx.sd_seq_begin(s, toks[s], s)
    ctx.sd_route_prompt(seqs, forced_task=[0] * n_seq)
    ctx.sd_prefill(seqs)
    x = np.stack([synth.make_prompt(V, gamma, seed=5, seq=s) for s in seqs]) if gamma else np.zeros((n_seq, 0), np.int32)
    logits = torch.zeros((n_seq, gamma + 1, V), dtype=torch.float32, device=DEV)
    ctx.sd_verify(seqs, gamma, torch.from_numpy(x).to(DEV), logits)
    got = logits.cpu().numpy().astype(np.float64)
    assert ctx.sd_device_status() == 0
    ctx.close()
    om = oracle.OracleModel(dims, w)
    for s in seqs:
        want = om.new_cache(128).forward(np.concatenate([toks[s], x[s]]), 0)[-(gamma + 1):]
        assert np.abs(got[s] - want).max() <= 1e-4, s          # logits of magnitude 1 over a few hundred fp32 terms per matrix


@pytest.mark.parametrize("hd,H,Hkv", [(16, 4, 2), (64, 2, 2), (256, 1, 1)])
def test_attention_over_long_contexts(hd, H, Hkv):
    """Contexts around the keys (256) and values (16 per group of threads) that are on their way at a time, and several times that."""
    from paper_2505_08600_b200 import binding
    dims = dict(n_layers=1, d_model=64, n_heads=H, n_kv_heads=Hkv, head_dim=hd, d_ffn=64, vocab=211)
    w = synth.make_weights(dims, seed=3, model_index=0, dtype="f32", std=0.2)
    lens = [16, 65, 256, 257, 900]
    om = oracle.OracleModel(dims, w)
    ctx = binding.Context(dims, [dims], "f32", 1, 1000, 1, 1.0, 7)
    ctx.load_weights(0, w); ctx.load_weights(1, w)
    for m in lens:
        toks, x = synth.make_prompt(211, m, seed=9, seq=m), np.array([[5]], dtype=np.int32)
        ctx.sd_seq_begin(0, toks, 0)
        ctx.sd_route_prompt([0], forced_task=[0])
        ctx.sd_prefill([0])
        logits = torch.zeros((1, 2, 211), dtype=torch.float32, device=DEV)
        ctx.sd_verify([0], 1, torch.from_numpy(x).to(DEV), logits)
        want = om.new_cache(1000).forward(np.concatenate([toks, x[0]]), 0)[-2:]
        assert np.abs(logits.cpu().numpy()[0].astype(np.float64) - want).max() <= 1e-4 * max(1.0, np.abs(want).max()), m      # a few hundred fp32 terms
    assert ctx.sd_device_status() == 0
    ctx.close()
