"""Prompt classifier (MLP variant) against the CPU oracle, at the edges of the split of its columns and tokens."""
import numpy as np
import pytest

import oracle
from paper_2505_08600_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [8, 128, 264, 2056, 10240])   # fewer columns than the cluster has CTAs x 8, ragged slices, more than 256 columns a CTA, more than 48 KB of shared memory
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_classifier_routes_like_the_oracle(d, dtype):
    from paper_2505_08600_b200 import binding
    V, K, dh = 64, 3, 37
    dims = dict(n_layers=1, d_model=d, n_heads=1, n_kv_heads=1, head_dim=8, d_ffn=64, vocab=V)
    w = synth.make_weights(dims, seed=5, dtype=dtype, std=1.0)
    ctx = binding.Context(dims, [dims] * K, dtype, 4, 96, 1, 1.0, 7, clf_d_hidden=dh)
    ctx.load_weights(0, w)
    c = synth.make_classifier(d, dh, K, seed=11)
    ctx.sd_load_classifier(c["w1"], c["b1"], c["w2"], c["b2"])
    lens = [2, 16, 33, 90]
    toks = [synth.make_prompt(V, m, seed=13, seq=i) for i, m in enumerate(lens)]
    for s, p in enumerate(toks):
        ctx.sd_seq_begin(s, p, s)
    got = ctx.sd_route_prompt([0, 1, 2, 3], forced_task=[-1, -1, 1, -1]).tolist()
    ctx.close()
    assert got[2] == 1                                       # given with the request
    for s in (0, 1, 3):
        want, probs = oracle.route_prompt(w["embed"], toks[s], c["w1"], c["b1"], c["w2"], c["b2"])
        top = np.sort(np.log(np.maximum(probs, 1e-300)))     # (differences of scores; fp32 sums of magnitude ~10 agree to far less)
        assert got[s] == want or top[-1] - top[-2] < 1e-3
