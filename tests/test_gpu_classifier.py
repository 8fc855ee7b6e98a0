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


def test_contexts_of_other_widths_on_several_threads():
    """Contexts of their own on several threads, one with more than 48 KB of shared memory per CTA: neither call changes what the other may launch."""
    import threading
    import torch
    from paper_2505_08600_b200 import binding
    ctxs = []
    for d in (10240, 8, 8, 8):
        dims = dict(n_layers=1, d_model=d, n_heads=1, n_kv_heads=1, head_dim=8, d_ffn=64, vocab=64)
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            ctx = binding.Context(dims, [dims] * 3, "f32", 1, 96, 1, 1.0, 7, clf_d_hidden=37)
            ctx.load_weights(0, synth.make_weights(dims, seed=5, dtype="f32", std=1.0))
            c = synth.make_classifier(d, 37, 3, seed=11)
            ctx.sd_load_classifier(c["w1"], c["b1"], c["w2"], c["b2"])
        ctxs.append((ctx, stream))
    wrong = []

    def loop(ctx, stream):
        try:
            with torch.cuda.stream(stream):
                for _ in range(2000):
                    ctx.sd_seq_begin(0, synth.make_prompt(64, 5, seed=13), 0)
                    ctx.sd_route_prompt([0])
        except RuntimeError as e:
            wrong.append(str(e))

    threads = [threading.Thread(target=loop, args=c) for c in ctxs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for ctx, _ in ctxs:
        ctx.close()
    assert not wrong
