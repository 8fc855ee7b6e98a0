"""The draft sampler and the accept rule with the vocabulary cut over a cluster: vocabularies at which the slices are ragged, the
smallest that takes that form, one that does not fit; exact against the oracle on shared probabilities."""
import numpy as np
import pytest
import torch

import oracle
from paper_2505_08600_b200 import synth
from gpu_util import DEV, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,gamma,V", [(3, 1, 4096), (2, 2, 4097), (2, 15, 20011), (2, 3, 50000), (1, 15, 32001)])
def test_accept_is_the_oracles(B, gamma, V):
    from paper_2505_08600_b200 import binding
    seed = 50 + V
    p = oracle.softmax_T(synth.make_logits((B, gamma + 1, V), seed=seed, std=1.4).astype(np.float64), 1.0)
    q = oracle.softmax_T(synth.make_logits((B, gamma, V), seed=seed, stream=1, std=1.4).astype(np.float64), 1.0)
    q[0] = p[0, :gamma]                                    # accepts everything: the draw from the last row
    x = np.array([[oracle.sample_icdf(q[b, s], oracle.uniform24(seed, b, s, 99, 0)) for s in range(gamma)] for b in range(B)], dtype=np.int32)
    if B > 1:
        x[1, 0] = V                                        # an impossible token counts as rejected
    it, sid = np.arange(B, dtype=np.uint32), np.full(B, 5, dtype=np.uint32)
    n_acc, out = torch.zeros(B, dtype=torch.int32, device=DEV), torch.zeros((B, gamma + 1), dtype=torch.int32, device=DEV)
    binding.sd_accept(to_dev(p), to_dev(q), to_dev(x), 1.0, seed, to_dev(it), to_dev(sid), n_acc, out, 0)
    n_acc, out = n_acc.cpu().numpy(), out.cpu().numpy()
    for b in range(B):
        if b == 1:
            assert n_acc[b] == 0 and 0 <= out[b, 0] < V and (out[b, 1:] == -1).all()
            continue
        n_ref, out_ref = oracle.accept(p[b], q[b], x[b], seed, b, 5)
        assert (n_acc[b], out[b].tolist()) == (n_ref, out_ref.tolist())
    assert n_acc[0] == gamma


@pytest.mark.parametrize("V", [4096, 4099, 32003])
@pytest.mark.parametrize("T", [0.0, 1.0])
def test_draft_draws_come_from_the_written_distribution(V, T):
    from paper_2505_08600_b200 import binding
    dims = dict(n_layers=1, d_model=64, n_heads=1, n_kv_heads=1, head_dim=64, d_ffn=64, vocab=V)
    ctx = binding.Context(dims, [dims], "bf16", 3, 64, 4, T, 7)
    w = synth.make_weights(dims, seed=3, dtype="bf16", std=0.3)
    ctx.load_weights(0, w); ctx.load_weights(1, w)
    for s in range(3):
        ctx.sd_seq_begin(s, synth.make_prompt(V, 5 + s, seed=9, seq=s), 40 + s)
    ctx.sd_route_prompt([0, 1, 2], forced_task=[0, 0, 0])
    ctx.sd_prefill([0, 1, 2])
    x, q = torch.zeros((3, 4), dtype=torch.int32, device=DEV), torch.zeros((3, 4, V), dtype=torch.float32, device=DEV)
    ctx.sd_draft_steps([0, 1, 2], 4, x, q)
    x, q = x.cpu().numpy(), q.cpu().numpy()
    ctx.close()
    for s in range(3):
        for j in range(4):
            if T == 0.0:
                assert q[s, j].sum() == 1.0 and q[s, j, x[s, j]] == 1.0
            else:
                assert abs(q[s, j].astype(np.float64).sum() - 1.0) <= 1e-5      # V fp32 roundings of 2^-24 relative each
                assert x[s, j] == oracle.sample_icdf(q[s, j], oracle.uniform24(7, 0, j, 40 + s, 0))
