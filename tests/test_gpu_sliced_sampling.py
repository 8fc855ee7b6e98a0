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


def _drafts(p, q, seed):
    B, gamma, _ = q.shape
    return np.array([[oracle.sample_icdf(q[b, s], oracle.uniform24(seed, b, s, 99, 0)) for s in range(gamma)] for b in range(B)], dtype=np.int32)


# vocabularies that do not divide into eight slices of fours, from two rows to as many as fit
@pytest.mark.parametrize("gamma,V", [(1, 4099), (1, 12001), (2, 20011), (3, 17003), (5, 50001), (12, 30003)])
def test_tokens_from_ragged_slices_are_the_oracles(gamma, V):
    """Ordinary drafts, and rejected ones whose residual is the whole row, or three tokens: the last of a slice, the first of the next, the
    last of the vocabulary."""
    from paper_2505_08600_b200 import binding
    B, seed = 12, 70 + V
    logits = synth.make_logits((B, gamma + 1, V), seed=seed, std=1.4).astype(np.float64)
    p = oracle.softmax_T(logits, 1.0)
    q = oracle.softmax_T(logits[:, :gamma] + synth.make_logits((B, gamma, V), seed=seed, stream=1, std=0.7), 1.0)
    x = _drafts(p, q, seed)
    slice_len = (V + 31) // 32 * 4
    edge = [slice_len - 1, slice_len, V - 1]
    x[8:, 0] = V                                           # an impossible token is rejected: the draw is the residual's, in slot 0
    for b in (10, 11):
        q[b, 0] = p[b, 0]
        q[b, 0, edge] = 0.0
    it, sid = np.arange(B, dtype=np.uint32), np.full(B, 5, dtype=np.uint32)
    n_acc, out = torch.zeros(B, dtype=torch.int32, device=DEV), torch.zeros((B, gamma + 1), dtype=torch.int32, device=DEV)
    binding.sd_accept(to_dev(p), to_dev(q), to_dev(x), 1.0, seed, to_dev(it), to_dev(sid), n_acc, out, 0)
    n_acc, out = n_acc.cpu().numpy(), out.cpu().numpy()
    for b in range(8):
        n_ref, out_ref = oracle.accept(p[b], q[b], x[b], seed, b, 5)
        assert (n_acc[b], out[b].tolist()) == (n_ref, out_ref.tolist()), b
    for b in range(8, B):
        y = oracle.sample_icdf(np.maximum(p[b, 0] - q[b, 0], np.float32(0)), oracle.uniform24(seed, b, 0, 5, 2))
        assert (n_acc[b], out[b, 0]) == (0, y) and (out[b, 1:] == -1).all(), b
        assert b < 10 or y in edge


@pytest.mark.parametrize("T", [0.0, 0.7])
@pytest.mark.parametrize("gamma,V", [(2, 20011), (5, 50001), (15, 24003)])
def test_logits_over_ragged_slices(gamma, V, T):
    """p from logits inside the kernel: greedy decisions are the oracle's; with a temperature they are wherever they do not lie within
    fp32 rounding of the comparison, and so is the token wherever the draw does not lie on the edge between two."""
    from paper_2505_08600_b200 import binding
    B, seed = 8, 30 + V
    logits = synth.make_logits((B, gamma + 1, V), seed=seed, std=1.4)
    logits[:, :, V - 1] += 9.0 * (np.arange(B) % 2)[:, None]          # the last value of the last slice is the likeliest one in every other sequence
    p = oracle.softmax_T(logits.astype(np.float64), T)
    q = oracle.softmax_T(logits[:, :gamma].astype(np.float64) + synth.make_logits((B, gamma, V), seed=seed, stream=1, std=0.5), T)
    x = _drafts(p, q, seed)
    it, sid = np.arange(B, dtype=np.uint32), np.full(B, 5, dtype=np.uint32)
    n_acc, out = torch.zeros(B, dtype=torch.int32, device=DEV), torch.zeros((B, gamma + 1), dtype=torch.int32, device=DEV)
    binding.sd_accept(to_dev(logits), to_dev(q), to_dev(x), T, seed, to_dev(it), to_dev(sid), n_acc, out, 1)
    n_acc, out = n_acc.cpu().numpy(), out.cpu().numpy()
    checked = 0
    for b in range(B):
        n_ref, out_ref = oracle.accept(p[b], q[b], x[b], seed, b, 5)
        if T > 0.0:
            u = np.array([oracle.uniform24(seed, b, s, 5, 1) for s in range(gamma)]) / 2.0**24
            lhs, rhs = u * q[b, np.arange(gamma), x[b]].astype(np.float64), p[b, np.arange(gamma), x[b]].astype(np.float64)
            if (np.abs(lhs - rhs) <= 1e-5 * rhs)[: min(n_ref + 1, gamma)].any():
                continue
            w = np.maximum(p[b, n_ref] - q[b, n_ref], 0).astype(np.float64) if n_ref < gamma else p[b, gamma].astype(np.float64)
            cdf = np.cumsum(w) / w.sum()
            at = oracle.uniform24(seed, b, n_ref, 5, 2) / 2.0**24
            if np.abs(cdf - at).min() <= 2e-6:             # V fp32 roundings of 2^-24 relative each, of p and of the sum, on weights that differ by less than p
                continue
        assert (n_acc[b], out[b].tolist()) == (n_ref, out_ref.tolist()), b
        checked += 1
    assert checked >= B // 2


@pytest.mark.parametrize("n,V", [(3, 8189), (3, 10007), (16, 50003)])       # a CTA per row; slices in one wave of clusters and in two
def test_draft_draws_on_both_sides_of_the_line(n, V):
    from paper_2505_08600_b200 import binding
    dims = dict(n_layers=1, d_model=64, n_heads=1, n_kv_heads=1, head_dim=64, d_ffn=64, vocab=V)
    ctx = binding.Context(dims, [dims], "bf16", n, 64, 3, 1.0, 7)
    w = synth.make_weights(dims, seed=3, dtype="bf16", std=0.3)
    ctx.load_weights(0, w); ctx.load_weights(1, w)
    seqs = list(range(n))
    for s in seqs:
        ctx.sd_seq_begin(s, synth.make_prompt(V, 5 + s, seed=9, seq=s), 40 + s)
    ctx.sd_route_prompt(seqs, forced_task=[0] * n)
    ctx.sd_prefill(seqs)
    x, q = torch.zeros((n, 3), dtype=torch.int32, device=DEV), torch.zeros((n, 3, V), dtype=torch.float32, device=DEV)
    ctx.sd_draft_steps(seqs, 3, x, q)
    x, q = x.cpu().numpy(), q.cpu().numpy()
    ctx.close()
    for s in seqs:
        for j in range(3):
            assert abs(q[s, j].astype(np.float64).sum() - 1.0) <= 1e-5
            assert x[s, j] == oracle.sample_icdf(q[s, j], oracle.uniform24(7, 0, j, 40 + s, 0))


def test_no_drafts_is_plain_sampling_over_slices():
    from paper_2505_08600_b200 import binding
    B, V, seed = 4, 20011, 8
    p = oracle.softmax_T(synth.make_logits((B, 1, V), seed=1).astype(np.float64), 1.0)
    it, sid = np.arange(B, dtype=np.uint32), np.full(B, 2, dtype=np.uint32)
    n_acc, out = torch.full((B,), -9, dtype=torch.int32, device=DEV), torch.full((B, 1), -9, dtype=torch.int32, device=DEV)
    binding.sd_accept(to_dev(p), None, None, 1.0, seed, to_dev(it), to_dev(sid), n_acc, out, 0)
    assert n_acc.tolist() == [0] * B
    assert out[:, 0].tolist() == [oracle.sample_icdf(p[b, 0], oracle.uniform24(seed, b, 0, 2, 2)) for b in range(B)]
