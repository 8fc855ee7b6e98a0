"""Attention over the cache in each form the launch picks (eight warps with clusters of four, two and one; four warps with clusters of four,
two and one; at most eight query vectors per tile and more), against the CPU oracle: lengths that end a chunk, one more and one less,
rows far from one another, an inactive row, a sequence of one position."""
import numpy as np
import pytest
import torch

import oracle
from paper_2505_08600_b200 import synth
from gpu_util import DEV, quantize, to_dev, widen

pytestmark = pytest.mark.gpu

TOL = 2e-2          # bf16 output rounding: 2^-9 relative on values up to ~3 (as in test_gpu_ops)


# heads, kv heads, head dim, rows per sequence, last positions of the sequences
FORMS = {
    "8w_c4": (8, 8, 128, 6, [300]),
    "8w_c2": (16, 16, 64, 6, [127, 128, 500, 6]),
    "8w_c1": (40, 40, 128, 2, [60, 5, 127]),
    "4w_c4": (32, 32, 128, 1, [899, 0, 255]),                       # 96 items, 384 CTAs
    "4w_c4_gqa": (32, 8, 64, 4, [700, 63, 64, 65, 400, 33, 511, 512, 3, 640, 256, 90]),      # 96 items of 16 query vectors
    "4w_c2": (32, 32, 128, 6, [400, 399, 401, 380, 350, 420]),       # 192 items
    "4w_c1": (40, 40, 64, 8, [255, 254, 129, 128, 127, 200]),        # 240 items
    "4w_many": (40, 40, 64, 9, [100, 64, 65, 63, 9, 120, 80, 127]),  # more than 2 per SM; nine query vectors
    "slices": (16, 16, 128, 3, [2500, 1024, 2047]),                  # contexts cut into slices
}


@pytest.mark.parametrize("name", sorted(FORMS))
def test_every_form_follows_the_oracle(name):
    from paper_2505_08600_b200 import binding as sd
    H, Hkv, hd, rps, last = FORMS[name]
    max_ctx, n = max(last) + 1, len(last)
    rng = np.random.default_rng(len(name))
    q = quantize(synth.make_logits((n * rps, H, hd), seed=21, stream=hd), "bf16")
    kc = quantize(synth.make_logits((n, Hkv, max_ctx, hd), seed=22, stream=hd), "bf16")
    vc = quantize(synth.make_logits((n, Hkv, max_ctx, hd), seed=23, stream=hd), "bf16")
    slots = np.repeat(np.arange(n, dtype=np.int32)[::-1], rps)
    pos = np.concatenate([np.arange(p - rps + 1, p + 1) for p in last]).astype(np.int32)
    pos[pos < 0] = -1                                               # (rows in front of a short sequence's first position are inactive)
    out = torch.full((n * rps, H, hd), 7.0, dtype=torch.bfloat16, device=DEV)
    args = (to_dev(q), to_dev(kc), to_dev(vc), out, to_dev(slots.copy()), to_dev(pos), H, Hkv, hd, max_ctx, sd.SD_BF16)
    sd.sd_op_attention(*args, rows_per_seq=rps)
    got = out.float().cpu().numpy().astype(np.float64)
    qf, kf, vf = widen(q), widen(kc), widen(vc)
    for r in range(n * rps):
        for h in sorted({0, H - 1, *rng.integers(0, H, 2).tolist()}):
            if pos[r] < 0:
                assert (got[r, h] == 0).all()
                continue
            m = pos[r] + 1
            ref = oracle.attention_head(qf[r, h], kf[slots[r], h // (H // Hkv), :m], vf[slots[r], h // (H // Hkv), :m])
            np.testing.assert_allclose(got[r, h], ref, rtol=0, atol=TOL, err_msg=f"row {r} head {h}")
    again = torch.zeros_like(out)
    sd.sd_op_attention(*args[:3], again, *args[4:], rows_per_seq=rps)
    assert torch.equal(out, again)


def test_scores_that_grow_and_shrink_from_tile_to_tile():
    """The running maximum moves in every tile, in none, and from far below: keys scaled up, down, and up at the very end."""
    from paper_2505_08600_b200 import binding as sd
    H, hd, m = 4, 128, 640
    q = quantize(synth.make_logits((3, H, hd), seed=31, stream=1), "bf16")
    base = synth.make_logits((3, H, m, hd), seed=32, stream=1)
    for s, scale in enumerate([np.linspace(0.1, 6, m), np.linspace(6, 0.1, m), np.where(np.arange(m) < m - 1, 1e-3, 8.0)]):
        base[s] *= scale[None, :, None]
    kc, vc = quantize(base, "bf16"), quantize(synth.make_logits((3, H, m, hd), seed=33, stream=1), "bf16")
    out = torch.zeros((3, H, hd), dtype=torch.bfloat16, device=DEV)
    sd.sd_op_attention(to_dev(q), to_dev(kc), to_dev(vc), out, to_dev(np.arange(3, dtype=np.int32)), to_dev(np.full(3, m - 1, dtype=np.int32)), H, H, hd, m,
                       sd.SD_BF16, rows_per_seq=1)
    got = out.float().cpu().numpy().astype(np.float64)
    qf, kf, vf = widen(q), widen(kc), widen(vc)
    for s in range(3):
        for h in range(H):
            np.testing.assert_allclose(got[s, h], oracle.attention_head(qf[s, h], kf[s, h], vf[s, h]), rtol=0, atol=TOL)


# Around one wave of CTAs (every launch of an operator counts all contexts as the longest): pairs of four warps, four warps alone, eight warps with
# more than eight query vectors and with heads of 64; below it four CTAs of four warps from 513 positions on, with heads of 128 from 769.
AROUND_ONE_WAVE = {
    "pairs": (40, 40, 128, 1, [1030, 15, 300, 1023]),                           # 320 items in two slices each: more than two per SM; the slices' merge
    "pairs_one_slice": (32, 32, 128, 8, [700, 31, 33, 512, 64]),                # 160 items
    "alone_512": (32, 32, 128, 6, [511, 64, 65, 127, 128, 500, 8, 300]),        # 256 items
    "alone_513": (32, 32, 128, 6, [512, 64, 65, 127, 128, 500, 8, 300]),
    "nine_vectors": (32, 32, 128, 9, [200, 64, 65, 127, 128]),
    "fours_513": (12, 12, 64, 2, [512, 63, 64, 65, 300, 127, 128, 15, 256]),     # 108 items
    "eight_512": (12, 12, 64, 2, [511, 63, 64, 65, 300, 127, 128, 15, 256]),
    "fours_769": (32, 32, 128, 1, [768, 63, 64]),                               # 96 items
    "eight_768": (32, 32, 128, 1, [767, 63, 64]),
    "heads_of_64": (40, 40, 64, 1, [255, 254, 129, 128, 127, 200]),             # 240 items
}


@pytest.mark.parametrize("name", sorted(AROUND_ONE_WAVE))
def test_forms_around_one_wave(name, monkeypatch):
    monkeypatch.setitem(FORMS, name, AROUND_ONE_WAVE[name])
    test_every_form_follows_the_oracle(name)


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("call", ["draft", "verify", "step", "verify_accept"])
def test_what_a_call_returns_does_not_depend_on_the_lengths_that_its_graph_was_captured_at(call, head_dim):
    """Attention's form follows the lengths of all sequences: the same five slots with one long context (eight warps), then with five (four warps in
    clusters of two), the longest alike.  The second call returns bit for bit what it returns in a context that never saw the first, and without graphs."""
    from paper_2505_08600_b200 import binding
    V, gamma, seqs = 512, 3, list(range(5))
    target = dict(n_layers=2, d_model=256, n_heads=32, n_kv_heads=32, head_dim=head_dim, d_ffn=256, vocab=V)      # 160 (head, sequence) items
    weights = [synth.make_weights(target, seed=3, model_index=k, dtype="bf16") for k in range(2)]

    def results(ctx, lens):
        for s in seqs:
            ctx.sd_seq_begin(s, synth.make_prompt(V, lens[s], seed=9, seq=s), s)
        ctx.sd_route_prompt(seqs, forced_task=[0] * 5)
        ctx.sd_prefill(seqs)
        if call == "draft":
            ctx.sd_draft_steps(seqs, gamma, x, q)
            return x.clone(), q.clone()
        if call == "step":
            ctx.sd_target_step(seqs, logits[:, 0])
            return (logits.flatten()[: 5 * V].clone(),)
        if call == "verify":
            ctx.sd_verify(seqs, gamma, given, logits)
        else:
            ctx.sd_verify_accept(seqs, gamma, given, given_q, logits, n_acc, out_tok)
        return logits.clone(), n_acc.clone(), out_tok.clone()

    x, q = torch.zeros((5, gamma), dtype=torch.int32, device=DEV), torch.zeros((5, gamma, V), device=DEV)
    given, given_q = torch.full((5, gamma), 7, dtype=torch.int32, device=DEV), torch.full((5, gamma, V), 1.0 / V, device=DEV)
    logits, n_acc, out_tok = torch.zeros((5, gamma + 1, V), device=DEV), torch.zeros(5, dtype=torch.int32, device=DEV), torch.zeros((5, gamma + 1), dtype=torch.int32, device=DEV)
    torch.cuda.synchronize()
    mixed, alike = [900, 40, 40, 40, 40], [900] * 5
    got = []
    for graphs, first in ((1, mixed), (1, None), (0, None)):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            ctx = binding.Context(target, [target], "bf16", 5, 1024, gamma, 1.0, 7, stream=stream)
            for k in range(2):
                ctx.load_weights(k, weights[k])
            ctx.sd_use_graphs(graphs)
            if first:
                results(ctx, first)
            got.append(results(ctx, alike))
            assert ctx.sd_device_status() == 0
            ctx.close()
        torch.cuda.synchronize()
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert torch.equal(a, b)
