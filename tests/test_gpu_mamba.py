"""Mamba-based prompt classifier of the CUDA library against the CPU oracle (through the C ABI)."""
import numpy as np
import pytest
import torch

from oracle import classifier_mamba as om
from paper_2505_08600_b200 import synth
from gpu_util import DEV

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sd():
    from paper_2505_08600_b200 import binding
    binding.lib()
    return binding


def _compare(sd, w, lens, vocab, seed):
    clf = sd.MambaClassifier(w)
    prompts = [synth.make_prompt(vocab, n, seed=seed, seq=i) for i, n in enumerate(lens)]
    gap = 5                                                      # prompts sit apart in the token buffer, as sequences do in the library
    starts, flat, at = [], [], 0
    for p in prompts:
        starts.append(at); flat += p.tolist() + [vocab - 1] * gap; at += len(p) + gap
    tokens = torch.tensor(flat, dtype=torch.int32, device=DEV)
    scores, labels = clf.classify(tokens, starts, lens)
    torch.cuda.synchronize()
    scores, labels = scores.cpu().numpy().astype(np.float64), labels.cpu().numpy()
    for i, p in enumerate(prompts):
        ref, _, _ = om.forward(w, p)
        tol = 2e-4 * (1.0 + np.abs(ref).max())                   # fp32 sums over up to 1000 tokens against fp64
        np.testing.assert_allclose(scores[i], ref, rtol=0, atol=tol)
        top2 = np.sort(ref)[-2:]
        if top2[1] - top2[0] > 2 * tol:
            assert labels[i] == int(np.argmax(ref))
        assert labels[i] == int(np.argmax(scores[i].astype(np.float32)))
    return scores, labels


def test_classifier_at_the_default_sizes_ragged_prompts_across_chunk_boundaries(sd):
    vocab = 3000
    w = synth.make_mamba_classifier(vocab, d_model=128, d_state=16, d_conv=4, expand=2, n_classes=4, seed=1)
    _compare(sd, w, [1, 2, 3, 4, 5, 63, 64, 65, 128, 129, 200, 1000], vocab, seed=3)


def test_short_prompts_only_take_the_single_chunk_path(sd):
    vocab = 500
    w = synth.make_mamba_classifier(vocab, d_model=128, d_state=16, d_conv=4, expand=2, n_classes=3, seed=2)
    _compare(sd, w, [32, 17, 64, 1], vocab, seed=4)


def test_other_sizes(sd):
    vocab = 300
    w = synth.make_mamba_classifier(vocab, d_model=48, d_state=5, d_conv=3, expand=1, n_classes=2, seed=7)      # odd sizes: 48 channels, 5 states, 3 taps
    _compare(sd, w, [70, 9, 300], vocab, seed=5)
    w = synth.make_mamba_classifier(vocab, d_model=256, d_state=8, d_conv=4, expand=2, n_classes=5, seed=8)
    _compare(sd, w, [150, 40], vocab, seed=6)


def test_long_prompt_many_chunks_and_batch_independence(sd):
    vocab = 1000
    w = synth.make_mamba_classifier(vocab, d_model=128, d_state=16, d_conv=4, expand=2, n_classes=4, seed=3)
    s_all, _ = _compare(sd, w, [4100, 77], vocab, seed=9)
    clf = sd.MambaClassifier(w)
    p1 = synth.make_prompt(vocab, 77, seed=9, seq=1)
    s1, _ = clf.classify(torch.from_numpy(p1).to(DEV), [0], [77])
    assert (s1.cpu().numpy()[0] == s_all[1].astype(np.float32)).all()          # a prompt's scores do not depend on its neighbours


def test_routing_through_the_context_and_unsupported_sizes(sd):
    cfg = synth.CONFIGS["tiny"]
    t = cfg["target"]
    ctx = sd.Context(t, cfg["drafts"], "f32", 3, 128, 4, 1.0, 9)
    w = synth.make_mamba_classifier(t["vocab"], d_model=64, d_state=8, d_conv=4, expand=2, n_classes=len(cfg["drafts"]), seed=4)
    clf = sd.MambaClassifier(w)
    prompts = [synth.make_prompt(t["vocab"], n, seed=6, seq=i) for i, n in enumerate([20, 70, 33])]
    for s, p in enumerate(prompts):
        ctx.sd_seq_begin(s, p, s)
    got = ctx.sd_route_prompt_mamba(clf, [0, 1, 2])
    want = [om.classify(w, p)[0] for p in prompts]
    margins = [np.sort(om.classify(w, p)[1])[-1] - np.sort(om.classify(w, p)[1])[-2] for p in prompts]
    for g, r, mg in zip(got.tolist(), want, margins):
        assert mg < 1e-3 or g == r
    ctx.sd_prefill([0, 1, 2])                                              # routed sequences continue down the normal path
    ctx.close()
    big = synth.make_mamba_classifier(100, d_model=64, d_state=32, d_conv=4, expand=2, n_classes=2, seed=1)      # 32 states: not supported
    with pytest.raises(RuntimeError):
        sd.MambaClassifier(big).classify(torch.zeros(8, dtype=torch.int32, device=DEV), [0], [8])


def test_workspace_at_a_multiple_of_eight_bytes(sd):
    """The workspace needs the alignment of its 64-bit words and no more: the same scores, bit for bit, from one eight bytes further on."""
    import ctypes
    vocab, lens = 500, np.array([70, 9, 300], dtype=np.int32)
    clf = sd.MambaClassifier(synth.make_mamba_classifier(vocab, d_model=64, d_state=16, d_conv=4, expand=2, n_classes=4, seed=5))
    tokens = torch.from_numpy(np.concatenate([synth.make_prompt(vocab, int(n), seed=6, seq=i) for i, n in enumerate(lens)])).to(DEV)
    starts = np.array([0, 70, 79], dtype=np.int64)
    want, _ = clf.classify(tokens, starts, lens)
    need = sd.lib().sd_mamba_workspace(ctypes.byref(clf.desc), int(lens.sum()), 3)
    buf, scores = torch.empty(need + 16, dtype=torch.uint8, device=DEV), torch.zeros((3, 4), dtype=torch.float32, device=DEV)
    assert buf.data_ptr() % 16 == 0
    status = sd.lib().sd_mamba_classify(ctypes.byref(clf.desc), ctypes.byref(clf.w), tokens.data_ptr(), starts.ctypes.data_as(ctypes.c_void_p),
                                        lens.ctypes.data_as(ctypes.c_void_p), 3, scores.data_ptr(), None, buf.data_ptr() + 8, need, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert status == 0 and torch.equal(scores, want)


def test_classifiers_of_other_sizes_on_several_threads(sd):
    """A large and a small classifier called from two threads on streams of their own: neither call changes what the other may launch."""
    import threading
    calls = []
    for d_model, seed in ((512, 3), (16, 4)):
        clf = sd.MambaClassifier(synth.make_mamba_classifier(100, d_model=d_model, d_state=16, d_conv=4, expand=2, n_classes=4, seed=seed))
        tokens = torch.from_numpy(synth.make_prompt(100, 90, seed=6)).to(DEV)
        calls.append((clf, tokens, clf.classify(tokens, [0], [90])[0], torch.cuda.Stream()))
    torch.cuda.synchronize()
    wrong = []

    def loop(clf, tokens, want, stream):
        try:
            with torch.cuda.stream(stream):
                for _ in range(1500):
                    scores, _ = clf.classify(tokens, [0], [90])
                stream.synchronize()
                if not torch.equal(scores, want):
                    wrong.append("scores")
        except RuntimeError as e:
            wrong.append(str(e))

    threads = [threading.Thread(target=loop, args=c) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong


@pytest.mark.parametrize("d_model,expand,d_state,d_conv", [(512, 2, 16, 4), (150, 2, 16, 3), (257, 1, 5, 4), (129, 6, 8, 6)])
def test_channels_of_several_ctas(sd, d_model, expand, d_state, d_conv):
    """More than 256 channels: two to four CTAs per chunk, the last with fewer channels, channels that are no multiple of four (257, 774)."""
    vocab = 200
    w = synth.make_mamba_classifier(vocab, d_model=d_model, d_state=d_state, d_conv=d_conv, expand=expand, n_classes=3, seed=12)
    _compare(sd, w, [1, 31, 33, 64, 150], vocab, seed=8)


@pytest.mark.parametrize("d_model,expand,d_state,d_conv", [(64, 2, 16, 4), (37, 1, 5, 3), (300, 1, 8, 4)])
def test_prompts_around_the_length_from_which_the_carry_has_a_kernel(sd, d_model, expand, d_state, d_conv):
    """15, 16 and 17 chunks, and 40, beside short prompts; channels that do not fill a CTA's eight; a prompt's scores do not depend on its
    neighbours' lengths."""
    vocab = 300
    w = synth.make_mamba_classifier(vocab, d_model=d_model, d_state=d_state, d_conv=d_conv, expand=expand, n_classes=4, seed=13)
    lens = [960, 961, 1024, 1025, 2500, 30, 100]
    scores, _ = _compare(sd, w, lens, vocab, seed=10)
    clf = sd.MambaClassifier(w)
    for i in (0, 1, 6):
        alone, _ = clf.classify(torch.from_numpy(synth.make_prompt(vocab, lens[i], seed=10, seq=i)).to(DEV), [0], [lens[i]])
        assert (alone.cpu().numpy()[0] == scores[i].astype(np.float32)).all()
