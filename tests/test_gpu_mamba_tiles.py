"""Chunks, tiles and tables of the Mamba classifier's kernels at the sizes where they begin and end, against the CPU oracle."""
import numpy as np
import pytest
import torch

from oracle import classifier_mamba as om
from paper_2505_08600_b200 import synth
from gpu_util import DEV

pytestmark = pytest.mark.gpu


def _check(w, lens, vocab, seed, oracle_of=None):
    """Scores of a queue within the fp32 bound of test_gpu_mamba (2e-4 of one plus the largest score) of the oracle's, for the prompts listed."""
    from paper_2505_08600_b200 import binding as sd
    prompts = [synth.make_prompt(vocab, n, seed=seed, seq=i) for i, n in enumerate(lens)]
    starts = np.concatenate([[0], np.cumsum([len(p) for p in prompts])[:-1]])
    scores, labels = sd.MambaClassifier(w).classify(torch.from_numpy(np.concatenate(prompts)).to(DEV), starts, lens)
    scores, labels = scores.cpu().numpy(), labels.cpu().numpy()
    for i in range(len(lens)) if oracle_of is None else oracle_of:
        ref, _, _ = om.forward(w, prompts[i])
        np.testing.assert_allclose(scores[i].astype(np.float64), ref, rtol=0, atol=2e-4 * (1.0 + np.abs(ref).max()))
    assert (labels == scores.argmax(1)).all()
    return scores


# (d_model, states, taps, expand): rank 8 with 16 states and 4 taps is the compiled form, rank 4 the same without it; 260 channels take two CTAs
@pytest.mark.parametrize("d_model,d_state,d_conv,expand", [(128, 16, 4, 2), (64, 16, 4, 2), (128, 16, 3, 1), (36, 7, 4, 1), (130, 15, 7, 2)])
@pytest.mark.parametrize("lens", [[1, 15, 16, 17, 31, 32, 33, 63, 64], [2, 65, 95, 96, 97, 127, 129, 161]], ids=["single_chunk", "several_chunks"])
def test_prompts_that_end_at_the_edges_of_tiles_and_chunks(d_model, d_state, d_conv, expand, lens):
    w = synth.make_mamba_classifier(200, d_model=d_model, d_state=d_state, d_conv=d_conv, expand=expand, n_classes=3, seed=d_model + d_conv)
    _check(w, lens, 200, seed=d_state)


@pytest.mark.parametrize("n", [32, 33, 1024, 1025])
def test_queues_that_fill_a_table_of_prompts(n):
    w = synth.make_mamba_classifier(100, d_model=32, d_state=4, d_conv=4, expand=1, n_classes=2, seed=n)
    lens = [1 + (7 * i) % 70 for i in range(n)]
    some = sorted({0, 1, 31, n // 2, n - 2, n - 1} & set(range(n)))
    all_scores = _check(w, lens, 100, seed=3, oracle_of=some)
    alone = _check(w, lens[:1], 100, seed=3)
    assert (alone[0] == all_scores[0]).all()                     # whatever table a prompt comes in


def test_a_capture_is_refused():
    from paper_2505_08600_b200 import binding as sd
    clf = sd.MambaClassifier(synth.make_mamba_classifier(50, d_model=16, d_state=4, d_conv=4, expand=1, n_classes=2, seed=1))
    tokens = torch.zeros(8, dtype=torch.int32, device=DEV)
    clf.classify(tokens, [0], [8])
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with pytest.raises(RuntimeError):
        with torch.cuda.graph(graph):
            clf.classify(tokens, [0], [8])
    torch.cuda.synchronize()


def test_the_call_waits_for_nothing_and_has_read_its_host_tables():
    """Offsets and lengths are overwritten as soon as the call returns, before the stream (held up for some ten milliseconds) has come to it."""
    from paper_2505_08600_b200 import binding as sd
    clf = sd.MambaClassifier(synth.make_mamba_classifier(90, d_model=32, d_state=4, d_conv=4, expand=1, n_classes=3, seed=2))
    for n in (3, 40):                                            # a table of up to 32 prompts, a longer one
        lens = np.array([5 + 31 * (i % 5) for i in range(n)], dtype=np.int32)
        starts = np.concatenate([[0], np.cumsum(lens)[:-1]]).astype(np.int64)
        tokens = torch.arange(int(lens.sum()), dtype=torch.int32, device=DEV) % 90
        want, _ = clf.classify(tokens, starts, lens)
        torch.cuda.synchronize()
        torch.cuda._sleep(20_000_000)
        got, _ = clf.classify(tokens, starts, lens)
        held = not torch.cuda.current_stream().query()
        starts[:], lens[:] = 0, 1
        assert held
        assert torch.equal(got, want)
