"""Time stamps of the launches of a pass: which records a draft pass (matrix and step in one kernel), a mixed verify pass and a prompt
pass leave, and that every record has a beginning, a dependency and an end in that order."""
import numpy as np
import pytest
import torch

from paper_2505_08600_b200 import synth
from gpu_util import DEV

pytestmark = pytest.mark.gpu

GEMM, STEP, ATTENTION, MATRIX = range(4)
PLAIN, QKV, RESIDUAL, SWIGLU = (k << 8 for k in range(4))


def _m(L, d, H, hd, F, V):
    return dict(n_layers=L, d_model=d, n_heads=H, n_kv_heads=H, head_dim=hd, d_ffn=F, vocab=V)


@pytest.mark.parametrize("adapters", [0, 2])
def test_records_of_every_kind_of_pass(adapters):
    from paper_2505_08600_b200 import binding
    V, gamma = 512, 2
    target, draft = _m(2, 1024, 4, 64, 4608, V), _m(2, 256, 4, 64, 320, V)         # the target streams gate/up and down
    lora = dict(lora_adapters=adapters, lora_rank=8, lora_scale=1.0) if adapters else {}
    ctx = binding.Context(target, [draft], "bf16", 1, 96, gamma, 1.0, 7, stream=torch.cuda.Stream(), **lora)
    ctx.load_weights(0, synth.make_weights(target, seed=3, model_index=0, dtype="bf16"))
    ctx.load_weights(1, synth.make_weights(draft, seed=3, model_index=1, dtype="bf16"))
    ctx.sd_launch_stamps(1)
    x, q = torch.zeros((1, gamma), dtype=torch.int32, device=DEV), torch.zeros((1, gamma, V), device=DEV)
    logits = torch.zeros((1, gamma + 1, V), device=DEV)
    torch.cuda.synchronize()
    t = [MATRIX | PLAIN] if adapters else []                                       # x A^T in front of a draft's matrix
    tg = [GEMM | PLAIN] if adapters else []
    prompt = tg + [MATRIX | QKV, ATTENTION] + tg + [GEMM | RESIDUAL, STEP | RESIDUAL] + tg + [MATRIX | SWIGLU] + tg + [GEMM | RESIDUAL, STEP | RESIDUAL]
    layer = t + [MATRIX | QKV, ATTENTION] + t + [MATRIX | RESIDUAL] + t + [MATRIX | SWIGLU] + t + [MATRIX | RESIDUAL]
    mixed = [MATRIX | QKV, ATTENTION, MATRIX | RESIDUAL, GEMM | SWIGLU, STEP | SWIGLU, GEMM | RESIDUAL, STEP | RESIDUAL]

    def check(want):
        stamps, kinds = ctx.sd_launch_stamps_read()
        assert kinds.tolist() == want
        s = stamps.astype(np.int64)
        assert (s[:, [0, 1, 2, 5, 6]] > 0).all()
        assert (s[:, 0] <= s[:, 1]).all() and (s[:, 1] <= s[:, 2]).all() and (s[:, 1] <= s[:, 5]).all() and (s[:, 5] <= s[:, 6]).all() and (s[:, 2] <= s[:, 6]).all()
        ring = np.array([k & 0xff == GEMM for k in kinds])
        assert (s[ring][:, 3] >= s[ring][:, 0]).all() and (s[ring][:, 3] > 0).all()

    ctx.sd_seq_begin(0, synth.make_prompt(V, 50, seed=9), 0)
    ctx.sd_route_prompt([0], forced_task=[0])
    ctx.sd_prefill([0])
    check(prompt + tg + [MATRIX | QKV])                                            # the draft's: its last layer ends with keys and values
    for _ in range(2):                                                             # captured, replayed
        ctx.sd_draft_steps([0], gamma, x, q)
        check(2 * layer + [MATRIX | PLAIN])
        ctx.sd_verify([0], gamma, x, logits)
        check(2 * mixed + [MATRIX | PLAIN])
    ctx.close()
