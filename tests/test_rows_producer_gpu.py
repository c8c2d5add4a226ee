"""Steps of 65 to 128 rows right behind a kernel that lets its dependents start
before it has written the rows they are to read: the merge of the
allocation-free head, whose confidences land in the step's hidden states here.
A step must wait for it, single-kernel or not."""
import numpy as np
import pytest
import torch

import synth
import paper_2608_22646_gb300 as cai

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("env", [{}, {"CAI_FUSED_MAX_BP": "128"},
                                 {"CAI_FUSED_MAX_BP": "128", "CAI_ROWS_HEAD": "0"}])
@pytest.mark.parametrize("norm", [False, True])
def test_rows_written_late(env, norm, monkeypatch):
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    B, P, H, V = 2, 33, 64, 3000
    W = synth.lm_head_weight(V, H, seed=71, device="cuda")
    cfg = cai.cai_config_default(cai.CAI_PRESET_LLADA, B, P, H, V, 4, 1)
    # A long head of few CTAs: every confidence rounds to 1, as bf16 (0, 1).
    Wp = synth.lm_head_weight(128, 16384, seed=72, device="cuda")
    rows = (Wp.float().repeat(2, 1) * 400.0).to(torch.bfloat16)
    argmax = torch.zeros(256, dtype=torch.int32, device="cuda")
    buf = torch.zeros(B * P * H // 2, dtype=torch.float32, device="cuda")
    hidden = buf.view(torch.bfloat16).reshape(B, P, H)
    start = synth.lm_head_weight(B * P, H, seed=73, device="cuda").reshape(B, P, H) * 50
    if norm:
        ctx = cai.cai_init_rmsnorm(cfg, W, synth.final_norm_weight(H, device="cuda"), 1e-5)
    else:
        ctx = cai.cai_init(cfg, W)
    with ctx:
        assert (cai.cai_get_stats(ctx)["kernels_per_step"] == 1) == bool(env)
        ends = []
        for sync in (True, False):
            cai.cai_reset(ctx)
            for t in range(3):
                hidden.copy_(start)
                torch.cuda.synchronize()
                cai.cai_head_rows_static(Wp, rows, buf[:256], argmax)
                if sync:
                    torch.cuda.synchronize()
                    assert torch.all(buf[:256] == 1.0)
                (cai.cai_denoise_step if t else cai.cai_first_step)(ctx, hidden)
                torch.cuda.synchronize()
                ends.append(cai.cai_state_download(ctx))
    for a, b in zip(ends[:3], ends[3:]):
        for f in ("tok", "conf", "cand", "m_hist"):
            assert np.array_equal(a[f], b[f]), f
