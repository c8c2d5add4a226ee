"""Single-kernel steps of up to 128 rows (several sequences committed in one
pass, alternating partial buffers, one or two K blocks per stage) and the
orientation rule of the pair head, against the oracle with the parity
tolerances."""
import numpy as np
import pytest
import torch

import synth
import paper_2608_22646_gb300 as cai
from tests import parity

pytestmark = pytest.mark.gpu


def _run(B, P, H, V, T, nb, flags=None, steps=None):
    wl = synth.Workload("single", B=B, H=H, V=V, gen_len=P * nb, P=P, T=T, a0="u04")
    W = synth.lm_head_weight(V, H, seed=91, device="cuda")
    cfg = cai.cai_config_default(cai.CAI_PRESET_LLADA, B, P, H, V, T, nb)
    if flags is not None:
        cfg.flags = flags
    hs = synth.HiddenStates(wl, W, "calibrated", seed=12)
    with cai.cai_init(cfg, W) as ctx:
        kernels = cai.cai_get_stats(ctx)["kernels_per_step"]
        for _ in range(2):  # a second generation starts on either buffer
            cai.cai_reset(ctx)
            rep, _ = parity.run_checked_trajectory(ctx, W, hs, max_steps=steps)
            assert rep.rows >= B * P
        assert cai.cai_test_check_guards(ctx) == 0
    return kernels


@pytest.mark.parametrize("B,P,H,V,flags", [
    (4, 32, 192, 1000, None),    # 128 rows, three K blocks: a stage of two and one of one
    (2, 64, 128, 3001, None),
    (1, 128, 64, 777, None),     # one K block
    (128, 1, 256, 520, None),    # as many sequences as rows
    (5, 13, 320, 2600, None),    # 65 rows, five K blocks
    (3, 33, 256, 40000, None),   # groups of more than one per CTA, 99 rows
    (3, 33, 256, 2600, cai.CAI_GATING | cai.CAI_POS_FACTOR | cai.CAI_DIAGNOSTICS),
    (3, 33, 256, 2600, cai.CAI_POS_FACTOR | cai.CAI_FLUSH_ON_EXIT),
])
def test_rows_up_to_128(B, P, H, V, flags, monkeypatch):
    monkeypatch.setenv("CAI_FUSED_MAX_BP", "128")
    assert _run(B, P, H, V, 6, 2, flags) == 1


@pytest.mark.parametrize("V,single", [(4096, True), (4095, False)])
def test_limit_by_weight(V, single):
    # 2 V H = 8 MiB at H = 1024, V = 4096: 99 rows run single-kernel from there.
    assert (_run(3, 33, 1024, V, 4, 1, steps=2) == 1) == single


def test_steps_back_to_back_equal_steps_alone(monkeypatch):
    # Small steps overlap their neighbours (two partial buffers, tickets and
    # commits in flight): the same generation, issued without a pause and with a
    # synchronisation after every step, ends in the same state bit for bit.
    monkeypatch.setenv("CAI_FUSED_MAX_BP", "128")
    B, P, H, V, T, nb = 4, 24, 128, 2000, 12, 3
    wl = synth.Workload("b2b", B=B, H=H, V=V, gen_len=P * nb, P=P, T=T, a0="u04")
    W = synth.lm_head_weight(V, H, seed=92, device="cuda")
    hs = synth.HiddenStates(wl, W, "calibrated", seed=13)
    hidden = [[hs(b, t) for t in range(T)] for b in range(nb)]
    cfg = cai.cai_config_default(cai.CAI_PRESET_LLADA, B, P, H, V, T, nb)
    ends = []
    with cai.cai_init(cfg, W) as ctx:
        for sync in (False, True, False):
            cai.cai_reset(ctx)
            for b in range(nb):
                if b:
                    cai.cai_block_advance(ctx)
                for t in range(T):
                    (cai.cai_denoise_step if t else cai.cai_first_step)(ctx, hidden[b][t])
                    if sync:
                        torch.cuda.synchronize()
            ends.append(cai.cai_state_download(ctx))
    for st in ends[1:]:
        for k in ("tok", "conf", "s0", "budget", "cstep", "cand", "ell", "eta", "exit_reason",
                  "exit_step", "unresolved", "m_hist"):
            assert np.array_equal(st[k], ends[0][k]), k


@pytest.mark.parametrize("B,P,H,V", [
    (7, 32, 3072, 900),    # 224 rows, H from 3072 on: one 224-wide swapped tile
    (7, 62, 3072, 600),    # 434 rows: two of them
    (5, 40, 320, 3000),    # H below 384: unswapped at every width
    (5, 40, 576, 3000),    # H below 768: swapped up to 64
    (5, 40, 1024, 1100),   # H below 1536: swapped up to 96
])
def test_orientation_rule(B, P, H, V):
    assert _run(B, P, H, V, 5, 1) > 1


def test_static_head_captured():
    # Both launches of the allocation-free head go into a captured graph.
    V, H, M = 5000, 256, 40
    W = synth.lm_head_weight(V, H, seed=93, device="cuda")
    wl = synth.Workload("cap", B=1, H=H, V=V, gen_len=M, P=M, T=4, a0="u04")
    hs = synth.HiddenStates(wl, W, "calibrated", seed=6)
    rows = hs(0, 1).reshape(M, H).contiguous()
    out = [(torch.zeros(M, device="cuda"), torch.zeros(M, dtype=torch.int32, device="cuda"))
           for _ in range(2)]
    cai.cai_head_rows_static(W, rows, *out[0])
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        cai.cai_head_rows_static(W, rows, *out[1])
    rows.copy_(hs(0, 2).reshape(M, H))
    for _ in range(3):
        g.replay()
    cai.cai_head_rows_static(W, rows, *out[0])
    torch.cuda.synchronize()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert float(out[0][0].min()) > 0.0
