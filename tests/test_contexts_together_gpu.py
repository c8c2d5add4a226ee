"""Contexts of different shapes alive at once, made in either order and stepped
in turn.  They share kernels (and so each kernel's launch limits on the device)
and nothing else: every step must run and agree with the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
import paper_2608_22646_gb300 as cai
from tests import parity

pytestmark = pytest.mark.gpu


def _make(B, P, H, V, T, norm):
    wl = synth.Workload("together", B=B, H=H, V=V, gen_len=P, P=P, T=T, a0="u04")
    W = synth.lm_head_weight(V, H, seed=H + V, device="cuda")
    cfg = cai.cai_config_default(cai.CAI_PRESET_LLADA, B, P, H, V, T, 1)
    hs = synth.HiddenStates(wl, W, "calibrated", seed=7)
    if norm:
        ctx = cai.cai_init_rmsnorm(cfg, W, synth.final_norm_weight(H, seed=9, device="cuda"), 1e-5)
        return ctx, W, synth.PreNormHidden(hs, seed=8)
    return cai.cai_init(cfg, W), W, hs


@pytest.mark.parametrize("order", [1, -1])
@pytest.mark.parametrize("rows_head,norm,shapes", [
    # (B, P, H, V).  Rows-operand head, the same 32 rows: a CTA's share of V
    # sets the stage size.  Then contexts of other row counts.
    ("1", False, [(1, 32, 256, 40000), (1, 32, 256, 4096), (1, 16, 128, 700), (2, 32, 512, 9000)]),
    ("1", True, [(1, 32, 256, 40000), (1, 32, 256, 4096)]),
    ("0", False, [(1, 16, 256, 4096), (2, 32, 256, 4096)]),
    # Pair head: unswapped below H = 384 (no exchange buffer), swapped above.
    ("1", False, [(5, 40, 512, 3000), (5, 40, 256, 3000)]),
    ("1", True, [(5, 40, 512, 3000), (5, 40, 256, 3000)]),
])
def test_steps_in_turn(order, rows_head, norm, shapes, monkeypatch):
    monkeypatch.setenv("CAI_ROWS_HEAD", rows_head)
    T = 4
    made = []
    try:
        for s in shapes[::order]:
            made.append(_make(*s, T, norm))
        pre = [cai.cai_state_download(ctx) for ctx, _, _ in made]
        for t in range(T):
            for k, (ctx, W, hs) in enumerate(made):
                h = hs(0, t)
                (cai.cai_denoise_step if t else cai.cai_first_step)(ctx, h)
                torch.cuda.synchronize()
                post = cai.cai_state_download(ctx)
                parity.check_step(parity.oracle_config(ctx.cfg), oracle.bf16_bits(W), h, pre[k],
                                  post, 0, t, norm_weight=ctx.norm_weight, eps=ctx.norm_eps)
                pre[k] = post
    finally:
        for ctx, _, _ in made:
            cai.cai_free(ctx)


@pytest.mark.parametrize("names", [("dream", "llada"), ("llada", "dream")])
def test_both_full_size_models(names):
    made = []
    try:
        for n in names:
            wl = synth.WORKLOADS[n]
            made.append(_make(wl.B, wl.P, wl.H, wl.V, 4, False))
        pre = [cai.cai_state_download(ctx) for ctx, _, _ in made]
        for t in range(2):
            for k, (ctx, W, hs) in enumerate(made):
                h = hs(0, t)
                (cai.cai_denoise_step if t else cai.cai_first_step)(ctx, h)
                torch.cuda.synchronize()
                post = cai.cai_state_download(ctx)
                parity.check_controller_step(parity.oracle_config(ctx.cfg), pre[k], post, 0, t)
                if t == 0:
                    parity.check_rows_sampled(W, h, post, 0, [(0, 0), (0, 17)], ctx.cfg.P)
                pre[k] = post
        assert all(np.isfinite(p["s0"][0, :32]).all() for p in pre)
    finally:
        for ctx, _, _ in made:
            cai.cai_free(ctx)


@pytest.mark.parametrize("B,flags", [(2, 0), (5, 0), (5, cai.CAI_DIAGNOSTICS)])
@pytest.mark.parametrize("host", [False, True])
def test_init_on_a_side_stream(B, flags, host):
    # A context made on one non-blocking stream while the default stream is
    # busy (its work is ordered before nothing of theirs), stepped on another
    # as soon as cai_init has returned: the states of a context made and
    # stepped on the default stream.
    P, H, V, T = 40, 256, 3000, 4
    wl = synth.Workload("side", B=B, H=H, V=V, gen_len=P, P=P, T=T, a0="u04")
    W = synth.lm_head_weight(V, H, seed=3, device="cuda")
    hidden = [synth.HiddenStates(wl, W, "calibrated", seed=4)(0, t) for t in range(T)]
    g = synth.final_norm_weight(H, seed=9, device="cuda")
    cfg = cai.cai_config_default(cai.CAI_PRESET_LLADA, B, P, H, V, T, 1)
    cfg.flags |= flags
    ends = []
    for side in (False, True):
        torch.cuda.synchronize()
        made, run = (torch.cuda.Stream(), torch.cuda.Stream()) if side else (None, None)
        if side:
            torch.cuda._sleep(400_000_000)
        ctx = cai.cai_init_rmsnorm(cfg, W.cpu() if host else W, g.cpu() if host else g, 1e-5, made)
        try:
            for t in range(T):
                (cai.cai_denoise_step if t else cai.cai_first_step)(ctx, hidden[t], run)
            ends.append(cai.cai_state_download(ctx))
            assert cai.cai_test_check_guards(ctx) == 0
        finally:
            cai.cai_free(ctx)
    for f in ends[0]:
        assert np.array_equal(ends[0][f], ends[1][f], equal_nan=f == "drift"), f
