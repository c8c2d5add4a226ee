"""Rows whose logits are not finite.  Box 1's softmax has no value there: the
confidence is NaN (never at or above a threshold, so such a row is not
committed by confidence) and the argmax is a vocabulary index, as the oracle
has it: 0 when every logit is NaN or -inf, the place of the +inf when there is
one.  The other rows of the call keep their values bit for bit."""
import numpy as np
import pytest
import torch

import oracle
import synth
import paper_2608_22646_gb300 as cai
from tests.test_zz_no_alloc import _check_against_oracle, _static

pytestmark = pytest.mark.gpu

TOP = 1234
SPECIAL = {3: 0, 7: 0, 11: TOP}  # row -> argmax


def _inputs(M, H, V):
    W = synth.lm_head_weight(V, H, seed=61, device="cuda")
    W[:, 0] = 1.0
    W[:, 1] = -1.0
    W[TOP, 1] = 1.0
    wl = synth.Workload("nonfinite", B=1, H=H, V=V, gen_len=M, P=M, T=4, a0="u04")
    good = synth.HiddenStates(wl, W, "calibrated", seed=6)(0, 0).reshape(M, H).contiguous()
    rows = good.clone()
    for r in SPECIAL:
        rows[r] = 0.0
    rows[3, 0] = float("nan")    # every logit NaN
    rows[7, 0] = float("-inf")   # every logit -inf
    rows[11, 1] = float("inf")   # one +inf, the others -inf
    return W, good, rows


def _check(conf, arg, conf0, arg0):
    rest = np.setdiff1d(np.arange(len(conf)), list(SPECIAL))
    for r, ix in SPECIAL.items():
        assert np.isnan(conf[r]) and arg[r] == ix, (r, conf[r], arg[r])
    assert np.array_equal(conf[rest], conf0[rest]) and np.array_equal(arg[rest], arg0[rest])


def test_oracle_has_the_same_values():
    W, _, rows = _inputs(12, 64, 2000)
    o = oracle.head_rows(W, rows)
    for r, ix in SPECIAL.items():
        assert np.isnan(o["conf"][r]) and o["idx"][r] == ix


@pytest.mark.parametrize("V,H,M", [
    (4100, 256, 40),    # unswapped
    (4100, 448, 40),    # swapped, two K blocks per stage
    (4100, 1024, 100),  # unswapped, H above 384
])
def test_static_head(V, H, M):
    W, good, rows = _inputs(M, H, V)
    conf0, arg0 = _static(W, good)
    _check_against_oracle(W, good, conf0, arg0)
    _check(*_static(W, rows), conf0, arg0)


@pytest.mark.parametrize("B,P,H,env", [
    (1, 32, 256, {}),                            # rows-operand head
    (3, 33, 256, {"CAI_FUSED_MAX_BP": "128"}),   # ... 99 rows
    (5, 40, 256, {}),                            # pair head, unswapped
    (5, 40, 256, {"CAI_PAIR_SWAP_MAX_N": "256"}),
    (12, 40, 448, {"CAI_PAIR_CLUSTERS": "3", "CAI_PAIR_SWAP_MAX_N": "256"}),  # per-tile partials
    (12, 40, 448, {"CAI_PAIR_CLUSTERS": "3", "CAI_PAIR_SWAP": "0"}),
])
def test_first_step(B, P, H, env, monkeypatch):
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    V = 4100
    W, good, rows = _inputs(B * P, H, V)
    cfg = cai.cai_config_default(cai.CAI_PRESET_LLADA, B, P, H, V, 8, 1)
    with cai.cai_init(cfg, W) as ctx:
        got = []
        for h in (good, rows):
            cai.cai_reset(ctx)
            cai.cai_first_step(ctx, h.reshape(B, P, H))
            torch.cuda.synchronize()
            st = cai.cai_state_download(ctx)
            assert np.array_equal(st["conf"], st["s0"], equal_nan=True)
            got += [st["conf"].reshape(-1), st["cand"].reshape(-1)]
        _check(got[2], got[3], got[0], got[1])
        assert all(st["tok"].reshape(-1)[r] == cai.CAI_MASK_TOKEN for r in SPECIAL)
