"""Vocabulary tiles of less than 128 rows per CTA (pair_even_rows): steps of
one row tile cut V evenly over the pairs, and the allocation-free head always
does.  Tile heights that are no multiple of 32, several tiles per pair, a
ragged last tile, both orientations and their edges in M; against the oracle
with the parity tolerances."""
import pytest

import synth
import paper_2608_22646_gb300 as cai
from tests import parity
from tests.test_zz_no_alloc import _check_against_oracle, _static

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("clusters,max_n,shape", [
    # V = 900 on one pair: four tiles of 2 x 120 rows, the last 2 x 90.
    (1, "256", (3, 70, 128, 900, 6, 1)),   # M = 210: 224-wide swapped tile
    (1, "0", (3, 70, 128, 900, 6, 1)),
    # V = 1301 on two pairs: tiles of 2 x 112 rows, three on one pair.
    (2, "192", (2, 40, 64, 1301, 6, 1)),
    (2, "0", (2, 40, 64, 1301, 6, 1)),
    # V = 72 on 76 pairs: tiles of 2 x 8 rows, the last CTA without any.
    (76, "192", (5, 30, 64, 72, 4, 1)),
    (76, "0", (5, 30, 64, 72, 4, 1)),
])
def test_context_steps(clusters, max_n, shape, monkeypatch):
    monkeypatch.setenv("CAI_PAIR_CLUSTERS", str(clusters))
    if max_n == "0":
        # min_M 1: the unswapped pair kernel decodes the narrow steps too
        monkeypatch.setenv("CAI_PAIR_SWAP", "0")
        monkeypatch.setenv("CAI_PAIR_MIN_M", "1")
    else:
        monkeypatch.setenv("CAI_PAIR_SWAP_MAX_N", max_n)
    B, P, H, V, T, nb = shape
    wl = synth.Workload("even", B=B, H=H, V=V, gen_len=P * nb, P=P, T=T, a0="u04")
    W = synth.lm_head_weight(V, H, seed=77, device="cuda")
    cfg = cai.cai_config_default(cai.CAI_PRESET_LLADA, B, P, H, V, T, nb)
    hs = synth.HiddenStates(wl, W, "calibrated", seed=4)
    with cai.cai_init(cfg, W) as ctx:
        rep, _ = parity.run_checked_trajectory(ctx, W, hs)
        assert rep.rows >= B * P
        assert cai.cai_test_check_guards(ctx) == 0


@pytest.mark.parametrize("V,H,M", [
    (128, 64, 1), (130, 64, 16), (4097, 128, 17), (4100, 64, 33),
    (21000, 192, 192), (21000, 192, 193), (21003, 64, 256),
])
def test_static_head(V, H, M):
    W = synth.lm_head_weight(V, H, seed=78, device="cuda")
    wl = synth.Workload("even", B=1, H=H, V=V, gen_len=M, P=M, T=4, a0="u04")
    h = synth.HiddenStates(wl, W, "calibrated", seed=6)(0, 1).reshape(M, H).contiguous()
    conf, arg = _static(W, h)
    _check_against_oracle(W, h, conf, arg)
