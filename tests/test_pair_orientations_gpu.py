"""The orientations of the CTA-pair LM head that the default limit keeps small
hidden sizes away from: swapped tiles at H <= 256 (edges, ring depths, random
shapes, the final norm, vocabulary shards), the norm with evict-first weights,
the norm on single-kernel steps of 65 to 128 rows, swapped tiles of the
allocation-free head with an odd number of K blocks, and a shard step whose two
halves run on different streams.  Against the oracle with the parity
tolerances."""
import numpy as np
import pytest
import torch

import synth
import paper_2608_22646_gb300 as cai
from tests import parity
from tests import test_parity_gpu as base
from tests import test_vocab_shard_gpu as shards
from tests.test_zz_no_alloc import _check_against_oracle, _static

pytestmark = pytest.mark.gpu


@pytest.fixture
def swapped(monkeypatch):
    monkeypatch.setenv("CAI_PAIR_SWAP_MAX_N", "192")


@pytest.mark.parametrize("shape", [
    (1, 65, 64, 130, 6, 2), (3, 22, 128, 128, 6, 2), (7, 41, 192, 777, 6, 1), (2, 200, 64, 1000, 5, 1),
])
def test_edge_shapes(shape, swapped):
    base.test_multi_kernel_edge_shapes(shape)


@pytest.mark.parametrize("ring_max", ["2", "12"])
def test_ring_depths(ring_max, swapped, monkeypatch):
    base.test_pair_ring_depths(ring_max, monkeypatch)


@pytest.mark.parametrize("shape", [s for s in base._random_shapes(14, seed=2609) if s[0] * s[1] > 64])
def test_random_shapes(shape, swapped):
    base.test_random_shape_trajectories(shape)


@pytest.mark.parametrize("g,shape", [
    (2, (5, 64, 256, 4096, 10, 2)), (3, (3, 32, 128, 5000, 8, 2)), (4, (13, 40, 256, 4096, 8, 1)),
])
def test_shards(g, shape, swapped):
    shards.test_vocab_shards_match_full_vocabulary(g, shape)


def test_shards_default_limit():
    # H = 832: swapped up to 96; 200 rows start unswapped and narrow into it.
    shards.test_vocab_shards_match_full_vocabulary(2, (5, 40, 832, 3000, 8, 1))


def _norm(B, P, H, V, T, steps=None):
    wl = synth.Workload("norm", B=B, H=H, V=V, gen_len=P, P=P, T=T, a0="bimodal")
    W = synth.lm_head_weight(V, H, seed=55, device="cuda")
    g = synth.final_norm_weight(H, seed=9, device="cuda")
    cfg = cai.cai_config_default(cai.CAI_PRESET_LLADA, B, P, H, V, T, 1)
    hs = synth.HiddenStates(wl, W, "calibrated", seed=13)
    with cai.cai_init_rmsnorm(cfg, W, g, 1e-5) as ctx:
        kernels = cai.cai_get_stats(ctx)["kernels_per_step"]
        rep, _ = parity.run_checked_trajectory(ctx, W, synth.PreNormHidden(hs, seed=21),
                                               max_steps=steps)
        assert rep.rows >= B * P
    return kernels


@pytest.mark.parametrize("B,P,H,V", [
    (5, 64, 256, 4096),    # two 160-wide tiles, then one
    (3, 50, 192, 1003),    # one 160-wide tile, V % 8 != 0
    (13, 40, 128, 2000),   # 520 rows: three row tiles
])
def test_norm_swapped(B, P, H, V, swapped):
    assert _norm(B, P, H, V, 8) > 1


@pytest.mark.parametrize("B,P,H,V", [
    (5, 32, 3200, 16001),  # evict-first (98 MiB): one 160-wide swapped tile
    (5, 32, 1024, 50003),  # ... unswapped at 160 rows, swapped from 96 on
])
def test_norm_evict_first(B, P, H, V):
    assert _norm(B, P, H, V, 4, steps=3) > 1


@pytest.mark.parametrize("B,P,H,V", [
    (4, 32, 192, 1000),    # 128 rows, three K blocks in stages of two
    (1, 100, 64, 777),     # one K block
    (5, 13, 320, 2600),    # 65 rows
    (3, 33, 256, 40000),   # two groups a CTA
])
def test_norm_rows_up_to_128(B, P, H, V, monkeypatch):
    monkeypatch.setenv("CAI_FUSED_MAX_BP", "128")
    assert _norm(B, P, H, V, 6) == 1


@pytest.mark.parametrize("V,H,M", [
    (4099, 448, 33), (4099, 448, 64), (5003, 1088, 1), (5003, 1088, 32), (5003, 1088, 96),
    (5003, 1088, 97), (3001, 3136, 96), (3001, 3136, 97), (3001, 3136, 224), (3001, 3136, 225),
])
def test_static_head_odd_k_blocks(V, H, M):
    # Widths on both sides of the limit by H and of the two-K-block stages (96);
    # 7, 17 or 49 K blocks leave a stage of one.
    W = synth.lm_head_weight(V, H, seed=78, device="cuda")
    wl = synth.Workload("oddk", B=1, H=H, V=V, gen_len=M, P=M, T=4, a0="u04")
    hs = synth.HiddenStates(wl, W, "calibrated", seed=6)
    for t in (0, 2):
        h = hs(0, t).reshape(M, H).contiguous()
        conf, arg = _static(W, h)
        _check_against_oracle(W, h, conf, arg)


def test_shard_step_over_two_streams():
    # Heads on one stream, commits on another, ordered by events only (as around
    # a collective on its own stream): the same states as on one stream.
    B, P, H, V, T, nb = 3, 40, 448, 3000, 8, 2
    wl = synth.Workload("twostreams", B=B, H=H, V=V, gen_len=P * nb, P=P, T=T, a0="u04")
    W = synth.lm_head_weight(V, H, device="cuda")
    hs = synth.HiddenStates(wl, W, "calibrated", seed=5)
    hidden = [[hs(b, t) for t in range(T)] for b in range(nb)]
    cfg = cai.cai_config_default(cai.CAI_PRESET_LLADA, B, P, H, V, T, nb)
    ctxs = shards._shard_ctxs(cfg, W, 2)
    try:
        gathered = torch.zeros((2, cai.cai_shard_rows(ctxs[0]), 4), device="cuda")
        torch.cuda.synchronize()
        ends = []
        for heads, commits in ((None, None), (torch.cuda.Stream(), torch.cuda.Stream())):
            for c in ctxs:
                cai.cai_reset(c, heads)
            for b in range(nb):
                if b:
                    for c in ctxs:
                        cai.cai_block_advance(c)
                for t in range(T):
                    for c, own in zip(ctxs, gathered):
                        cai.cai_shard_head(c, hidden[b][t], own, heads)
                    if heads is not None:
                        commits.wait_event(heads.record_event())
                    for c in ctxs:
                        cai.cai_shard_commit(c, gathered, commits)
                    if heads is not None:
                        heads.wait_event(commits.record_event())
            torch.cuda.synchronize()
            ends.append([cai.cai_state_download(c) for c in ctxs])
        for a, b in zip(ends[0] + ends[0][:1], ends[1] + ends[0][1:]):
            for f in shards.FIELDS:
                assert np.array_equal(a[f], b[f]), f
    finally:
        for c in ctxs:
            cai.cai_free(c)
