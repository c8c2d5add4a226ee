"""cai_pair_swap_limit: the orientation limit that a context's steps use, on both
sides of every line of the rule by H."""
import ctypes

import pytest

import synth
import paper_2608_22646_gb300 as cai


def test_arguments():
    from paper_2608_22646_gb300 import build
    build.build()
    n = ctypes.c_int32(7)
    assert cai.lib().cai_pair_swap_limit(None, ctypes.byref(n)) == cai.CAI_ERR_ARG and n.value == 7


@pytest.mark.gpu
@pytest.mark.parametrize("H,env,limit", [
    (320, {}, 0), (384, {}, 64), (704, {}, 64), (768, {}, 96), (1472, {}, 96), (1536, {}, 192),
    (3008, {}, 192), (3072, {}, 224), (4096, {}, 224),
    (256, {"CAI_PAIR_SWAP_MAX_N": "192"}, 192), (4096, {"CAI_PAIR_SWAP_MAX_N": "64"}, 64),
    (4096, {"CAI_PAIR_SWAP": "0"}, 0), (4096, {"CAI_PAIR": "0"}, 0),
])
def test_limit_in_use(H, env, limit, monkeypatch):
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    W = synth.lm_head_weight(512, H, seed=5, device="cuda")
    cfg = cai.cai_config_default(cai.CAI_PRESET_LLADA, 5, 40, H, 512, 4, 1)
    with cai.cai_init(cfg, W) as ctx:
        assert cai.cai_pair_swap_limit(ctx) == limit
        st = cai.cai_get_stats(ctx)
        off = "CAI_PAIR_SWAP" in env or "CAI_PAIR" in env
        assert st["pair_swap_max_n"] == (0 if off else int(env.get("CAI_PAIR_SWAP_MAX_N", 192)))
    with cai.cai_init_vocab_shard(cfg, W[:256].contiguous(), 0) as ctx:
        # a shard's steps are the pair head's alone: turned off means "as not set" here
        assert cai.cai_pair_swap_limit(ctx) == (limit if not off else 224)
