"""Runs of one key tile right behind longer ones, no soft prompts: the last tile of either is ragged (its V rows past the
sequence's last slot have to be zeroed), so a work unit has several repaired V tiles close together."""
import pytest
import torch

from paper_2603_08899_b200 import binding as cb
from paper_2603_08899_b200 import inputs
from tests import harness as H
from tests import test_gpu_fp8 as F8

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    g = H.Gpu()
    yield g
    g.close()


# key tiles of the sequences; with 8 kv heads the line of the first is cut so that units get [.., a] and [b] with both ragged
TILES = [[10, 1] * 4, [3, 1, 1, 2, 1, 1, 4, 1], [1] * 9 + [2] * 4, [6, 1, 1, 1, 1, 1, 1, 1, 1]]


@pytest.mark.parametrize("D", [128, 64])
@pytest.mark.parametrize("tiles", TILES)
@pytest.mark.parametrize("path", ["auto", "one_cta_per_sm"])
def test_ragged_tiles_of_neighbouring_runs(gpu, tiles, path, D):
    B, R = len(tiles), 64
    cfg = inputs.VerifyConfig("short", B=B, L=1, Hq=32, Hkv=8, D=D, T=60, C=4, S=0, V=32, prefix=(1, 2), tree="random",
                              kv_dtype=torch.bfloat16, logit_dtype=torch.float32, sigma_logit=1.0, draft="independent",
                              temperatures=(1.0,), seed=720 + B, max_depth=7, fanout=(1, 4))
    parent, owner = inputs.trees(cfg)
    plen = torch.tensor([128 * n - R - 5 - 7 * b for b, n in enumerate(tiles)], dtype=torch.int32).clamp_(min=1)
    seq_start, n_slots = inputs.cache_layout(cfg, plen)
    t = inputs.layer_tensors(cfg, 0, n_slots, device="cuda", seq_start=seq_start, prefix_len=plen)
    for b in range(B):                       # keys that grow along the prefix: the reference maximum moves in most tiles
        n = int(plen[b]) + R
        s = int(seq_start[b])
        t["k_cache"][s:s + n] *= torch.linspace(0.5, 4.0, n, device="cuda", dtype=torch.bfloat16)[:, None, None]
    want, want_lse, _ = H.oracle_attention(cfg, t, seq_start, plen, parent, owner)
    gpu.set_path(cb.ATTENTION_AUTO if path == "auto" else cb.ATTENTION_TENSOR)
    cb.confu_set_option(gpu.ctx, cb.OPT_WAIT_LIMIT_NS, 50_000_000)
    try:
        for _ in range(20):
            out, lse, st = H.gpu_attention(gpu, cfg, t, seq_start, plen, parent, owner, n_slots, use_plan=True)
            assert st.tolist() == [0] * B
            H.assert_attention_close(out, lse, want, want_lse, cfg.kv_dtype, f"{tiles}")
    finally:
        cb.confu_set_option(gpu.ctx, cb.OPT_WAIT_LIMIT_NS, 2_000_000_000)
        gpu.set_path(cb.ATTENTION_AUTO)


@pytest.mark.parametrize("D,G", [(128, 4), (64, 4), (64, 1)])
def test_many_short_runs_per_cta(gpu, D, G):
    """More pairs than CTAs with two M tiles hold, one to three key tiles each, nearly all with a ragged last tile."""
    cfg = inputs.VerifyConfig("many", B=60, L=1, Hq=8 * G, Hkv=8, D=D, T=60, C=4, S=0, V=32, prefix=(1, 260), tree="random",
                              kv_dtype=torch.bfloat16, logit_dtype=torch.float32, sigma_logit=1.0, draft="independent",
                              temperatures=(1.0,), seed=730 + D + G, max_depth=7, fanout=(1, 4))
    parent, owner, plen, seq_start, n_slots, t = H.setup_case(cfg)
    want, want_lse, _ = H.oracle_attention(cfg, t, seq_start, plen, parent, owner)
    cb.confu_set_option(gpu.ctx, cb.OPT_WAIT_LIMIT_NS, 50_000_000)
    try:
        for _ in range(10):
            out, lse, st = H.gpu_attention(gpu, cfg, t, seq_start, plen, parent, owner, n_slots, use_plan=True)
            assert st.tolist() == [0] * cfg.B
            H.assert_attention_close(out, lse, want, want_lse, cfg.kv_dtype, "many short runs")
    finally:
        cb.confu_set_option(gpu.ctx, cb.OPT_WAIT_LIMIT_NS, 2_000_000_000)


def test_many_short_runs_e4m3(gpu):
    cfg = F8._cfg(B=60, Hq=32, Hkv=8, T=60, C=4, S=0, prefix=(1, 260), max_depth=7, fanout=(1, 4), seed=740)
    *case, want, want_lse = F8._setup(cfg)
    cb.confu_set_option(gpu.ctx, cb.OPT_WAIT_LIMIT_NS, 50_000_000)
    try:
        for _ in range(10):
            out, lse, st = F8._run(gpu, cfg, *case, True)
            assert st.tolist() == [0] * cfg.B
            F8._assert_close(out, lse, want, want_lse, "many short runs")
    finally:
        cb.confu_set_option(gpu.ctx, cb.OPT_WAIT_LIMIT_NS, 2_000_000_000)
