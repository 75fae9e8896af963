"""Tensor-core attention for every number of query heads per kv head and both head dims, at the edges of
the row packing (128 / G query rows per M tile, two tiles per row group), against the fp64 oracle."""
import pytest
import torch

from paper_2603_08899_b200 import binding as cb
from paper_2603_08899_b200 import inputs
from tests import harness as H

pytestmark = pytest.mark.gpu

# (G, D, T, C): all rows in one tile, one row more, one full group, one row more, several groups
CASES = [(1, 128, 60, 4), (1, 64, 64, 64), (2, 128, 32, 32), (2, 64, 40, 25), (3, 64, 42, 0), (3, 128, 43, 0), (4, 64, 32, 32),
         (4, 64, 60, 5), (5, 128, 25, 0), (5, 64, 50, 1), (7, 128, 18, 18), (7, 64, 20, 17), (8, 128, 16, 0), (8, 128, 60, 4),
         (8, 64, 64, 64), (16, 128, 9, 8), (32, 128, 5, 4), (32, 64, 64, 64), (33, 64, 6, 2)]


@pytest.fixture(scope="module")
def gpu():
    g = H.Gpu()
    yield g
    g.close()


@pytest.mark.parametrize("G,D,T,C", CASES)
@pytest.mark.parametrize("prefix", [(1, 300), 700])
def test_groups_match_oracle(gpu, G, D, T, C, prefix):
    Hkv = 2 if G <= 8 else 1
    cfg = inputs.VerifyConfig("groups", B=2, L=1, Hq=G * Hkv, Hkv=Hkv, D=D, T=T, C=C, S=5, V=32, prefix=prefix, tree="random",
                              kv_dtype=torch.bfloat16, logit_dtype=torch.float32, sigma_logit=1.0, draft="independent",
                              temperatures=(1.0,), seed=600 + G + D + T, max_depth=7, fanout=(1, 4))
    parent, owner, plen, seq_start, n_slots, t = H.setup_case(cfg)
    want, want_lse, _ = H.oracle_attention(cfg, t, seq_start, plen, parent, owner)
    paths = [cb.ATTENTION_AUTO]
    if G <= 32:
        assert cb.confu_attention_path(gpu.ctx, H.dims_of(cfg)) != cb.ATTENTION_GENERIC
        paths.append(cb.ATTENTION_TENSOR)
        if D == 128 and cfg.R > 128 // G:
            paths.append(cb.ATTENTION_TENSOR_PAIR)
    for path in paths:
        gpu.set_path(path)
        try:
            out, lse, st = H.gpu_attention(gpu, cfg, t, seq_start, plen, parent, owner, n_slots)
        finally:
            gpu.set_path(cb.ATTENTION_AUTO)
        assert st.tolist() == [0] * cfg.B
        H.assert_attention_close(out, lse, want, want_lse, cfg.kv_dtype, f"G {G} D {D} path {path}")


@pytest.mark.parametrize("G,D", [(1, 64), (4, 64), (8, 64), (5, 128), (8, 128), (32, 128)])
@pytest.mark.parametrize("path", ["auto", "one_cta_per_sm"])
def test_weights_keep_more_than_bf16(gpu, G, D, path):
    """Head dim 64 and more than four heads per kv head: weights travel as two bf16 numbers, 16 bits or more of each, so the error against 64 bits is
    that of rounding the output to bf16 (2^-9 at most, 2^-17 from the weights: together at most 1 + 2^-8 times the first, and
    far less in the 2-norm; with weights of 8 bits it is 1.03 to 1.4 times).  lse, in absolute terms: fp32 rounding of a number near 8."""
    cfg = inputs.VerifyConfig("split", B=2, L=1, Hq=2 * G, Hkv=2, D=D, T=30, C=10, S=5, V=32, prefix=(200, 1500), tree="random",
                              kv_dtype=torch.bfloat16, logit_dtype=torch.float32, sigma_logit=1.0, draft="independent",
                              temperatures=(1.0,), seed=650 + G + D, max_depth=7, fanout=(1, 4))
    parent, owner, plen, seq_start, n_slots, t = H.setup_case(cfg)
    want, want_lse, _ = H.oracle_attention(cfg, t, seq_start, plen, parent, owner)
    gpu.set_path(cb.ATTENTION_AUTO if path == "auto" else cb.ATTENTION_TENSOR)
    try:
        out, lse, st = H.gpu_attention(gpu, cfg, t, seq_start, plen, parent, owner, n_slots)
    finally:
        gpu.set_path(cb.ATTENTION_AUTO)
    assert st.tolist() == [0, 0]
    rounding = (want.to(torch.bfloat16).double() - want).norm().item()
    assert (out.double() - want).norm().item() <= 1.001 * rounding
    assert (lse.double() - want_lse).abs().max().item() <= 4e-6
