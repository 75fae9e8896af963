"""Acceptance walks where the vocabulary's slices have edges: one entry below, at and past what a strip of every CTA
holds, 8 and 16 CTAs per sequence, ragged rows; all rules, against the fp64 oracle."""
import pytest
import torch

from oracle import ref
from paper_2603_08899_b200 import inputs
from tests import harness as H

pytestmark = pytest.mark.gpu
LAZY = 0x100


@pytest.fixture(scope="module")
def gpu():
    g = H.Gpu()
    yield g
    g.close()


@pytest.mark.parametrize("B,V", [(2, 1), (2, 9), (2, 32768), (2, 32769), (1, 65544), (2, 131073), (8, 65540), (8, 98312), (8, 131080),
                                 (8, 163840), (8, 163848), (1, 262144),
                                 # many sequences: 4, 2 and 1 CTAs each, either side of what 16 entries per thread hold
                                 (38, 32768), (38, 32769), (75, 16384), (75, 16385), (149, 8192), (149, 8193), (300, 1000), (297, 37)])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_slice_edges(gpu, B, V, dtype):
    T = 1 if V < 9 else 6
    cfg = inputs.VerifyConfig("slices", B=B, L=1, Hq=4, Hkv=1, D=64, T=T, C=1, S=0, V=V, prefix=4, tree="random",
                              kv_dtype=torch.bfloat16, logit_dtype=dtype, sigma_logit=4.0, draft="noise", temperatures=(1.0,),
                              seed=800 + B + V % 97, max_depth=3, fanout=(1, 3))
    parent, owner = inputs.trees(cfg)
    tl, dl = inputs.logits(cfg)
    tok = inputs.draft_tokens(cfg, parent, dl, 0.8)
    u = inputs.uniforms(cfg)
    for mode in (1, 1 | LAZY, 0 | LAZY):
        exact, border = H.compare_accept(H.gpu_accept(gpu, cfg, tl, dl, tok, parent, owner, u, 0.8, mode),
                                         ref.tree_accept(tl, dl, tok, parent, owner, u, temperature=0.8, sibling_mode=mode))
        assert exact + border == B and border <= 1
    for mode in (1, 1 | LAZY):
        exact, border = H.compare_accept(H.gpu_accept(gpu, cfg, tl, None, tok, parent, owner, None, 0.0, mode),
                                         ref.tree_accept(tl, None, tok, parent, owner, None, temperature=0.0, sibling_mode=mode))
        assert exact == B
    for temperature in (0.8, 0.0):
        uu = u if temperature > 0 else None
        exact, border = H.compare_match(H.gpu_accept_match(gpu, cfg, tl, tok, parent, owner, uu, temperature),
                                        ref.tree_accept_match(tl, tok, parent, owner, uu, temperature=temperature))
        assert exact + border == B and border <= 1
