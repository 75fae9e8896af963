"""Row statistics of the acceptance step where a sum can go wrong: logits whose product with the scale leaves fp32, and long sums."""
import pytest
import torch

from oracle import ref
from paper_2603_08899_b200 import binding as cb
from paper_2603_08899_b200 import inputs
from tests import harness as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    g = H.Gpu()
    yield g
    g.close()


# masks within the finite range whose product with log2(e) / temperature is beyond it, and a temperature at which the product's
# rounding is as large as the exponents themselves
@pytest.mark.parametrize("mask,temperature", [(-2.5e38, 1.0), (-1e38, 0.1), (-50.0, 1e-9)])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("V", [96, 250, 5000, 32000, 32003])
def test_masked_rows(gpu, V, dtype, mask, temperature):
    """All but a few dozen entries of every row masked, the others anywhere (the first that a lane reads are nearly always masked)."""
    cfg = inputs.VerifyConfig("mask", B=8, L=1, Hq=4, Hkv=1, D=64, T=9, C=2, S=0, V=V, prefix=4, tree="random", kv_dtype=torch.bfloat16,
                              logit_dtype=dtype, sigma_logit=2.0 * min(temperature, 1.0), draft="noise", temperatures=(temperature,),
                              seed=900 + V % 89, max_depth=4, fanout=(1, 3))
    parent, owner = inputs.trees(cfg)
    tl, dl = inputs.logits(cfg)
    g = torch.Generator()
    g.manual_seed(V)
    keep = torch.zeros((cfg.B, cfg.T, V), dtype=torch.bool)
    keep.scatter_(2, torch.rand((cfg.B, cfg.T, V), generator=g).topk(min(40, V // 3), dim=2).indices, True)
    if temperature < 1e-6:                           # only the largest count: draws among equals
        tl, dl = (torch.randint(29, 31, tl.shape, generator=g).to(dtype) for _ in range(2))
    tl, dl = tl.masked_fill(~keep, mask), dl.masked_fill(~keep, mask)
    tok = inputs.draft_tokens(cfg, parent, dl, temperature)
    u = inputs.uniforms(cfg)
    for lazy in (0, cb.ACCEPT_LAZY):
        want = ref.tree_accept(tl, dl, tok, parent, owner, u, temperature=temperature, sibling_mode=1 | lazy)
        got = H.gpu_accept(gpu, cfg, tl, dl, tok, parent, owner, u, temperature, 1 | lazy)
        assert got["status"].tolist() == want["status"].tolist()
        assert H.compare_accept(got, want) == (cfg.B, 0)
