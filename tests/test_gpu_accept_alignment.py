"""Acceptance where a row of logits starts anywhere between two 16-byte boundaries: vocabulary sizes around the edges of
vectors, of a CTA's slice and of the slices together, every rule, against the oracle."""
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


def _case(V, dtype, temperature, B=9, T=7):
    cfg = inputs.VerifyConfig("align", B=B, L=1, Hq=4, Hkv=1, D=64, T=T, C=2, S=0, V=V, prefix=4, tree="random", kv_dtype=torch.bfloat16,
                              logit_dtype=dtype, sigma_logit=2.0, draft="noise", temperatures=(1.0,), seed=800 + V % 97, max_depth=4,
                              fanout=(1, 3))
    parent, owner = inputs.trees(cfg)
    tl, dl = inputs.logits(cfg)
    return cfg, parent, owner, tl, dl, inputs.draft_tokens(cfg, parent, dl, temperature), inputs.uniforms(cfg)


def _check(gpu, case, temperature):
    cfg, parent, owner, tl, dl, tok, u = case
    sampled = temperature > 0
    d, un = (dl, u) if sampled else (None, None)
    for lazy in (0, cb.ACCEPT_LAZY):
        want = ref.tree_accept(tl, d, tok, parent, owner, un, temperature=temperature, sibling_mode=1 | lazy)
        got = H.gpu_accept(gpu, cfg, tl, d, tok, parent, owner, un, temperature, 1 | lazy)
        exact, border = H.compare_accept(got, want)
        assert exact + border == cfg.B and border <= 1
    want = ref.tree_accept_match(tl, tok, parent, owner, un, temperature=temperature)
    got = H.gpu_accept_match(gpu, cfg, tl, tok, parent, owner, un, temperature)
    exact, border = H.compare_match(got, want)
    assert exact + border == cfg.B and border <= 1


@pytest.mark.parametrize("temperature", [1.0, 0.0])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("V", [9, 11, 14, 15, 17, 250, 255, 257, 2047, 4095, 4097, 4099, 32761, 32766, 32769, 32775, 65531, 65537, 131075])
def test_rows_start_anywhere(gpu, V, dtype, temperature):
    _check(gpu, _case(V, dtype, temperature), temperature)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("V", [13, 1003, 40001])
def test_ends_of_a_row_belong_to_it_alone(gpu, V, dtype):
    """A value that is not finite next to a row's ends is its sequence's, not its neighbours'; the largest at either end is found."""
    for first in (True, False):
        case = list(_case(V, dtype, 1.0))
        for m in (3, 4):
            case[m] = case[m].clone()
        at = 0 if first else V - 1
        case[3][4, 0 if first else -1, at] = float("inf")          # the sequence's first row begins, its last row ends with it
        case[4][2, 0 if first else -1, at] = float("nan")
        case[3][6, :, at] = 40.0
        cfg, parent, owner, tl, dl, tok, u = case
        want = ref.tree_accept(tl, dl, tok, parent, owner, u, temperature=1.0, sibling_mode=1)
        got = H.gpu_accept(gpu, cfg, tl, dl, tok, parent, owner, u, 1.0, 1)
        assert [b for b in range(cfg.B) if got["status"][b]] == [2, 4]
        assert got["next_token"][6] == want["next_token"][6] == at
        H.compare_accept(got, want)
        want = ref.tree_accept(tl, None, tok, parent, owner, None, temperature=0.0, sibling_mode=1)
        got = H.gpu_accept(gpu, cfg, tl, None, tok, parent, owner, None, 0.0, 1)
        assert [b for b in range(cfg.B) if got["status"][b]] == [4] and got["next_token"][6] == at
        H.compare_accept(got, want)


# rows of lengths that leave the last round of the statistics, the last chunk and the last batch of loads all unfinished
@pytest.mark.parametrize("temperature", [1.0, 0.0])
@pytest.mark.parametrize("B,T,V", [(48, 7, 93477), (55, 8, 171133), (16, 17, 148937), (2, 47, 5000), (16, 3, 3017), (40, 64, 300)])
def test_rounds_of_statistics(gpu, B, T, V, temperature):
    cfg, parent, owner, tl, dl, tok, u = _case(V, torch.bfloat16, temperature, B, T)
    d, un = (dl, u) if temperature > 0 else (None, None)
    want = ref.tree_accept(tl, d, tok, parent, owner, un, temperature=temperature, sibling_mode=1)
    got = H.gpu_accept(gpu, cfg, tl, d, tok, parent, owner, un, temperature, 1)
    exact, border = H.compare_accept(got, want)
    assert exact + border == B and border <= max(1, B // 8)


# rounds x warps per chunk of the statistics, sampling and greedy (148 SMs): 7 x 2 and 4 x 2, 5 x 2 and 5 x 4, 5 x 4 and 3 x 1, 4 x 1 and 2 x 1 (the
# buffers in which warps meet are used again from the third item on)
@pytest.mark.parametrize("temperature", [1.0, 0.0])
@pytest.mark.parametrize("B,T,V", [(149, 60, 18), (101, 59, 4116), (66, 45, 4122), (147, 63, 607)])
def test_many_items_to_a_warp(gpu, B, T, V, temperature):
    cfg, parent, owner, tl, dl, tok, u = _case(V, torch.bfloat16, temperature, B, T)
    d, un = (dl, u) if temperature > 0 else (None, None)
    want = ref.tree_accept(tl, d, tok, parent, owner, un, temperature=temperature, sibling_mode=1)
    got = H.gpu_accept(gpu, cfg, tl, d, tok, parent, owner, un, temperature, 1)
    exact, border = H.compare_accept(got, want)
    assert exact + border == B and border <= max(1, B // 8)
