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


def _row_sums(gpu, tl, dl, temperature):
    """Sum of exp((x - maximum) / temperature) of every target and draft row, from the statistics that the call leaves in its workspace:
    16 entries of 16 bytes a row (maximum of a chunk, its sum, two integers), the first ones used."""
    B, T, V = tl.shape
    ws = torch.zeros(cb.confu_accept_workspace_bytes(B, T, V), dtype=torch.uint8, device="cuda")
    ws.view(torch.float32)[0::4] = -float("inf")
    i32 = dict(dtype=torch.int32, device="cuda")
    out = [torch.zeros(n, **i32) for n in ((B,), (B, cb.MAX_DEPTH + 1), (B,), (B,), (B, 4))]
    tokens = torch.arange(T, **i32).expand(B, T).contiguous()
    parent = torch.arange(-1, T - 1, **i32).expand(B, T).contiguous()
    uniforms = torch.full((B, T), 0.5, device="cuda")
    status = torch.zeros(B, **i32)
    cb.confu_tree_accept(gpu.ctx, B, T, 0, V, tl.dtype, tl, dl, tokens, parent, None, uniforms, temperature, 1, *out, ws, status)
    torch.cuda.synchronize()
    assert not status.any()
    part = ws.view(torch.float32)[:2 * B * T * 64].view(2 * B * T, 16, 4).double()
    m, s = part[..., 0], part[..., 1]
    top = m.max(1, keepdim=True).values
    return top[:, 0], (s * torch.exp((m - top) / temperature)).sum(1)


# A warp to a row, to chunks of whole and of broken batches, in one round and in two, two and eight warps to a chunk (148 SMs).  Half of the
# rows: one logit far above all others, read among the first, so that its lane's sum takes in hundreds of weights that are next to
# nothing beside it (eight of an fp32 row, 32 of a bf16 row at a time: a little less than half a unit in its last place).  The other
# half: deviation 5.
@pytest.mark.parametrize("dtype,low", [(torch.bfloat16, -20.125), (torch.float32, -18.75)])
@pytest.mark.parametrize("B,T,V", [(49, 60, 48003), (3, 60, 128256), (2, 47, 5000), (1, 5, 151937), (37, 32, 4099), (32, 3, 12878),
                                   (55, 8, 171133)])
def test_error_of_sums(gpu, B, T, V, dtype, low):
    g = torch.Generator(device="cuda")
    g.manual_seed(B + V)
    x = torch.randn((2, B, T, V), generator=g, device="cuda") * 5
    x[:, :, ::2] = low
    at = torch.randint(0, min(V, 256), (2, B, T, 1), generator=g, device="cuda")
    x[:, :, ::2] = x[:, :, ::2].scatter(3, at[:, :, ::2], 0.0)
    x = x.to(dtype)
    top, got = _row_sums(gpu, x[0].clone(), x[1].clone(), 1.0)
    rows = x.view(2 * B * T, V)
    want = torch.stack([torch.exp(r.double() - t).sum() for r, t in zip(rows, top)])
    assert torch.equal(top, rows.max(1).values.double())
    err = (got / want - 1).abs()
    # In units of 2^-24 of the sum: 8 + 2 for the additions in front of a lane's sum, 1 for that sum with its correction, 5 and 3 for a
    # warp's and a chunk's (fp64 after that); a weight's own error is the exponential unit's 2 and, of its argument a, |a| ln 2 twice:
    # next to nothing where the sum is its largest weight (|a| of the mean weight some 4 at deviation 5, and as often up as down).
    lone = torch.arange(2 * B * T, device="cuda") % T % 2 == 0
    assert err[lone].max().item() <= 19 * 2.0 ** -24
    assert err[~lone].max().item() <= (19 + 2 + 6) * 2.0 ** -24
    assert err[~lone].square().mean().sqrt().item() <= 4 * 2.0 ** -24
