"""CUDA-core attention at the edges of its blocks (16, 32 or 64 row-head pairs) and of its 64-key tiles, with
clusters of every size, against the fp64 oracle; and that slots a row does not see may hold anything."""
import pytest
import torch

from paper_2603_08899_b200 import binding as cb
from paper_2603_08899_b200 import inputs
from tests import harness as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    g = H.Gpu()
    yield g
    g.close()


def _cfg(B, Hq, Hkv, D, T, C, S, prefix, dtype):
    return inputs.VerifyConfig("generic", B=B, L=1, Hq=Hq, Hkv=Hkv, D=D, T=T, C=C, S=S, V=32, prefix=prefix, tree="random",
                               kv_dtype=dtype, logit_dtype=torch.float32, sigma_logit=1.0, draft="independent",
                               temperatures=(1.0,), seed=700 + B + D + T, max_depth=7, fanout=(1, 4))


F, H16 = torch.float32, torch.bfloat16
CASES = [_cfg(1, 1, 1, 64, 1, 0, 0, 0, F), _cfg(1, 1, 1, 128, 16, 0, 0, 48, F), _cfg(1, 1, 1, 128, 17, 0, 3, 44, F),
         _cfg(1, 4, 2, 64, 8, 2, 2, 700, F), _cfg(2, 32, 4, 64, 33, 31, 16, (1, 600), F), _cfg(12, 16, 8, 128, 30, 30, 16, (1, 300), F),
         _cfg(3, 8, 8, 128, 64, 64, 130, (60, 200), F), _cfg(2, 4, 2, 128, 20, 20, 150, (60, 200), H16),
         _cfg(1, 40, 1, 64, 5, 3, 2, 333, H16)]


@pytest.mark.parametrize("cfg", CASES, ids=lambda c: f"B{c.B}_{c.Hq}x{c.Hkv}x{c.D}_R{c.R}_S{c.S}")
def test_generic_matches_oracle(gpu, cfg):
    parent, owner, plen, seq_start, n_slots, t = H.setup_case(cfg)
    assert cb.confu_attention_path(gpu.ctx, H.dims_of(cfg)) == cb.ATTENTION_GENERIC
    out, lse, st = H.gpu_attention(gpu, cfg, t, seq_start, plen, parent, owner, n_slots)
    want, want_lse, _ = H.oracle_attention(cfg, t, seq_start, plen, parent, owner)
    assert st.tolist() == [0] * cfg.B
    H.assert_attention_close(out, lse, want, want_lse, cfg.kv_dtype, cfg.name)


@pytest.mark.parametrize("where", ["root", "tile"])
def test_nan_that_is_all_a_cta_sees_of_a_row_shows(gpu, where):
    """The keys are dealt out over a cluster; a CTA may see nothing of a row but NaN: the root's row in the tile of the tree
    slots, or any row in a tile of 64 NaN keys."""
    cfg = inputs.VerifyConfig("generic", B=1, L=1, Hq=4, Hkv=2, D=64, T=8, C=2, S=2, V=32, prefix=256 - 2, tree="chain",
                              kv_dtype=torch.float32, logit_dtype=torch.float32, sigma_logit=1.0, draft="independent",
                              temperatures=(1.0,), seed=570)
    parent, owner, plen, seq_start, n_slots, t = H.setup_case(cfg)       # soft prompts and prefix: four whole tiles of 64 keys
    at = int(seq_start[0]) + int(plen[0])
    if where == "root":
        t["k_cache"][at, 1] = float("nan")
    else:
        t["k_cache"][at - 64:at, 1] = float("nan")
    out, lse, st = H.gpu_attention(gpu, cfg, t, seq_start, plen, parent, owner, n_slots)
    assert st.tolist() == [0]
    assert out[0, :, :2].isfinite().all() and lse[0, :, :2].isfinite().all()
    assert out[0, :, 2:].isnan().all() and lse[0, :, 2:].isnan().all()


def test_more_blocks_than_a_grid_dimension_holds(gpu):
    """33000 kv heads and 65 rows: two blocks of rows per head, 66000 of them."""
    heads, D, T, C, P = 33000, 64, 33, 32, 3
    R = T + C
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    q, k, v = (torch.randn((1, n, heads, D), generator=g, device="cuda") for n in (R, P + R, P + R))
    dims = cb.make_dims(1, heads, heads, D, T, C, 0, torch.float32)
    gpu.ensure_ws(dims)
    parent, owner = torch.arange(-1, T - 1, dtype=torch.int32).cuda(), torch.arange(C, dtype=torch.int32).cuda()
    out, status = torch.empty_like(q), torch.zeros(1, dtype=torch.int32, device="cuda")
    cb.confu_tree_attention(gpu.ctx, dims, q, k[0], v[0], P + R, torch.zeros(1, dtype=torch.int64, device="cuda"),
                            torch.tensor([P], dtype=torch.int32, device="cuda"), None, None, parent, owner, None, out, None, status)
    assert status.tolist() == [0]
    row, key = torch.arange(R, device="cuda")[:, None], torch.arange(P + R, device="cuda")[None, :] - P
    depth = torch.where(row < T, row, row - T)       # a chain: row r sees rows 0..r, contemplate row k rows 0..k and itself
    sees = (key <= depth) & (key < T) | (key == row)
    for h in (0, 1, 16383, 32767, 32768, heads - 1):
        s = (q[0, :, h].double() @ k[0, :, h].double().T) * D ** -0.5
        want = torch.softmax(s.masked_fill(~sees, float("-inf")), dim=-1) @ v[0, :, h].double()
        assert (out[0, :, h].double() - want).abs().max().item() <= 1e-5 * want.abs().max().item()
