"""The planning kernel at the edges of its split (a warp per sequence, shares found by bisection, tables in shared
memory up to 1024 sequences), and confu_kv_append at the edges of its blocks; against the oracle and against the definition."""
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


@pytest.mark.parametrize("B,prefix", [(8, (0, 300)), (9, 0), (33, (1, 400)), (1024, (0, 3)), (1025, (0, 3))])
def test_plan_splits_cover_every_key(gpu, B, prefix):
    """Some sequences have malformed trees (no tiles: nothing of the line is theirs); they give zeros and a status."""
    cfg = inputs.VerifyConfig("plan", B=B, L=1, Hq=2, Hkv=1, D=64, T=3, C=1, S=1, V=32, prefix=prefix, tree="random",
                              kv_dtype=torch.bfloat16, logit_dtype=torch.float32, sigma_logit=1.0, draft="independent",
                              temperatures=(1.0,), seed=500 + B, max_depth=2, fanout=(1, 2))
    parent, owner, plen, seq_start, n_slots, t = H.setup_case(cfg)
    for b in {0, B // 2, B - 1}:
        parent[b, 1] = 2
    want, want_lse, want_st = H.oracle_attention(cfg, t, seq_start, plen, parent, owner)
    out, lse, st = H.gpu_attention(gpu, cfg, t, seq_start, plen, parent, owner, n_slots, use_plan=True)
    assert st.tolist() == want_st.tolist()
    ok = [b for b in range(B) if want_st[b] == 0]
    assert (out[[b for b in range(B) if want_st[b] != 0]] == 0).all()
    H.assert_attention_close(out[ok], lse[ok], want[ok], want_lse[ok], cfg.kv_dtype, "plan")


@pytest.mark.parametrize("R,Hkv,D,dtype", [(1, 1, 64, torch.bfloat16), (128, 8, 128, torch.bfloat16), (37, 3, 64, torch.float32), (65, 5, 128, torch.bfloat16)])
def test_append_writes_the_rows_and_nothing_else(gpu, R, Hkv, D, dtype):
    B, T = 3, (R + 1) // 2
    g = torch.Generator().manual_seed(R)
    plen = torch.tensor([5, 0, 131], dtype=torch.int32)
    size = plen.to(torch.int64) + R + 2
    start = torch.cumsum(size, 0) - size
    rows = [torch.randn(B, R, Hkv, D, generator=g).to(dtype) for _ in range(2)]
    pools = [torch.randn(int(size.sum()), Hkv, D, generator=g).to(dtype) for _ in range(2)]
    dims = cb.make_dims(B, Hkv, Hkv, D, T, R - T, 0, dtype)
    dev = [p.cuda() for p in pools]
    cb.confu_kv_append(gpu.ctx, dims, rows[0].cuda(), rows[1].cuda(), dev[0], dev[1], start.cuda(), plen.cuda())
    torch.cuda.synchronize()
    for p, r, d in zip(pools, rows, dev):
        for b in range(B):
            lo = int(start[b]) + int(plen[b])
            p[lo:lo + R] = r[b]
        assert torch.equal(d.cpu(), p)


@pytest.mark.parametrize("B,Hkv,G,prefix,R", [(1, 8, 4, 4096, (60, 4)), (1, 1, 4, 20000, (20, 20)), (2, 8, 3, (1, 900), (40, 30)), (9, 8, 4, (100, 300), (20, 20)), (18, 4, 4, (1, 1200), (60, 4)), (19, 4, 4, (1, 200), (60, 4)), (7, 4, 8, (0, 1500), (30, 4))])
def test_shares_of_their_own(gpu, B, Hkv, G, prefix, R):
    """Few (sequence, kv head) pairs for the machine: each gets a number of equal shares; an uneven one per pair, one tile per
    share, and batches that just fit or just do not."""
    cfg = inputs.VerifyConfig("own", B=B, L=1, Hq=G * Hkv, Hkv=Hkv, D=128, T=R[0], C=R[1], S=3, V=32, prefix=prefix, tree="random",
                              kv_dtype=torch.bfloat16, logit_dtype=torch.float32, sigma_logit=1.0, draft="independent",
                              temperatures=(1.0,), seed=560 + B, max_depth=7, fanout=(1, 4))
    parent, owner, plen, seq_start, n_slots, t = H.setup_case(cfg)
    if B > 1:
        parent[1, 1] = 7
    want, want_lse, want_st = H.oracle_attention(cfg, t, seq_start, plen, parent, owner)
    for path in (cb.ATTENTION_AUTO, cb.ATTENTION_TENSOR, cb.ATTENTION_TENSOR_PAIR):
        gpu.set_path(path)
        try:
            out, lse, st = H.gpu_attention(gpu, cfg, t, seq_start, plen, parent, owner, n_slots, use_plan=True)
        finally:
            gpu.set_path(cb.ATTENTION_AUTO)
        assert st.tolist() == want_st.tolist()
        ok = [b for b in range(B) if want_st[b] == 0]
        H.assert_attention_close(out[ok], lse[ok], want[ok], want_lse[ok], cfg.kv_dtype, "own shares")
