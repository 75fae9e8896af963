"""Shares of a plan that hold several whole (sequence, kv head) stretches or one piece of a stretch: every key tile is walked
exactly once, the merge is told who walked it, and attention over such plans agrees with the oracle."""
import numpy as np
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


def _config(tiles, Hkv, G, T=60, C=4, S=0, D=128):
    return inputs.VerifyConfig("shares", B=len(tiles), L=1, Hq=Hkv * G, Hkv=Hkv, D=D, T=T, C=C, S=S, V=32, prefix=(1, 2),
                               tree="random", kv_dtype=torch.bfloat16, logit_dtype=torch.float32, sigma_logit=1.0,
                               draft="independent", temperatures=(1.0,), seed=760 + len(tiles) + Hkv, max_depth=7, fanout=(1, 4))


def _prefix(tiles, R):
    return torch.tensor([max(128 * n - R - 3 * b, 1) for b, n in enumerate(tiles)], dtype=torch.int32)


def _up(x):
    return (x + 255) // 256 * 256


def _runs(plan, B, Hkv):
    """The runs of every work unit, and the words that tell the merge who walked a stretch."""
    raw = plan.cpu().numpy()
    at = 256 + _up(B * 128 * 8) + 2 * _up(B * 4) + _up((B + 1) * 8)
    cta = raw[at:at + 256 * 64].view(np.int32).reshape(256, 16)
    at += _up(256 * 64)
    parts = raw[at:at + B * Hkv * 4].view(np.int32)
    at += _up(B * Hkv * 4)
    segs = raw[at:at + (raw.size - at) // 48 * 48].view(np.int32).reshape(-1, 12)
    return [[cta[c, :12]] + [segs[cta[c, 13] + i] for i in range(1, cta[c, 12])] if cta[c, 12] else [] for c in range(256)], parts


LENGTHS = [[22, 3, 18, 11, 6, 8, 5, 3], [40, 1, 1, 2, 1], [9, 2, 2, 1], [1] * 30, [30, 1] * 3, [2], [5, 5, 4, 4, 3], [17] * 7, [60, 3, 1] * 5]


@pytest.mark.parametrize("Hkv,G,S", [(8, 4, 16), (3, 8, 0), (5, 3, 0), (1, 32, 0), (12, 1, 5)])
@pytest.mark.parametrize("tiles", LENGTHS)
def test_every_tile_once(gpu, tiles, Hkv, G, S):
    cfg = _config(tiles, Hkv, G, S=S)
    B, R = cfg.B, cfg.R
    parent, owner = inputs.trees(cfg)
    if B > 2:
        parent[1, 5] = 7                             # a malformed tree in between: no shares
    plen = _prefix(tiles, R)
    seq_start, _ = inputs.cache_layout(cfg, plen)
    dims = cb.make_dims(B, cfg.Hq, Hkv, cfg.D, cfg.T, cfg.C, S, cfg.kv_dtype)
    plan = torch.zeros(cb.confu_plan_bytes(gpu.ctx, dims), dtype=torch.uint8, device="cuda")
    status = torch.zeros(B, dtype=torch.int32, device="cuda")
    cb.confu_tree_plan(gpu.ctx, dims, seq_start.cuda(), plen.cuda(), parent.cuda(), owner.cuda(), plan, status)
    torch.cuda.synchronize()
    per_tile = 128 // G * (1 if cb.confu_attention_path(gpu.ctx, dims) == cb.ATTENTION_TENSOR_NARROW else 2)
    n_rg = (R + per_tile - 1) // per_tile
    runs, parts = _runs(plan, B, Hkv)
    seen, walkers = {}, {}
    for c, of_c in enumerate(runs):
        slots = [int(r[6]) for r in of_c if r[6] >= 0]
        assert len(slots) == len(set(slots)) <= 2 and all(s // 2 == c for s in slots)
        for r in of_c:
            b, g, rg, t0, t1, nt, P = int(r[0]), int(r[1]) & 0xffff, int(r[1]) >> 16, int(r[2]), int(r[3]), int(r[4]), int(r[5])
            assert rg == c % n_rg and P == int(plen[b]) and nt == (P + R + 127) // 128 + (S > 0) and 0 <= t0 < t1 <= nt
            assert (r[6] < 0) == (t0 == 0 and t1 == nt)
            if r[6] >= 0:
                assert int(r[6]) == 2 * c + (t1 < nt)
            walkers.setdefault((b, g, rg), []).append(c)
            for t in range(t0, t1):
                assert (b, g, rg, t) not in seen
                seen[b, g, rg, t] = c
    good = [b for b in range(B) if not (B > 2 and b == 1)]
    assert len(seen) == sum((int(plen[b]) + R + 127) // 128 + (S > 0) for b in good) * Hkv * n_rg
    for u, word in enumerate(parts.tolist()):
        b, g = divmod(u, Hkv)
        first, n = word & 0xfff, (word >> 12) & 0xfff
        assert n == (0 if b not in good else len(walkers[b, g, 0]))
        for rg in range(n_rg if b in good else 0):
            assert walkers[b, g, rg] == [(first + p) * n_rg + rg for p in range(n)]


@pytest.mark.parametrize("tiles,Hkv,G,D", [([22, 3, 9, 11, 1, 2], 8, 4, 128), ([9, 2, 2, 1], 3, 8, 128), ([14, 1, 1, 2, 1], 8, 4, 64)])
def test_attention_over_packed_shares(gpu, tiles, Hkv, G, D):
    cfg = _config(tiles, Hkv, G, S=16, D=D)
    parent, owner = inputs.trees(cfg)
    plen = _prefix(tiles, cfg.R)
    seq_start, n_slots = inputs.cache_layout(cfg, plen)
    t = inputs.layer_tensors(cfg, 0, n_slots, device="cuda", seq_start=seq_start, prefix_len=plen)
    want, want_lse, _ = H.oracle_attention(cfg, t, seq_start, plen, parent, owner)
    for path in (cb.ATTENTION_AUTO, cb.ATTENTION_TENSOR):
        gpu.set_path(path)
        out, lse, st = H.gpu_attention(gpu, cfg, t, seq_start, plen, parent, owner, n_slots, use_plan=True)
        gpu.set_path(cb.ATTENTION_AUTO)
        assert st.tolist() == [0] * cfg.B
        H.assert_attention_close(out, lse, want, want_lse, cfg.kv_dtype, f"{tiles}")


@pytest.mark.parametrize("path", ["auto", "one_cta_per_sm"])
def test_plan_rewritten_between_layers(gpu, path):
    """One plan buffer, plans of other lengths and attention calls right behind one another: what a CTA fetches ahead of time by the
    plan before must not be what it works with."""
    cfg = _config([9, 3, 5], 8, 4, S=16)
    parent, owner = (x.cuda() for x in inputs.trees(cfg))
    gpu.set_path(cb.ATTENTION_AUTO if path == "auto" else cb.ATTENTION_TENSOR)
    dims = cb.make_dims(cfg.B, cfg.Hq, cfg.Hkv, cfg.D, cfg.T, cfg.C, cfg.S, cfg.kv_dtype)
    gpu.ensure_ws(dims)
    room = _prefix([9, 9, 9], cfg.R)
    seq_start, n_slots = inputs.cache_layout(cfg, room)
    t = inputs.layer_tensors(cfg, 0, n_slots, device="cuda", seq_start=seq_start, prefix_len=room)
    ss = seq_start.cuda()
    lengths = [_prefix(x, cfg.R).cuda() for x in ([9, 3, 5], [1, 9, 2], [4, 4, 9])]
    plan = torch.zeros(cb.confu_plan_bytes(gpu.ctx, dims), dtype=torch.uint8, device="cuda")
    status = torch.zeros(cfg.B, dtype=torch.int32, device="cuda")

    def step(n, out):
        cb.confu_tree_plan(gpu.ctx, dims, ss, n, parent, owner, plan, status)
        cb.confu_tree_attention(gpu.ctx, dims, t["q"], t["k_cache"], t["v_cache"], n_slots, ss, n, t["k_soft"], t["v_soft"], None, None,
                                plan, out, None, status)

    try:
        alone = [torch.empty_like(t["q"]) for _ in lengths]
        for n, out in zip(lengths, alone):
            step(n, out)
            torch.cuda.synchronize()
            want, _, _ = H.oracle_attention(cfg, t, seq_start, n.cpu(), parent.cpu(), owner.cpu())
            H.assert_attention_close(out.cpu(), None, want, None, cfg.kv_dtype)
        outs = [[torch.empty_like(t["q"]) for _ in lengths] for _ in range(5)]
        for o in outs:
            for n, out in zip(lengths, o):
                step(n, out)
        torch.cuda.synchronize()
        assert status.tolist() == [0] * cfg.B
        for o in outs:
            assert all(torch.equal(a, b) for a, b in zip(o, alone))
    finally:
        gpu.set_path(cb.ATTENTION_AUTO)


@pytest.mark.parametrize("kv", [torch.bfloat16, torch.float8_e4m3fn])
@pytest.mark.parametrize("paged", [False, True])
def test_fetch_ahead_by_a_stale_record(gpu, kv, paged):
    """Plan and block table rewritten in stream order between attention calls right behind one another: the record that a CTA reads ahead
    of time, and the table's entry that it names, may be those of the call before (or of none: the first plan is zeros)."""
    fp8 = kv == torch.float8_e4m3fn
    cfg = inputs.VerifyConfig("stale", B=3, L=1, Hq=32, Hkv=8, D=128, T=60, C=4, S=16, V=32, prefix=(1, 2), tree="random", kv_dtype=kv,
                              logit_dtype=torch.float32, sigma_logit=1.0, draft="independent", temperatures=(1.0,), seed=771, max_depth=7,
                              fanout=(1, 4))
    parent, owner = (x.cuda() for x in inputs.trees(cfg))
    dims = cb.make_dims(cfg.B, cfg.Hq, cfg.Hkv, cfg.D, cfg.T, cfg.C, cfg.S, torch.uint8 if fp8 else kv)
    pages, max_pages = 27, 9                         # of 128 slots, nine to a sequence
    t = inputs.layer_tensors(cfg, 0, pages * 128, device="cuda")
    seq_start = torch.arange(3, device="cuda") * max_pages * 128
    packed = torch.arange(pages, dtype=torch.int32, device="cuda").view(3, max_pages)
    lengths = [_prefix(x, cfg.R).cuda() for x in ([9, 3, 5], [1, 9, 2], [4, 4, 9])]
    order = [torch.from_numpy(np.random.default_rng(i).permutation(pages)).cuda() for i in range(3)]
    # pool i holds page p of the packed one at order[i][p]
    pools = [{n: torch.empty_like(t[n]).view(pages, 128, 8, 128).index_copy_(0, o, t[n].view(pages, 128, 8, 128)).view_as(t[n])
              for n in ("k_cache", "v_cache")} if paged else t for o in order]
    tables = [o.to(torch.int32)[packed.long()].contiguous() for o in order]
    table = torch.zeros_like(packed)
    if fp8:
        cb.confu_set_kv_scales(gpu.ctx, t["k_scale"], t["v_scale"])
    gpu.ensure_ws(dims)
    plan = torch.zeros(cb.confu_plan_bytes(gpu.ctx, dims), dtype=torch.uint8, device="cuda")
    status = torch.zeros(cfg.B, dtype=torch.int32, device="cuda")

    def step(i, pool, ss, out):
        cb.confu_tree_plan(gpu.ctx, dims, ss, lengths[i], parent, owner, plan, status)
        cb.confu_tree_attention(gpu.ctx, dims, t["q"], pool["k_cache"], pool["v_cache"], pages * 128, ss, lengths[i], t["k_soft"], t["v_soft"],
                                None, None, plan, out, None, status)

    try:
        alone = [torch.empty_like(t["q"]) for _ in lengths]          # packed, one call at a time: tested against the oracle elsewhere
        for i, out in enumerate(alone):
            step(i, t, seq_start, out)
            torch.cuda.synchronize()
        if paged:
            cb.confu_set_paging(gpu.ctx, table, max_pages)
        plan.zero_()
        outs = [[torch.empty_like(t["q"]) for _ in lengths] for _ in range(5)]
        for o in outs:
            for i, out in enumerate(o):
                table.copy_(tables[i])
                step(i, pools[i], None if paged else seq_start, out)
        torch.cuda.synchronize()
        assert status.tolist() == [0] * cfg.B
        for o in outs:
            assert all(torch.equal(a, b) for a, b in zip(o, alone))
    finally:
        cb.confu_set_paging(gpu.ctx, None)
        cb.confu_set_kv_scales(gpu.ctx, None, None)


@pytest.mark.parametrize("kv", [torch.bfloat16, torch.float8_e4m3fn])
@pytest.mark.parametrize("B,Hkv,G,T,C", [(1, 8, 1, 4, 0), (1, 8, 1, 60, 3), (1, 8, 1, 60, 4), (3, 2, 1, 20, 4), (1, 2, 3, 20, 1), (1, 2, 3, 20, 2),
                                         (1, 2, 4, 15, 0), (1, 2, 4, 16, 0), (2, 2, 8, 7, 0), (1, 2, 4, 60, 60), (2, 2, 3, 50, 10)])
def test_few_rows_of_q(gpu, kv, B, Hkv, G, T, C):
    """Boxes of Q with 63, 64 and other few rows inside the tensor, under a plan made beforehand (what is asked for ahead of time depends on
    them) and under the call's own (nothing is)."""
    fp8 = kv == torch.float8_e4m3fn
    if fp8 and G > 4:
        pytest.skip("E4M3 caches: up to four query heads per kv head")
    cfg = inputs.VerifyConfig("few", B=B, L=1, Hq=Hkv * G, Hkv=Hkv, D=128, T=T, C=C, S=3, V=32, prefix=(100, 900), tree="chain", kv_dtype=kv,
                              logit_dtype=torch.float32, sigma_logit=1.0, draft="independent", temperatures=(1.0,), seed=780 + T)
    parent, owner, plen, seq_start, n_slots, t = H.setup_case(cfg)
    parent, owner, plen, seq_start = parent.cuda(), owner.cuda() if C else None, plen.cuda(), seq_start.cuda()
    dims = cb.make_dims(B, cfg.Hq, Hkv, 128, T, C, 3, torch.uint8 if fp8 else kv)
    gpu.ensure_ws(dims)
    if fp8:
        cb.confu_set_kv_scales(gpu.ctx, t["k_scale"], t["v_scale"])
    plan = torch.zeros(cb.confu_plan_bytes(gpu.ctx, dims), dtype=torch.uint8, device="cuda")
    status = torch.zeros(B, dtype=torch.int32, device="cuda")
    outs = [torch.empty_like(t["q"]) for _ in range(3)]
    try:
        for path in (cb.ATTENTION_AUTO, cb.ATTENTION_TENSOR):
            gpu.set_path(path)
            cb.confu_tree_plan(gpu.ctx, dims, seq_start, plen, parent, owner, plan, status)
            for out, own in zip(outs, (False, False, True)):
                cb.confu_tree_attention(gpu.ctx, dims, t["q"], t["k_cache"], t["v_cache"], n_slots, seq_start, plen, t["k_soft"], t["v_soft"],
                                        parent if own else None, owner if own else None, None if own else plan, out, None, status)
            torch.cuda.synchronize()
            assert not status.any() and all(torch.equal(outs[0], x) for x in outs[1:])
            if not fp8:
                want, _, _ = H.oracle_attention(cfg, t, seq_start.cpu(), plen.cpu(), parent.cpu(), owner.cpu() if C else torch.zeros((B, 0)))
                H.assert_attention_close(outs[0].cpu(), None, want, None, kv)
    finally:
        gpu.set_path(cb.ATTENTION_AUTO)
        cb.confu_set_kv_scales(gpu.ctx, None, None)
