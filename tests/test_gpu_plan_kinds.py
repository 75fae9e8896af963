"""A plan only fits the kind of work unit it was built for (two M tiles per CTA, one M tile per CTA, CTA pairs): any other
kernel refuses it with CONFU_ST_BAD_PLAN, computes nothing, and neither reads nor writes outside its buffers."""
import pytest
import torch

from paper_2603_08899_b200 import binding as cb
from paper_2603_08899_b200 import inputs
from tests import harness as H

pytestmark = pytest.mark.gpu

PATHS = {"auto": cb.ATTENTION_AUTO, "one_cta": cb.ATTENTION_TENSOR, "pairs": cb.ATTENTION_TENSOR_PAIR}


@pytest.fixture(scope="module")
def gpu():
    g = H.Gpu()
    yield g
    g.close()


@pytest.mark.parametrize("launched", list(PATHS))
@pytest.mark.parametrize("built", list(PATHS))
@pytest.mark.parametrize("B,prefix", [(8, (500, 2000)), (1, 3000)])
def test_plan_of_another_kind_is_refused(gpu, built, launched, B, prefix):
    """B 8: nearly as many shares as the GPU has SMs.  A plan for two M tiles per CTA numbers them 0 .. SMs - 1; with the one-M-tile
    kernel's two row groups those numbers, followed, would lead past the partial results in the workspace."""
    if built == launched:
        pytest.skip("the plan fits")
    cfg = inputs.VerifyConfig("kinds", B=B, L=1, Hq=32, Hkv=8, D=128, T=60, C=4, S=16, V=32, prefix=prefix, tree="random",
                              kv_dtype=torch.bfloat16, logit_dtype=torch.float32, sigma_logit=1.0, draft="independent",
                              temperatures=(1.0,), seed=700 + B, max_depth=7, fanout=(1, 4))
    parent, owner, plen, seq_start, n_slots, t = H.setup_case(cfg)
    dims = H.dims_of(cfg)
    gpu.ensure_ws(dims)
    gpu.ws.fill_(0)
    reg = []
    out, lse = H.guarded(reg, t["q"].shape, t["q"].dtype, 7.0), H.guarded(reg, (B, cfg.R, cfg.Hq), torch.float32, 7.0)
    status = H.guarded(reg, (B,), torch.int32, 0)
    plan = H.guarded(reg, (cb.confu_plan_bytes(gpu.ctx, dims),), torch.uint8)
    ss, pl = seq_start.cuda(), plen.cuda()
    try:
        gpu.set_path(PATHS[built])
        cb.confu_tree_plan(gpu.ctx, dims, ss, pl, parent.cuda(), owner.cuda(), plan, status)
        gpu.set_path(PATHS[launched])
        cb.confu_tree_attention(gpu.ctx, dims, t["q"], t["k_cache"], t["v_cache"], n_slots, ss, pl, t["k_soft"], t["v_soft"], None,
                                None, plan, out, lse, status)
        torch.cuda.synchronize()
    finally:
        gpu.set_path(cb.ATTENTION_AUTO)
    H.assert_guards(reg, "refused plan")
    assert gpu.ws_intact()
    assert status.cpu().tolist() == [cb.ST_BAD_PLAN] * B
    assert (out == 7.0).all() and (lse == 7.0).all()


@pytest.mark.parametrize("B,G,narrow", [(1, 4, True), (13, 4, True), (14, 4, False), (6, 8, True), (7, 8, False)])
def test_path_tells_which_plans_fit(gpu, B, G, narrow):
    """Up to three M tiles of query rows per two SMs (148 of them: 222) the automatic choice is one tile per CTA: confu_attention_path
    says so, and a plan built under AUTO fits a forced _TENSOR exactly when both paths have the same name."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms != 148:
        pytest.skip("the batches are those on either side of the rule for 148 SMs")
    cfg = inputs.VerifyConfig("paths", B=B, L=1, Hq=8 * G, Hkv=8, D=128, T=60, C=4, S=0, V=32, prefix=(1, 200), tree="random",
                              kv_dtype=torch.bfloat16, logit_dtype=torch.float32, sigma_logit=1.0, draft="independent",
                              temperatures=(1.0,), seed=710 + B, max_depth=7, fanout=(1, 4))
    dims = H.dims_of(cfg)
    parent, owner, plen, seq_start, n_slots, t = H.setup_case(cfg)
    gpu.ensure_ws(dims)
    plan = torch.empty(cb.confu_plan_bytes(gpu.ctx, dims), dtype=torch.uint8, device="cuda")
    status = torch.zeros(B, dtype=torch.int32, device="cuda")
    ss, pl = seq_start.cuda(), plen.cuda()
    auto = cb.confu_attention_path(gpu.ctx, dims)
    assert auto == (cb.ATTENTION_TENSOR_NARROW if narrow else cb.ATTENTION_TENSOR)
    cb.confu_tree_plan(gpu.ctx, dims, ss, pl, parent.cuda(), owner.cuda(), plan, status)
    try:
        gpu.set_path(cb.ATTENTION_TENSOR)
        assert cb.confu_attention_path(gpu.ctx, dims) == cb.ATTENTION_TENSOR
        out = torch.zeros_like(t["q"])
        cb.confu_tree_attention(gpu.ctx, dims, t["q"], t["k_cache"], t["v_cache"], n_slots, ss, pl, None, None, None, None, plan, out,
                                None, status)
        torch.cuda.synchronize()
        with pytest.raises(cb.ConfuError):
            gpu.set_path(cb.ATTENTION_TENSOR_NARROW)
    finally:
        gpu.set_path(cb.ATTENTION_AUTO)
    assert status.cpu().tolist() == [cb.ST_BAD_PLAN if narrow else 0] * B
