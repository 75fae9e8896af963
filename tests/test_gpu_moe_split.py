"""Contemplate-token embedding where the split over a cluster has remainders: fewer experts than CTAs, experts and
columns that do not divide by eight, one / two / four sequences per cluster with a ragged last cluster."""
import pytest
import torch

from oracle import ref
from tests import harness as H
from tests.test_gpu_moe import _case, _gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    g = H.Gpu()
    yield g
    g.close()


@pytest.mark.parametrize("B,H_in,H_out,n,k,dtype", [
    (1, 8, 8, 3, 2, torch.bfloat16), (16, 264, 72, 9, 3, torch.bfloat16), (17, 1032, 40, 65, 4, torch.bfloat16),
    (33, 520, 136, 17, 5, torch.float32), (35, 49, 19, 130, 8, torch.bfloat16), (64, 3000, 1000, 100, 1, torch.float32),
    # one CTA per sequence, 512 or 256 threads, or per four (small routers, large batches): dot products whole and in 2 to 16
    # parts, the last three sequences of four missing, rows that do not divide by a vector
    (5, 4096, 64, 1, 1, torch.bfloat16), (3, 2056, 24, 3, 2, torch.float32), (7, 1531, 33, 5, 2, torch.bfloat16), (444, 64, 48, 20, 4, torch.bfloat16),
    (445, 1024, 40, 2, 2, torch.float32), (500, 72, 16, 33, 3, torch.bfloat16), (889, 520, 24, 4, 2, torch.bfloat16), (1001, 40, 17, 9, 9, torch.float32)])
def test_split_matches_oracle(gpu, B, H_in, H_out, n, k, dtype):
    h, w, b, e = _case(B, H_in, H_out, n, seed=900 + B + n, dtype=dtype)
    want, wsel, wgate, gap = ref.con_embedding(h, w, b, e, k, True)
    out, sel, gate = _gpu(gpu, h, w, b, e, k, True)
    # the bounds of tests/test_gpu_moe.py: bf16 rounds the sum once (2^-9 of it), fp32 sums up to 3000 products
    tol = 1e-2 if dtype == torch.bfloat16 else 1e-5
    close = 0
    for i in range(B):
        if not torch.equal(sel[i], wsel[i]):
            assert gap[i].item() < 1e-4 or sorted(sel[i].tolist()) == sorted(wsel[i].tolist())
            close += 1
            continue
        assert torch.allclose(gate[i].double(), wgate[i], rtol=1e-4, atol=1e-6)
        assert (out[i].double() - want[i]).abs().max().item() <= tol * max(want[i].abs().max().item(), 1e-3)
    assert close <= max(1, B // 8)
