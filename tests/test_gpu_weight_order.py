"""A weight's fp16 split is complete before the product that follows it on the stream reads it, although the products
load their first weight tiles before they wait for the kernel before them."""

import pytest
import torch

pytestmark = pytest.mark.gpu

from paper_2609_15039_gb300 import workloads as wl  # noqa: E402


@pytest.fixture(scope="module")
def spl():
    from paper_2609_15039_gb300 import spl as s
    return s


# the swapped kernel, clusters of single SMs, pairs of SMs; the left operand split before, or by the call itself
@pytest.mark.parametrize("M", [16, 64, 1024])
@pytest.mark.parametrize("presplit", [True, False])
def test_a_product_sees_the_weight_split_just_before_it(spl, M, presplit):
    K, N = 3072, 16384
    old, new = (wl.weight(N, K, seed=s, device="cuda") for s in (1, 2))
    X, C = wl.activations(M, K, seed=3, device="cuda"), torch.zeros((M, N), device="cuda")
    W = spl.Weight.prepare(old, tf32=False)
    A = spl.Weight(None)
    A.f16_hi, A.f16_lo = (torch.empty((M, K), dtype=torch.int16, device="cuda") for _ in range(2))
    A.f16_exp = torch.empty(M, dtype=torch.int32, device="cuda")
    spl.spl_split_fp16(A.f16_hi, A.f16_lo, A.f16_exp, X)
    ws = spl.workspace(spl.spl_linear_workspace_bytes(M, K, N, "fp16x3"))

    def product(out):
        if presplit:
            spl.spl_masked_linear_unmask_split(out, A, W, C, path="fp16x3", workspace=ws)
        else:
            spl.spl_masked_linear_unmask(out, X, W, C, path="fp16x3", workspace=ws)

    got = [torch.empty((M, N), device="cuda") for _ in range(8)]
    for i, out in enumerate(got):  # the weight changes under the split buffers from call to call
        torch.cuda.synchronize()
        spl.spl_split_fp16(W.f16_hi, W.f16_lo, W.f16_exp, new if i % 2 == 0 else old)
        product(out)
    torch.cuda.synchronize()
    want = torch.empty((M, N), device="cuda")
    for i, w in enumerate((new, old)):
        spl.spl_split_fp16(W.f16_hi, W.f16_lo, W.f16_exp, w)
        torch.cuda.synchronize()
        product(want)
        for out in got[i::2]:
            assert torch.equal(out, want)
