"""The decode kernel's masked forms for grids of few and of many waves: one result, that of the mask and the product as
two calls."""

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def spl():
    from paper_2609_15039_gb300 import spl as s
    return s


# N on both sides of 0.82 (one row at eps = inf) and 2 waves of the blocks that the plan counts on, ragged in both; K at
# one slice, past one, and of more than 16 (the sums taken 16 at a time there)
@pytest.mark.parametrize("mech,eps", [("laplace", 1.0), ("gaussian", 1.0), ("laplace", float("inf"))])
@pytest.mark.parametrize("K,N", [(64, 130), (1540, 40003), (2048, 17000), (2048, 33001), (26000, 1100)])
@pytest.mark.parametrize("rows,bank", [(1, 0), (2, 0), (3, 0), (4, 0), (1, 1), (2, 2), (1, 2)])
def test_masked_call_equals_mask_then_product(spl, mech, eps, K, N, rows, bank):
    g = torch.Generator(device="cuda").manual_seed(K + N + rows)
    W = torch.randn((N, K), generator=g, device="cuda") * 0.02
    X, C = torch.randn((rows, K), generator=g, device="cuda"), torch.randn((rows, N), generator=g, device="cuda")
    M = rows + bank
    ws = spl.workspace(spl.spl_linear_workspace_bytes(M, K, N, "fp32"))
    Y, Xt = torch.full((M, N), float("nan"), device="cuda"), torch.full((M, K), float("nan"), device="cuda")
    kw = dict(path="fp32", workspace=ws)
    delta = rows * K // 4 + 3
    if bank:
        spl.spl_noise_mask_linear_unmask_precompute(Y, Xt, X, W, C, 825.0, eps, mech, 7, bank, delta, **kw)
    else:
        spl.spl_noise_mask_linear_unmask(Y, Xt, X, W, C, 825.0, eps, mech, 7, **kw)
    want = torch.empty((M, K), device="cuda")
    spl.spl_noise_mask(want[:rows], None, X, 825.0, eps, mech, 7)
    if bank:
        spl.spl_noise(want[rows:], 825.0, eps, mech, 7, offset=delta)
    assert torch.equal(Xt, want)
    P = torch.empty((M, N), device="cuda")
    spl.spl_masked_linear(P, want, W, **kw)
    assert torch.equal(Y[rows:], P[rows:])
    assert torch.equal(Y[:rows], P[:rows] - C)
