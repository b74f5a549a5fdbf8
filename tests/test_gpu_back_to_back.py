"""Calls of the swapped kernel and of the binary64 slices right behind one another, so that each CTA follows others on
its SM with barriers at the same places in shared memory: every result as in a call that runs alone."""

import pytest
import torch

pytestmark = pytest.mark.gpu

from paper_2609_15039_gb300 import workloads as wl  # noqa: E402


@pytest.fixture(scope="module")
def spl():
    from paper_2609_15039_gb300 import spl as s
    return s


# one K block, one chain, two chains; fewer CTAs than SMs and more (binary64)
@pytest.mark.parametrize("K,N", [(64, 640), (1024, 2560), (2176, 9984)])
def test_calls_without_a_pause_equal_calls_alone(spl, K, N):
    M = 16
    W = spl.Weight.prepare(wl.weight(N, K, seed=1, device="cuda"), tf32=False)
    X, C = wl.activations(M, K, seed=2, device="cuda"), wl.activations(M, N, seed=3, norm="none", device="cuda")
    X64, C64 = X.double(), C.double()
    ws = spl.workspace(max(spl.spl_linear_workspace_bytes(M, K, N, "fp16x3"), spl.spl_f64_workspace_bytes(M, K, N)))

    def calls(y, z):
        spl.spl_masked_linear_unmask(y, X, W, C, path="fp16x3", workspace=ws)
        spl.spl_masked_linear_unmask_f64(z, X64, W.w, C64, workspace=ws)

    alone, alone64 = torch.empty((M, N), device="cuda"), torch.empty((M, N), device="cuda")
    torch.cuda.synchronize()
    spl.spl_masked_linear_unmask(alone, X, W, C, path="fp16x3", workspace=ws)
    torch.cuda.synchronize()
    spl.spl_masked_linear_unmask_f64(alone64, X64, W.w, C64, workspace=ws)
    torch.cuda.synchronize()
    outs = [(torch.zeros((M, N), device="cuda"), torch.zeros((M, N), device="cuda")) for _ in range(40)]
    torch.cuda.synchronize()
    for y, z in outs:
        calls(y, z)
    assert spl.spl_get_device_status() == 0
    for y, z in outs:
        assert torch.equal(y, alone) and torch.equal(z, alone64)
