"""The launch model does not buy speed with longer accumulation chains: FP16X3 corrections against 64 bits."""

import math

import pytest
import torch

pytestmark = pytest.mark.gpu

from paper_2609_15039_gb300 import workloads as wl  # noqa: E402


@pytest.fixture(scope="module")
def spl():
    from paper_2609_15039_gb300 import spl as s
    return s


def _limit(K, splits):
    """Error of a K-split over `splits` CTAs of chains of at most 1024: each chain truncates in proportion to its length
    times its size (the square root of its length), 3.55e-9 measured (3.54 to 3.63 over 13 splits and chains), and 4%."""
    kps = -(-(-(-K // splits)) // 32) * 32
    total, k0 = 0, 0
    while k0 < K:
        n = min(kps, K - k0)
        total += (n // 1024) * 1024 ** 3 + (n % 1024) ** 3
        k0 += kps
    return 1.04 * 3.55e-9 * math.sqrt(total / K)


# rows of the online product, K, N, and the split of K that fills the chip with single SMs: 128-row products (whose
# order the banks follow), odd row counts, pairs, a K of no round size
@pytest.mark.parametrize("M,K,N,splits", [(128, 3072, 5120, 5), (128, 3072, 3072, 6), (128, 3072, 16384, 2),
                                          (61, 4096, 2560, 8), (61, 2560, 6144, 4), (61, 2560, 19456, 2),
                                          (17, 4096, 2560, 8), (256, 3072, 3072, 4), (1024, 3072, 5120, 1),
                                          (832, 2120, 11472, 1), (138, 4752, 5880, 3), (22, 2160, 4518, 5)])
def test_corrections_round_no_more_than_the_split_that_fills_the_chip(spl, M, K, N, splits):
    W = spl.Weight.prepare(wl.weight(N, K, seed=1, device="cuda"), tf32=False)
    eta = torch.randn((M, K), generator=torch.Generator(device="cuda").manual_seed(2), device="cuda") * 825.0
    C = torch.empty((M, N), device="cuda")
    ws = spl.workspace(spl.spl_precompute_matched_workspace_bytes(M, K, N, M, "fp16x3"))
    spl.spl_precompute_noise_product_matched(C, eta, W, M, path="fp16x3", workspace=ws)
    exact = eta.double() @ W.w.double().T
    err = float((C.double() - exact).norm() / exact.norm())
    assert err <= _limit(K, splits), (err, _limit(K, splits), spl.spl_test_tc_shape(M, K, N))
