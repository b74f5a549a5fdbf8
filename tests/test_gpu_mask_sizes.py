"""The mask kernel's two launch shapes draw the same noise: sizes on both sides of the lines between them."""

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def spl():
    from paper_2609_15039_gb300 import spl as s
    return s


@pytest.mark.parametrize("mech,eps", [("laplace", 1.0), ("gaussian", 1.0), ("gaussian", float("inf"))])
@pytest.mark.parametrize("n", [2 ** 23 - 4, 2 ** 23 - 1, 2 ** 23, 2 ** 23 + 5, 2 ** 24 - 1, 2 ** 24, 2 ** 24 + 7, 5 * 10 ** 7 + 3])
def test_large_masks_equal_their_parts(spl, mech, eps, n):
    """Masked at once, and as parts of fewer entries (the other shape, and part trips) with their block offsets."""
    g = torch.Generator(device="cuda").manual_seed(3)
    X = torch.randn((1, n), generator=g, device="cuda")
    Xt, N = torch.full_like(X, float("nan")), torch.full_like(X, float("nan"))
    spl.spl_noise_mask(Xt, N, X, 2.0, eps, mech, 11, offset=5)
    step = 4 * 1_000_003
    for a in range(0, n, step):
        b = min(n, a + step)
        xt, nz = torch.full_like(X[:, a:b], float("nan")), torch.full_like(X[:, a:b], float("nan"))
        spl.spl_noise_mask(xt, nz, X[:, a:b].contiguous(), 2.0, eps, mech, 11, offset=5 + a // 4)
        assert torch.equal(Xt[:, a:b], xt) and torch.equal(N[:, a:b], nz), (a, b)
