"""Products with fewer rows than the 128 of a tile: the tensor-core kernels copy only the rows there are, the
tile's other rows keep what shared memory held; and the swapped kernel's split of 9 to 16 rows."""

import pytest
import torch

pytestmark = pytest.mark.gpu

from paper_2609_15039_gb300 import workloads as wl  # noqa: E402

from tests._util import assert_product_close, f32  # noqa: E402


@pytest.fixture(scope="module")
def spl():
    from paper_2609_15039_gb300 import spl as s
    return s


# around the 8-row steps of the copies and the warps' 32 rows; the last height that is cut and the first that is not
@pytest.mark.parametrize("M", [1, 7, 8, 9, 17, 24, 31, 33, 120, 121, 127, 128, 129])
@pytest.mark.parametrize("path,tile_n,ring_kb,splits,persistent", [
    ("fp16x3", 128, 224, 1, False), ("fp16x3", 128, 96, 2, False), ("fp16x3", 192, 224, 3, False),
    ("fp16x3", 224, 224, 1, True), ("tf32x3", 256, 192, 1, False), ("tf32x3", 160, 224, 2, False)])
def test_rows_that_are_not_there_do_not_matter(spl, M, path, tile_n, ring_kb, splits, persistent):
    """Equal bit for bit to the same rows of a full tile's product, after a product that leaves NaN and infinities
    in every row of every stage."""
    K, N = 1160, 2 * tile_n + 4
    W = spl.Weight.prepare(wl.weight(N, K, seed=3, device="cuda"))
    X = wl.activations(160, K, seed=4, device="cuda")
    C = wl.activations(160, N, seed=5, norm="none", device="cuda")
    ws = spl.workspace(spl.spl_linear_workspace_bytes(160, K, N, path))
    kw = dict(path=path, tile_n=tile_n, ring_kb=ring_kb, splits=splits, persistent=persistent, workspace=ws)
    full, Y = torch.empty((160, N), device="cuda"), torch.full((M, N), float("nan"), device="cuda")
    spl.spl_test_tc_product(full, X, W, C, **kw)
    bad = torch.full((160, K), float("nan"), device="cuda")
    bad[::3] = float("inf")
    spl.spl_test_tc_product(torch.empty_like(full), bad, W, C, **kw)
    spl.spl_test_tc_product(Y, X[:M], W, C[:M], **kw)
    assert torch.equal(Y, full[:M])
    spl.spl_test_tc_product(Y, X[:M], W, None, **kw)
    assert_product_close(f32(Y), f32(X[:M]), f32(W.w), path, what=f"{M} rows")
    assert spl.spl_get_device_status() == 0


# one tile; pieces of one k-block; several whole pieces a tile; a short last tile and k-block; one tile a CTA; more
# tiles than SMs; a width where no whole number of CTAs keeps the chains short
@pytest.mark.parametrize("K,N", [(8, 4), (256, 512), (1024, 1024), (2560, 6144), (1000, 2500), (256, 19456),
                                 (128, 20000), (512, 11008)])
@pytest.mark.parametrize("M", [9, 16])
def test_swapped_split_matches_bank(spl, M, K, N):
    """The library's product of 9 and 16 rows, and the same noise rows in a bank of 5 draws, whose sums must agree
    bit for bit."""
    W = spl.Weight.prepare(wl.weight(N, K, seed=7, device="cuda"), tf32=False)
    X = wl.activations(5 * M, K, seed=8, device="cuda")
    ws = spl.workspace(max(spl.spl_linear_workspace_bytes(M, K, N, "fp16x3"),
                           spl.spl_precompute_matched_workspace_bytes(5 * M, K, N, M, "fp16x3")))
    bank, Y = torch.empty((5 * M, N), device="cuda"), torch.full((M, N), float("nan"), device="cuda")
    spl.spl_precompute_noise_product_matched(bank, X, W, M, path="fp16x3", workspace=ws)
    zero = torch.zeros((M, N), device="cuda")
    for d in (0, 4):
        rows = X[d * M:(d + 1) * M].contiguous()
        spl.spl_masked_linear_unmask(Y, rows, W, zero, path="fp16x3", workspace=ws)
        assert torch.equal(Y, bank[d * M:(d + 1) * M])
        assert_product_close(f32(Y), f32(rows), f32(W.w), "fp16x3", what=f"{K} by {N}")
    assert spl.spl_get_device_status() == 0
