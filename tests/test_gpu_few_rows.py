"""Products with fewer rows than the 128 of a tile: the tensor-core kernels copy only the rows there are, the
tile's other rows keep what shared memory held."""

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
