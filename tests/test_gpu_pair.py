"""The pair kernel (256-row tiles on two SMs) against the single-SM product it must equal bit for bit, and
against the fp64 product, at the edges of its tiles, chains and correction rows."""

import pytest
import torch

pytestmark = pytest.mark.gpu

from paper_2609_15039_gb300 import workloads as wl  # noqa: E402

from tests._util import assert_product_close, f32  # noqa: E402

WIDTHS = (256, 224, 192, 160, 128)
PAIR_RING = 448


@pytest.fixture(scope="module")
def spl():
    from paper_2609_15039_gb300 import spl as s
    return s


def _problem(spl, M, K, N, seed):
    W = spl.Weight.prepare(wl.weight(N, K, seed=seed, device="cuda"), tf32=False)
    X = wl.activations(M, K, seed=seed + 1, device="cuda")
    C = wl.activations(M, N, seed=seed + 2, norm="none", device="cuda")
    ws = spl.workspace(spl.spl_linear_workspace_bytes(M, K, N, "fp16x3"))
    return W, X, C, ws


# (rows, K, outputs past a whole tile): one row, the two CTAs' boundary, a ragged second row tile; one k-block,
# an odd number of them, one element of K past a chain, several chains; a last tile of 4 columns or none, output rows
# that are no whole number of 16-byte units
@pytest.mark.parametrize("bn", WIDTHS)
@pytest.mark.parametrize("M,K,extra", [(1, 32, 4), (128, 8, 0), (129, 96, 36), (256, 1024, 0), (257, 1032, 4),
                                       (300, 3080, 100), (161, 64, 1), (290, 1096, 35)])
def test_pair_equals_unsplit_product(spl, bn, M, K, extra):
    N = bn + extra
    W, X, C, ws = _problem(spl, M, K, N, seed=11)
    for Cx in (C, None):
        ref, Y = torch.empty((M, N), device="cuda"), torch.full((M, N), float("nan"), device="cuda")
        spl.spl_test_tc_product(ref, X, W, Cx, tile_n=256, ring_kb=192, splits=1, workspace=ws)
        spl.spl_test_tc_product(Y, X, W, Cx, tile_n=bn, ring_kb=PAIR_RING, persistent=True, workspace=ws)
        assert torch.equal(Y, ref), float((Y - ref).abs().max())
    assert_product_close(f32(Y), f32(X), f32(W.w), "fp16x3", what=f"pair {bn}")
    assert spl.spl_get_device_status() == 0


@pytest.mark.parametrize("bn", WIDTHS)
def test_pair_over_several_tiles_a_pair(spl, bn):
    """More tiles than pairs, ragged in every direction, 3 chains of K: the ring and the accumulators run on."""
    M, K, N = 1290, 2100 // 8 * 8, 12 * 76 // 5 * 32 + 20
    W, X, C, ws = _problem(spl, M, K, N, seed=21)
    assert -(-M // 256) * -(-N // bn) > spl.spl_test_tc_capacity(bn, PAIR_RING, 2)
    ref, Y = torch.empty((M, N), device="cuda"), torch.full((M, N), float("nan"), device="cuda")
    spl.spl_test_tc_product(ref, X, W, C, tile_n=256, ring_kb=192, splits=1, workspace=ws)
    spl.spl_test_tc_product(Y, X, W, C, tile_n=bn, ring_kb=PAIR_RING, persistent=True, workspace=ws)
    assert torch.equal(Y, ref), float((Y - ref).abs().max())
    assert spl.spl_get_device_status() == 0


@pytest.mark.parametrize("K,s", [(2560, 3), (3072, 8), (1032, 2)])
def test_pair_segments_equal_split_product(spl, K, s):
    """The bank's form: segments at a split's K ranges (27 k-blocks, 12, 17: odd ones end inside a stage)."""
    M, N = 270, 1000
    W, X, _C, ws = _problem(spl, M, K, N, seed=31)
    ref, Y = torch.empty((M, N), device="cuda"), torch.full((M, N), float("nan"), device="cuda")
    spl.spl_test_tc_product(ref, X, W, None, tile_n=256, ring_kb=192, splits=s, workspace=ws)
    spl.spl_test_tc_product(Y, X, W, None, tile_n=192, ring_kb=PAIR_RING, persistent=True, seg_splits=s, workspace=ws)
    assert torch.equal(Y, ref), float((Y - ref).abs().max())
    assert spl.spl_get_device_status() == 0


@pytest.mark.parametrize("N", [16384, 16383])
@pytest.mark.parametrize("M", [4, 100, 128, 488])
def test_library_pair_product_with_fewer_correction_rows(spl, M, N):
    """The stacked call on the pair kernel: C has M rows, the rows after them are corrections, equal to the
    product without C bit for bit (the boundary inside a warp's 32 rows, at a CTA's and past a tile's end)."""
    rows, K = 1000, 1024
    assert spl.spl_test_tc_shape(rows, K, N)[1] == PAIR_RING
    W, X, C, ws = _problem(spl, rows, K, N, seed=41)
    plain, YC = torch.empty((rows, N), device="cuda"), torch.full((rows, N), float("nan"), device="cuda")
    spl.spl_masked_linear(plain, X, W, path="fp16x3", workspace=ws)
    spl.spl_masked_linear_unmask_precompute(YC, spl.Weight(X), W, C[:M].contiguous(), M, path="fp16x3", workspace=ws)
    assert torch.equal(YC[M:], plain[M:])
    assert torch.equal(YC[:M], plain[:M] - C[:M])
    assert spl.spl_get_device_status() == 0


def test_pair_variant_is_refused_outside_its_forms(spl):
    W, X, C, ws = _problem(spl, 64, 64, 64, seed=51)
    Y = torch.empty((64, 64), device="cuda")
    for kw in (dict(splits=2), dict(persistent=False), dict(full_tiles=1), dict(path="tf32x3")):
        args = dict(tile_n=128, ring_kb=PAIR_RING, persistent=True, workspace=ws)
        args.update(kw)
        with pytest.raises(spl.SplError):
            spl.spl_test_tc_product(Y, X, W, C, **args)
