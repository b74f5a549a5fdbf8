"""Outputs whose rows are no whole 16-byte units (N % 4 != 0): the epilogues that go by single elements."""

import pytest
import torch

pytestmark = pytest.mark.gpu

from paper_2609_15039_gb300 import workloads as wl  # noqa: E402


@pytest.fixture(scope="module")
def spl():
    from paper_2609_15039_gb300 import spl as s
    return s


# every cluster size, one SM and pairs; row tiles of 1 and of 7 rows (ranks without any), a ragged last tile
@pytest.mark.parametrize("path,tile_n,ring_kb,splits", [
    ("fp16x3", 128, 224, 1), ("fp16x3", 128, 96, 2), ("fp16x3", 160, 224, 3), ("fp16x3", 192, 224, 4),
    ("fp16x3", 224, 224, 5), ("fp16x3", 256, 192, 6), ("fp16x3", 128, 224, 7), ("fp16x3", 256, 192, 8),
    ("fp16x3", 128, 448, 1), ("fp16x3", 256, 448, 1), ("tf32x3", 192, 224, 1), ("tf32x3", 128, 96, 8)])
@pytest.mark.parametrize("M,extra", [(1, 1), (33, 2), (135, 35), (257, 127)])
def test_ragged_rows_equal_padded_ones(spl, path, tile_n, ring_kb, splits, M, extra):
    """Bit for bit the columns of the product with the weight padded to a multiple of 4 rows; nothing else is
    written, in front of the output's first row or behind its last."""
    K, N = 1064, tile_n + extra
    Np = (N + 3) // 4 * 4
    wp = wl.weight(Np, K, seed=3, device="cuda")
    X = wl.activations(M, K, seed=4, device="cuda")
    Cp = wl.activations(M, Np, seed=5, norm="none", device="cuda")
    ws = spl.workspace(spl.spl_linear_workspace_bytes(M, K, Np, path))
    kw = dict(path=path, tile_n=tile_n, ring_kb=ring_kb, splits=splits, persistent=ring_kb == 448, workspace=ws)
    W, Wp = spl.Weight.prepare(wp[:N].contiguous()), spl.Weight.prepare(wp)
    for C in (Cp, None):
        ref = torch.empty((M, Np), device="cuda")
        spl.spl_test_tc_product(ref, X, Wp, C, **kw)
        buf = torch.full((M * N + 512,), 7.0, device="cuda")
        Y = buf[256:256 + M * N].view(M, N)
        spl.spl_test_tc_product(Y, X, W, None if C is None else C[:, :N].contiguous(), **kw)
        assert torch.equal(Y, ref[:, :N])
        assert bool((buf[:256] == 7.0).all()) and bool((buf[256 + M * N:] == 7.0).all())
    assert spl.spl_get_device_status() == 0


@pytest.mark.parametrize("M,c_rows", [(40, 20), (200, 100), (600, 300), (600, 64)])
def test_fewer_ragged_correction_rows(spl, M, c_rows):
    """The stacked call: rows past C's are plain products."""
    K, N = 2056, 5003
    W = spl.Weight.prepare(wl.weight(N, K, seed=6, device="cuda"), tf32=False)
    X = wl.activations(M, K, seed=7, device="cuda")
    C = wl.activations(c_rows, N, seed=8, norm="none", device="cuda")
    ws = spl.workspace(spl.spl_linear_workspace_bytes(M, K, N, "fp16x3"))
    plain, Y = torch.empty((M, N), device="cuda"), torch.full((M, N), float("nan"), device="cuda")
    spl.spl_masked_linear(plain, X, W, path="fp16x3", workspace=ws)
    spl.spl_masked_linear_unmask_precompute(Y, spl.Weight(X), W, C, c_rows, path="fp16x3", workspace=ws)
    assert torch.equal(Y[c_rows:], plain[c_rows:])
    assert torch.equal(Y[:c_rows], plain[:c_rows] - C)
    assert spl.spl_get_device_status() == 0
