"""Planning a call on the host: the choices, and what they cost (no GPU work)."""

import time

import pytest

from paper_2609_15039_gb300 import spl

SMS = 152  # what the library assumes without a device


def _swap_ctas(K, N):
    """CTAs of the swapped kernel as its comment states them: the model's best whole number of CTAs per weight tile."""
    cd = lambda a, b: -(-a // b)
    tiles, nkb = cd(N, 128), cd(K, 64)
    total = tiles * nkb
    even = SMS if tiles > SMS else max(1, min(3 * SMS // 4, total))
    longest = min(16, nkb if 4 * tiles >= 3 * SMS else cd(total, even))
    hbm, best, pick, k = total * 32768.0 / 6.7e6, float("inf"), even, 1
    while k * tiles <= SMS and k <= nkb:
        if min(16, cd(nkb, k)) <= longest:
            c = ((0.37 * cd(nkb, k)) ** 4 + hbm ** 4) ** 0.25 + (2.4 + 0.15 * k if k > 1 else 0.0)
            if c < best * (1.0 - 1e-9):
                best, pick = c, k * tiles
        k += 1
    return min(pick, total)


@pytest.mark.parametrize("N", [1, 64, 128, 129, 512, 2560, 4096, 6144, 14592, 14593, 19456, 19457, 32768])
@pytest.mark.parametrize("K", [64, 72, 256, 1024, 1032, 2560, 4096, 9728])
def test_swapped_kernel_ctas(K, N):
    got = spl.spl_split_workspace_bytes(16, K, N, path="fp16x3") - 64 * 1024
    assert got == _swap_ctas(K, N) * 2 * 16 * 128 * 4  # two slots of 16 x 128 sums a CTA


def test_planning_a_few_row_call_costs_no_more_with_many_candidates():
    """One weight tile and 152 k-blocks have 152 candidates; they took seven times as long as a single one."""
    L, path = spl.lib(), spl._path("fp16x3")

    def best(K, N):
        t = []
        for _ in range(30):
            t0 = time.perf_counter()
            for _ in range(300):
                L.spl_linear_workspace_bytes(16, K, N, path)
            t.append(time.perf_counter() - t0)
        return min(t)

    assert best(9728, 64) <= 3.0 * best(64, 64)
