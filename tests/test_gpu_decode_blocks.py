"""The decode kernel's masked instances against the plan, which sizes their grids by the unmasked instance."""

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def spl():
    from paper_2609_15039_gb300 import spl as s
    return s


@pytest.mark.parametrize("M", [1, 2, 3, 4])
@pytest.mark.parametrize("ks", [64, 320, 768, 1536])
@pytest.mark.parametrize("mask", [0, 1, 2])
def test_masked_instances_fill_the_planned_blocks(spl, M, ks, mask):
    """Fewer resident blocks than planned: a second, mostly empty wave (2 of 3 at one row and eps = inf took 133 us for
    106); more: fewer registers than the loads in flight need."""
    assert spl.spl_test_gemv_blocks(M, ks, mask) == spl.spl_test_gemv_blocks(M, ks)


def test_blocks_hook_refuses_what_has_no_instance(spl):
    for args in ((0, 64, -1), (17, 64, -1), (1, 63, -1), (1, 1537, -1), (8, 64, 0), (1, 64, 3), (1, 64, -2)):
        with pytest.raises(spl.SplError):
            spl.spl_test_gemv_blocks(*args)
