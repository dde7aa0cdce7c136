"""da_set_draw_warp takes one-warp shapes up to N = 1024 and changes nothing above, where no
one-warp shape holds the instance."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def da():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1806_08815_gb300 import binding
    return binding


@pytest.mark.parametrize("N", [40, 300, 1024, 1025, 2049, 3000, 4096, 4097])
def test_draw_warp_changes_one_warp_sizes_only(da, N):
    ctx = da.da_create(np.triu(np.ones((N, N), np.int32)))
    for R in (1, 38, 39, 152, 153, 304, 305, 2000):
        da.da_set_draw_warp(ctx, 1)
        on = da.da_diag_launch_shape(ctx, R)
        da.da_set_draw_warp(ctx, 0)
        off = da.da_diag_launch_shape(ctx, R)
        if N > 1024:
            assert on == off
        else:
            assert on[1] == 1 and on[3] == 1 and on[0] == max(4, 1 << ((N - 1).bit_length() - 5)), on
