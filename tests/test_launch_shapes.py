"""The automatic launch shape as a rule on sizes alone (host code, no device): every choice covers N
with the narrowest lane width of its group, is a shape the kernels exist for, has the padded width of
every other choice for that N (the row-ordered copies are shared by width), and takes clusters only
where there are few replicas of the widest shapes."""
import numpy as np
import pytest


@pytest.fixture(scope="module")
def da():
    from paper_1806_08815_gb300 import binding, build
    build.build()
    return binding


def test_automatic_shapes_over_all_sizes(da):
    widths = {1: (4, 8, 16, 32), 2: (4, 8, 16, 32), 4: (4, 8, 16, 32), 8: (8, 16, 32)}
    rs = [1, 2, 5, 37, 38, 39, 64, 151, 152, 153, 303, 304, 305, 608, 1000, 1216, 1217, 4096, 65536]
    for N in list(range(1, 70)) + [k + d for k in (128, 256, 512, 1024, 2048, 4096, 8192) for d in (-1, 0, 1) if k + d <= 8192]:
        pad = max(128, 1 << (N - 1).bit_length())
        for R in rs:
            V, G, rpb, ws, blocks = da.da_diag_launch_shape(None, R, N)
            assert V in widths[G] and 32 * V * G == pad, (N, R)
            assert 1 <= rpb <= {1: 4, 2: 2}.get(G, 1) and ws == 0
            assert blocks == (4 if N > 2048 and R <= 38 else 1), (N, R)
            if N <= 256:
                assert G == 1
            if 1024 < N <= 2048:
                assert (G, rpb) == ((4, 1) if R <= 1216 else (2, 2))


def test_arguments_are_checked(da):
    for N, R in ((0, 1), (8193, 1), (64, 0), (64, -3)):
        with pytest.raises(da.DAError):
            da.da_diag_launch_shape(None, R, N)
    assert da.lib().da_diag_launch_shape(None, 64, 1, None) == 1
