"""The tensor-core recompute at the ends of its digit planes' range: states of all ones over
couplings that are one power of two, so that every term of a plane's sum over the couplings
is the lowest digit -2^(b-1) (or the highest power below the highest digit), with one large
coupling that fixes the scale.  The fields have a closed form, exact in 64-bit integers."""
import math

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


@pytest.mark.parametrize("N", [63, 1024, 2000, 4096, 8192])
@pytest.mark.parametrize("sign", [-1.0, 1.0])
@pytest.mark.parametrize("plane", [0, 1, 2, 3, 4])
def test_extreme_digit_sums_are_exact(da, N, sign, plane):
    # the fixed-point grid of an instance whose largest entry is 1: 2^-S, S = 62 - L - 1
    # (entries below 2^1), 2^L >= N + 1; b bits per plane
    L = math.ceil(math.log2(N + 1))
    S = 62 - L - 1
    b = min(12, 23 - math.ceil(math.log2(N)))
    e = b - 1 + b * plane - S                 # coupling 2^e: digit 2^(b-1) of the plane, as -2^(b-1)
    if e >= 0:
        pytest.skip("above the largest entry")
    c = sign * 2.0 ** e
    Q = np.triu(np.full((N, N), c, np.float32), 1)
    Q[0, 1] = 1.0
    np.fill_diagonal(Q, np.float32(c))
    ctx = da.da_create(Q)
    words = da.da_words(N)
    x = np.full((3, words), 0xFFFFFFFF, np.uint32)
    if N % 32:
        x[:, -1] = (1 << (N % 32)) - 1
    x[1, 0] &= ~np.uint32(1)                  # without variable 0
    x[2] = 0
    h = da.da_field_recompute(ctx, x)
    unit = int(c * 2.0 ** S)                  # exact: the coupling in units of the grid
    one = 1 << S
    for r, bits in enumerate((np.ones(N, bool), np.r_[False, np.ones(N - 1, bool)], np.zeros(N, bool))):
        n = int(bits.sum())
        for i in {0, 1, 2, N // 2, N - 1}:
            s = unit + unit * (n - int(bits[i]))
            if i == 0 and bits[1]:
                s += one - unit
            if i == 1 and bits[0]:
                s += one - unit
            assert h[r, i] == _round(s, S), (r, i)


def _round(v, S):
    """fl32(v) 2^-S of an exact integer v."""
    if v == 0:
        return np.float32(0)
    m, k = abs(v), abs(v).bit_length() - 24
    if k > 0:
        q, rem = divmod(m, 1 << k)
        half = 1 << (k - 1)
        q += rem > half or (rem == half and q & 1)
        m = q << k
    return np.float32(math.copysign(math.ldexp(float(m), -S), v))
