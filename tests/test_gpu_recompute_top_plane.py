"""The top digit plane of the tensor-core recompute at its largest sums: states of all ones over
couplings that are all the largest an instance of that scale can hold (or 1, its smallest largest
entry), of either sign.  The fields and energies have a closed form, exact in integers."""
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


@pytest.mark.parametrize("N", [1, 63, 64, 65, 1023, 1024, 2000, 2048, 2049, 4095, 4096, 4097, 8191, 8192])
@pytest.mark.parametrize("sign", [-1.0, 1.0])
@pytest.mark.parametrize("top", [1.0, 2.0 - 2.0 ** -23])
def test_largest_couplings_are_summed_exactly(da, N, sign, top):
    # entries below 2^1: the grid is 2^-S, S = 62 - L - 1 with 2^L >= N + 1
    S = 62 - math.ceil(math.log2(N + 1)) - 1
    c = np.float32(sign * top)
    ctx = da.da_create(np.triu(np.full((N, N), c, np.float32)))
    words = da.da_words(N)
    x = np.full((3, words), 0xFFFFFFFF, np.uint32)
    if N % 32:
        x[:, -1] = (1 << (N % 32)) - 1
    x[1, 0] &= ~np.uint32(1)
    x[2] = 0
    h, E = da.da_field_recompute(ctx, x), da.da_energy(ctx, x)
    unit = int(float(c) * 2 ** 24) << (S - 24) if S >= 24 else None
    assert unit is not None
    for r, bits in enumerate((np.ones(N, bool), np.r_[False, np.ones(N - 1, bool)], np.zeros(N, bool))):
        n = int(bits.sum())
        for i in {0, N // 2, N - 1}:
            assert h[r, i] == _f32(unit * (1 + n - int(bits[i])), S), (r, i)
        # sum over the set bits of the diagonal and half the couplings among them
        assert E[r] == math.ldexp(float(unit * (2 * n + n * (n - 1))), -(S + 1)), r


def _f32(v, S):
    """fl32(v) 2^-S of an exact integer v (Python's int to float rounds to nearest even at 53 bits,
    so the rounding to 24 is made on the integer)."""
    m = abs(v)
    k = m.bit_length() - 24
    if k > 0:
        q, rem = divmod(m, 1 << k)
        half = 1 << (k - 1)
        q += rem > half or (rem == half and q & 1)
        m = q << k
    return np.float32(math.copysign(math.ldexp(float(m), -S), v)) if v else np.float32(0)
