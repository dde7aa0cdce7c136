"""The results of a blocking call as one staged copy (small) and array by array (large), for every
subset of the arrays a caller may ask for: each equals the call that asks for all of them, at sizes
on both sides of the line with padded and unpadded state words, also at the end of a segment."""
import ctypes

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


KEYS = ("final_E", "best_E", "final_x", "best_x", "max_drift", "flips")


def _arrays(R, W):
    return dict(final_E=np.full(R, np.nan), best_E=np.full(R, np.nan), final_x=np.full((R, W), 0xABABABAB, np.uint32),
                best_x=np.full((R, W), 0xABABABAB, np.uint32), max_drift=np.full(R, np.nan),
                flips=np.full(R, -7, np.int64))


# (4 R 8 + 32 per replica and state word) bytes around 768 KB, N = 64 (2 of 4 words used) and N = 1024
@pytest.mark.parametrize("N,R", [(33, 3), (64, 5000), (64, 12287), (64, 12288), (64, 20000), (64, 30000), (1024, 2730),
                                 (1024, 2731), (1000, 9000)])
def test_every_subset_of_results(da, N, R):
    from paper_1806_08815_gb300 import instances as inst
    T, W = 6, da.da_words(N)
    q = inst.sk_gaussian(N, 1)
    beta = inst.beta_linear(0.1, 1.0, T)
    ctx = da.da_create(q.Q)
    L = da.lib()
    want = None
    subsets = [KEYS, ("best_E",), ("final_x",), ("best_x",), ("flips", "best_x"), ("max_drift", "final_E", "final_x"), ()]
    for sub in subsets:
        for segment in (False, True):
            a = _arrays(R, W)
            res = da.da_result(*(da._ptr(a[k]) if k in sub else None for k in KEYS), None, 0.0)
            if segment:
                rc = L.da_anneal_segment(ctx.handle, da._ptr(beta), T, 0, T, 0.25, R, 5, 3, None, None, ctypes.byref(res))
            else:
                rc = L.da_anneal(ctx.handle, da._ptr(beta), T, 0.25, R, 5, 3, ctypes.byref(res))
            assert rc == 0 and res.elapsed_s > 0
            want = want or {k: v.copy() for k, v in a.items()}
            untouched = _arrays(R, W)
            for k in KEYS:
                ref = want[k] if k in sub else untouched[k]
                assert np.array_equal(a[k], ref, equal_nan=a[k].dtype.kind == "f"), (sub, k)
    assert np.all(want["flips"] > 0) and np.isfinite(want["final_E"]).all()
    assert L.da_anneal(ctx.handle, da._ptr(beta), T, 0.25, R, 5, 3, None) == 0
    e = da.da_energy(ctx, want["best_x"][:200])
    assert np.array_equal(e, want["best_E"][:200])
