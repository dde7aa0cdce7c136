"""The producer-warp form at its widest, V = 32: without padding, with a lane straddling N, with
whole lanes beyond N (they load their part of each row and leave it), down to one variable; int8,
fp32 and int16 couplings of both forms, bit for bit against the oracle."""
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


@pytest.mark.parametrize("kind", ["int8", "fp32", "int16", "int16 wide"])
@pytest.mark.parametrize("N", [1, 31, 33, 513, 992, 1000, 1023, 1024])
def test_widest_producer_form_matches_the_oracle(da, kind, N):
    import oracle
    from paper_1806_08815_gb300 import instances as inst
    T, R, P = 400, 4, 100
    beta = np.linspace(0.05, 6.0, T).astype(np.float32)
    dtype = None
    if kind == "int8":
        Q, beta = inst.sk_bimodal(N, 2).Q, (beta / np.sqrt(N)).astype(np.float32)
    else:
        Q = inst.sk_gaussian(N, 2).Q
        if kind != "fp32":
            Q, s = da.da_quantize(Q) if N > 1 else (np.array([[-7]], np.int32), 1.0)
            beta, dtype = (beta / s).astype(np.float32), da.DA_INT16
            if kind == "int16 wide":           # a row sum of 2^24 or more: int16 couplings
                Q = Q.copy()
                Q[0, 0] = -(1 << 24)
    ctx = da.da_create(Q, dtype)
    da.da_set_launch_shape(ctx, 32, 1, 1)
    da.da_set_draw_warp(ctx, 1)
    assert da.da_diag_launch_shape(ctx, R)[3] == 1
    res = da.da_anneal(ctx, beta, 0.25, R, 9, recompute_every=P, trace=True)
    ref = oracle.da_anneal(Q, beta, R=R, seed=9, inc=0.25, recompute_every=P, nthreads=R, trace=True)
    assert np.array_equal(res["trace"], ref["trace"])
    for k, o in (("final_x", "x_final"), ("best_x", "x_best"), ("flips", "flips")):
        assert np.array_equal(res[k], ref[o]), k
