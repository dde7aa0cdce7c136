"""DA_INT16 contexts anneal on exact fp32 couplings while every |Q_ii| + sum_j |Q_ij| stays
below 2^24 and on int16 couplings with int32 fields from there on: both sides of the line,
in the context path (results, and a checkpoint's integer fields) and in one batched launch,
bit for bit against the oracle's integer anneal."""
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


def _instance(N, row, over):
    """Couplings +-c and a first linear term that puts row 0's sum at 2^24 - 1 (or 2^24)."""
    rng = np.random.default_rng(N)
    c = min(32767, row // N)
    Q = np.triu(rng.choice(np.array([-c, c], np.int64), size=(N, N)), 1)
    np.fill_diagonal(Q, rng.integers(-1000, 1001, N))
    Q[0, 0] = (1 << 24) - 1 + over - (N - 1) * c
    return Q.astype(np.int32)


@pytest.mark.parametrize("over", [0, 1])
@pytest.mark.parametrize("N", [40, 200, 480, 1300])
def test_int16_on_both_sides_of_the_fp32_line(da, N, over):
    import oracle
    Q = _instance(N, 12_000_000, over)
    T, R, cut = 240, 4, 101
    beta = np.linspace(1e-6, 2e-4, T).astype(np.float32)
    ctx = da.da_create(Q, da.DA_INT16)
    ref = oracle.da_anneal(Q, beta, R=R, seed=3, inc=500.0, trace=True, nthreads=R)
    got = da.da_anneal(ctx, beta, 500.0, R, 3, trace=True)
    assert np.array_equal(got["trace"], ref["trace"])
    assert np.array_equal(got["best_x"], ref["x_best"]) and np.array_equal(got["final_E"], ref["E_final"])
    _, ck = da.da_anneal_segment(ctx, beta, 0, cut, 500.0, R, 3)
    d = np.diag(Q).astype(np.int64)
    for r in range(R):
        assert np.array_equal(ck["fields"][r].astype(np.int64), oracle.fields_int(Q, ck["x"][r]) + d)
    res, _ = da.da_anneal_segment(ctx, beta, cut, T, 500.0, R, 3, checkpoint=ck)
    assert np.array_equal(res["final_x"], ref["x_final"]) and np.array_equal(res["best_E"], ref["E_best"])
    if N <= 1024:
        jobs = [dict(ctx=ctx, beta=beta, offset_inc=500.0, replicas=R, seed=3),
                dict(ctx=da.da_create(_instance(N, 12_000_000, 1 - over), da.DA_INT16), beta=beta, offset_inc=500.0,
                     replicas=R, seed=3)]
        outs, _ = da.da_batch_anneal(jobs)
        assert np.array_equal(outs[0]["final_x"], ref["x_final"]) and np.array_equal(outs[0]["best_E"], ref["E_best"])
