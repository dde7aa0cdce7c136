"""Few replicas of more than 2048 variables on clusters of four blocks: only by the automatic or the
tuned choice (a fixed shape runs as named), bit for bit the oracle's anneal in every coupling form, in
two segments whose cut falls inside a flip window and with a trace."""
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


@pytest.mark.parametrize("kind", ["int8", "fp32"])
@pytest.mark.parametrize("N,R", [(2049, 38), (2100, 5), (4096, 3), (4097, 4), (8192, 2)])
def test_automatic_clusters_match_the_oracle(da, kind, N, R):
    import oracle
    from paper_1806_08815_gb300 import instances as inst
    Q = (inst.sk_bimodal if kind == "int8" else inst.sk_gaussian)(N, 3).Q
    T, rec, inc, n = 151, 50, 0.25, min(R, 3)
    beta = (np.linspace(0.2, 6.0, T) / (np.sqrt(N) if kind == "int8" else 1.0)).astype(np.float32)
    ctx = da.da_create(Q)
    assert da.da_diag_launch_shape(ctx, R)[4] == 4
    ref = oracle.da_anneal(Q, beta, R=n, seed=9, inc=inc, recompute_every=rec, nthreads=n, trace=True)
    _, ck = da.da_anneal_segment(ctx, beta, 0, 71, inc, R, 9, recompute_every=rec)
    res, ck = da.da_anneal_segment(ctx, beta, 71, T, inc, R, 9, recompute_every=rec, checkpoint=ck)
    whole = da.da_anneal(ctx, beta, inc, R, 9, recompute_every=rec, trace=True)
    assert np.array_equal(whole["trace"][:n], ref["trace"])
    for k, o in (("final_x", "x_final"), ("best_x", "x_best"), ("flips", "flips")):
        assert np.array_equal(res[k][:n], ref[o]) and np.array_equal(whole[k], res[k]), k
    bits = ck["scalars"] if kind == "int8" else ck["scalars"].view(np.float64)
    assert np.array_equal(bits[:n, 0], ref["E_final"]) and np.array_equal(bits[:n, 1], ref["E_best"])


def test_fixed_and_tuned_shapes_run_as_named(da):
    from paper_1806_08815_gb300 import instances as inst
    N, R = 3000, 8
    q = inst.sk_bimodal(N, 1)
    beta = inst.beta_linear(0.05, 3.0, 200)
    ctx = da.da_create(q.Q)
    assert da.da_diag_launch_shape(ctx, R) == (16, 8, 1, 0, 4)
    ref = da.da_anneal(ctx, beta, 0.5, R, 1)
    assert da.da_diag_launch_shape(ctx, 39) == (16, 8, 1, 0, 1)
    for shape in ((16, 8, 1), (32, 8, 1), (32, 4, 1)):
        da.da_set_launch_shape(ctx, *shape)
        assert da.da_diag_launch_shape(ctx, R) == shape + (0, 1)
        out = da.da_anneal(ctx, beta, 0.5, R, 1)
        assert all(np.array_equal(out[k], ref[k]) for k in ("final_x", "best_x", "flips", "best_E"))
    da.da_set_launch_shape(ctx, 0, 0, 0)
    tuned = da.da_tune_shape(ctx, R, 300)
    run = da.da_diag_launch_shape(ctx, R)
    assert run[:2] == (tuned["V"], tuned["G"]) and run[4] in (1, 4)
    out = da.da_anneal(ctx, beta, 0.5, R, 1)
    assert all(np.array_equal(out[k], ref[k]) for k in ("final_x", "best_x", "flips", "best_E"))
