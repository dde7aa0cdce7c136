"""The kernels on int16 couplings with int32 fields, which take DA_INT16 instances with a row sum of
2^24 or more and those beyond N = 4096 (the others anneal on exact fp32 couplings): over the launch
shapes, on clusters, with the producer warp and under PTDA, bit for bit against the oracle."""
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


def _instance(da, N, seed, wide=True):
    """Gaussian couplings in 16 bits; wide: one linear term of 2^24, so that its row's fields need int32."""
    from paper_1806_08815_gb300 import instances as inst
    Q, scale = da.da_quantize(inst.sk_gaussian(N, seed).Q)
    if wide:
        Q = Q.copy()
        Q[N // 2, N // 2] = -(1 << 24)
    return Q, scale


def _check(da, ctx, Q, beta, inc, R, n):
    import oracle
    got = da.da_anneal(ctx, beta, inc, R, 8, trace=True)
    ref = oracle.da_anneal(Q, beta, R=n, seed=8, inc=np.float32(inc), trace=True, nthreads=n)
    assert np.array_equal(got["trace"][:n], ref["trace"])
    for k, o in (("final_x", "x_final"), ("best_x", "x_best"), ("flips", "flips"), ("final_E", "E_final"),
                 ("best_E", "E_best")):
        assert np.array_equal(got[k][:n], ref[o]), k
    assert np.all(got["max_drift"] == 0)


@pytest.mark.parametrize("N,shape", [(100, (4, 1, 4)), (100, (4, 2, 2)), (128, (4, 1, 1)), (200, (8, 1, 2)), (256, (8, 1, 4)),
                                     (200, (8, 2, 1)), (250, (4, 4, 1)), (500, (16, 1, 4)), (512, (16, 1, 4)),
                                     (512, (16, 2, 2)), (1000, (32, 1, 4)), (1024, (32, 1, 4)), (1024, (8, 4, 1)),
                                     (1024, (32, 2, 2)), (2048, (16, 4, 1)), (2048, (8, 8, 1)), (2100, (32, 4, 1)),
                                     (2100, (16, 8, 1)), (2100, (32, 8, 1))])
def test_trajectories_over_launch_shapes(da, N, shape):
    Q, scale = _instance(da, N, 5)
    beta = (np.linspace(0.1, 10.0, 600) / scale).astype(np.float32)
    ctx = da.da_create(Q, da.DA_INT16)
    da.da_set_launch_shape(ctx, *shape)
    _check(da, ctx, Q, beta, 0.3 * scale, 7 if N <= 1024 else 3, 7 if N <= 1024 else 3)


@pytest.mark.parametrize("N,R,wide,want", [(60, 9, True, (4, 1)), (300, 9, True, (4, 4)), (300, 305, True, (16, 1)),
                                           (1500, 9, True, (16, 4)), (2049, 5, True, (16, 8)), (2100, 39, True, (16, 8)),
                                           (3000, 153, True, (32, 4)), (4096, 3, True, (16, 8)), (4097, 4, False, (32, 8)),
                                           (4097, 39, False, (32, 8)), (6000, 38, False, (32, 8)), (8192, 2, False, (32, 8)),
                                           (8192, 40, False, (32, 8))])
def test_automatic_shapes(da, N, R, wide, want):
    """Clusters (5, 3, 4, 38 and 2 replicas beyond N = 2048) and single blocks, padded and full widths."""
    Q, scale = _instance(da, N, 6, wide)
    beta = (np.linspace(0.1, 10.0, 130) / scale).astype(np.float32)
    ctx = da.da_create(Q, da.DA_INT16)
    shape = da.da_diag_launch_shape(ctx, R)
    assert shape[:2] == want and shape[4] == (4 if N > 2048 and R <= 38 else 1)
    _check(da, ctx, Q, beta, 0.3 * scale, R, min(R, 3))


@pytest.mark.parametrize("N", [60, 200, 256, 500, 512])
def test_draw_warp_and_ptda(da, N):
    import oracle
    Q, scale = _instance(da, N, 7)
    beta = (np.linspace(0.1, 10.0, 500) / scale).astype(np.float32)
    ctx = da.da_create(Q, da.DA_INT16)
    da.da_set_draw_warp(ctx, 1)
    assert da.da_diag_launch_shape(ctx, 5)[3] == 1
    _check(da, ctx, Q, beta, 0.5 * scale, 5, 5)
    da.da_set_draw_warp(ctx, 0)
    betas = (np.geomspace(0.2, 5.0, 6) / scale).astype(np.float32)
    g = da.da_pt(ctx, betas, 6, 3, 4, swap_trace=True)
    r = oracle.ptda(Q, betas, 6, L=3, seed=4, nthreads=3)
    assert np.array_equal(g["swap_trace"], r["swap_trace"]) and np.array_equal(g["best_x"], r["x_best"])
    assert np.array_equal(g["best_E"], r["E_best"]) and np.array_equal(g["final_E"], r["E_final"])


@pytest.mark.parametrize("N", [300, 1024, 2100])
def test_wide_rows_keep_no_fp32_couplings(da, N):
    """What tells the two forms apart from outside: the fp32 couplings' 4 N^2 bytes."""
    sizes = []
    for wide in (False, True):
        Q, _ = _instance(da, N, 8, wide)
        before = da.da_diag_live_allocations()["bytes"]
        ctx = da.da_create(Q, da.DA_INT16)
        sizes.append(da.da_diag_live_allocations()["bytes"] - before)
        del ctx
    assert sizes[0] - sizes[1] >= 4 * N * N
