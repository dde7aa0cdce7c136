"""The step kernels settle the tracked energy and the best state 32 flips at a time
(FlipLog): as integers where every fp64 addition of the in-order sum is exact, one
addition after the other elsewhere.  Checked against the oracle, which adds and tests
after every step, bit for bit: tracked energies (the checkpoint's scalars), best states,
flips.  The instances reach both forms: energies on one grid, energies that gain and lose
binary places (couplings of mixed magnitude), exponents outside the integer form's range,
numbers of steps and recompute periods around the 32-flip window, steps without flips, one
and several warps per replica (each warp restores its own words of the best state)."""
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


def _instance(kind, N):
    from paper_1806_08815_gb300 import instances
    if kind == "int8":
        return instances.sk_bimodal(N, 3).Q, 1.0
    Q = instances.sk_gaussian(N, 3).Q
    rng = np.random.default_rng(N)
    if kind == "mixed":        # couplings from 1 down to 2^-40: sums that cannot be exact on one grid
        Q = np.triu(Q * np.exp2(-rng.integers(0, 41, Q.shape))).astype(np.float32)
        return Q, 0.2
    if kind == "tiny":         # energies near 2^-120
        return (Q * np.float32(2.0 ** -120)).astype(np.float32), 2.0 ** -119
    if kind == "huge":         # energies near 2^110
        return (Q * np.float32(2.0 ** 105)).astype(np.float32), 2.0 ** 106
    return Q, 1.0


@pytest.mark.parametrize("kind", ["int8", "sk", "mixed", "tiny", "huge"])
@pytest.mark.parametrize("N,shape", [(33, (4, 1, 4)), (100, (8, 1, 2)), (500, (16, 1, 1)), (1000, (32, 1, 4)),
                                     (200, (4, 2, 2)), (509, (4, 4, 1)), (700, (8, 4, 1)), (1024, (16, 2, 1)),
                                     (1023, (16, 4, 1)), (1500, (8, 8, 1))])
@pytest.mark.parametrize("T,rec", [(1, 0), (33, 1), (700, 31)])
def test_tracked_energy_and_best_state_match_the_oracle(da, kind, N, shape, T, rec):
    import oracle
    Q, scale = _instance(kind, N)
    beta = (np.linspace(0.2, 6.0, T) / scale).astype(np.float32)
    inc, R = 0.25 * min(scale, 1.0), 5
    ctx = da.da_create(Q)
    da.da_set_launch_shape(ctx, *shape)
    res, ck = da.da_anneal_segment(ctx, beta, 0, T, inc, R, 9, recompute_every=rec)
    ref = oracle.da_anneal(Q, beta, R=R, seed=9, inc=inc, recompute_every=rec, nthreads=5)
    tracked = ck["scalars"][:, 0] if kind == "int8" else ck["scalars"][:, 0].view(np.float64)
    best = ck["scalars"][:, 1] if kind == "int8" else ck["scalars"][:, 1].view(np.float64)
    assert np.array_equal(res["final_x"], ref["x_final"])
    assert np.array_equal(res["flips"], ref["flips"])
    assert np.array_equal(res["best_x"], ref["x_best"])
    assert np.array_equal(tracked, ref["E_final"])
    assert np.array_equal(best, ref["E_best"])


@pytest.mark.parametrize("kind", ["int8", "sk", "mixed"])
@pytest.mark.parametrize("N,shape,R", [(2049, (16, 8, 1), 5), (4096, (16, 8, 1), 3), (1100, (32, 8, 1), 4),
                                       (4200, (32, 8, 1), 2), (2100, (16, 8, 1), 40)])
def test_replicas_on_clusters_match_the_oracle(da, kind, N, shape, R):
    """The widest shapes run few replicas on clusters of four blocks (the last case, with more
    replicas, on one block each): tracked and best energies, states and flips, in two segments
    whose cut falls inside a flip window."""
    import oracle
    T, rec = 151, 50
    Q, scale = _instance(kind, N)
    beta = (np.linspace(0.2, 6.0, T) / scale).astype(np.float32)
    ctx = da.da_create(Q)
    da.da_set_launch_shape(ctx, *shape)
    _, ck = da.da_anneal_segment(ctx, beta, 0, 71, 0.25, R, 9, recompute_every=rec)
    res, ck = da.da_anneal_segment(ctx, beta, 71, T, 0.25, R, 9, recompute_every=rec, checkpoint=ck)
    n = min(R, 3)
    ref = oracle.da_anneal(Q, beta, R=n, seed=9, inc=0.25, recompute_every=rec, nthreads=n)
    assert np.array_equal(res["final_x"][:n], ref["x_final"])
    assert np.array_equal(res["flips"][:n], ref["flips"])
    assert np.array_equal(res["best_x"][:n], ref["x_best"])
    bits = ck["scalars"] if kind == "int8" else ck["scalars"].view(np.float64)
    assert np.array_equal(bits[:n, 0], ref["E_final"])
    assert np.array_equal(bits[:n, 1], ref["E_best"])

