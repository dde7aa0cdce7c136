"""The batched launch recomputes the fp32 fields inside each replica's warp, with every
coupling split into three integers summed in 32-bit accumulators (and in 64-bit integers
where the scale leaves the fp32 range); the context path recomputes on the tensor cores.
Both follow one exact definition, so every result agrees bit for bit: instances on one
scale, with couplings that the fixed-point grid rounds, at extreme scales, at sizes around
the lane widths and the 32-variable words, alone and in one launch with others."""
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
    Q = instances.sk_gaussian(N, 4).Q if N > 1 else np.array([[-0.7]], np.float32)
    if kind == "mixed":      # magnitudes from 1 down to 2^-60: far below the grid, ties among them
        rng = np.random.default_rng(N)
        s = np.exp2(-rng.integers(0, 61, Q.shape))
        Q = np.triu(np.where(rng.random(Q.shape) < 0.3, np.sign(Q) * s, Q * s)).astype(np.float32)
    scale = {"sk": 0, "mixed": 0, "small": -50, "tiny": -110, "huge": 100}[kind]
    return (Q * np.float32(2.0 ** scale)).astype(np.float32), 2.0 ** scale


@pytest.mark.parametrize("kind", ["sk", "mixed", "small", "tiny", "huge"])
def test_batched_recompute_equals_the_context_path(da, kind):
    jobs = []
    for i, N in enumerate((1, 31, 33, 100, 129, 200, 256, 257, 500, 513, 1000, 1024)):
        Q, scale = _instance(kind, N)
        beta = (np.linspace(0.2, 5.0, 150) / scale).astype(np.float32)
        jobs.append(dict(ctx=da.da_create(Q), beta=beta, offset_inc=0.1 * scale, replicas=5, seed=i,
                         recompute_every=17 if i % 2 else 50))
    outs, _ = da.da_batch_anneal(jobs)
    for j, o in zip(jobs, outs):
        ref = da.da_anneal(j["ctx"], j["beta"], j["offset_inc"], 5, j["seed"], recompute_every=j["recompute_every"])
        for key in ("final_x", "best_x", "flips", "final_E", "best_E", "max_drift"):
            assert np.array_equal(o[key], ref[key]), (kind, j["ctx"].N, key)
