"""Traces of a batched launch: items with and without one in the same classes (every coupling form
and kernel source of rows), with recomputes inside the run, against da_anneal's and the oracle's, the
untraced items' results untouched; and a traced launch makes each step's draws once."""
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


def _item(da, kind, N):
    from paper_1806_08815_gb300 import instances as inst
    beta = np.linspace(0.05, 6.0, 500).astype(np.float32)
    if kind == "int8":
        return inst.sk_bimodal(N, 2).Q, None, (beta / np.sqrt(N)).astype(np.float32)
    Q = inst.sk_gaussian(N, 2).Q
    if kind == "fp32":
        return Q, None, beta
    Q, s = da.da_quantize(Q)
    Q = Q.copy()
    Q[0, 0] = -(1 << 24)                       # int16 couplings, not exact fp32
    return Q, da.DA_INT16, (beta / s).astype(np.float32)


@pytest.mark.parametrize("staging", [-1, 0, 1, 2])
@pytest.mark.parametrize("N", [50, 128, 250, 256, 500, 1000])
def test_traces_in_mixed_classes(da, staging, N):
    import oracle
    from paper_1806_08815_gb300 import binding
    jobs, refs = [], []
    for kind in ("int8", "fp32", "int16"):
        Q, dtype, beta = _item(da, kind, N)
        ctx = da.da_create(Q, dtype)
        for traced in (True, False):
            jobs.append(dict(ctx=ctx, beta=beta, offset_inc=0.25, replicas=5, seed=9, trace=traced,
                             recompute_every=100 if kind == "fp32" else 0))
            refs.append(oracle.da_anneal(Q, beta, R=5, seed=9, inc=0.25, recompute_every=jobs[-1]["recompute_every"],
                                         nthreads=5, trace=True))
    try:
        binding._check(binding.lib().da_batch_force(staging, 0))
        outs, _ = da.da_batch_anneal(jobs)
    finally:
        binding.lib().da_batch_force(-1, 0)
    for j, o, ref in zip(jobs, outs, refs):
        if j["trace"]:
            assert np.array_equal(o["trace"], ref["trace"])
        for k, r in (("final_x", "x_final"), ("best_x", "x_best"), ("flips", "flips")):
            assert np.array_equal(o[k], ref[r]), k


def test_a_trace_costs_less_than_the_draws(da):
    """A step's draws are about as long as the rest of it, so drawing twice doubles it; storing the
    flipped index adds a few percent.  The line is drawn at half the step (best of five runs)."""
    Q, dtype, _ = _item(da, "fp32", 1000)
    ctx = da.da_create(Q)
    beta = np.linspace(0.05, 6.0, 4000).astype(np.float32)
    best = {}
    for traced in (False, True):
        job = [dict(ctx=ctx, beta=beta, offset_inc=0.0, replicas=64, seed=9, trace=traced, recompute_every=0)]
        best[traced] = min(da.da_batch_anneal(job)[1] for _ in range(5))
    assert best[True] < 1.5 * best[False], best
