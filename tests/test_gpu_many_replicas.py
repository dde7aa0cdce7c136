"""More replicas than two full waves of the four-warp shape at 1025..2048 variables: the two-warp
shape with two replicas to a block, an odd one at the end, results per replica as with one replica
alone (keyed by its index) and as the oracle's."""
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
@pytest.mark.parametrize("N,R", [(1025, 1217), (1500, 1301), (2048, 1217)])
def test_many_replicas_match_few_and_the_oracle(da, kind, N, R):
    import oracle
    from paper_1806_08815_gb300 import instances as inst
    Q = (inst.sk_bimodal if kind == "int8" else inst.sk_gaussian)(N, 3).Q
    beta = (np.linspace(0.2, 6.0, 120) / (np.sqrt(N) if kind == "int8" else 1.0)).astype(np.float32)
    ctx = da.da_create(Q)
    assert da.da_diag_launch_shape(ctx, R) == (32, 2, 2, 0, 1)
    assert da.da_diag_launch_shape(ctx, 1216) == (16, 4, 1, 0, 1)
    many = da.da_anneal(ctx, beta, 0.25, R, 9, recompute_every=50)
    few = da.da_anneal(ctx, beta, 0.25, 40, 9, recompute_every=50)
    for k in ("final_x", "best_x", "flips", "final_E", "best_E"):
        assert np.array_equal(many[k][:40], few[k]), k
    last = oracle.da_anneal(Q, beta, R=1, seed=9, inc=0.25, recompute_every=50, replica_base=R - 1)
    for k, o in (("final_x", "x_final"), ("best_x", "x_best"), ("flips", "flips")):
        assert np.array_equal(many[k][-1], last[o][0]), k
