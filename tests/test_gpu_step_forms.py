"""The forms of a step chosen by padding: without padding variables (N = 32 V G) V = 16 takes the
wide form of the one-warp step and the early exact test of the several-warp step, with them
V = 8 takes packed field updates.  Each against the oracle bit for bit at the padded width and
one variable below it, over enough trials (about 4e-5 of them) that the exact test is taken,
with steps on which nothing flips, at hot and cold ends of a schedule."""
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
@pytest.mark.parametrize("shape", [(4, 1, 4), (8, 1, 4), (16, 1, 4), (32, 1, 4), (16, 2, 2), (16, 4, 1)])
@pytest.mark.parametrize("short", [0, 1])
def test_full_and_padded_widths_match_the_oracle(da, kind, shape, short):
    import oracle
    from paper_1806_08815_gb300 import instances
    N = 32 * shape[0] * shape[1] - short
    T, R, inc = 1500, 5, 0.25
    Q = instances.sk_bimodal(N, 4).Q if kind == "int8" else instances.sk_gaussian(N, 4).Q
    beta = np.linspace(0.05, 6.0, T).astype(np.float32) / (np.sqrt(N) if kind == "int8" else 1.0)
    beta = beta.astype(np.float32)
    ctx = da.da_create(Q)
    da.da_set_launch_shape(ctx, *shape)
    res = da.da_anneal(ctx, beta, inc, R, 9, recompute_every=500)
    ref = oracle.da_anneal(Q, beta, R=R, seed=9, inc=inc, recompute_every=500, nthreads=5)
    for k, o in (("final_x", "x_final"), ("best_x", "x_best"), ("flips", "flips")):
        assert np.array_equal(res[k], ref[o]), k


@pytest.mark.parametrize("N", [256, 255, 512, 511])
def test_allocation_free_form_at_both_widths(da, N):
    """The int8 rows of the allocation-free anneal against the context's anneal (exact fp32)."""
    import torch
    from paper_1806_08815_gb300 import instances
    Q = instances.sk_bimodal(N, 5).Q
    T, R, inc = 1500, 320, 0.5                # more replicas than take several warps each
    beta = (np.linspace(0.05, 6.0, T) / np.sqrt(N)).astype(np.float32)
    want = da.da_anneal(da.da_create(Q), beta, inc, R, 9)
    ldw = da.da_static_pitch(N)
    U = np.triu(Q, 1)
    W = np.zeros((N, ldw), np.int8)
    W[:, :N] = U + U.T
    out = dict(final_x=torch.zeros((R, da.da_words(N)), dtype=torch.int32, device="cuda"),
               best_x=torch.zeros((R, da.da_words(N)), dtype=torch.int32, device="cuda"),
               flips=torch.zeros(R, dtype=torch.int64, device="cuda"))
    stream = torch.cuda.current_stream()
    da.da_anneal_static(torch.from_numpy(W).cuda(), torch.from_numpy(np.diag(Q).astype(np.int32)).cuda(), N, ldw,
                        torch.from_numpy(beta).cuda(), T, inc, R, 9, out, stream)
    torch.cuda.synchronize()
    for k in ("final_x", "best_x", "flips"):
        got = out[k].cpu().numpy()
        assert np.array_equal(got.view(want[k].dtype), want[k]), k
