"""da_server_resident: every request of at most max_n variables runs as one launch, whatever
its replicas, seen in the server's launch count, and gives da_anneal's results."""
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


@pytest.mark.parametrize("N,R", [(33, 3), (128, 8), (256, 32), (257, 2), (300, 24), (512, 304), (513, 5), (1000, 20),
                                 (1024, 32), (1024, 305)])
def test_requests_up_to_max_n_take_one_launch(da, N, R):
    from paper_1806_08815_gb300 import instances as inst
    q = inst.sk_gaussian(N, N)
    T, P = 400, 16                       # 25 chunks of a step launch and a recompute, or one launch
    beta = inst.beta_linear(0.1, 6.0, T)
    srv = da.Server(8 << 30, 4)
    outs, launches = [], []
    for max_n in (1024, N, N - 1):
        srv.resident(max_n)
        before = srv.stats()["kernel_launches"]
        outs.append(da.da_poll(da.da_submit(srv, q.Q, beta, 0.5, R, 7, P), 60_000_000))
        launches.append(srv.stats()["kernel_launches"] - before)
    srv.close()
    assert launches[0] == launches[1] < T // P < launches[2], launches
    ref = da.da_anneal(da.da_create(q.Q), beta, 0.5, R, 7, recompute_every=P)
    for o in outs:
        for k in ("final_x", "best_x", "flips", "final_E", "best_E", "max_drift"):
            assert np.array_equal(o[k], ref[k]), k


def test_a_cancelled_resident_request_leaves_within_its_launch(da):
    """One launch of 3e7 steps (tens of seconds): cancelled, it is gone within a second."""
    import time
    from paper_1806_08815_gb300 import instances as inst
    q = inst.sk_bimodal(512, 8)
    srv = da.Server(8 << 30, 4)
    srv.resident(1024)
    before = srv.stats()["kernel_launches"]
    req = da.da_submit(srv, q.Q, np.full(30_000_000, 1.0, np.float32), 1.0, 32, 1)
    time.sleep(0.3)
    t0 = time.perf_counter()
    da.da_cancel(req)
    with pytest.raises(da.DAError) as e:
        da.da_poll(req, 60_000_000)
    assert e.value.status == 8 and time.perf_counter() - t0 < 1.0
    launches = srv.stats()["kernel_launches"] - before
    srv.close()
    assert launches < 20, launches        # chunked: 1832 step launches
