"""A full batch of the decode server fits its slot: requests with many chunks stay
within the pinned staging buffer, and a small memory budget holds what is put into
it, instead of the server failing for good once enough requests wait."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("restarts,max_batch,budget", [(256, 64, 0), (1024, 16, 0), (32, 1024, 192 << 10), (128, 256, 256 << 10)])
def test_waiting_requests_fill_a_slot(restarts, max_batch, budget):
    import paper_2509_17837_gb300 as X
    noise = X.noise_from_eta(0.1, 10.0)
    sv = X.Server(7, restarts, 40, 0.05, 20.0, max_batch=max_batch, n_slots=1, hbm_budget_bytes=budget, resident_waves=64)
    try:
        cid = sv.add_class(3, noise)
        sv.start()
        n = 400
        _, syn = X.sample_errors(X.Code(3), noise, 7, 0, n, want_errors=False)
        words = np.zeros((n, 32), np.uint32)
        words[:, :1] = syn.cpu().numpy().view(np.uint32)
        sv.replay(list(range(n)), [cid] * n, words, np.zeros(n))  # all at once: they wait for the one slot
        got = []
        for _ in range(300):
            got += sv.poll(timeout_ms=100)
            if len(got) == n:
                break
        assert sorted(r["req_id"] for r in got) == list(range(n))
        assert sv.stats()["batches"] < n // 4
    finally:
        sv.close()
