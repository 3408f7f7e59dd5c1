"""The annealing launch forms agree bit for bit: one thread per chain (launches
that fill the GPU), several lanes per chain with every warp sweeping, and several
lanes per chain with producing warps (small launches).  The last two are pinned
to the oracle by test_gpu_parity.py; here the first is compared with them at the
sizes where the choice changes."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    import paper_2509_17837_gb300 as X
    return X, torch


@pytest.mark.parametrize("d", range(3, 32, 2))
def test_thread_and_lane_forms_agree(env, d):
    X, torch = env
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    restarts = 37  # 148 chains per shot: ragged warps and CTAs in every form
    shots = (144 * n_sm) // (4 * restarts) + 2  # past the lane forms' range at every distance
    code, noise = X.Code(d), X.noise_from_eta(0.17, 10.0)
    sched = X.Schedule(noise, 11, 0.05, 3.0)  # 11 sweeps: a partial set of tables
    _, syn = X.sample_errors(code, noise, 5, 7, shots)
    init, _ = X.greedy_init(code, noise, 5, 7, syn, restarts)
    kw = dict(want_cfg=True, want_final=True)
    thread = X.anneal(code, sched, 5, 7, init, **kw)
    lanes = X.anneal(code, sched, 5, 7, init, per_warp=True, **kw)
    few = X.anneal(code, sched, 5, 7, init[:1].contiguous(), **kw)
    for k in thread:
        assert torch.equal(thread[k], lanes[k]), k
        assert torch.equal(thread[k][:1], few[k]), k
