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
    shots = (280 * n_sm) // (4 * restarts) + 2  # past the lane forms' range at every distance
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


@pytest.mark.parametrize("d", range(3, 16, 2))
def test_one_warp_and_wide_ctas_agree(env, d):
    """One thread per chain: CTAs of one warp up to 384 chains per SM, wide ones above."""
    X, torch = env
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    restarts = 37
    wide, narrow = (384 * n_sm) // (4 * restarts) + 1, (384 * n_sm) // (4 * restarts)
    code, noise = X.Code(d), X.noise_from_eta(0.17, 10.0)
    sched = X.Schedule(noise, 11, 0.05, 3.0)
    _, syn = X.sample_errors(code, noise, 5, 7, wide)
    init, _ = X.greedy_init(code, noise, 5, 7, syn, restarts)
    kw = dict(want_cfg=True, want_final=True)
    a, b = X.anneal(code, sched, 5, 7, init, **kw), X.anneal(code, sched, 5, 7, init[:narrow].contiguous(), **kw)
    for k in a:
        assert torch.equal(a[k][:narrow], b[k]), k


@pytest.mark.parametrize("d", range(3, 32, 2))
def test_planar_forms_agree(env, d):
    """On the planar lattice (d <= 15: one thread per chain, then several lanes;
    above: lanes with every warp sweeping, then with producing warps)."""
    X, torch = env
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    restarts = 37
    shots = (128 * n_sm) // (4 * restarts) + 2
    code, noise = X.Code(d, X.LAYOUT_PLANAR), X.noise_from_eta(0.13, 5.0, X.CONVENTION_PAPER)
    _, syn = X.sample_errors(code, noise, 5, 7, shots)
    init, _ = X.greedy_init(code, noise, 5, 7, syn, restarts)
    for n, b0, b1 in ((11, 0.9, 1.0), (60, 0.1, 60.0)):  # the second freezes
        sched = X.Schedule(noise, n, b0, b1)
        many = X.anneal(code, sched, 5, 7, init, want_cfg=True, want_final=True)
        no_final = X.anneal(code, sched, 5, 7, init, want_cfg=True)
        assert torch.equal(no_final["best_E"], many["best_E"]) and torch.equal(no_final["best_cfg"], many["best_cfg"])
        for take in (1, 1 + 40 * n_sm // (4 * restarts)):
            few = X.anneal(code, sched, 5, 7, init[:take].contiguous(), want_cfg=True, want_final=True)
            for k in many:
                assert torch.equal(many[k][:take], few[k]), (k, take)
            few = X.anneal(code, sched, 5, 7, init[:take].contiguous(), want_cfg=False)
            assert torch.equal(many["best_E"][:take], few["best_E"])


@pytest.mark.parametrize("d,eta", [(3, 10.0), (5, 100.0), (11, 100.0), (15, 1.0), (17, 100.0), (21, 1.0), (31, 1000.0)])
def test_stopping_in_the_frozen_sweeps_changes_no_minimum(env, d, eta):
    """Past the last sweep with a threshold above zero a warp whose chains all
    repeat stops, unless the final states are asked for: the minima with and
    without them are the same, in the thread form, both lane forms and a batch."""
    X, torch = env
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    restarts = 32
    shots = (280 * n_sm) // (4 * restarts) + 1
    code, noise = X.Code(d), X.noise_from_eta(0.15, eta)
    sched = X.Schedule(noise, 150, 0.1, 60.0)  # frozen from about a fifth of the sweeps
    _, T = sched.table()
    assert not T[-1].any() and T[0].any()
    _, syn = X.sample_errors(code, noise, 9, 0, shots)
    init, cbits = X.greedy_init(code, noise, 9, 0, syn, restarts)
    full = X.anneal(code, sched, 9, 0, init, want_cfg=True, want_final=True)
    for per_warp in (False, True):
        got = X.anneal(code, sched, 9, 0, init, want_cfg=True, per_warp=per_warp)
        assert torch.equal(got["best_E"], full["best_E"]) and torch.equal(got["best_cfg"], full["best_cfg"])
        got = X.anneal(code, sched, 9, 0, init, want_cfg=False, per_warp=per_warp)
        assert torch.equal(got["best_E"], full["best_E"])
        few = X.anneal(code, sched, 9, 0, init[:2].contiguous(), want_cfg=True, per_warp=per_warp)
        assert torch.equal(few["best_E"], full["best_E"][:2]) and torch.equal(few["best_cfg"], full["best_cfg"][:2])
    want = X.decode_reduce(code, init, cbits, full["best_E"])
    b = X.Batch([dict(code=code, noise=noise, sched=sched, shot0=0, syndromes=syn, restarts=restarts)], 9)
    for mode in (0, 1, 2):
        b.run(mode)
        torch.cuda.synchronize()
        assert all(torch.equal(b.outputs[0][k], want[k]) for k in ("cls", "E4", "recovery"))
    b.close()
