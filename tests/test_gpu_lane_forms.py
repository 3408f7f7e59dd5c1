"""The lane-parallel annealing forms on both sides of the sizes where the launch
rule changes from one to the next: three producing CTAs per SM, four, and every
warp sweeping.  Each launch equals the first shots of a launch that takes the
one-thread-per-chain form (planar d > 15: the form where every warp sweeps)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    import paper_2509_17837_gb300 as X
    return X, torch


def chains_per_cta(planar, d):
    lanes = 4 if planar else 2
    while lanes < (d if planar else (d + 1) // 2):
        lanes *= 2
    return 32 // lanes


@pytest.mark.parametrize("planar", [False, True])
@pytest.mark.parametrize("d", range(3, 32, 2))
def test_producing_forms_at_their_limits(env, planar, d):
    X, torch = env
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    code, noise = X.Code(d, X.LAYOUT_PLANAR if planar else X.LAYOUT_ROTATED), X.noise_from_eta(0.15, 10.0)
    shots = 70 * n_sm + 1  # 280 chains per SM at one restart
    _, syn = X.sample_errors(code, noise, 5, 7, shots)
    init, _ = X.greedy_init(code, noise, 5, 7, syn, 1)
    for sweeps, b0, b1 in ((11, 0.05, 3.0), (37, 0.1, 60.0)):  # a partial set of sweeps; frozen from about a third
        sched = X.Schedule(noise, sweeps, b0, b1)
        many = X.anneal(code, sched, 5, 7, init, want_cfg=True, want_final=True)
        for per_sm in (3, 4):
            last = per_sm * n_sm * chains_per_cta(planar, d) // 4
            for take in (last, last + 1):
                few = X.anneal(code, sched, 5, 7, init[:take].contiguous(), want_cfg=True, want_final=True)
                for k in many:
                    assert torch.equal(many[k][:take], few[k]), (k, take)
                few = X.anneal(code, sched, 5, 7, init[:take].contiguous(), want_cfg=False)
                assert torch.equal(many["best_E"][:take], few["best_E"])


@pytest.mark.parametrize("d", [5, 7, 9, 13, 15, 17, 21, 31])
def test_planar_sweeping_forms_at_their_limits(env, d):
    """Every warp sweeping: two to six CTAs per SM and one more of each."""
    X, torch = env
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    code, noise = X.Code(d, X.LAYOUT_PLANAR), X.noise_from_eta(0.15, 10.0)
    shots = 70 * n_sm + 1
    _, syn = X.sample_errors(code, noise, 5, 7, shots)
    init, _ = X.greedy_init(code, noise, 5, 7, syn, 1)
    sched = X.Schedule(noise, 37, 0.1, 60.0)
    many = X.anneal(code, sched, 5, 7, init, want_cfg=True, want_final=True)
    for per_sm in (2, 3, 4, 5, 6):
        last = per_sm * n_sm * chains_per_cta(True, d)
        for take in (last, last + 1):
            few = X.anneal(code, sched, 5, 7, init[:take].contiguous(), want_cfg=True, want_final=True)
            for k in many:
                assert torch.equal(many[k][:take], few[k]), (k, take)


@pytest.mark.parametrize("d", [7, 11, 17, 31])
def test_batch_lane_forms_at_their_limits(env, d):
    """Batch mode 2, whose chunks of 128 chains are cut into the same forms."""
    X, torch = env
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    code, noise = X.Code(d), X.noise_from_eta(0.15, 10.0)
    sched = X.Schedule(noise, 37, 0.1, 60.0)
    ctas_per_chunk = 128 // chains_per_cta(False, d)
    sizes = sorted({n for per_sm in (3, 4) for n in (per_sm * n_sm // ctas_per_chunk, per_sm * n_sm // ctas_per_chunk + 1)})
    _, syn = X.sample_errors(code, noise, 5, 7, sizes[-1])
    for shots in sizes:  # 32 restarts: one chunk per shot
        b = X.Batch([dict(code=code, noise=noise, sched=sched, shot0=7, syndromes=syn[:shots].contiguous(), restarts=32)], 5)
        b.run(1)
        want = {k: b.outputs[0][k].clone() for k in ("cls", "E4", "recovery")}
        for k in want:
            b.outputs[0][k].zero_()
        b.run(2)
        torch.cuda.synchronize()
        for k in want:
            assert torch.equal(b.outputs[0][k], want[k]), (k, shots)
        b.close()
