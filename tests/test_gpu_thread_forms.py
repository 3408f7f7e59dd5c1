"""One thread per chain against the oracle: launches large enough to take those
kernels (CTAs of one warp and wide ones, the row layout past d = 21, the planar
register kernel) over the schedules, scales and chain ids of the small parity
tests, a sample of their chains compared bit for bit; and the checked build's
bounds checks in the same kernels and in the literal forms."""
import ctypes

import numpy as np
import pytest

import oracle as O
from layout import words_to_labels
from test_gpu_device_errors import _checked_lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    import paper_2509_17837_gb300 as X
    return X, torch


# (planar, d, chains per SM): past the lane-parallel launches; up to 384 CTAs of one warp at rotated d <= 15
FORMS = [(False, 3, 330), (False, 3, 400), (False, 7, 330), (False, 7, 400), (False, 15, 330), (False, 15, 400),
         (False, 17, 300), (False, 21, 300), (False, 23, 300), (False, 31, 300), (True, 3, 260), (True, 9, 260),
         (True, 15, 260)]
EDGES = [(0, 0, 0.1, 1.0), (0, 1, 0.4, 9.0), (0, 3, 0.0, 0.0), (0, 12, 1e6, 1e6), (1, 30, 0.9, 1.0), (0, 60, 0.05, 20.0)]


def launch(X, torch, planar, d, per_sm, noise, seed, shot0):
    code = X.Code(d, X.LAYOUT_PLANAR if planar else X.LAYOUT_ROTATED)
    shots = per_sm * torch.cuda.get_device_properties(0).multi_processor_count // 4 + 1  # one restart; a ragged last CTA
    _, syn = X.sample_errors(code, noise, seed, shot0, shots)
    init, _ = X.greedy_init(code, noise, seed, shot0, syn, 1)
    return code, shots, init


def against_the_oracle(X, torch, planar, d, per_sm, noise, kind, n, b0, b1, seed=3, shot0=11):
    code, shots, init = launch(X, torch, planar, d, per_sm, noise, seed, shot0)
    out = X.anneal(code, X.Schedule(noise, n, b0, b1, kind=kind), seed, shot0, init, want_cfg=True, want_final=True)
    cid, pxyz = O.planar(d) if planar else d, (noise.px, noise.py, noise.pz)
    LX, LZ = O.logicals(cid)
    cosets = [0 * LX, LX, LX ^ LZ, LZ]
    for s in (0, shots // 3, shots - 1):
        ref0 = words_to_labels(init[s].cpu().numpy(), code.n_qubits)[0]
        best = words_to_labels(out["best_cfg"][s].cpu().numpy().reshape(4, -1), code.n_qubits)
        last = words_to_labels(out["final_cfg"][s].cpu().numpy().reshape(4, -1), code.n_qubits)
        for P in range(4):
            ref = O.anneal_chain_variant(cid, pxyz, noise.scale, kind, n, b0, b1, seed, (shot0 + s) * 4 + P,
                                         ref0 ^ cosets[P], 0, 0)
            assert out["best_E"][s, 0, P] == ref["best_E"] and out["final_E"][s, 0, P] == ref["final_E"], (s, P)
            assert np.array_equal(best[P], ref["best"]) and np.array_equal(last[P], ref["final"]), (s, P)


@pytest.mark.parametrize("planar,d,per_sm", FORMS)
def test_thread_kernels_at_the_edge_schedules(env, planar, d, per_sm):
    X, torch = env
    for kind, n, b0, b1 in EDGES:
        against_the_oracle(X, torch, planar, d, per_sm, X.noise_from_eta(0.2, 100.0), kind, n, b0, b1)


@pytest.mark.parametrize("planar,d,per_sm", FORMS)
def test_thread_kernels_chain_ids_and_scale(env, planar, d, per_sm):
    """Chain ids above 2^32 (the counter's high word), and energies at scale 4096."""
    X, torch = env
    against_the_oracle(X, torch, planar, d, per_sm, X.noise_from_eta(0.15, 10.0), 0, 20, 0.1, 8.0, shot0=(1 << 31) + 7)
    against_the_oracle(X, torch, planar, d, per_sm, X.noise_from_eta(0.25, 1000.0, 0, 4096), 0, 30, 0.02, 30.0)


@pytest.mark.parametrize("planar,d,per_sm,literal", [(p, d, n, False) for p, d, n in FORMS if d in (7, 9, 21, 31)]
                         + [(False, 7, 20, True), (False, 31, 2, True), (True, 9, 20, True), (True, 31, 2, True),
                            (True, 21, 20, False), (True, 9, 4, False)])
def test_checked_build_in_every_annealing_kernel(env, planar, d, per_sm, literal):
    """Equal results and no flag from the checked build; its check, made to fail,
    is recorded."""
    X, torch = env
    from paper_2509_17837_gb300._lib import XZZX_DEVERR_BOUNDS, XZZX_OK, Noise
    L = _checked_lib()
    noise = X.noise_from_eta(0.16, 100.0)
    code, shots, init = launch(X, torch, planar, d, per_sm, noise, 5, 0)
    form = dict(order=X.ORDER_RANDOM_SITE, emin=X.EMIN_PER_ATTEMPT) if literal else {}
    want = X.anneal(code, X.Schedule(noise, 9, 0.05, 20.0), 5, 0, init, want_final=True, **form)
    got = {k: torch.zeros_like(v) for k, v in want.items()}
    hc, hs, nz = ctypes.c_void_p(), ctypes.c_void_p(), Noise()
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    flags, count = ctypes.c_uint32(), ctypes.c_uint32()

    def ok(st):
        assert st == XZZX_OK, L.xzzx_last_error()

    def run():
        ok(L.xzzx_anneal_variant(hc, hs, 5, 0, shots, 1, int(literal), int(literal), p(init), p(got["best_E"]),
                                 p(got["best_cfg"]), p(got["final_E"]), p(got["final_cfg"]), stream))
        ok(L.xzzx_device_errors(hc, ctypes.byref(flags), ctypes.byref(count), 1, stream))

    try:
        ok(L.xzzx_make_code(d, int(planar), ctypes.byref(hc)))
        ok(L.xzzx_noise_from_eta(0.16, 100.0, 0, 1024, ctypes.byref(nz)))
        ok(L.xzzx_make_schedule(ctypes.byref(nz), 0, 9, 0.05, 20.0, ctypes.byref(hs)))
        run()
        assert (flags.value, count.value) == (0, 0)
        for k in want:
            assert torch.equal(got[k], want[k]), k
        ok(L.xzzx_debug_inject(hc, XZZX_DEVERR_BOUNDS, stream))
        run()
        assert flags.value == XZZX_DEVERR_BOUNDS and count.value > 0
    finally:
        L.xzzx_free_schedule(hs)
        L.xzzx_free_code(hc)
