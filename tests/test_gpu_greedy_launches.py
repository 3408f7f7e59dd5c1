"""Greedy references in the launches that take a way of their own: boundary
references of large codes in narrow CTAs without lists, launches that scan every
colour, and small codes in CTAs of four warps.  Each equals the same
shots a few at a time, and the oracle on a sample."""
import numpy as np
import pytest

import oracle as O
from layout import syn_words_to_bits, words_to_labels

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    import paper_2509_17837_gb300 as X
    return X, torch


def check(env, layout, d, restarts, shots, mode, p, eta):
    X, torch = env
    code, noise = X.Code(d, layout), X.noise_from_eta(p, eta)
    _, syn = X.sample_errors(code, noise, 4, 11, shots)
    init, cbits = X.greedy_init(code, noise, 4, 11, syn, restarts, randomised=mode)
    for first, n in ((0, 1), (shots - 1, 1), (shots // 2, 6)):
        # more restarts than needed: another cut of the same references
        a, c = X.greedy_init(code, noise, 4, 11 + first, syn[first:first + n].contiguous(), restarts + 7, randomised=mode)
        assert torch.equal(a[:, :restarts], init[first:first + n]) and torch.equal(c[:, :restarts], cbits[first:first + n])
    cid = O.planar(d) if layout else d
    bits = syn_words_to_bits(syn.cpu().numpy(), code.n_stab)
    for s in (0, shots - 1):
        ref, _ = O.greedy(cid, (noise.px, noise.py, noise.pz), noise.scale, 4, 11 + s, restarts - 1, mode, bits[s])
        assert np.array_equal(words_to_labels(init[s, restarts - 1].cpu().numpy(), code.n_qubits), ref)
        assert int(cbits[s, restarts - 1]) == O.class_bits(cid, ref)
    assert code.device_errors() == (0, 0)


@pytest.mark.parametrize("layout,d,restarts,shots", [(0, 19, 1, 305), (0, 31, 1, 700), (0, 25, 40, 110), (1, 13, 3, 500),
                                                     (1, 27, 64, 100), (1, 31, 1, 400)])
def test_boundary_references_of_large_codes(env, layout, d, restarts, shots):
    check(env, layout, d, restarts, shots, 2, 0.14, 5.0)


@pytest.mark.parametrize("layout,d,restarts,shots,p", [(1, 27, 1, 300, 0.17), (1, 27, 4, 60, 0.17), (1, 25, 2, 160, 0.25),
                                                       (1, 27, 4, 60, 0.06), (1, 29, 1, 300, 0.12), (1, 31, 9, 40, 0.12),
                                                       (1, 31, 64, 20, 0.04)])
@pytest.mark.parametrize("mode", [0, 1])
def test_scans(env, layout, d, restarts, shots, p, mode):
    """Planar d >= 29, and d = 25, 27 with few restarts where the noise fills the
    colours (p = 0.06: lists)."""
    check(env, layout, d, restarts, shots, mode, p, 5.0)


@pytest.mark.parametrize("layout,d,restarts,shots", [(0, 3, 8, 700), (0, 3, 3, 609), (0, 5, 3, 800), (0, 9, 1, 700),
                                                     (0, 17, 2, 650), (1, 3, 20, 400), (1, 11, 1, 700)])
@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("p", [0.02, 0.15])
def test_narrow_launches_of_small_codes(env, layout, d, restarts, shots, mode, p):
    """Four-warp CTAs; at the low rate most colours have no more than two vertices."""
    check(env, layout, d, restarts, shots, mode, p, 5.0)
