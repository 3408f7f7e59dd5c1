"""Greedy references at the sizes where the kernel changes its way: colours just
under and over the room of the candidate lists and the widths of their sorts, and
launches that give a restart two warps, one warp, or share a CTA among many."""
import numpy as np
import pytest

import oracle as O
from inputs import random_syndromes
from layout import syn_bits_to_words, words_to_labels

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    import paper_2509_17837_gb300 as X
    return X, torch


def room(faces):
    """Vertices per colour that the lists hold (0: every colour is scanned)."""
    n = (faces * 35 // 64 + 31) // 32 * 32
    return 0 if faces > 800 else min(max(n, 64), 256)


# (layout, d, vertices per colour aimed at): a sort width or the room, a little under and over
CASES = [(0, 9, 32), (0, 17, 64), (0, 21, 64), (0, 19, 128), (0, 23, 128), (0, 25, 192), (0, 31, 256),
         (1, 7, 32), (1, 11, 64), (1, 13, 96), (1, 15, 128), (1, 21, 256), (1, 27, 256), (1, 29, 200)]


@pytest.mark.parametrize("layout,d,aim", CASES)
@pytest.mark.parametrize("equal_weights", [True, False])
def test_lists_and_scan_equal_the_oracle(env, layout, d, aim, equal_weights):
    X, torch = env
    code = X.Code(d, layout)
    faces = code.n_stab // 2
    assert room(faces) in (0, 64, 96, 128, 160, 192, 224, 256)
    cid = O.planar(d) if layout else d
    noise = X.make_noise(0.05, 0.05, 0.05) if equal_weights else X.make_noise(0.03, 0.05, 0.09)
    pxyz = (noise.px, noise.py, noise.pz)
    bits = np.concatenate([random_syndromes(code.n_stab, 1, min(1.0, f * aim / faces), seed=d + k)
                           for k, f in enumerate((0.93, 1.0, 1.07))])
    syn = torch.from_numpy(syn_bits_to_words(bits).view(np.int32)).cuda()
    restarts = 2
    for randomised in (0, 1):
        init, cbits = X.greedy_init(code, noise, 9, 3, syn, restarts, randomised=randomised)
        init, cbits = init.cpu().numpy(), cbits.cpu().numpy()
        for s in range(len(bits)):
            for i in range(restarts):
                ref, _ = O.greedy(cid, pxyz, noise.scale, 9, 3 + s, i, randomised, bits[s])
                assert np.array_equal(words_to_labels(init[s, i], code.n_qubits), ref), (s, i, randomised)
                assert cbits[s, i] == O.class_bits(cid, ref)
    assert code.device_errors() == (0, 0)


@pytest.mark.parametrize("layout,d,restarts,shots", [(0, 3, 8, 600), (0, 11, 100, 700), (0, 19, 37, 200), (0, 31, 256, 20),
                                                     (1, 5, 100, 500), (1, 13, 50, 100), (1, 21, 37, 100), (1, 31, 33, 12)])
@pytest.mark.parametrize("mode", [0, 1, 2])
def test_cuts_of_a_launch_agree(env, layout, d, restarts, shots, mode):
    """Many shots at once (restarts sharing CTAs) equal the same shots a few at a
    time (one warp per restart) and one at a time (two)."""
    X, torch = env
    code, noise = X.Code(d, layout), X.noise_from_eta(0.14, 5.0)
    _, syn = X.sample_errors(code, noise, 4, 11, shots)
    init, cbits = X.greedy_init(code, noise, 4, 11, syn, restarts, randomised=mode)
    for first, n in ((0, 1), (shots - 1, 1), (shots // 2, 6)):
        a, c = X.greedy_init(code, noise, 4, 11 + first, syn[first:first + n].contiguous(), restarts, randomised=mode)
        assert torch.equal(a, init[first:first + n]) and torch.equal(c, cbits[first:first + n])
    assert code.device_errors() == (0, 0)
