"""Anyon sets that ask the history decoder for old syndromes, and noise with a
given anyon set."""
import numpy as np


def patch_and_far(L, rng, far):
    """Anyon indicator: a patch of balanced anyons that stays dense for many steps,
    and a few anyons so far from it that they need old syndromes."""
    s = np.zeros((L, L), np.uint8)
    w, h = int(rng.integers(L // 6, L // 2)), int(rng.integers(L // 2, L + 1))
    s[:h, :w][::2, ::2] = 1
    for _ in range(far):
        s[int(rng.integers(L)), int(rng.integers(w + 10, L))] ^= 1
    if s.sum() % 2:
        s[0, L - 3] ^= 1
    return s


def strip_and_far(L, rng, far):
    """Anyon indicator: a strip of balanced anyons along the lattice that never thins
    out, and anyons half the torus from it, which ask for more old syndromes than the
    decoder keeps (from L = 129 on)."""
    s = np.zeros((L, L), np.uint8)
    s[:, : L // 4][::2, ::2] = 1
    for _ in range(far):
        s[int(rng.integers(L)), int(rng.integers(L // 2, 3 * L // 4))] ^= 1
    if s.sum() % 2:
        s[0, 5 * L // 8] ^= 1
    return s


def noise_of(s):
    """Links uint8 [2][L][L] of the torus whose anyons are s (an even number)."""
    L = s.shape[0]
    N = np.zeros((2, L, L), np.uint8)
    along = np.bitwise_xor.accumulate(s, axis=1)
    N[0, :, : L - 1] = along[:, : L - 1]
    N[1, :, L - 1] = np.bitwise_xor.accumulate(along[:, L - 1])
    assert not N[1, L - 1, L - 1]
    return N


def open_noise_of(s):
    """The same on the open lattice, whose columns 0 and L - 1 hold no anyons."""
    L = s.shape[0]
    N = np.zeros((2, L, L), np.uint8)
    N[0, :, 1: L - 1] = np.bitwise_xor.accumulate(s[:, 1: L - 1], axis=1)
    return N
