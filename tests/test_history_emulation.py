"""The history decoder's device code run on the CPU, lane by lane in a drawn
order, against the oracle: whole outputs, and no lane of a warp or block left
behind at a collective.  A shot it leaves pending is not compared."""
import shutil

import numpy as np
import pytest

import history_emulation as emu
import oracle
from history_states import open_noise_of, patch_and_far, strip_and_far

pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")


@pytest.fixture(scope="module", autouse=True)
def built():
    oracle.build()


def compare_noise(N, **kw):
    """Decodes noise; every shot that is not pending equals the oracle's.  Returns
    the number of pending shots."""
    okw = dict(max_steps=kw.get("max_steps", 400), m_max=kw.get("m_max", 255),
               move_thr=kw.get("move_thr", 0), seed=kw.get("seed", 0), tie_order=kw.get("tie", 0),
               balance_rule=kw.get("bal", 0))
    C, s, f = emu.decode(N, **kw)
    Co, so, fo = oracle.decode_batch(N, **okw)
    done = s != emu.PENDING
    np.testing.assert_array_equal(s[done], so[done])
    np.testing.assert_array_equal(f[done], fo[done])
    np.testing.assert_array_equal(C[done], Co[done])
    return int((~done).sum())


def compare_sigma(s, **kw):
    C, st, ex = emu.decode(s[None], sigma=True, **kw)
    if st[0] == emu.PENDING:
        return 1
    Co, so, fo = oracle.decode_syndrome_shot(s, max_steps=kw.get("max_steps", 400),
                                             m_max=kw.get("m_max", 255),
                                             tie_order=kw.get("tie", 0))[:3]
    assert (int(st[0]), bool(ex[0])) == (so, fo == 2)
    np.testing.assert_array_equal(C[0], Co)
    return 0


@pytest.mark.parametrize("L,p,shots", [(8, .15, 20), (16, .08, 20), (33, .08, 5), (64, .07, 4),
                                       (65, .07, 2), (128, .05, 1), (200, .04, 1)])
def test_noise_against_oracle(L, p, shots):
    N = oracle.sample_errors(L, shots, p, seed=L)
    thr = oracle.prob_threshold(0.1)
    for kw in (dict(), dict(tie=1), dict(bal=1, seed=4), dict(move_thr=thr, tie=1, seed=5)):
        compare_noise(N, max_steps=150, skew=L % 3, order=L, **kw)
    if L <= 32:
        compare_noise(N, max_steps=150, all_slots=True)


@pytest.mark.parametrize("L", [8, 17, 33, 64, 100, 161])
def test_random_moves_of_dense_steps(L):
    """Draws that replace a decided move, a balanced axis and no move."""
    N = oracle.sample_errors(L, 3 if L < 100 else 1, 0.1, seed=L)
    for p in (0.02, 0.5, 1.0):
        for kw in (dict(), dict(bal=1), dict(tie=1), dict(tie=1, bal=1)):
            compare_noise(N, max_steps=20, move_thr=oracle.prob_threshold(p), seed=9, order=L, **kw)


@pytest.mark.parametrize("L", [64, 96, 128])
@pytest.mark.parametrize("m_max", [15, 16, 18, 19, 21, 22])
def test_caps_around_the_slots(L, m_max):
    """Caps whose oldest slice is about the oldest syndrome that dense and listed
    steps keep in slots; the correction holds 0xFF before."""
    rng = np.random.default_rng(100 * L + m_max)
    for i in range(6):
        s = patch_and_far(L, rng, 1 + i % 5)
        compare_sigma(s, max_steps=70, m_max=m_max, tie=i & 1, order=i)
    N = open_noise_of(patch_and_far(L, rng, 4))
    C, st, f = emu.decode(N[None], max_steps=40, m_max=m_max, open=True)
    Co, so, fo = oracle.open_decode_shot(N, max_steps=40, m_max=m_max)
    assert (st[0], f[0]) == (so, fo)
    np.testing.assert_array_equal(C[0], Co)


@pytest.mark.parametrize("L,far,tie,seed", [(129, 80, 0, 3), (129, 80, 1, 1), (229, 80, 0, 2),
                                            (229, 80, 1, 3)])
def test_warps_stay_together_when_a_shot_is_left(L, far, tie, seed):
    """One warp finds that a syndrome is no longer kept while others search."""
    s = strip_and_far(L, np.random.default_rng(seed), far)
    for order in range(10):
        assert compare_sigma(s, max_steps=130, tie=tie, order=1000 + 17 * order) == 1


@pytest.mark.parametrize("L", [129, 136, 144, 152, 160, 176, 177, 208])
def test_no_shot_of_random_noise_is_left(L):
    for p in (0.08, 0.12):
        assert compare_noise(oracle.sample_errors(L, 2, p, seed=L), max_steps=100) == 0


@pytest.mark.parametrize("L", [9, 23, 33, 50, 80, 97, 128, 129, 170, 192, 256])
def test_archive_against_oracle(L):
    """Sets that stay large while a few anyons ask for old ones: entries of all sizes,
    the ring's end, and entries that others have covered."""
    rng = np.random.default_rng(L)
    for i in range(6):
        make = strip_and_far if i & 1 or L < 24 else patch_and_far
        s = make(L, rng, 1 + 3 * i)
        compare_sigma(s, max_steps=100, tie=i % 3 == 2, skew=i, order=i, m_max=255 - 60 * (i % 3))


@pytest.mark.parametrize("L,threads", [(8, 128), (17, 128), (32, 128), (33, 128), (64, 128),
                                       (65, 256), (100, 256), (128, 256), (129, 512), (144, 256),
                                       (177, 512), (224, 256), (256, 512)])
def test_threads_of_small_batches(L, threads):
    N = oracle.sample_errors(L, 2 if L < 130 else 1, 0.1, seed=L)
    for kw in (dict(), dict(tie=1), dict(bal=1, seed=4),
               dict(move_thr=oracle.prob_threshold(0.1), tie=1, seed=5)):
        compare_noise(N, max_steps=40, threads=threads, skew=L % 3, order=L, **kw)
    if L <= 32:
        compare_noise(N, max_steps=100, threads=threads, all_slots=True)
    if L >= 24:
        rng = np.random.default_rng(L)
        for i, make in enumerate((patch_and_far, strip_and_far)):
            compare_sigma(make(L, rng, 5), max_steps=60, threads=threads, order=i, tie=i)
