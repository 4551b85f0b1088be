"""Shots that the history decoder leaves to the sweeps with message fields, in every
form of call that may leave some: their syndromes ask for more old ones than are
kept (L from 129 on).  The device code on the CPU says which shots are left, so that
the tests cannot pass without any; outputs equal the oracle's."""
import shutil

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")]

import history_emulation as emu  # noqa: E402
import oracle  # noqa: E402
import paper_2506_03266_gb300 as qca  # noqa: E402
from history_states import noise_of, open_noise_of, strip_and_far  # noqa: E402

STEPS = 130


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qca.build()
    oracle.build()
    yield
    torch.cuda.synchronize()


def states(L, n, make=noise_of):
    return np.stack([make(strip_and_far(L, np.random.default_rng(i), 6)) for i in range(n)])


def host(out):
    torch.cuda.synchronize()
    return [x.cpu().numpy() for x in out]


def same(got, ref, label=""):
    for x, y, name in zip(got, ref, ("correction", "steps", "flag")):
        np.testing.assert_array_equal(x, y, err_msg=f"{label} {name}")


# two-CTA clusters, the sweep for any size, and rows of whole 16-byte groups
@pytest.mark.parametrize("L", [131, 136, 192, 200, 256])
def test_noise(L):
    N = states(L, 3)
    thr = oracle.prob_threshold(0.001)
    for kw, ekw, okw in [({}, {}, {}), (dict(tie_order=1), dict(tie=1), dict(tie_order=1)),
                         (dict(p_move=0.001, rng_seed=4), dict(move_thr=thr, seed=4),
                          dict(move_thr=thr, seed=4))]:
        assert (emu.decode(N, max_steps=STEPS, **ekw)[1] == emu.PENDING).any()
        got = host(qca.decode_batch(torch.from_numpy(N).cuda(), max_steps=STEPS, **kw))
        same(got, oracle.decode_batch(N, max_steps=STEPS, **okw), f"L{L} {kw}")


def test_arrays_off_a_word_boundary():
    """Such arrays go to the sweep that reads bytes."""
    L, N = 136, states(136, 3)
    buf = torch.zeros(N.size + 8, dtype=torch.uint8, device="cuda")
    view = buf[1: 1 + N.size].view(N.shape)
    view.copy_(torch.from_numpy(N))
    assert (emu.decode(N, max_steps=STEPS, skew=1)[1] == emu.PENDING).any()
    same(host(qca.decode_batch(view, max_steps=STEPS)), oracle.decode_batch(N, max_steps=STEPS))


def test_left_shots_spread_over_a_large_batch():
    """Every seventh shot of a batch longer than a cluster's threads is left."""
    L, n = 136, 1200
    N = np.zeros((n, 2, L, L), np.uint8)
    S = states(L, 2)
    assert (emu.decode(S, max_steps=STEPS)[1] == emu.PENDING).all()
    ref = oracle.decode_batch(S, max_steps=STEPS)
    N[::7] = S[np.arange(len(N[::7])) % 2]
    C, s, f = host(qca.decode_batch(torch.from_numpy(N).cuda(), max_steps=STEPS))
    for i in range(n):
        if i % 7:
            assert s[i] == 0 and f[i] == 0 and not C[i].any()
        else:
            same((C[i], s[i], f[i]), [x[i // 7 % 2] for x in ref], f"shot {i}")


@pytest.mark.parametrize("L", [131, 160])
def test_open_lattice(L):
    N = states(L, 3, open_noise_of)
    assert (emu.decode(N, max_steps=STEPS, open=True)[1] == emu.PENDING).any()
    C, s, f = host(qca.decode_open_batch(torch.from_numpy(N).cuda(), max_steps=STEPS))
    for i in range(len(N)):
        same((C[i], s[i], f[i]), oracle.open_decode_shot(N[i], max_steps=STEPS), f"shot {i}")


@pytest.mark.parametrize("mode", ["mixed", "per_size"])
def test_packed_batch(mode):
    """Pairs of CTAs (200, 256), groups of one (136, 160) and odd sizes, among shots
    of sizes that are never left."""
    sizes = [24, 64, 131, 136, 160, 200, 256, 33]
    L = np.array([s for s in sizes for _ in range(2)], np.int32)
    plan = qca.UnevenPlan(L)
    plan.set_mode(mode)
    shots, refs, left = [], [], 0
    for i, l in enumerate(L):
        n = states(l, 2)[i % 2: i % 2 + 1] if l > 128 else oracle.sample_errors(int(l), 1, 0.05, seed=i)
        shots.append(n)
        refs.append(oracle.decode_batch(n, max_steps=STEPS))
        if l > 128:
            left += int(emu.decode(n, max_steps=STEPS)[1][0] == emu.PENDING)
    assert left == 10
    N = torch.zeros(plan.total_bytes, dtype=torch.uint8)
    for o, n in zip(plan.offsets, shots):
        N[o: o + n.size] = torch.from_numpy(n.reshape(-1))
    C, s, f = host(plan.decode(N.cuda(), max_steps=STEPS))
    for i, (o, n, ref) in enumerate(zip(plan.offsets, shots, refs)):
        same((C[o: o + n.size].reshape(n.shape[1:]), s[i], f[i]), [x[0] for x in ref],
             f"shot {i} L{L[i]}")
    plan.close()
