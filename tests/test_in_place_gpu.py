"""Decodes whose correction takes the place of the noise: every output equals the
oracle's, also where the history decoder could leave a shot to a second decode."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

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


def noise(L, make=noise_of):
    """Two syndromes that outgrow the archive (L from 129 on), two of random noise, and
    two without anyons: a cycle around the torus, and the empty one."""
    N = np.zeros((6, 2, L, L), np.uint8)
    for i in range(2):
        N[i] = make(strip_and_far(L, np.random.default_rng(i), 6))
    N[2:4] = oracle.sample_errors(L, 2, 0.06, seed=L)
    N[4, 0, 0] = 1
    return N


def outputs(C, shots):
    return (C, torch.empty(shots, dtype=torch.int32, device="cuda"),
            torch.empty(shots, dtype=torch.uint8, device="cuda"))


def same(got, ref, label=""):
    for x, y, name in zip(got, ref, ("correction", "steps", "flag")):
        np.testing.assert_array_equal(x, y, err_msg=f"{label} {name}")


@pytest.mark.parametrize("L", [24, 40, 65, 128, 131, 136, 192, 256, 300])
@pytest.mark.parametrize("shift", [0, 1])
def test_torus(L, shift):
    N = noise(L)
    buf = torch.zeros(N.size + 4, dtype=torch.uint8, device="cuda")
    x = buf[shift: shift + N.size].view(N.shape)
    x.copy_(torch.from_numpy(N))
    got = qca.decode_batch(x, max_steps=STEPS, out=outputs(x, len(N)))
    same([g.cpu().numpy() for g in got], oracle.decode_batch(N, max_steps=STEPS))


@pytest.mark.parametrize("L", [24, 131])
def test_open(L):
    N = noise(L, open_noise_of)
    x = torch.from_numpy(N).cuda()
    got = [g.cpu().numpy() for g in
           qca.decode_open_batch(x, max_steps=STEPS, out=outputs(x, len(N)))]
    for i in range(len(N)):
        same([g[i] for g in got], oracle.open_decode_shot(N[i], max_steps=STEPS), f"shot {i}")


@pytest.mark.parametrize("mode", ["mixed", "per_size"])
def test_packed(mode):
    L = np.array([24, 136, 256, 33, 131, 24], np.int32)
    shots = [noise(int(l))[i % 3: i % 3 + 1] for i, l in enumerate(L)]
    plan = qca.UnevenPlan(L)
    plan.set_mode(mode)
    x = torch.from_numpy(np.concatenate([n.reshape(-1) for n in shots])).cuda()
    got = plan.decode(x, max_steps=STEPS, out=outputs(x, len(L)))
    C, s, f = [g.cpu().numpy() for g in got]
    for i, (o, n) in enumerate(zip(plan.offsets, shots)):
        same((C[o: o + n.size].reshape(n.shape), s[i: i + 1], f[i: i + 1]),
             oracle.decode_batch(n, max_steps=STEPS), f"shot {i} L{L[i]}")
    plan.close()


@pytest.mark.parametrize("L", [64, 131, 192])
def test_syndrome(L):
    """One shot whose anyons lie in the first half of the correction array."""
    s = strip_and_far(L, np.random.default_rng(0), 6)
    x = torch.zeros(2 * L * L, dtype=torch.uint8, device="cuda")
    x[: L * L] = torch.from_numpy(s.reshape(-1))
    steps = torch.zeros(1, dtype=torch.int32, device="cuda")
    cut, exhausted = (torch.zeros(2, dtype=torch.uint8, device="cuda") for _ in range(2))
    rc = qca.lib().qca_decode_syndrome_batch_async(
        ctypes.c_void_p(x.data_ptr()), L, 1, STEPS, 0,
        *(ctypes.c_void_p(t.data_ptr()) for t in (x, steps, cut, exhausted)), None, None)
    assert rc == 0
    torch.cuda.synchronize()
    ref = qca.decode_syndrome_batch(torch.from_numpy(s[None]).cuda(), max_steps=STEPS)
    Co, so, _ = oracle.decode_batch(noise_of(s)[None], max_steps=STEPS)
    np.testing.assert_array_equal(x.cpu().numpy(), Co.reshape(-1))
    assert int(steps) == int(so[0]) == int(ref[1])
    assert cut.tolist() == ref[2][0].tolist() and int(exhausted[0]) == int(ref[3])
