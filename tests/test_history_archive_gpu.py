"""Shots that ask the history decoder for syndromes which have left shared memory:
caps at the edge of what it keeps there."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2506_03266_gb300 as qca  # noqa: E402
from history_states import noise_of, patch_and_far  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qca.build()
    oracle.build()
    yield
    torch.cuda.synchronize()


def decode_filled(N, **kw):
    """decode_batch into arrays that hold 0xFF (steps: -1) before."""
    t = torch.from_numpy(N).cuda()
    C = torch.full_like(t, 0xFF)
    s = torch.full((len(N),), -1, dtype=torch.int32, device="cuda")
    f = torch.full((len(N),), 0xFF, dtype=torch.uint8, device="cuda")
    qca.decode_batch(t, out=(C, s, f), **kw)
    torch.cuda.synchronize()
    return [x.cpu().numpy() for x in (C, s, f)]


def same(got, ref, label):
    for x, y, name in zip(got, ref, ("correction", "steps", "flag")):
        np.testing.assert_array_equal(x, y, err_msg=f"{label} {name}")


@pytest.mark.parametrize("L", [40, 64, 96, 128])
@pytest.mark.parametrize("m_max", range(15, 23))
def test_caps_around_the_slots(L, m_max):
    rng = np.random.default_rng(100 * L + m_max)
    N = np.stack([noise_of(patch_and_far(L, rng, 1 + i % 5)) for i in range(6)])
    for tie in (0, 1):
        got = decode_filled(N, max_steps=70, m_max=m_max, tie_order=tie)
        same(got, oracle.decode_batch(N, max_steps=70, m_max=m_max, tie_order=tie),
             f"L{L} m{m_max} tie{tie}")
