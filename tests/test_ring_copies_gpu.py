"""Rings whose words fill a warp, and those that one holds 2 to 16 times over, at the
sizes where a word, the number of copies or the kernel changes; against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2506_03266_gb300 as qca  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qca.build()
    oracle.build()
    yield
    torch.cuda.synchronize()


@pytest.mark.parametrize("L", [64, 65, 95, 128, 129, 160, 255, 256, 257, 511, 512, 513, 1024, 1025])
@pytest.mark.parametrize("v,m_max", [(1, 255), (3, 255), (3, 1), (3, 20), (5, 7), (8, 255), (8, 3)])
def test_against_oracle(L, v, m_max):
    for p, p_move, shots in ((0.05, 0.0, 6), (0.4, 0.0, 4), (0.3, 0.1, 4)):
        N = oracle.sample_errors_1d(L, shots, p, seed=L + v)
        got = qca.decode_1d_batch(torch.from_numpy(N).cuda(), max_steps=120, v=v, m_max=m_max,
                                  p_move=p_move, rng_seed=L)
        C, s, f, m = [x.cpu().numpy() for x in got]
        for i in range(shots):
            Co, so, fo, mo = oracle.decode_shot_1d(N[i], v=v, m_max=m_max, max_steps=120,
                                                   move_thr=oracle.prob_threshold(p_move),
                                                   seed=L, shot=i)
            assert (s[i], f[i], m[i]) == (so, fo, mo), (p, p_move, i)
            np.testing.assert_array_equal(C[i], Co, err_msg=f"p={p} p_move={p_move} shot {i}")
