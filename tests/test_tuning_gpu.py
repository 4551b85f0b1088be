"""The tuner times the sweep whose settings it chooses."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2506_03266_gb300 as qca  # noqa: E402


def test_autotune_times_the_on_chip_sweep():
    """At L = 256, p = 0.05 the sweep with message fields takes about ten times as long
    as the history decoder that a default call runs; a third of that tells them apart."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qca.build()
    L, shots, steps = 256, 2000, 512
    N = qca.sample_errors(L, shots, 0.05, seed=1)
    times = []
    for _ in range(4):
        t = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        t[0].record()
        qca.decode_batch(N, max_steps=steps)
        t[1].record()
        t[1].synchronize()
        times.append(t[0].elapsed_time(t[1]))
    try:
        H, div, ms = qca.autotune(L, shots, 0.05, seed=1, max_steps=steps)
        assert qca.get_tuning(L)[:2] == (H, div)
    finally:
        qca.set_tuning(L, 0, 0)
    assert ms > 3 * min(times)
