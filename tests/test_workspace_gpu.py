"""The device memory that the library keeps."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2506_03266_gb300 as qca  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qca.build()
    yield
    torch.cuda.synchronize()
    torch.cuda.empty_cache()


def test_large_lattices_with_little_memory():
    """160 shots of L = 1024 want 1.8 GB; with 0.7 GB left they are decoded in turns."""
    L, shots = 1024, 160
    N = qca.sample_errors(L, shots, 0.02, seed=3)
    want = [x.clone() for x in qca.decode_batch(N, max_steps=64)]
    out = tuple(torch.empty_like(x) for x in want)
    assert qca.lib().qca_free_workspace() == 0
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (700 << 20), dtype=torch.uint8,
                       device="cuda")
    try:
        for _ in range(2):
            for x in out:
                x.fill_(0xFF if x.dtype == torch.uint8 else -7)
            qca.decode_batch(N, max_steps=64, out=out)
            torch.cuda.synchronize()
    finally:
        del hold
        torch.cuda.empty_cache()
        assert qca.lib().qca_free_workspace() == 0
    for x, y in zip(out, want):
        assert torch.equal(x, y)
