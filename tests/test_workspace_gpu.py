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


def test_training_buffers_are_released():
    """512 tori of 64 x 64 are 2^21 sites, the most whose buffers a net keeps: 3 bytes,
    seven times 32 bf16 channels and four floats a site, and some more.  The library
    gives them back on request, and the next call returns the same gradients (the loss
    is a sum in no fixed order)."""
    net = qca.Net(seed=1)
    N = qca.sample_errors(64, 512, 0.05, seed=2)
    _, want = net.gradients(N)
    torch.cuda.synchronize()
    held = torch.cuda.mem_get_info()[0]
    assert qca.lib().qca_free_workspace() == 0
    assert torch.cuda.mem_get_info()[0] - held >= (3 + 7 * 32 * 2 + 4 * 4) << 21
    _, again = net.gradients(N)
    assert (again == want).all()
    net.close()
