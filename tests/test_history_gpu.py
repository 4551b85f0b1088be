"""The decode from the syndrome history (v = 3, L from 8 up) against the sweeps
that keep message fields and the CPU oracle, at the sizes and states where it can
go wrong: bitmap rows with a few bits in their last word, unaligned blocks,
message caps that cut a slice, the anyon counts where its modes change, searches
that wrap the torus, shots that never move, and a shot that needs a syndrome it
no longer keeps.  Outputs are whole numbers and must be equal."""
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


def decode(N, path=None, **kw):
    L = N.shape[-1]
    if path is not None:
        qca.set_kernel_path(L, path)
    try:
        out = qca.decode_batch(N, **kw)
        torch.cuda.synchronize()
    finally:
        if path is not None:
            qca.set_kernel_path(L, -1)
    return [t.cpu().numpy() for t in out]


def same(a, b, label):
    for x, y, name in zip(a, b, ("correction", "steps", "flag")):
        np.testing.assert_array_equal(x, y, err_msg=f"{label} {name}")


@pytest.mark.parametrize("L", [8, 9, 15, 16, 17, 31, 32, 33, 35, 48, 63, 64, 65, 66, 97, 127, 128,
                               129, 130, 161, 192, 225, 255, 256, 257, 288, 385])
def test_sizes_against_literal_sweep(L):
    shots = max(4, min(400, 200000 // L ** 2))
    for p, kw in [(0.02, {}), (0.07, {}), (0.07, dict(tie_order=1)),
                  (0.06, dict(balance_rule=1, rng_seed=3)),
                  (0.05, dict(p_move=0.1, tie_order=1, rng_seed=4))]:
        N = qca.sample_errors(L, shots, p, seed=L)
        same(decode(N, max_steps=150, **kw), decode(N, path=0, max_steps=150, **kw),
             f"L{L} p{p} {kw}")


@pytest.mark.parametrize("m_max", [1, 2, 3, 4, 6, 40, 254])
def test_message_caps(m_max):
    for L in (8, 24, 33, 70):
        for tie in (0, 1):
            N = qca.sample_errors(L, 200, 0.09, seed=m_max)
            kw = dict(max_steps=200, m_max=m_max, tie_order=tie)
            same(decode(N, **kw), decode(N, path=0, **kw), f"L{L} m{m_max} tie{tie}")


@pytest.mark.parametrize("L", [24, 64, 192, 256])
def test_heavy_noise_fills_the_lists(L):
    N = qca.sample_errors(L, 16, 0.5, seed=L)
    same(decode(N, max_steps=120), decode(N, path=0, max_steps=120), f"L{L}")


def test_stationary_belt_of_many_anyons():
    """Shot 2878 of this draw ends in 22 anyons that never move: budget, flag 2."""
    N = qca.sample_errors(16, 1, 0.05, seed=0, shot0=2878)
    for budget in (90, 91, 500, 4096):
        got = decode(N, max_steps=budget)
        same(got, oracle.decode_batch(N.cpu().numpy(), max_steps=budget), f"budget {budget}")
        assert got[2][0] == 2


def dense_and_sparse(L):
    """Anyon indicator: a stationary lattice of balanced anyons (every second
    site of every second row of a quarter) and two anyons as far from it and from
    each other as the torus allows, which therefore need old syndromes that are
    too large for the archive's lists and too many for its bitmaps."""
    s = np.zeros((L, L), np.uint8)
    s[:, : L // 4][::2, ::2] = 1
    s[1, 5 * L // 8] = s[1 + L // 2, 5 * L // 8] = 1
    return s


@pytest.mark.parametrize("L", [128, 192, 256])
def test_syndromes_that_outgrow_the_archive(L):
    s = np.stack([dense_and_sparse(L), np.zeros((L, L), np.uint8)])
    t = torch.from_numpy(s).cuda()
    got = [x.cpu().numpy() for x in qca.decode_syndrome_batch(t, max_steps=130)]
    qca.set_kernel_path(L, 0)
    try:
        ref = [x.cpu().numpy() for x in qca.decode_syndrome_batch(t, max_steps=130)]
    finally:
        qca.set_kernel_path(L, -1)
    for x, y in zip(got, ref):
        np.testing.assert_array_equal(x, y)


def test_unaligned_blocks():
    for L in (24, 49, 64):
        n = 2 * L * L
        buf = torch.zeros(8 * n + 64, dtype=torch.uint8, device="cuda")
        N = qca.sample_errors(L, 8, 0.06, seed=5)
        ref = decode(N, path=0, max_steps=200)
        for off in (1, 2, 3, 5, 8):
            view = buf[off: off + 8 * n].view(8, 2, L, L)
            view.copy_(N)
            out = torch.zeros(8 * n + 64, dtype=torch.uint8, device="cuda")
            C = out[off: off + 8 * n].view(8, 2, L, L)
            steps = torch.zeros(8, dtype=torch.int32, device="cuda")
            flag = torch.zeros(8, dtype=torch.uint8, device="cuda")
            qca.decode_batch(view, max_steps=200, out=(C, steps, flag))
            torch.cuda.synchronize()
            same([x.cpu().numpy() for x in (C, steps, flag)], ref, f"L{L} off {off}")
            assert int(out[:off].sum()) == 0 and int(out[off + 8 * n:].sum()) == 0


@pytest.mark.parametrize("L", [63, 64, 65, 95, 96, 127, 1024, 1025, 4096, 4099, 16384])
def test_ring_history_against_oracle(L):
    shots = 40 if L < 2000 else 4
    for p, v, m_max, p_move in [(0.3, 3, 255, 0.1), (0.2, 3, 255, 0.0), (0.2, 2, 9, 0.0),
                                (0.25, 8, 255, 0.05), (0.2, 1, 255, 0.0)]:
        N = oracle.sample_errors_1d(L, shots, p, seed=L)
        got = qca.decode_1d_batch(torch.from_numpy(N).cuda(), max_steps=60, v=v, m_max=m_max,
                                  p_move=p_move, rng_seed=3)
        C, s, f, m = [x.cpu().numpy() for x in got]
        thr = oracle.prob_threshold(p_move) if p_move else 0
        for i in range(shots):
            Co, so, fo, mo = oracle.decode_shot_1d(N[i], v=v, m_max=m_max, max_steps=60,
                                                   move_thr=thr, seed=3, shot=i)
            assert (s[i], f[i], m[i]) == (so, fo, mo), (L, p, v, m_max, p_move, i)
            np.testing.assert_array_equal(C[i], Co)


@pytest.mark.parametrize("L", [8, 9, 16, 31, 33, 64, 65, 96, 130, 200, 256])
def test_open_history_against_oracle(L):
    """Tile and word edges of the open lattice, and caps that cut a slice."""
    shots = 24 if L <= 64 else 3
    for p, m_max in [(0.03, 255), (0.08, 255), (0.08, 2), (0.08, 7)]:
        N = oracle.sample_errors(L, shots, p, seed=L)
        got = qca.decode_open_batch(torch.from_numpy(N).cuda(), max_steps=80, m_max=m_max)
        C, s, f = [x.cpu().numpy() for x in got]
        for i in range(shots if L <= 64 else 1):
            Co, so, fo = oracle.open_decode_shot(N[i], m_max=m_max, max_steps=80)
            assert (s[i], f[i]) == (so, fo), (L, p, m_max, i)
            np.testing.assert_array_equal(C[i], Co)


def test_mixed_sizes_with_odd_ones_and_both_cta_shapes():
    rng = np.random.default_rng(3)
    Ls = rng.choice(np.array([9, 15, 24, 33, 48, 64, 65, 81, 96, 128, 130, 192, 255, 256, 257, 7, 10,
                              11, 12, 13, 14, 18, 19, 20, 21, 22, 23, 25], dtype=np.int32), 300)
    plan = qca.UnevenPlan(Ls)
    N = plan.sample(np.full(len(Ls), oracle.prob_threshold(0.05), dtype=np.uint64), seed=2)
    C, s, f = plan.decode(N, max_steps=200)
    torch.cuda.synchronize()
    for i in rng.permutation(len(Ls))[:120]:
        L = int(Ls[i])
        n = N[plan.offsets[i]: plan.offsets[i] + 2 * L * L].view(1, 2, L, L).contiguous()
        ref = decode(n, path=0, max_steps=200)
        c = C[plan.offsets[i]: plan.offsets[i] + 2 * L * L].view(2, L, L).cpu().numpy()
        assert (int(s[i]), int(f[i])) == (ref[1][0], ref[2][0]), (i, L)
        np.testing.assert_array_equal(c, ref[0][0])
    plan.close()
