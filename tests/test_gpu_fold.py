"""Folding a band's sums over the lanes: totals past FP32's range and near its
lower end, where the long bands' fold (beyond FP64) has to hold what FP64 held.

Constant rows make every product the same power of two, so lane sums, totals
and y are exact: y must equal the FP64 product exactly (lift: 2G mixing and the
scaling are exact too)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need CUDA")
    import paper_1902_08018_gb300 as W

    W.library()
    return W, torch


@pytest.mark.parametrize("fmt,rate", [(1, 16), (5, 8), (5, 16), (6, 16), (8, 0)])
@pytest.mark.parametrize("exp", [112, 0, -80])
@pytest.mark.parametrize("R", [1, 8])
def test_totals_beyond_fp32(env, orc, fmt, rate, exp, R):
    W, torch = env
    M, N = 9, 1 << 16  # 16384 blocks per band: the FP64 default; totals of 2^(16 + exp) times 1 or 2
    A = np.full((M, N), 2.0**exp)
    A[4] = -A[4]
    blob = W.whff_compress_accuracy(A, 0.0) if fmt == 8 else W.whff_compress(A, fmt, rate)
    Ahat = orc.wz3_decode(blob.tobytes())[0] if fmt == 8 else orc.decode(blob.tobytes())
    assert (Ahat == A).all()
    X = np.full((R, N), 1.0, dtype=np.float32) * np.array([2.0**(r % 2) for r in range(R)], dtype=np.float32)[:, None]
    with W.whff_create(blob, max_rhs=R) as h:
        if R > 1 and fmt in (5, 6):
            h.crossover = 33  # CUDA cores
        y = torch.zeros((R, M), dtype=torch.float64, device="cuda")
        h.step(torch.from_numpy(X).cuda(), y)
        torch.cuda.synchronize()
        got = y.cpu().numpy()
    assert (got == X.astype(np.float64) @ A.T).all()


@pytest.mark.parametrize("fmt,rate", [(5, 8), (5, 16), (6, 24), (2, 0), (4, 0), (7, 0), (8, 0)])
@pytest.mark.parametrize("M,N", [(30, 40000), (700, 3001), (5000, 378)])
def test_shared_bands_pass_after_pass(env, fmt, rate, M, N):
    """A band's last segment adds them all up and leaves its counter at zero: whole
    steps, row views and other column counts on one handle repeat bit for bit."""
    W, torch = env
    A = np.random.default_rng(M + fmt).standard_normal((M, N))
    blob = W.whff_compress_accuracy(A, 1e-4) if fmt == 8 else W.whff_compress(A, fmt, rate or 16)
    x = torch.from_numpy(np.random.default_rng(N).standard_normal((8, N)).astype(np.float32)).cuda()
    with W.whff_create(blob, max_rhs=8) as h:
        if fmt in (2, 4, 5, 6):
            h.crossover = 33  # CUDA cores
        rows = min(M, 256)
        first = None
        for _ in range(3):
            out = []
            for R in (1, 8, 2):
                y = torch.zeros((R, M), dtype=torch.float64, device="cuda")
                h.step(x[:R], y)
                v = torch.zeros((R, rows), dtype=torch.float64, device="cuda")
                h.step_rows(0, rows, x[:R], v)
                out += [y, v]
            torch.cuda.synchronize()
            if first is None:
                first = out
                for y, v in zip(out[::2], out[1::2]):  # two partitions of the same sums
                    assert (y[:, :rows] - v).norm() <= 1e-6 * v.norm()
            assert all(torch.equal(a, b) for a, b in zip(first, out))


@pytest.mark.parametrize("M,N", [(257, 516), (1000, 1027)])
@pytest.mark.parametrize("rate", [8, 16])
def test_x_of_any_alignment(env, M, N, rate):
    """The one-column kernel that transforms x itself: x at an odd address, same bits."""
    W, torch = env
    A = np.random.default_rng(rate + N).standard_normal((M, N))
    buf = torch.from_numpy(np.random.default_rng(N).standard_normal(N + 1).astype(np.float32)).cuda()
    with W.whff_create(W.whff_compress(A, 5, rate), max_rhs=1) as h:
        y = torch.zeros((2, M), dtype=torch.float64, device="cuda")
        h.step(buf[1:], y[0])
        h.step(buf[1:].clone(), y[1])
        torch.cuda.synchronize()
    assert torch.equal(y[0], y[1])
