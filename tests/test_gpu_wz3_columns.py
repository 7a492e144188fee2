"""Fixed accuracy with eight right-hand sides: the pass that shares x between the
bands of a CTA, at the edges of its groups of 8 bands and runs of 32 blocks.

Every column has the products of the one-column pass, each rounded the same way,
and both sum them without rounding error above 2^-46 of the terms' magnitude
(TwoSum, pairs folded over the lanes), so the two agree to 1e-12 of
sum_j |a_ij x_j| entry by entry."""
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


# (M, N): one band; 8 and 9 bands, ragged; one block; runs of 31, 32, 33 blocks; groups cut by many CTAs
SHAPES = [(1, 3), (4, 128), (29, 124), (32, 128), (33, 132), (35, 257), (16, 20000), (70, 9001), (3001, 40),
          (515, 1030)]


@pytest.mark.parametrize("M,N", SHAPES)
@pytest.mark.parametrize("tol", [1e-2, 1e-7, 0.0])
def test_eight_columns_match_single_ones(env, orc, M, N, tol):
    W, torch = env
    rng = np.random.default_rng(1000 * M + N)
    A = rng.standard_normal((M, N)) * np.exp(rng.uniform(-4, 4, size=(M, 1)))
    if M >= 8:
        A[4:8, : N // 2] = 0.0  # a band of zero blocks
    blob = W.whff_compress_accuracy(A, tol)
    Ahat = orc.wz3_decode(blob.tobytes())[0]
    X = rng.standard_normal((8, N)).astype(np.float32)
    S0 = rng.standard_normal(M)
    with W.whff_create(blob, max_rhs=8) as h:
        x = torch.from_numpy(X).cuda()
        y8 = torch.zeros((8, M), dtype=torch.float64, device="cuda")
        s8 = torch.from_numpy(S0.copy()).cuda()
        h.step(x, y8, s8, 0.9)
        y1 = torch.zeros((8, M), dtype=torch.float64, device="cuda")
        s1 = torch.from_numpy(S0.copy()).cuda()
        for r in range(8):
            h.step(x[r], y1[r], s1, 0.9)
        rows = max(4, (M // 2) // 4 * 4) if M > 4 else M
        yr = torch.zeros((8, M - (M - rows) // 4 * 4), dtype=torch.float64, device="cuda")
        r0 = (M - rows) // 4 * 4
        h.step_rows(r0, M - r0, x, yr)
        torch.cuda.synchronize()
        y8, y1, yr, s8, s1 = (t.cpu().numpy() for t in (y8, y1, yr, s8, s1))
    bound = 1e-12 * (np.abs(X).astype(np.float64) @ np.abs(Ahat).T)
    assert (np.abs(y8 - y1) <= bound).all()
    assert (np.abs(yr - y1[:, r0:]) <= bound[:, r0:]).all()
    assert (np.abs(s8 - s1) <= 8 * bound.max(axis=0) + 1e-15 * np.abs(s1)).all()
    ref = X.astype(np.float64) @ Ahat.T
    for r in range(8):
        assert np.linalg.norm(y8[r] - ref[r]) <= 1e-6 * max(np.linalg.norm(ref[r]), 1e-300)
