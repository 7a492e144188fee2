"""Tensor-core passes: the words of a stage brought in by one tiled copy, by two
(odd numbers of blocks per band at rates 12 and 20, whose rows are 8 bytes off
16), and in 16-byte pieces (host-resident streams) -- the same words, so the same
bits -- at the edges of stages, tiles and row views, and against the FP64 oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 1e-6  # relative L2 per right-hand side, as for every pass


@pytest.fixture(scope="module")
def env():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need CUDA")
    import paper_1902_08018_gb300 as W

    W.library()
    return W, torch


# (M, N, first row of the view, its rows): one band and one block; a last stage of 1 and of 15 blocks;
# odd and even blocks per band; a tile's last band, one band past a tile, views from odd bands
SHAPES = [(3, 4, 0, 3), (127, 68, 4, 60), (132, 60, 128, 4), (260, 1284, 12, 248), (516, 1280, 4, 129),
          (70, 9004, 36, 34)]


@pytest.mark.parametrize("fmt,rate", [(5, 8), (5, 12), (6, 12), (5, 16), (5, 20), (6, 24)])
@pytest.mark.parametrize("M,N,row0,nrows", SHAPES)
@pytest.mark.parametrize("R", [5, 20])
def test_copies_agree(env, orc, fmt, rate, M, N, row0, nrows, R):
    W, torch = env
    rng = np.random.default_rng(M + N + rate)
    A = rng.standard_normal((M, N)) * np.exp(rng.uniform(-3, 3, size=(M, 1)))
    blob = W.whff_compress(A, fmt, rate)
    Ahat = orc.decode(blob.tobytes())
    X = rng.standard_normal((R, N)).astype(np.float32)
    out = []
    for host in (False, True):
        with W.whff_create(blob, max_rhs=32, host_resident=host) as h:
            x = torch.from_numpy(X).cuda()
            y = torch.zeros((R, M), dtype=torch.float64, device="cuda")
            h.step(x, y)
            v = torch.zeros((R, nrows), dtype=torch.float64, device="cuda")
            h.step_rows(row0, nrows, x, v)
            torch.cuda.synchronize()
            assert h.sync_status() == 0
            out.append((y.cpu().numpy(), v.cpu().numpy()))
    assert (out[0][0] == out[1][0]).all() and (out[0][1] == out[1][1]).all()
    ref = X.astype(np.float64) @ Ahat.T
    for r in range(R):
        for got, want in ((out[0][0][r], ref[r]), (out[0][1][r], ref[r, row0:row0 + nrows])):
            assert np.linalg.norm(got - want) <= TOL * np.linalg.norm(want)


# (M, N): one row and less than a 16-byte piece; an odd last stage; a last row past a tile; many
# stages a tile; more tiles than item ranges
@pytest.mark.parametrize("M,N", [(1, 5), (127, 65), (129, 700), (300, 9001), (40000, 100)])
@pytest.mark.parametrize("R", [5, 20, 32])
def test_fp8_copies_agree(env, orc, M, N, R):
    """FP8 by tiled copies (device memory) and through registers (host memory): the same bits."""
    W, torch = env
    rng = np.random.default_rng(M + N)
    A = rng.standard_normal((M, N)) * np.exp(rng.uniform(-3, 3, size=(M, 1)))
    blob = W.whff_compress(A, 4, 0)
    X = rng.standard_normal((R, N)).astype(np.float32)
    out = []
    for host in (False, True):
        with W.whff_create(blob, max_rhs=32, host_resident=host) as h:
            x = torch.from_numpy(X).cuda()
            y = torch.zeros((R, M), dtype=torch.float64, device="cuda")
            h.step(x, y)
            torch.cuda.synchronize()
            assert h.sync_status() == 0
            out.append(y.cpu().numpy())
    assert (out[0] == out[1]).all()
    ref = X.astype(np.float64) @ orc.decode(blob.tobytes()).T
    for r in range(R):
        assert np.linalg.norm(out[0][r] - ref[r]) <= TOL * np.linalg.norm(ref[r])
