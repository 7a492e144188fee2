"""FP8 tensor-core passes on row views: the tiled copies take the view's first row as a
coordinate of the whole matrix's map, so views from several scale tiles on, and
time-sliced steps, give the bits of the host-resident handle, whose register-fed kernel
reads the view's own pointer, and the sliced step meets the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N", [(700, 600), (513, 1030)])
@pytest.mark.parametrize("R", [5, 20, 32])
def test_fp8_views_and_slices(orc, M, N, R):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need CUDA")
    import paper_1902_08018_gb300 as W

    rng = np.random.default_rng(M + R)
    A = rng.standard_normal((M, N)) * np.exp(rng.uniform(-3, 3, size=(M, 1)))
    blob = W.whff_compress(A, 4, 0)
    X = rng.standard_normal((R, N)).astype(np.float32)
    ref = X.astype(np.float64) @ orc.decode(blob.tobytes()).T
    views = [(128, 100), (256, M - 256), (384, 129), (512, 1)]
    out = []
    for host in (False, True):
        with W.whff_create(blob, max_rhs=32, host_resident=host) as h:
            assert h.crossover <= R
            x = torch.from_numpy(X).cuda()
            got = []
            for row0, nrows in views:
                y = torch.zeros((R, nrows), dtype=torch.float64, device="cuda")
                h.step_rows(row0, nrows, x, y)
                got.append(y)
            h.slice_rows = 256
            y = torch.zeros((R, M), dtype=torch.float64, device="cuda")
            h.step(x, y)
            got.append(y)
            torch.cuda.synchronize()
            assert h.sync_status() == 0
            out.append([g.cpu().numpy() for g in got])
    for a, b in zip(*out):
        assert (a == b).all()
    for r in range(R):  # the bar is on whole columns: the sliced step
        assert np.linalg.norm(out[0][-1][r] - ref[r]) <= 1e-6 * np.linalg.norm(ref[r])
