"""A band's sums over the lanes keep FP64's digits: the lanes of a warp hold 1, 2^-27 and
2^-52 (times powers of two), whose sum FP64 holds exactly and a pair of FP32 numbers
does not (1 + 2^-27 (1 + 2^-25) needs 26 digits below the leading one).

Constant blocks make every product a power of two, so y must equal the FP64 product
exactly: 4096 blocks per band and more take the fold beyond FP64, and fixed accuracy
takes it with any number."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fmt,rate,N", [(8, 0, 128), (8, 0, 4096), (5, 8, 16384), (5, 16, 16384), (6, 16, 16384),
                                        (1, 16, 128), (7, 0, 16384)])
@pytest.mark.parametrize("R", [1, 8])
def test_sums_keep_the_digits_of_fp64(orc, fmt, rate, N, R):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need CUDA")
    import paper_1902_08018_gb300 as W

    M = 36
    A = np.ones((M, N))
    A[8:12] = -2.0
    blob = W.whff_compress_accuracy(A, 0.0) if fmt == 8 else W.whff_compress(A, fmt, rate)
    assert ((orc.wz3_decode(blob.tobytes())[0] if fmt == 8 else orc.decode(blob.tobytes())) == A).all()
    X = np.zeros((R, N), dtype=np.float32)
    for r in range(R):
        X[r, 4 * r:4 * r + 4] = 1.0  # lanes r, r + 5 and r + 17 of a warp
        X[r, 4 * (r + 5):4 * (r + 5) + 4] = 2.0**-27
        X[r, 4 * (r + 17):4 * (r + 17) + 4] = 2.0**-52
    with W.whff_create(blob, max_rhs=R) as h:
        if R > 1 and fmt in (5, 6):
            h.crossover = 33  # CUDA cores
        y = torch.zeros((R, M), dtype=torch.float64, device="cuda")
        h.step(torch.from_numpy(X).cuda(), y)
        torch.cuda.synchronize()
        got = y.cpu().numpy()
    want = np.zeros((R, M))
    want[:] = 4.0 * (1.0 + 2.0**-27 + 2.0**-52)
    want[:, 8:12] *= -2.0
    assert (got == want).all()
