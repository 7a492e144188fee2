"""whff_decompress into outputs of every alignment, bit for bit against the oracle.

The decode kernels write 32-byte stores when the output's address and leading
dimension allow it and turn the rows round in shared memory otherwise; both
paths at the edges of a warp's 32 units, for each format's FP64 assembly (FP32
and integer block transforms, products with a tile scale, values whose scale or
significand leaves the normal FP32 range)."""
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


def matrix(M, N, seed, tiny):
    rng = np.random.default_rng(seed)
    A = rng.standard_normal((M, N)) * np.exp(rng.uniform(-6, 6, size=(M, N)))
    if M > 4 and N > 4:
        A[:4, :4] = 0.0
    return A * (2.0**-121 if tiny else 1.0)  # tile scales (and BF16 values) below the normal FP32 range


FORMATS = [(1, 8), (1, 16), (1, 64), (5, 8), (5, 12), (5, 16), (5, 20), (5, 24), (6, 16), (6, 24), (2, 0), (3, 0),
           (4, 0), (7, 0), (8, 0)]
# (M, N, first column, padding): 32-byte aligned rows; an odd leading dimension; an odd first entry
SHAPES = [(5, 3, 0, 1), (9, 128, 0, 0), (130, 260, 4, 4), (37, 131, 0, 0), (66, 516, 1, 3), (13, 16, 2, 2)]


@pytest.mark.parametrize("fmt,rate", FORMATS)
@pytest.mark.parametrize("M,N,first,pad", SHAPES)
@pytest.mark.parametrize("tiny", [False, True])
def test_decode_every_alignment(env, orc, fmt, rate, M, N, first, pad, tiny):
    W, torch = env
    A = matrix(M, N, 100 * fmt + rate + M, tiny and fmt in (2, 3, 4, 7))
    if fmt == 8:
        blob = W.whff_compress_accuracy(A, 1e-6)
        ref = orc.wz3_decode(blob.tobytes())[0]
    else:
        blob = W.whff_compress(A, fmt, rate or 16)
        ref = orc.decode(blob.tobytes())
    with W.whff_create(blob, max_rhs=1) as h:
        buf = torch.full((M + 1, first + N + pad), np.nan, dtype=torch.float64, device="cuda")
        h.decompress(buf[:M, first:])
        torch.cuda.synchronize()
        got = buf.cpu().numpy()
    assert (got[:M, first:first + N].view(np.uint64) == ref.view(np.uint64)).all()
    rest = got.copy()
    rest[:M, first:first + N] = np.nan
    assert np.isnan(rest).all()  # nothing written outside
