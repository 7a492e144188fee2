"""Fixed accuracy with eight columns at sizes whose one-column plan shares no band (its
ranges are whole bands): the eight-column plan has a workspace of its own for its shared
groups of 8 bands, so that it keeps the whole grid -- without one it went down to as
little as an eighth of it -- and its results agree with single columns."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N", [(17000, 512), (14674, 512)])
def test_eight_columns_have_their_workspace(M, N):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need CUDA")
    import paper_1902_08018_gb300 as W

    A = np.random.default_rng(M).standard_normal((M, N))
    blob = W.whff_compress_accuracy(A, 1e-3)
    x = torch.from_numpy(np.random.default_rng(N).standard_normal((8, N)).astype(np.float32)).cuda()
    bands, runs = -(-M // 4), -(-N // 128)
    # all but the partials: stream, counters, staged x and y, transformed x, status word
    other = (blob.size - 64) + 4 * bands + 4 * 8 * N + 8 * 8 * M + 8 * 4 * 4 * 32 * runs + 4
    with W.whff_create(blob, max_rhs=8) as h:
        assert h.device_bytes >= other + bands * 2 * 256  # two segments of 8 columns and 4 rows a band
        y8 = torch.zeros((8, M), dtype=torch.float64, device="cuda")
        y1 = torch.zeros((8, M), dtype=torch.float64, device="cuda")
        h.step(x, y8)
        for r in range(8):
            h.step(x[r], y1[r])
        torch.cuda.synchronize()
    with W.whff_create(blob, max_rhs=7) as h:  # no eight-column pass: no workspace for one
        assert h.device_bytes < other + bands * 2 * 256
    # products rounded alike, sums good to 2^-46 of the terms' magnitude (as for other shapes)
    bound = 1e-12 * (np.abs(x.cpu().numpy()).astype(np.float64) @ (np.abs(A).T + 1e-2))
    assert (np.abs(y8.cpu().numpy() - y1.cpu().numpy()) <= bound).all()
