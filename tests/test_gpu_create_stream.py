"""whff_create works on its own stream: all its uploads, the tensor maps among them, are
enqueued there and have landed when it returns.  So it neither waits for the legacy
stream (a pageable copy there would, and may return before its bytes have reached the
device) nor leaves an upload that a step on a non-blocking stream could overtake."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fmt,rate", [(5, 16), (6, 12), (4, 0)])
def test_create_beside_a_busy_legacy_stream(orc, fmt, rate):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need CUDA")
    import paper_1902_08018_gb300 as W

    M, N, R = 256, 260, 16
    A = np.random.default_rng(rate).standard_normal((M, N))
    blob = W.whff_compress(A, fmt, rate)
    X = np.random.default_rng(R).standard_normal((R, N)).astype(np.float32)
    side = torch.cuda.Stream()  # non-blocking: not ordered with the legacy stream
    x = torch.from_numpy(X).cuda()
    y = torch.zeros((R, M), dtype=torch.float64, device="cuda")
    with W.whff_create(blob, max_rhs=R) as warm:  # kernels loaded, attributes set
        warm.step(x, y)
    torch.cuda.synchronize()
    done = torch.cuda.Event()
    torch.cuda._sleep(1_000_000_000)  # the legacy stream: about half a second
    done.record()
    h = W.whff_create(blob, max_rhs=R, stream=side)
    busy = not done.query()
    assert busy
    h.step(x, y, stream=side)
    side.synchronize()
    torch.cuda.synchronize()
    ref = X.astype(np.float64) @ orc.decode(blob.tobytes()).T
    got = y.cpu().numpy()
    h.destroy()
    for r in range(R):
        assert np.linalg.norm(got[r] - ref[r]) <= 1e-6 * np.linalg.norm(ref[r])
