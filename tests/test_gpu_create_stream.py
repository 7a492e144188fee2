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


def test_batches_step_at_once_on_a_stream_of_their_own(orc):
    """The batch's tables are on the device when whff_batch_create returns: its first step
    may run on a non-blocking stream (shown by reading; a copy still under way is a race)."""
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need CUDA")
    import paper_1902_08018_gb300 as W

    side = torch.cuda.Stream()
    work = []
    for k, (M, N, R) in enumerate([(256, 260, 16), (132, 516, 1), (300, 128, 5)]):
        rng = np.random.default_rng(k)
        blob = W.whff_compress(rng.standard_normal((M, N)), 5, 12)
        X = rng.standard_normal((R, N)).astype(np.float32)
        work.append((W.whff_create(blob, max_rhs=16, stream=side), torch.from_numpy(X).cuda(),
                     torch.zeros((R, M), dtype=torch.float64, device="cuda"),
                     X.astype(np.float64) @ orc.decode(blob.tobytes()).T))
    torch.cuda.synchronize()
    for _ in range(4):
        for w in work:
            w[2].zero_()
        torch.cuda.synchronize()
        with W.Batch([w[0] for w in work], [w[1].shape[0] for w in work]) as b:
            b.step([w[1] for w in work], [w[2] for w in work], None, stream=side)
            side.synchronize()
        for w in work:
            got = w[2].cpu().numpy()
            for r in range(len(got)):
                assert np.linalg.norm(got[r] - w[3][r]) <= 1e-6 * np.linalg.norm(w[3][r])
    for w in work:
        w[0].destroy()
