"""Tensor maps in device memory whose address an earlier matrix used: each of many
short-lived matrices of changing shapes gets the results of its own stream, alone and in
batches, though the allocator hands the same memory to the next one's map."""
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


SHAPES = [(256, 516), (132, 1028), (260, 512), (384, 260)]  # odd and even blocks per band


@pytest.mark.parametrize("rate", [12, 16])
def test_maps_at_a_reused_address(env, orc, rate):
    W, torch = env
    R = 16
    work = []
    for k, (M, N) in enumerate(SHAPES):
        rng = np.random.default_rng(k)
        blob = W.whff_compress(rng.standard_normal((M, N)), 5, rate)
        X = rng.standard_normal((R, N)).astype(np.float32)
        work.append((blob, torch.from_numpy(X).cuda(), X.astype(np.float64) @ orc.decode(blob.tobytes()).T))

    def check(y, ref):
        got = y.cpu().numpy()
        for r in range(R):
            assert np.linalg.norm(got[r] - ref[r]) <= 1e-6 * np.linalg.norm(ref[r])

    for k in range(24):
        blob, x, ref = work[k % len(work)]
        with W.whff_create(blob, max_rhs=R) as h:
            y = torch.zeros(ref.shape, dtype=torch.float64, device="cuda")
            h.step(x, y)
            check(y, ref)
    for k in range(6):
        two = [work[k % len(work)], work[(k + 1 + k // 4) % len(work)]]
        hs = [W.whff_create(w[0], max_rhs=R, host_resident=(i + k) % 3 == 2) for i, w in enumerate(two)]  # no map
        with W.Batch(hs, [R, R]) as b:
            ys = [torch.zeros(w[2].shape, dtype=torch.float64, device="cuda") for w in two]
            b.step([w[1] for w in two], ys, None)
            for y, w in zip(ys, two):
                check(y, w[2])
        for h in hs:
            h.destroy()
