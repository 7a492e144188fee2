"""Where the lift's one-column kernel transforms x itself: an x that it cannot load 16
bytes at a time (N not a multiple of 4, or an unaligned x) goes through the transform's
own launch above 2^22 blocks, an aligned one does not; the bits are the same."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# blocks: 2048^2 = 2^22 and one column of blocks more
@pytest.mark.parametrize("M,N,launches", [(8192, 8192, 1), (8192, 8191, 1), (8192, 8196, 1), (8192, 8195, 2),
                                          (8192, 8193, 2),
                                          # lane groups: 20971 x 25 blocks (2^19 less 13), 20972 x 25, aligned
                                          (83884, 99, 1), (83888, 99, 2), (83888, 100, 1)])
def test_route_and_bits(M, N, launches):
    import ctypes

    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need CUDA")
    import paper_1902_08018_gb300 as W

    A = np.random.default_rng(N).standard_normal((M, N), dtype=np.float32).astype(np.float64)
    buf = torch.from_numpy(np.random.default_rng(M).standard_normal(N + 1).astype(np.float32)).cuda()
    with W.whff_create(W.whff_compress(A, 5, 8), max_rhs=1) as h:
        k, n = ctypes.c_int(), ctypes.c_int()
        assert W.library().whff_plan(h.ptr, ctypes.byref(k), ctypes.byref(n)) == 0
        assert n.value == launches
        out = []
        for x in (buf[1:].clone(), buf[1:]):  # aligned, 4 bytes off
            for unroll, fold in ((2, h.config()[2]), (4, 0)) if N > 1000 else ((2, 2),):
                h.set_config(unroll, 1, fold)  # four blocks in flight always take the transform's launch
                y = torch.zeros(M, dtype=torch.float64, device="cuda")
                h.step(x, y)
                out.append(y)
        torch.cuda.synchronize()
        assert all(torch.equal(y, out[0]) for y in out)
