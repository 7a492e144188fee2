"""Tensor-core passes of a host-resident matrix cross the link once: its bytes take the
link's time, which the one-column pass over the same matrix shows (653 us for 134 MB;
the 32-column pass 662 us, and 1124 us when every 16-byte piece fetched a sector of its
own).  The line is at 1.35 times the one-column pass."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rate", [8, 16])
def test_many_columns_take_the_links_time(rate):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need CUDA")
    import paper_1902_08018_gb300 as W

    n = 8192
    A = np.random.default_rng(rate).standard_normal((n, n), dtype=np.float32).astype(np.float64)
    x = torch.randn((32, n), device="cuda")
    y = torch.zeros((32, n), dtype=torch.float64, device="cuda")
    with W.whff_create(W.whff_compress(A, 5, rate), max_rhs=32, host_resident=True) as h:

        def best(R):
            times = []
            for _ in range(8):
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record()
                h.step(x[:R], y[:R])
                e1.record()
                torch.cuda.synchronize()
                times.append(e0.elapsed_time(e1))
            return min(times)

        best(32)
        one, many = best(1), best(32)
    assert many <= 1.35 * one, (one, many)
