"""Bounded waits that run out after copies and MMAs have begun: with a limit of a few
polls (about a quarter of a microsecond each) the waits on free slots succeed, stages are
in flight when the next wait gives up, and the kernel has to let them land before its
CTAs go.  The status word reports the timeout, and with the default limit restored the
same handle gives the bits that it gave before.

Zero polls, where the first waits give up before anything has begun, are tried too, for
FP8's kernel above all (test_gpu_wait_timeout.py does not take it)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TIMEOUT = -7  # WHFF_ETIMEOUT


@pytest.fixture(scope="module")
def env():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need CUDA")
    import paper_1902_08018_gb300 as W

    W.library()
    return W, torch


# one tiled copy a stage; two (rates 12 and 20, odd number of blocks per band); three A
# pieces; 16-byte pieces (host-resident); FP8's own kernel
CASES = [(5, 8, 4096, False), (5, 16, 4096, False), (6, 12, 4100, False), (5, 20, 4100, False), (5, 24, 4096, False),
         (5, 16, 4096, True), (4, 0, 4096, False)]


@pytest.mark.parametrize("fmt,rate,N,host", CASES)
@pytest.mark.parametrize("R", [8, 32])
def test_waits_that_run_out_midway(env, fmt, rate, N, host, R):
    W, torch = env
    M = 1024
    A = np.random.default_rng(N + rate).standard_normal((M, N))
    with W.whff_create(W.whff_compress(A, fmt, rate), max_rhs=32, host_resident=host) as h:
        assert h.crossover <= R  # the pass runs on the tensor cores
        x = torch.from_numpy(np.random.default_rng(R).standard_normal((R, N)).astype(np.float32)).cuda()
        y0 = torch.zeros((R, M), dtype=torch.float64, device="cuda")
        h.step(x, y0)
        assert h.sync_status() == 0
        seen = []
        for polls in (0, 1, 2, 3, 5, 8, 16):
            h.set_wait_limit(polls)
            y = torch.zeros_like(y0)
            h.step(x, y)
            seen.append(h.sync_status())
            h.set_wait_limit(-1)
            h.step(x, y)
            assert h.sync_status() == 0
            assert torch.equal(y, y0)
        assert set(seen) <= {0, TIMEOUT}
        assert seen[0] == TIMEOUT  # nothing has begun
        assert seen[1] == TIMEOUT  # a copy from HBM takes longer than one poll
