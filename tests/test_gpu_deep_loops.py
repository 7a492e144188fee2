"""One-column passes with four or eight blocks in flight: shared bands added up in the
kernel up to 2^21 blocks and by a launch of their own above, the same bits as with two
in flight (the blocks in flight change the schedule, not the arithmetic), pass after
pass, with the state and on row views of the same handle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# 1448^2 blocks (2^21 less 448) and 1449 x 1448, 1449^2 above; wide; a last column of one entry
@pytest.mark.parametrize("M,N", [(5792, 5792), (5796, 5792), (5793, 5793), (260, 140001), (31, 4001)])
@pytest.mark.parametrize("fmt,rate", [(5, 8), (5, 16), (6, 12), (5, 24)])
def test_blocks_in_flight_change_no_bits(M, N, fmt, rate):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need CUDA")
    import paper_1902_08018_gb300 as W

    rng = np.random.default_rng(M + rate)
    A = rng.standard_normal((M, N), dtype=np.float32).astype(np.float64)
    x = torch.from_numpy(rng.standard_normal(N).astype(np.float32)).cuda()
    s0 = torch.from_numpy(rng.standard_normal(M)).cuda()
    with W.whff_create(W.whff_compress(A, fmt, rate), max_rhs=1) as h:
        for fold in (0, 1):
            out = []
            for unroll in (2, 4, 8):
                h.set_config(unroll, 1, fold)  # one CTA per SM: the same ranges for each
                for _ in range(2):
                    y, s = torch.zeros(M, dtype=torch.float64, device="cuda"), s0.clone()
                    h.step(x, y, s, 0.5)
                    v = torch.zeros(M - M // 8 * 4, dtype=torch.float64, device="cuda")
                    h.step_rows(M // 8 * 4, M - M // 8 * 4, x, v)
                    torch.cuda.synchronize()
                    out.append((y, s, v))
            for got in out[1:]:
                assert all(torch.equal(a, b) for a, b in zip(got, out[0]))
            assert torch.equal(out[0][1], 0.5 * s0 + out[0][0])
