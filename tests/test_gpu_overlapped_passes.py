"""Passes of one handle that overlap on two streams share its workspace, so their results
mean nothing; but they leave nothing behind: once both streams are idle, the next passes
of every kind give the bits they gave before, direct and replayed from graphs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fmt,rate", [(5, 8), (5, 16), (6, 16), (2, 0), (7, 0), (8, 0)])
@pytest.mark.parametrize("M,N", [(256, 20000), (1000, 2052), (3000, 512)])
def test_overlap_leaves_nothing_behind(fmt, rate, M, N):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need CUDA")
    import paper_1902_08018_gb300 as W

    A = np.random.default_rng(M).standard_normal((M, N))
    blob = W.whff_compress_accuracy(A, 1e-4) if fmt == 8 else W.whff_compress(A, fmt, rate)
    x = torch.from_numpy(np.random.default_rng(N).standard_normal((8, N)).astype(np.float32)).cuda()
    with W.whff_create(blob, max_rhs=8) as h:
        if fmt in (2, 5, 6):
            h.crossover = 33  # CUDA cores
        rows = 128
        ys = [torch.zeros((R, n), dtype=torch.float64, device="cuda")
              for n in (M, rows) for R in (1, 8)]
        yg = torch.zeros(M, dtype=torch.float64, device="cuda")
        graph = W.whff_graph_create(h, x[0], yg)

        def passes():
            out = []
            for R, y, v in ((1, ys[0], ys[2]), (8, ys[1], ys[3])):
                y.zero_(), v.zero_()
                h.step(x[:R], y)
                h.step_rows(0, rows, x[:R], v)
                out += [y.clone(), v.clone()]
            yg.zero_()
            graph.launch()
            torch.cuda.synchronize()
            return out + [yg.clone()]

        first = passes()
        a, b = torch.cuda.Stream(), torch.cuda.Stream()
        junk = [torch.empty_like(y) for y in ys]
        for what in range(3):
            torch.cuda.synchronize()
            for k in range(60):
                h.step(x[:1 + 7 * (k % 2)], junk[k % 2], stream=a)
                if what == 0:
                    h.step_rows(0, rows, x[:1], junk[2], stream=b)
                elif what == 1:
                    graph.launch(stream=b)
                else:
                    h.step_rows(0, rows, x, junk[3], stream=b)
            torch.cuda.synchronize()
            for _ in range(2):
                for got, want in zip(passes(), first):
                    assert torch.equal(got, want)
