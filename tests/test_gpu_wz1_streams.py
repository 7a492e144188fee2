"""The embedded decoder on arbitrary streams, bit for bit against the oracle.

The encoder writes only streams that its data leads to; here the block payloads
are random bits of several densities, so that group tests of every length, scans
that end at the last coefficient, planes without a test and budgets that end
inside a plane all occur at every place."""
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


@pytest.mark.parametrize("rate", [4, 8, 12, 16, 20, 64])
@pytest.mark.parametrize("ones", [0.03, 0.2, 0.5, 0.8, 0.97])
def test_random_streams(env, orc, rate, ones):
    W, torch = env
    M, N = 130, 259
    blob = W.whff_compress(np.zeros((M, N)), W.FMT_ZFP, rate)
    rng = np.random.default_rng(int(1000 * ones) + rate)
    bits = rng.random((blob.size - 64, 8)) < ones
    blob[64:] = np.packbits(bits, axis=1, bitorder="little")[:, 0]
    block = 2 * rate
    first = blob[64::block]
    blob[64::block] = first | (rng.random(first.size) < 0.95)  # most blocks carry the nonzero flag
    blob[65::block] |= 1  # a block exponent of at least 1 + 2^7 - 127: results stay in the normal range
    assert W.library().whff_blob_seal(blob.ctypes.data, blob.size) == 0
    ref = orc.decode(blob.tobytes())
    with W.whff_create(blob, max_rhs=1) as h:
        out = torch.empty((M, N), dtype=torch.float64, device="cuda")
        h.decompress(out)
        torch.cuda.synchronize()
        got = out.cpu().numpy()
    assert (got.view(np.uint64) == ref.view(np.uint64)).all()
