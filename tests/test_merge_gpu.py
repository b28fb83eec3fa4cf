"""The merge of chunk records at the edges of its split: subvolumes of one
chunk, of the most that one warp merges, of one more (pieces), of pieces that
start inside a window, without samples, and more correlation distances than a
warp has lanes.  Records against the oracle, totals against the host merge."""
import numpy as np
import pytest

import workloads
from test_parity_gpu import FP64_ERR_ATOL, FP64_RTOL, assert_slots_close, run_gpu, run_oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CHUNK = 1024  # samples of a chunk in jobs below 2^21 samples
WHOLE = 64    # chunks of a subvolume that one warp merges


@pytest.fixture(scope="module")
def dev(bfi):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


@pytest.mark.parametrize("nx,nt,chunks", [
    (4, 1, [WHOLE]), (4, 1, [WHOLE + 1]), (4, 2, [1, WHOLE, 0, WHOLE + 1, 3, 2 * WHOLE + 31, 1]),
    (2, 1, [97, 33, 31, 129, 0]), (64, 2, [2, WHOLE + 2, 1]), (128, 1, [1, 0, 5])])
def test_merge_pieces(bfi, dev, nx, nt, chunks):
    samples = np.array([max(0, c * CHUNK - 7 * (s % 2)) for s, c in enumerate(chunks)], dtype=np.uint64)
    assert bfi.chunking(samples).chunks == sum(chunks) and bfi.chunking(samples).chunk_samples == CHUNK
    k = int(np.ceil(np.log2(len(chunks))))
    lo, hi = workloads.bisected_boxes(nx * nt, k)
    job = workloads.Job(nx, nt, lo[:len(chunks)], hi[:len(chunks)], samples, seed=11)
    g_s, g_t, _ = run_gpu(bfi, dev, job, 0)
    o_s, _ = run_oracle(job)
    assert_slots_close(g_s, o_s, nx // 2 + 1, FP64_RTOL)
    h_t, R = bfi.merge_host(nx, g_s), nx // 2 + 1
    np.testing.assert_allclose(h_t[:4 + R], g_t[:4 + R], rtol=1e-13, atol=1e-13 * abs(g_t[4]))
    np.testing.assert_allclose(h_t[4 + R:], g_t[4 + R:], rtol=1e-9, atol=FP64_ERR_ATOL * abs(g_t[4]))
