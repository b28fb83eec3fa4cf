"""The generic kernel's batched draws at their edges: two and sixteen Philox
blocks a sample (the most and the fewest points at once), one block more (no
batch), ragged last blocks, and budgets below one batch, one short of a chunk,
a chunk and one more.  Records against the oracle in both precisions."""
import numpy as np
import pytest

import workloads
from test_parity_gpu import FP32_RTOL, FP64_RTOL, assert_slots_close, run_gpu, run_oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev(bfi):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nx,nt", [(5, 1), (7, 1), (5, 3), (9, 3), (9, 7), (8, 8), (13, 5)])
def test_generic_batches(bfi, dev, nx, nt, precision):
    samples = np.array([1, 2, 5, 63, 0, 1023, 1024, 1025], dtype=np.uint64)
    lo, hi = workloads.bisected_boxes(nx * nt, 3)
    job = workloads.Job(nx, nt, lo, hi, samples, seed=17, nu=0.7)
    g_s, _, plan = run_gpu(bfi, dev, job, precision)
    assert plan.info().kernel == 1
    o_s, _ = run_oracle(job, fp32_points=precision == 1)
    assert_slots_close(g_s, o_s, nx // 2 + 1, FP32_RTOL if precision else FP64_RTOL)
