"""Totals where the actions are so large (tiny D) that log V - log n - m is far
outside the range of an integer exponent, and where its form changes (2^60):
against the estimator's definition on the records."""
import numpy as np
import pytest

import oracle
import workloads
from test_parity_gpu import run_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [2.0 ** -k for k in (8, 18, 22, 23, 24, 25, 26, 30, 45, 48, 49, 50, 51, 52, 53, 54, 55, 100, 400)])
@pytest.mark.parametrize("precision", [0, 1])
def test_large_actions(bfi, D, precision):
    """Subvolumes 0 and 3 are the same job; the others' weights are of other orders altogether."""
    if precision == 1 and D < 1e-30:
        pytest.skip("the action is beyond float's range")
    dev = torch.device("cuda:0")
    lo, hi = workloads.bisected_boxes(8, 2)
    lo, hi = lo + 7.0, hi + 7.0 + np.arange(4)[:, None]
    lo[3], hi[3] = lo[0], hi[0]
    samples = np.array([3000, 2, 2500, 3000], dtype=np.uint64)
    job = workloads.Job(4, 2, lo, hi, samples, sub_id=np.array([5, 1, 2, 5], dtype=np.uint32), seed=11, D=D)
    g_s, g_t, _ = run_gpu(bfi, dev, job, precision)
    assert np.array_equal(g_s[0], g_s[3])
    ls = g_s[:, 2] - np.log(g_s[:, 0]) - g_s[:, 1]
    top = int(np.argmax(ls))
    rest = np.abs(ls - ls[top])
    assert np.all((rest == 0.0) | (rest > 1e3)), "no subvolume between"  # so f_s is 1 or 0
    with np.errstate(under="ignore"):
        want = oracle.merge(4, g_s)
    # the logarithms of ls and Z may be an ulp apart
    np.testing.assert_allclose(g_t[0], want[0], rtol=1e-14)
    np.testing.assert_allclose(g_t[[1, 2, 3]], want[[1, 2, 3]], rtol=1e-12)
    np.testing.assert_allclose(g_t[4:7], want[4:7], rtol=0, atol=1e-12 * want[4])
    # one sample carries nearly all weight: the variance of C(r) is the rounding of terms of size C(0)^2
    np.testing.assert_allclose(g_t[7:], want[7:], rtol=1e-9, atol=np.sqrt(16 * 2.0 ** -52) * want[4])


def test_no_volume(bfi):
    """A box of no width carries no weight beside others, and gives no number alone."""
    dev = torch.device("cuda:0")
    lo, hi = workloads.bisected_boxes(8, 1)
    hi[1] = lo[1]
    job = workloads.Job(4, 2, lo, hi, np.array([700, 700], dtype=np.uint64), seed=3)
    g_s, g_t, _ = run_gpu(bfi, dev, job, 0)
    np.testing.assert_allclose(g_t[:4], oracle.merge(4, g_s)[:4], rtol=1e-12)
    alone = workloads.Job(4, 2, lo[1:], hi[1:], np.array([700], dtype=np.uint64), seed=3)
    assert np.isnan(run_gpu(bfi, dev, alone, 0)[1][0])
