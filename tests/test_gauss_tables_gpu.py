"""The Gaussian sampler's Box-Muller tables at their edges, through the
records: factors that leave single coordinates of z visible, an odd last
coordinate (the pair whose second normal is dropped), every quadrant, boxes
whose bounds are zero, equal to a coordinate's sign, infinite, or NaN.  Records
against the oracle's plain log, sqrt, sin and cos."""
import numpy as np
import pytest

import oracle
from oracle.maps import GAUSSIAN, integrate_mapped
from test_parity_gpu import FP64_RTOL, assert_slots_close
from test_samplers_gpu import _run_plan

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nt,scale,upper", [(2, 1, 1.0, True), (3, 1, 0.7, True), (4, 1, 1.3, False),
                                               (2, 2, 1.0, False), (3, 2, 1.0, True), (6, 2, 0.5, True)])
def test_box_muller_records(bfi, nx, nt, scale, upper):
    d = nx * nt
    F = scale * np.eye(d) + (0.1 * np.triu(np.ones((d, d)), 1) if upper else 0.05 * np.ones((d, d)))
    inf = np.inf
    lo = np.stack([np.full(d, -inf), np.zeros(d), np.full(d, -inf), np.full(d, -0.0), np.full(d, -3.0)])
    hi = np.stack([np.full(d, inf), np.full(d, inf), np.zeros(d), np.full(d, 2.0), np.full(d, 3.0)])
    lo[4, 0] = np.nan  # admits nothing
    samples = np.array([70_001, 30_000, 30_000, 20_000, 1000], dtype=np.uint64)
    lat_o = oracle.lattice(nx, nt, mass2=0.5)
    g_s, _ = _run_plan(bfi, bfi.lattice(nx, nt, mass2=0.5), lo, hi, samples, 13, None, bfi.SAMPLE_GAUSSIAN, factor=F)
    o_s, _ = integrate_mapped(lat_o, lo, hi, samples, 13, kind=GAUSSIAN, factor=F)
    assert np.array_equal(np.isfinite(g_s[:, 1]), np.isfinite(o_s[:, 1])) and g_s[4, 3] == 0.0
    used = np.isfinite(o_s[:, 1])
    assert used.sum() >= 3
    assert_slots_close(g_s[used], o_s[used], nx // 2 + 1, FP64_RTOL)
