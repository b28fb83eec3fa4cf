"""The range map's FP32 screen against the plain FP64 estimator, where it can
go wrong: every compiled shape's stencil, chunks of one row and of ragged
rows, wide and narrow boxes, actions far apart and close together, chunks
wholly outside the window, a mass term, and the records' shift, which is
defined by the samples alone (per chunk and thread: the first sample's action,
then any more than 16 below) and compared with that rule in numpy."""
import numpy as np
import pytest

import oracle
from oracle.maps import TRANSFORM, integrate_mapped, log_jacobian, transform
from test_parity_gpu import FP64_RTOL, assert_slots_close
from test_samplers_gpu import _run_plan

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _shift(lat, lo, hi, n, sid, seed, chunk):
    """Smallest thread shift of the subvolume (256 threads a chunk, margin 16)."""
    y = oracle.points(lat.nx * lat.nt, lo, hi, sid, seed, 0, 0, n)
    S = oracle.eval_points(lat, transform(y))[0] - log_jacobian(y).sum(axis=1)
    best = np.inf
    for c in range(0, n, chunk):
        part = S[c:c + chunk]
        for t in range(min(256, part.size)):
            m = np.inf
            for s in part[t::256]:
                if s < m - 16.0:
                    m = s
            best = min(best, m)
    return best


@pytest.mark.parametrize("nx,nt,nu,mass2,half,n", [
    (2, 1, 1.0, 0.5, 1.0, 1), (3, 1, 1.0, 0.3, 1.0, 255), (4, 1, 0.2, 0.0, 1.0, 257), (2, 2, 1.0, 0.0, 1.0, 1025),
    (3, 2, 1.0, 0.0, 1.0, 5000), (4, 2, 1.0, 0.0, 0.3, 5000), (6, 2, 3.0, 0.0, 1.0, 7001), (8, 2, 0.1, 0.0, 1.0, 9000),
    (10, 2, 1.0, 0.0, 1.0, 20011), (10, 2, 8.0, 0.0, 1.0, 20011), (10, 2, 1.0, 0.0, 1e-4, 3000),
    (16, 2, 1.0, 0.2, 1.0, 9001), (32, 2, 1.0, 0.0, 1.0, 3001), (4, 4, 1.0, 0.0, 1.0, 9001),
    (6, 4, 5.0, 0.0, 1.0, 9001), (8, 4, 1.0, 0.0, 0.9, 9001), (10, 4, 0.3, 0.0, 1.0, 5001),
    (16, 4, 1.0, 0.0, 1.0, 3001)])
def test_transform_screen(bfi, nx, nt, nu, mass2, half, n):
    d = nx * nt
    lo = np.stack([np.full(d, -half), np.where(np.arange(d) % 2 == 0, 0.0, -half), np.full(d, -half)])
    hi = np.stack([np.full(d, half), np.full(d, half), np.where(np.arange(d) % 3 == 0, 0.0, half)])
    samples = np.array([n, max(1, n // 3), n + 256], dtype=np.uint64)
    sid = np.array([4, 0, 7], dtype=np.uint32)
    g_s, _ = _run_plan(bfi, bfi.lattice(nx, nt, nu=nu, mass2=mass2), lo, hi, samples, 21, sid, bfi.SAMPLE_TRANSFORM)
    lat = oracle.lattice(nx, nt, nu=nu, mass2=mass2)
    o_s, _ = integrate_mapped(lat, lo, hi, samples, 21, sub_id=sid, kind=TRANSFORM)
    R = nx // 2 + 1
    assert_slots_close(g_s, o_s, R, FP64_RTOL)
    chunk = bfi.chunking(samples).chunk_samples
    for s in range(3):
        m = _shift(lat, lo[s], hi[s], int(samples[s]), int(sid[s]), 21, chunk)
        assert abs(g_s[s, 1] - m) <= 1e-10 * max(1.0, abs(m)), (s, g_s[s, 1], m)
