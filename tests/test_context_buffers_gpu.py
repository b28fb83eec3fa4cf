"""A context's reused buffers: one context through jobs that grow, shrink, cross
the size up to which arrays go through the page-locked buffer, change shape,
precision and sampler, with and without sub_ids and records.  Every call equals
the plan path bit for bit."""
import numpy as np
import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _plan(bfi, lat, lo, hi, samples, seed, sid, precision, sampler):
    plan = bfi.Plan(lat, samples, precision)
    if sampler[0] != bfi.SAMPLE_BOX:
        plan.set_sampler(sampler[0], factor=sampler[1])
    dev = torch.device("cuda:0")
    s, t = plan.execute(torch.tensor(lo, device=dev), torch.tensor(hi, device=dev), seed,
                        sub_id=None if sid is None else torch.tensor(sid.astype(np.int32), device=dev))
    torch.cuda.synchronize()
    plan.close()
    return s.cpu().numpy(), t.cpu().numpy()


# bytes up: tables 8 (2 nsub + 1), boxes 16 nsub d, sub_ids 4 nsub; the page-locked path ends at 64 KiB
@pytest.mark.parametrize("sizes", [[1, 3, 190, 191, 700, 2, 191], [700, 5], [189, 190, 192]])
def test_context_buffers(bfi, sizes):
    ctx = bfi.Context(0)
    try:
        for i, n in enumerate(sizes):
            nx, nt = (10, 2) if i % 3 != 1 else (4, 2)
            d = nx * nt
            lo, hi = workloads.bisected_boxes(d, int(np.ceil(np.log2(max(n, 1)))))
            lo, hi = lo[:n].copy(), hi[:n].copy()
            samples = np.array([300 + 7 * (s % 5) for s in range(n)], dtype=np.uint64)
            sid = None if i % 2 else np.arange(n, dtype=np.uint32)[::-1].copy() + 5
            precision = 1 if i % 4 == 3 else 0
            sampler = (bfi.SAMPLE_BOX, None)
            lat = bfi.lattice(nx, nt)
            if i % 4 == 2:
                sampler = (bfi.SAMPLE_GAUSSIAN, bfi.gaussian_proposal(lat, 4.0))
            ctx.set_sampler(sampler[0], d, factor=sampler[1])
            p_s, p_t = _plan(bfi, lat, lo, hi, samples, 9, sid, precision, sampler)
            for want in (True, False, True):  # planned, then the plan kept
                c_s, c_t = ctx.integrate(lat, lo, hi, samples, 9, sub_id=sid, precision=precision, want_slots=want)
                assert np.array_equal(c_t, p_t, equal_nan=True), (i, n, want)
                assert not want or np.array_equal(c_s, p_s, equal_nan=True), (i, n)
    finally:
        ctx.close()
