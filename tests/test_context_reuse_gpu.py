"""What a context costs and keeps between calls: its creation, the plan that it
keeps while lattice, precision and budgets stay, and its device memory."""
import time

import numpy as np
import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_creation_time(bfi):
    """A stream and no page-locked memory (about 10 us; page-locking 128 KiB takes 100)."""
    bfi.Context(0).close()
    times = []
    for _ in range(30):
        t = time.perf_counter()
        ctx = bfi.Context(0)
        times.append(time.perf_counter() - t)
        ctx.close()
    assert np.median(times) < 60e-6, times


def test_kept_plan(bfi):
    """Calls in a row that differ in one thing only, small jobs (copied in one piece) and larger ones, against a
    context of their own each."""
    lat, other = bfi.lattice(10, 2), bfi.lattice(10, 2, nu=0.5)
    for n in (3, 300):
        lo, hi = workloads.bisected_boxes(20, int(np.ceil(np.log2(n))))
        lo, hi = lo[:n].copy(), hi[:n].copy()
        samples = np.full(n, 700, dtype=np.uint64)
        more = samples.copy()
        more[1] += 300
        sid = np.arange(n, dtype=np.uint32) + 7
        base = dict(lat=lat, lo=lo, hi=hi, samples=samples, seed=1, sub_id=None, precision=0, want_slots=True)
        steps = [{}, {}, dict(lo=lo - 0.25, hi=hi + 0.125), dict(seed=2), dict(sub_id=sid), {}, dict(want_slots=False),
                 dict(precision=1), {}, dict(samples=more), dict(lat=other), {}, dict(sub_id=sid, seed=3), dict(sub_id=sid + 1)]
        ctx = bfi.Context(0)
        for i, step in enumerate(steps):
            kw = {**base, **step}
            fresh = bfi.Context(0)
            a_s, a_t = ctx.integrate(**kw)
            b_s, b_t = fresh.integrate(**kw)
            fresh.close()
            assert np.array_equal(a_t, b_t, equal_nan=True), (n, i)
            assert not kw["want_slots"] or np.array_equal(a_s, b_s, equal_nan=True), (n, i)
        ctx.close()


def test_device_memory(bfi):
    """A context's buffer follows its jobs: little over a large job's need after a smaller one, and given back by a
    small job."""
    lat, small = bfi.lattice(10, 2), np.array([300], dtype=np.uint64)
    one = np.ones((1, 20))

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info(0)[0]

    def large(ctx, n):
        ctx.integrate(lat, np.repeat(-one, n, axis=0), np.repeat(one, n, axis=0), np.ones(n, dtype=np.uint64), 1)
        return n * (2 * 8 * 20 + 8 * 23 + 8 * 22 + 44)  # boxes, slots, chunk records, tables and factors

    ctx = bfi.Context(0)
    ctx.integrate(lat, -one, one, small, 1)
    before = free()
    large(ctx, 200_000)
    need = large(ctx, 210_000)
    assert before - free() < need + (40 << 20), (before - free(), need)
    ctx.integrate(lat, -one, one, small, 1)
    assert abs(before - free()) <= 4 << 20, before - free()
    ctx.close()
