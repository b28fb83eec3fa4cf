"""The range map over boxes next to y = +-1, where v and the Jacobian grow
without bound: slabs whose samples' FP32 Jacobian products overflow, and slabs
whose samples' intervals are about as wide as a record's margin, records and
shifts against the plain FP64 estimator and the shift rule."""
import numpy as np
import pytest

import oracle
from oracle.maps import TRANSFORM, integrate_mapped, log_jacobian, transform

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(bfi, lat, lo, hi, samples, seed, sid):
    plan = bfi.Plan(lat, samples, bfi.FP64)
    plan.set_sampler(bfi.SAMPLE_TRANSFORM)
    dev = torch.device("cuda:0")
    s, t = plan.execute(torch.tensor(lo, device=dev), torch.tensor(hi, device=dev), seed,
                        sub_id=torch.tensor(sid.astype(np.int32), device=dev))
    torch.cuda.synchronize()
    evaluated = plan.stats()[0]
    plan.close()
    return s.cpu().numpy(), t.cpu().numpy(), evaluated


def _action(lat, lo, hi, sid, seed, n):
    """Points, S_eff, and the magnitude that a relative error of every v and 1 - y^2 is multiplied by in S_eff."""
    y = oracle.points(lat.nx * lat.nt, lo, hi, sid, seed, 0, 0, n)
    v = transform(y).reshape(n, lat.nx, lat.nt)
    c_adv, c_dif = lat.nonlinear * lat.tau / (2 * lat.a), lat.nu * lat.tau / lat.a ** 2
    nxt, right, left = np.roll(v, -1, 2), np.roll(v, -1, 1), np.roll(v, 1, 1)
    R = nxt + v * (c_adv * (right - left) + 2 * c_dif - 1) - c_dif * (right + left)
    T = abs(nxt) + abs(v) * (2 * c_adv * (abs(right) + abs(left)) + abs(2 * c_dif - 1)) + c_dif * (abs(right) + abs(left))
    S = oracle.eval_points(lat, v.reshape(n, -1))[0]
    lj = log_jacobian(y).sum(axis=1)
    size = (2 * abs(R) * T).sum(axis=(1, 2)) / (2 * lat.D * lat.tau) + S + abs(lj) + 2 * y.shape[1]
    return y, S - lj, size


def _shift(S, chunk):
    """Smallest thread shift (256 threads a chunk: the first action, then any more than 16 below)."""
    rows = chunk // 256
    pad = np.full(-(-S.size // chunk) * chunk, np.inf)
    pad[:S.size] = S
    pad = pad.reshape(-1, rows, 256)
    m = np.full((pad.shape[0], 256), np.inf)
    for r in range(rows):
        m = np.where(pad[:, r] < m - 16.0, pad[:, r], m)
    return m.min()


def _check(bfi, nx, nt, nu, D, nonlinear, lo, hi, samples, seed=21):
    d = nx * nt
    sid = np.arange(4, 4 + len(samples), dtype=np.uint32)
    par = dict(nu=nu, D=D, nonlinear=nonlinear)
    g_s, g_t, evaluated = _run(bfi, bfi.lattice(nx, nt, **par), lo, hi, samples, seed, sid)
    lat = oracle.lattice(nx, nt, **par)
    o_s, _ = integrate_mapped(lat, lo, hi, samples, seed, sub_id=sid, kind=TRANSFORM)
    assert np.all(np.isfinite(g_s)) and np.all(np.isfinite(g_t))
    R, chunk, facts = nx // 2 + 1, bfi.chunking(samples).chunk_samples, []
    for s, n in enumerate(samples.astype(int)):
        y, S, size = _action(lat, lo[s], hi[s], int(sid[s]), seed, n)
        facts.append((y, S))
        m = _shift(S, chunk)
        # v and S_eff carry some ten roundings on either side, each of 2^-53 of 'size': an error of the weights'
        # exponents, twice of their squares'; 1e-12 is the rest's
        err = 20 * 2.0 ** -53 * size[S <= S.min() + 60].max()
        assert abs(g_s[s, 1] - m) <= err + 1e-12 * abs(m), (s, g_s[s, 1], m)
        a, b = g_s[s], o_s[s]
        f = np.exp(b[1] - a[1])  # records at one shift
        for k in range(3, 5 + 3 * R):
            sq = k == 4 or k >= 5 + R
            want = b[k] * (1.0 / (f * f) if sq else 1.0 / f)
            scale = {0: a[3], 1: a[4]}.get(k - 3, None)
            if scale is None:  # |P_r| <= P_0
                scale = a[5] if k < 5 + R else (a[5 + R] if k < 5 + 2 * R else a[5 + 2 * R])
            tol = 1e-12 + 2 * err
            assert abs(a[k] - want) <= tol * abs(scale), (s, k, a[k], want, tol)
    return facts, evaluated


@pytest.mark.parametrize("nx,nt,nu,D,nonlinear,k,at,side,n", [
    (2, 2, 0.1, 30.0, 1.0, 10, 4, 1, 1 << 22), (2, 2, 1.0, 100.0, 1.0, 10, 4, -1, 1 << 21),
    (2, 2, 0.1, 1.0, 1.0, 8, 4, 1, 1 << 21), (4, 2, 0.1, 10.0, 0.0, 10, 4, 1, 1 << 20),
    (4, 2, 1.0, 1.0, 0.0, 8, 4, -1, 1 << 20), (4, 2, 1.0, 100.0, 1.0, 6, 8, 1, 1 << 20),
    (10, 2, 0.1, 1000.0, 0.0, 9, 4, 1, 200_003)])
def test_slabs(bfi, nx, nt, nu, D, nonlinear, k, at, side, n):
    """The first 'at' coordinates within 2^-k of +1 or -1, the others over (-1, 1)."""
    d = nx * nt
    lo, hi = -np.ones((2, d)), np.ones((2, d))
    if side > 0:
        lo[:, :at] = 1.0 - 2.0 ** -k
    else:
        hi[:, :at] = -1.0 + 2.0 ** -k
    _check(bfi, nx, nt, nu, D, nonlinear, lo, hi, np.array([n, 3001], dtype=np.uint64))


@pytest.mark.parametrize("nx,nt,k", [(4, 2, 12), (10, 2, 12), (32, 2, 12)])
def test_path(bfi, nx, nt, k):
    """The whole cube is screened; a cube within 2^-k of +1, whose hint has an interval far wider than a record's
    margin (S ~ 4^k, its relative width above 2^-14), is evaluated throughout."""
    d, n = nx * nt, np.array([40_001], dtype=np.uint64)
    lat, sid, one = bfi.lattice(nx, nt), np.zeros(1, dtype=np.uint32), np.ones((1, d))
    assert 0 < _run(bfi, lat, -one, one, n, 3, sid)[2] < 40_001 // 2
    assert _run(bfi, lat, one - 2.0 ** -k, one, n, 3, sid)[2] == 40_001


@pytest.mark.parametrize("nx,nt,D,k,n", [
    (2, 2, 4.0 ** 12, 12, 20_000), (2, 2, 1e6, 12, 1 << 21), (2, 2, 1e6, 13, 70_001), (2, 2, 1e7, 14, 70_001), (2, 2, 4.0 ** 16, 16, 1 << 15), (4, 2, 4.0 ** 18, 12, 70_001),
    (2, 2, 4.0 ** 16, 16, 1 << 22)])
def test_open_threads(bfi, nx, nt, D, k, n):
    """Slabs where samples may or may not have moved their threads' shifts."""
    d = nx * nt
    _check(bfi, nx, nt, 0.1, D, 1.0, np.full((2, d), 1.0 - 2.0 ** -k), np.ones((2, d)), np.array([n, 700], dtype=np.uint64))


def test_open_threads_time(bfi):
    """Following the open threads costs no more than a few times an evaluation of every sample (which a box that
    leaves [-1, 1] gets)."""
    lat, n, dev = bfi.lattice(2, 2, D=4.0 ** 16), np.full(8, 1 << 15, dtype=np.uint64), torch.device("cuda:0")
    plan = bfi.Plan(lat, n, bfi.FP64)
    plan.set_sampler(bfi.SAMPLE_TRANSFORM)
    hi = torch.ones((8, 4), dtype=torch.float64, device=dev)
    ms = []
    for lo in (hi - 2.0 ** -16, -1.5 * hi):
        times = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            plan.execute(lo, hi, 9)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        ms.append(min(times[2:]))
    plan.close()
    assert ms[0] < 3.0 * ms[1], ms


@pytest.mark.parametrize("nx,nt,nonlinear,k,D,n", [
    (2, 2, 1.0, 32, 2.0 ** 48, 1 << 18), (2, 2, 1.0, 34, 2.0 ** 52, 1 << 18), (10, 2, 0.0, 34, 2.0 ** 52, 1 << 16),
    (2, 2, 1.0, 36, 2.0 ** 56, 5000), (2, 2, 1.0, 24, 2.0 ** 32, 1 << 18), (2, 2, 1.0, 12, 2.0 ** 8, 1 << 22)])
def test_rounded_points(bfi, nx, nt, nonlinear, k, D, n):
    """One coordinate within 2^-k of 1: samples so close to 1 that the rounding of y itself leaves the screen no bound
    (1 / (1 - y^2) > 2^40) are evaluated, whatever their action."""
    d = nx * nt
    lo = -np.ones((1, d))
    lo[0, 0] = 1.0 - 2.0 ** -k
    facts, evaluated = _check(bfi, nx, nt, 0.1, D, nonlinear, lo, np.ones((1, d)), np.array([n], dtype=np.uint64))
    y, S = facts[0]
    r = (1.0 / ((1.0 - y) * (1.0 + y))).max(axis=1)
    # the screen's 1 - y is not rounded as the evaluation's is: 2^-12 at 2^-41
    needed = (S <= S.min() + 34.0 + np.log(n)) | (r > 2.0 ** 40 * (1.0 + 2.0 ** -11))
    assert evaluated >= needed.sum(), (evaluated, needed.sum())


@pytest.mark.parametrize("nx,nt", [(2, 1), (3, 1), (4, 1), (2, 2)])
def test_residency(bfi, nx, nt):
    """The smallest lattices run three CTAs an SM (80 registers), which jobs of short chunks need."""
    plan = bfi.Plan(bfi.lattice(nx, nt), np.array([300], dtype=np.uint64), bfi.FP64)
    plan.set_sampler(bfi.SAMPLE_TRANSFORM)
    assert plan.info().ctas_per_sm_max >= 3
    plan.close()


@pytest.mark.parametrize("k,D,screened", [(0, 1.0, True), (0, 4.0 ** 8, False), (12, 1e6, True), (16, 4.0 ** 16, False),
                                          (20, 4.0 ** 30, False)])
def test_where_the_screen_gains(bfi, k, D, screened):
    """Every sample is evaluated where nearly all lie within the window, or many do and their intervals are wide."""
    n, one = np.array([300_000], dtype=np.uint64), np.ones((1, 4))
    lo = -one if k == 0 else one - 2.0 ** -k
    evaluated = _run(bfi, bfi.lattice(2, 2, D=D), lo, one, n, 3, np.zeros(1, dtype=np.uint32))[2]
    assert (evaluated < 300_000) == screened, evaluated
