"""Performance cases: the integrations that a user of the package runs.

A case is a dict of plain values; its "kind" says which public entry point the
pass goes through:

  plan       Plan.execute on boxes that lie on the device (box sampler)
  call       Context.integrate, host arrays in and out
  transform  Plan.execute with the range map over [-1, 1]^d
  gaussian   Plan.execute with Gaussian importance sampling
  adaptive   Context.adaptive_integrate (subdivision with the convergence test)
  batch      Batch.launch, uneven jobs in one CUDA graph
  serving    Server.submit of a burst of jobs with adaptive splitting, then
             every result

prepare() makes what the caller holds before the call (boxes, budgets, the
plan, batch or server); run() is one pass; exact() is the same estimator in
plain 64-bit torch on the same Philox points, for cases small enough.
"""
import math
import random

import numpy as np
import torch

import paper_1803_07560_gb300 as bfi

# Nx, Nt of the mixed workloads (batching and serving)
MIX_NX = (4, 6, 8, 10, 16, 32)
MIX_NT = (2, 4)
# shapes of drawn single plans: the mixed workloads', the big serving lattice
# and shapes without a kernel of their own
FAST_SHAPES = ((4, 2), (6, 2), (8, 2), (10, 2), (16, 2), (32, 2), (4, 4), (6, 4), (8, 4), (10, 4), (16, 4))
LANE_SHAPES = ((32, 4), (64, 8), (64, 4))
OTHER_SHAPES = ((5, 3), (7, 3), (12, 2), (12, 3), (20, 4))
# coordinates (samples x d) that exact() works through in about 20 s
EXACT_LIMIT = 3 << 33


def listed():
    return [
        # The smallest job of the paper's method: one volume, no subdivision, a million points.
        {"name": "plan_4x2_one_volume_f64", "kind": "plan", "nx": 4, "nt": 2, "nsub": 1, "per": 1 << 20,
         "ragged": 0, "nu": 1.0, "fp32": False},
        # A single small request from host arrays, a few subvolumes with uneven budgets: what one line of the
        # line protocol or one refinement step costs, launches and copies included.
        {"name": "call_10x2_ragged_f64", "kind": "call", "nx": 10, "nt": 2, "nsub": 3, "per": 40003,
         "ragged": 1237, "nu": 1.0, "fp32": False},
        # The paper's shape: 1024 subvolumes with a million points each (Sec. 4), full precision.
        {"name": "plan_10x2_paper_f64", "kind": "plan", "nx": 10, "nt": 2, "nsub": 1024, "per": 1 << 20,
         "ragged": 0, "nu": 1.0, "fp32": False},
        # The same with the doubled budget of the convergence test (2 10^6 points), single-precision evaluation:
        # the form that long runs use.
        {"name": "plan_10x2_paper_f32", "kind": "plan", "nx": 10, "nt": 2, "nsub": 1024, "per": 1 << 21,
         "ragged": 0, "nu": 1.0, "fp32": True},
        # A shape without a kernel of its own, odd sizes and budgets: a user's own lattice.
        {"name": "plan_7x3_odd_f64", "kind": "plan", "nx": 7, "nt": 3, "nsub": 37, "per": 54321, "ragged": 17,
         "nu": 0.7, "fp32": False},
        # The wide lattice of the mixed workloads, alone, in double precision.
        {"name": "plan_32x4_f64", "kind": "plan", "nx": 32, "nt": 4, "nsub": 256, "per": 1 << 16, "ragged": 0,
         "nu": 1.0, "fp32": False},
        # The big lattice of the serving stream, alone.
        {"name": "plan_64x8_f32", "kind": "plan", "nx": 64, "nt": 8, "nsub": 256, "per": 1 << 14, "ragged": 0,
         "nu": 1.0, "fp32": True},
        # The infinite range mapped to (-1, 1) as in Sec. 4, over bisected boxes.
        {"name": "transform_10x2_f64", "kind": "transform", "nx": 10, "nt": 2, "nsub": 256, "per": 1 << 16,
         "ragged": 0, "nu": 1.0},
        # Importance sampling of the whole box as one volume (Sec. 5).
        {"name": "gaussian_10x2_f64", "kind": "gaussian", "nx": 10, "nt": 2, "nsub": 1, "per": 1 << 22,
         "ragged": 0, "nu": 1.0, "sigma0": 6.0},
        # Adaptive subdivision with the convergence test (Sec. 3): many rounds, each planned from host arrays.
        {"name": "adaptive_10x2_f64", "kind": "adaptive", "nx": 10, "nt": 2, "n": 1 << 16, "nu": 1.0,
         "rel_tol": 0.2, "max_depth": 10, "max_leaves": 4096},
        # Uneven jobs of the batching workload in one graph.
        {"name": "batch_32_jobs_f32", "kind": "batch", "jobs": 32, "pick": 3, "log2_lo": 20.0, "log2_hi": 28.0,
         "fp32": True},
        # A burst of the serving stream: mixed jobs and a 64x8, subvolumes of high variance split.
        {"name": "serving_16_jobs_f32", "kind": "serving", "jobs": 16, "pick": 5, "log2_lo": 20.0, "log2_hi": 25.0,
         "big": 1},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plan", "plan", "plan", "plan", "plan", "call", "call", "transform", "gaussian", "adaptive",
                       "batch", "serving"])
    nu = round(math.exp(rng.uniform(math.log(0.1), math.log(10.0))), 4)
    if kind in ("plan", "call"):
        shape, cap = rng.choice([(FAST_SHAPES, 1 << 34), (FAST_SHAPES, 1 << 34), (((10, 2),), 1 << 34),
                                 (LANE_SHAPES, 1 << 33), (OTHER_SHAPES, 1 << 30)])
        nx, nt = rng.choice(shape)
        # samples in total: 2^16 to the cap's worth of coordinates (at most 2^30 samples)
        total = _log_int(rng, 1 << 16, min(1 << 30, cap // (nx * nt)))
        if kind == "call":
            total = min(total, 1 << 24)
        nsub = _log_int(rng, 1, 1024)
        return {"kind": kind, "nx": nx, "nt": nt, "nsub": nsub, "per": max(64, total // nsub),
                "ragged": rng.choice([0, 0, 1, 17]), "nu": nu, "fp32": rng.random() < 0.5}
    if kind == "transform":
        nx, nt = rng.choice([(4, 2), (8, 2), (10, 2), (10, 2), (6, 4), (8, 4)])
        total = _log_int(rng, 1 << 17, (1 << 28) // (nx * nt))
        nsub = _log_int(rng, 1, 1024)
        return {"kind": kind, "nx": nx, "nt": nt, "nsub": nsub, "per": max(64, total // nsub),
                "ragged": rng.choice([0, 1, 17]), "nu": nu}
    if kind == "gaussian":
        nx, nt = rng.choice([(4, 2), (8, 2), (10, 2), (10, 2), (6, 4), (8, 4)])
        total = _log_int(rng, 1 << 17, (1 << 27) // (nx * nt))
        nsub = _log_int(rng, 1, 16)
        return {"kind": kind, "nx": nx, "nt": nt, "nsub": nsub, "per": max(64, total // nsub),
                "ragged": rng.choice([0, 1, 17]), "nu": nu, "sigma0": round(rng.uniform(3.0, 8.0), 3)}
    if kind == "adaptive":
        nx, nt = rng.choice([(4, 2), (6, 2), (8, 2), (10, 2)])
        return {"kind": kind, "nx": nx, "nt": nt, "n": _log_int(rng, 1 << 11, 1 << 17), "nu": nu,
                "rel_tol": round(rng.uniform(0.1, 0.4), 3), "max_depth": rng.randint(5, 10), "max_leaves": 4096}
    if kind == "batch":
        hi = rng.uniform(22.0, 26.0)
        return {"kind": kind, "jobs": rng.randint(6, 32), "pick": rng.randrange(1 << 20), "log2_lo": 20.0,
                "log2_hi": round(hi, 3), "fp32": rng.random() < 0.75}
    return {"kind": kind, "jobs": rng.randint(4, 16), "pick": rng.randrange(1 << 20), "log2_lo": 18.0,
            "log2_hi": round(rng.uniform(20.0, 24.0), 3), "big": rng.choice([0, 1])}


def _boxes(d, nsub, half):
    """nsub subvolumes of [-half, half]^d: the first nsub of 2^k bisections along the coordinates in turn."""
    k = max(0, (nsub - 1).bit_length())
    s = np.arange(nsub)
    lo, hi = np.full((nsub, d), -half), np.full((nsub, d), half)
    for j in range(min(d, k)):
        at, bits = np.zeros(nsub, dtype=np.int64), list(range(j, k, d))
        for b in bits:
            at = 2 * at + ((s >> b) & 1)
        width = 2.0 * half / (1 << len(bits))
        lo[:, j], hi[:, j] = -half + at * width, -half + (at + 1) * width
    return lo, hi


def _budgets(case):
    return np.array([case["per"] + case["ragged"] * s for s in range(case["nsub"])], dtype=np.uint64)


def _mixed_jobs(case):
    """The jobs of a batch or a burst: shapes, viscosities, subvolumes and budgets of the mixed workloads."""
    rng, jobs = random.Random(case["pick"]), []
    for k in range(case["jobs"]):
        nx, nt = rng.choice(MIX_NX), rng.choice(MIX_NT)
        if k < case.get("big", 0):
            nx, nt = 64, 8
        nu = math.exp(rng.uniform(math.log(0.1), math.log(10.0)))
        levels = rng.randint(6, 10)
        total = math.exp(rng.uniform(case["log2_lo"] * math.log(2.0), case["log2_hi"] * math.log(2.0)))
        if (nx, nt) == (64, 8):
            total = min(total, float(1 << 22))
        nsub = 1 << min(levels, nx * nt)
        jobs.append({"nx": nx, "nt": nt, "nu": nu, "nsub": nsub, "per": max(64, int(total) // nsub), "ragged": 0})
    return jobs


def _precision(case):
    return bfi.FP32 if case.get("fp32") else bfi.FP64


def _on_gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def prepare(case, seed):
    kind, seed = case["kind"], int(seed) & 0xFFFFFFFF
    state = {"kind": kind, "seed": seed}
    if kind in ("plan", "call", "transform", "gaussian"):
        lat = bfi.lattice(case["nx"], case["nt"], nu=case["nu"])
        d = case["nx"] * case["nt"]
        lo, hi = _boxes(d, case["nsub"], 1.0 if kind == "transform" else 5.0)
        budgets = _budgets(case)
        if kind == "call":
            state.update(ctx=bfi.Context(), lat=lat, lo=lo, hi=hi, budgets=budgets, precision=_precision(case))
            return state
        plan = bfi.Plan(lat, budgets, _precision(case))
        if kind == "transform":
            plan.set_sampler(bfi.SAMPLE_TRANSFORM)
        elif kind == "gaussian":
            plan.set_sampler(bfi.SAMPLE_GAUSSIAN, factor=bfi.gaussian_proposal(lat, case["sigma0"]))
        state.update(plan=plan, lo=_on_gpu(lo), hi=_on_gpu(hi))
    elif kind == "adaptive":
        d = case["nx"] * case["nt"]
        state.update(ctx=bfi.Context(), lat=bfi.lattice(case["nx"], case["nt"], nu=case["nu"]), lo=np.full(d, -5.0),
                     hi=np.full(d, 5.0), n=case["n"],
                     conv=bfi.convergence(2.0, rel_tol=case["rel_tol"], max_depth=case["max_depth"],
                                          max_leaves=case["max_leaves"]))
    elif kind == "batch":
        jobs = []
        for k, j in enumerate(_mixed_jobs(case)):
            lo, hi = _boxes(j["nx"] * j["nt"], j["nsub"], 5.0)
            jobs.append({"lattice": bfi.lattice(j["nx"], j["nt"], nu=j["nu"]), "samples": _budgets(j),
                         "lo": _on_gpu(lo), "hi": _on_gpu(hi), "seed": seed, "job_id": k})
        state.update(batch=bfi.Batch(jobs, _precision(case)))
    else:
        jobs = []
        for j in _mixed_jobs(case):
            lo, hi = _boxes(j["nx"] * j["nt"], j["nsub"], 5.0)
            jobs.append((bfi.lattice(j["nx"], j["nt"], nu=j["nu"]), lo, hi, _budgets(j)))
        state.update(server=bfi.Server(precision=bfi.FP32, split_rel_var=1e-2, max_split_rounds=2), jobs=jobs)
    return state


def run(state):
    kind, seed = state["kind"], state["seed"]
    if kind in ("plan", "transform", "gaussian"):
        return state["plan"].execute(state["lo"], state["hi"], seed)
    if kind == "call":
        return state["ctx"].integrate(state["lat"], state["lo"], state["hi"], state["budgets"], seed,
                                      precision=state["precision"])
    if kind == "adaptive":
        totals, stats = state["ctx"].adaptive_integrate(state["lat"], state["lo"], state["hi"], state["n"], seed,
                                                        state["conv"])
        return totals, stats.as_dict()
    if kind == "batch":
        state["batch"].launch()
        return state["batch"].slots, state["batch"].totals
    requests = [state["server"].submit(lat, lo, hi, budgets, seed, job_id=k)
                for k, (lat, lo, hi, budgets) in enumerate(state["jobs"])]
    results = []
    for r in requests:
        r.wait(120_000)
        results.append(r.result())  # the totals; how many leaf records there are follows from the splitting
        r.release()
    return results


def _parts(case):
    """(nx, nt, nsub, samples) of every integration of a pass, as far as the case fixes them."""
    if case["kind"] in ("batch", "serving"):
        return [(j["nx"], j["nt"], j["nsub"], int(_budgets(j).sum())) for j in _mixed_jobs(case)]
    if case["kind"] == "adaptive":  # the first evaluation of every subvolume of a full tree is the least it can do
        return [(case["nx"], case["nt"], 1 << case["max_depth"], 3 * case["n"] << case["max_depth"])]
    return [(case["nx"], case["nt"], case["nsub"], int(_budgets(case).sum()))]


def work(case):
    """Bytes: boxes and budgets in, records and totals out.  Flops: the definition's own for each sample, the
    point (2 per coordinate) and the action (8 per coordinate); the random words and the few evaluations of
    samples that carry weight are not counted."""
    nbytes = flops = 0
    for nx, nt, nsub, n in _parts(case):
        d, r = nx * nt, nx // 2 + 1
        nbytes += 8 * (nsub * (2 * d + 1 + 5 + 3 * r) + 4 + 2 * r)
        flops += n * 10 * d
    return {"bytes": nbytes, "flops": flops}


# ---- exact(): the estimator in 64 bits, in plain torch ----

def _philox(seed, job, sub, first, count, blocks, device):
    """Words of samples first .. first + count - 1: [count, 4 blocks] int64 (Philox4x32-10 of Salmon et al.,
    counter (block, index low, index high, sub), key (seed, job))."""
    mask = 0xFFFFFFFF
    i = torch.arange(first, first + count, device=device, dtype=torch.int64)[:, None]
    c0 = torch.arange(blocks, device=device, dtype=torch.int64)[None, :].expand(count, blocks)
    c1 = (i & mask).expand(count, blocks)
    c2 = (i >> 32).expand(count, blocks)
    c3 = torch.full((1, 1), sub, device=device, dtype=torch.int64).expand(count, blocks)
    k0, k1 = seed & mask, job & mask
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57  # 64 bits, wrapped: the high halves are masked below
        c0, c1, c2, c3 = (((p1 >> 32) & mask) ^ c1 ^ k0, p1 & mask, ((p0 >> 32) & mask) ^ c3 ^ k1, p0 & mask)
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return torch.stack((c0, c1, c2, c3), dim=2).reshape(count, 4 * blocks)


def _proposal(nx, nt, nu, sigma0):
    """F = L^-T of the Cholesky factor of the linear limit's quadratic form plus I / sigma0^2."""
    d = nx * nt
    b = np.zeros((d, d))
    for j in range(d):
        m, l = divmod(j, nt)
        b[j, m * nt + (l + 1) % nt] += 1.0
        b[j, j] += 2.0 * nu - 1.0
        b[j, ((m + 1) % nx) * nt + l] -= nu
        b[j, ((m - 1) % nx) * nt + l] -= nu
    return np.linalg.inv(np.linalg.cholesky(b.T @ b + np.eye(d) / sigma0 ** 2)).T


def _sums(part, case, lo, hi, n, sub, seed, job, device):
    """(n, shift, log volume, [sum w, w^2, w P_r, w^2 P_r, w^2 P_r^2]) of one subvolume."""
    nx, nt = part["nx"], part["nt"]
    d, r_max, kind = nx * nt, nx // 2, case["kind"]
    lo_t, hi_t = torch.from_numpy(lo).to(device), torch.from_numpy(hi).to(device)
    log_v, factor = float(np.sum(np.log(hi - lo))), None
    if kind == "gaussian":
        f = _proposal(nx, nt, part["nu"], case["sigma0"])
        factor, log_v = torch.from_numpy(f).to(device), 0.5 * d * math.log(2.0 * math.pi) + np.linalg.slogdet(f)[1]
    step = max(1, min(n, (1 << 25) // d))
    shift, sums = math.inf, torch.zeros(2 + 3 * (r_max + 1), dtype=torch.float64, device=device)
    for first in range(0, n, step):
        count = min(step, n - first)
        w = _philox(seed, job, sub, first, count, (d + (d % 2 if kind == "gaussian" else 0) + 3) // 4, device)
        log_j = 0.0
        if kind == "gaussian":
            u = (w[:, :d + d % 2].double() + 0.5) * 2.0 ** -32
            r = torch.sqrt(-2.0 * torch.log(u[:, 0::2]))
            t = 2.0 * math.pi * u[:, 1::2]
            z = torch.stack((r * torch.cos(t), r * torch.sin(t)), dim=2).reshape(count, -1)[:, :d]
            v, log_j = z @ factor.T, 0.5 * (z * z).sum(1)
        elif case.get("fp32"):  # the points of the single-precision form are floats
            u = ((w[:, :d] >> 9).double() + 0.5) * 2.0 ** -23
            v = (u * (hi_t - lo_t).float().double() + lo_t.float().double()).float().double()
        else:
            v = (w[:, :d].double() + 0.5) * 2.0 ** -32 * (hi_t - lo_t) + lo_t
            if kind == "transform":
                one_m = (1.0 - v) * (1.0 + v)
                log_j = (torch.log1p(v * v) - 2.0 * torch.log(one_m)).sum(1)
                v = v / one_m
        del w
        f = v.reshape(count, nx, nt)
        right, left = f.roll(-1, 1), f.roll(1, 1)
        res = f.roll(-1, 2) - f + f * (right - left) / 2.0 - part["nu"] * (right - 2.0 * f + left)
        s = 0.5 * (res * res).sum((1, 2)) - log_j
        if kind == "gaussian":
            keep = ((v >= lo_t) & (v < hi_t)).all(1)
            f, s = f[keep], s[keep]
        if not s.numel():
            continue
        low = min(shift, float(s.min()))
        if shift < math.inf:
            a = math.exp(low - shift)
            sums[0], sums[1] = sums[0] * a, sums[1] * a * a
            sums[2:3 + r_max] *= a
            sums[3 + r_max:] *= a * a
        shift, weight = low, torch.exp(low - s)
        near = weight > 1e-30  # the others are below the last bit of every sum
        f, weight = f[near], weight[near]
        sums[0] += weight.sum()
        sums[1] += (weight * weight).sum()
        for r in range(r_max + 1):
            p = (f * f.roll(-r, 1)).sum((1, 2)) / d
            sums[2 + r] += (weight * p).sum()
            sums[3 + r_max + r] += (weight * weight * p).sum()
            sums[4 + 2 * r_max + r] += (weight * weight * p * p).sum()
    return float(n), shift, log_v, sums.cpu().numpy()


def _totals(records, r_max):
    """ln Z, its relative error, samples, subvolumes, C(r) and their errors (delta method)."""
    records = [q for q in records if q[0] > 0]
    some = [q for q in records if q[3][0] > 0]
    top = max(v - math.log(n) - m for n, m, v, _ in some)
    f = np.array([math.exp(v - math.log(n) - m - top) for n, m, v, _ in some])
    n = np.array([q[0] for q in some])
    s = np.stack([q[3] for q in some])
    z = float((f * s[:, 0]).sum())
    g = f * f / np.maximum(n - 1.0, 1e-300)
    v_z = n * s[:, 1] - s[:, 0] ** 2
    out = np.zeros(4 + 2 * (r_max + 1))
    out[:4] = top + math.log(z), math.sqrt(max(0.0, float((g * v_z).sum()))) / z, sum(q[0] for q in records), len(records)
    for r in range(r_max + 1):
        a, b, c2 = s[:, 2 + r], s[:, 3 + r_max + r], s[:, 4 + 2 * r_max + r]
        c = float((f * a).sum()) / z
        var = float((g * (n * c2 - a * a - 2.0 * c * (n * b - s[:, 0] * a) + c * c * v_z)).sum())
        out[4 + r], out[5 + r_max + r] = c, math.sqrt(max(0.0, var)) / z
    return out


def exact(case, seed):
    """The totals in 64 bits; the records have no such value, since each is relative to a shift of the
    implementation's choice.  None for adaptive and serving runs, whose subvolumes follow from the results."""
    kind, seed = case["kind"], int(seed) & 0xFFFFFFFF
    if kind in ("adaptive", "serving"):
        return None
    parts = _mixed_jobs(case) if kind == "batch" else [case]
    if sum(int(_budgets(p).sum()) * p["nx"] * p["nt"] for p in parts) > EXACT_LIMIT:
        return None
    device = "cuda" if torch.cuda.is_available() else "cpu"
    totals = []
    for k, p in enumerate(parts):
        lo, hi = _boxes(p["nx"] * p["nt"], p["nsub"], 1.0 if kind == "transform" else 5.0)
        records = [_sums(p, case, lo[s], hi[s], int(n), s, seed, k, device) for s, n in enumerate(_budgets(p))]
        totals.append(_totals(records, p["nx"] // 2))
    return ([None] * len(parts), totals) if kind == "batch" else (None, totals[0])
