"""Timed workloads of the multi-function Monte Carlo library, through its public calls.

Each case is one call (or submit / poll sequence) that a program integrating tables of
functions makes, on tables drawn as ``paper_2104_10073_gb300.workloads`` draws them: the
paper's Fig. 1 and Eq. 2 sets, single families and the mix of all four, dimensions 1..7,
budgets of 10^4 .. 10^7 samples, user functions in FP32 and FP64, stratified refinement in
up to 10 dimensions, and serving.  A seed fixes the parameters, the boxes, the budgets and
the Philox key.

``exact`` recomputes the results in FP64 with PyTorch alone: the Philox4x32-10 stream, the
23-bit fields, the box map, the integrand and the two moments.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2104_10073_gb300 import workloads as W
from paper_2104_10073_gb300 import zmc

MAX_SAMPLES = 1.4e10  # samples of the largest case
FAMILIES = {"harmonic": W.HARMONIC, "abslin": W.ABSLIN, "gauss": W.GAUSS, "poly": W.POLY}

USER_HARMONIC = {
    "f32": "__device__ float zmc_user_f(const float *x, const float *p) {\n"
           "  float ph = 0.0f;\n"
           "  for (int i = 0; i < ZMC_UDF_DIM; ++i) ph = fmaf(p[2 + i], x[i], ph);\n"
           "  float s, c; sincosf(ph, &s, &c); return p[0] * c + p[1] * s;\n}\n",
    "f64": "__device__ double zmc_user_f(const double *x, const double *p) {\n"
           "  double ph = 0.0;\n"
           "  for (int i = 0; i < ZMC_UDF_DIM; ++i) ph = fma(p[2 + i], x[i], ph);\n"
           "  return p[0] * cos(ph) + p[1] * sin(ph);\n}\n",
}
USER_PEAK = ("__device__ float zmc_user_f(const float *x, const float *p) {\n"
             "  float r2 = 0.0f;\n"
             "  for (int i = 0; i < ZMC_UDF_DIM; ++i) r2 = fmaf(x[i] - p[0], x[i] - p[0], r2);\n"
             "  return expf(-r2 / (2.0f * p[1] * p[1]));\n}\n")


def listed():
    return [
        # One function, the smallest budget in use: a program that calls the library from an
        # inner loop of its own and waits for each integral.  Latency only.
        {"name": "one_gauss_1e4", "call": "integrate", "kind": "gauss", "rows": 1, "dim": 3,
         "n_lo": 10000, "n_hi": 10000},
        # The paper's Fig. 1 set at 10^5 samples each, one blocking call.
        {"name": "fig1_1e5", "call": "integrate", "kind": "fig1", "rows": 100, "dim": 4,
         "n_lo": 10**5, "n_hi": 10**5},
        # Eq. 2: abs-linear functions in 2 and 3 dimensions at 10^6 samples, one blocking call.
        {"name": "eq2_1e6", "call": "integrate", "kind": "eq2", "rows": 100, "dim": 0,
         "n_lo": 10**6, "n_hi": 10**6},
        # A small mixed job, ragged budgets, one blocking call: what an interactive user sends.
        {"name": "mixed_job_64", "call": "integrate", "kind": "mixed", "rows": 64, "dim": 0,
         "n_lo": 10**4, "n_hi": 10**7},
        # The Fig. 1 set at its stated size with ten keys: the benchmark's table, a plan
        # prepared once and run again and again.
        {"name": "fig1x10_plan", "call": "plan", "kind": "fig1", "rows": 1000, "dim": 4,
         "n_lo": 10**6, "n_hi": 10**6},
        # 10^4 different integrations: all families, dimensions 1..7, budgets 10^4 .. 10^7.
        {"name": "mixed_1e4_plan", "call": "plan", "kind": "mixed", "rows": 10**4, "dim": 0,
         "n_lo": 10**4, "n_hi": 10**7},
        # The second half of each stream: one rank's share of a sharded table, or the next
        # piece of a progressive refinement.
        {"name": "moments_poly_5d", "call": "moments", "kind": "poly", "rows": 96, "dim": 5,
         "n_lo": 400003, "n_hi": 400003},
        # Parameter scan: one harmonic form over a lattice of wave vectors, common streams.
        {"name": "functional_1000", "call": "functional", "kind": "harmonic", "rows": 1000,
         "dim": 3, "n_lo": 10**5, "n_hi": 10**5},
        # The integrand as user code, FP32: Eq. 1 compiled at run time.
        {"name": "udf_f32_1e6", "call": "udf", "kind": "f32", "rows": 100, "dim": 4,
         "n_lo": 10**6, "n_hi": 10**6},
        # The same in FP64, for users who want every sample in double precision.
        {"name": "udf_f64_1e5", "call": "udf", "kind": "f64", "rows": 100, "dim": 4,
         "n_lo": 10**5, "n_hi": 10**5},
        # Stratified sampling with tree refinement, a localised peak in 10 dimensions.
        {"name": "normal_udf_10d", "call": "normal", "kind": "peak", "rows": 1, "dim": 10,
         "n_lo": 1 << 14, "n_hi": 1 << 14},
        # Serving: 24 jobs of different sizes arrive together, every result is waited for.
        {"name": "serving_24_jobs", "call": "serving", "kind": "mixed", "rows": 60, "dim": 0,
         "n_lo": 10**4, "n_hi": 10**7, "jobs": 24},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mean_budget(case):
    lo, hi = float(case["n_lo"]), float(case["n_hi"])
    return lo if hi <= lo else (hi - lo) / math.log(hi / lo)


def _mean_dim(case):
    return 2.5 if case["kind"] == "eq2" else float(case["dim"] or 4)


def draw(rng):
    call = rng.choice(["integrate", "integrate", "integrate", "plan", "plan", "moments",
                       "functional", "udf", "normal", "serving"])
    case = {"call": call, "kind": "mixed", "dim": 0}
    if call in ("integrate", "plan", "moments"):
        case["kind"] = rng.choice(["mixed", "mixed", "harmonic", "abslin", "gauss", "poly", "fig1"])
        case["rows"] = _log_int(rng, 1, 2000)
        if case["kind"] == "fig1":
            case["dim"] = 4
        elif case["kind"] != "mixed":
            case["dim"] = rng.randint(0, W.MAX_DIM)  # 0: a dimension per row
        if call == "moments" or rng.random() < 0.5:  # one budget for every row
            case["n_lo"] = case["n_hi"] = _log_int(rng, 10**4, 10**7)
        else:
            case["n_lo"], case["n_hi"] = sorted(_log_int(rng, 10**4, 10**7) for _ in range(2))
    elif call == "functional":
        case.update(kind=rng.choice(["harmonic", "gauss"]), dim=rng.randint(1, W.MAX_DIM),
                    rows=_log_int(rng, 10, 2000))
        case["n_lo"] = case["n_hi"] = _log_int(rng, 10**4, 10**6)
    elif call == "udf":
        case.update(kind=rng.choice(["f32", "f32", "f64"]), dim=rng.randint(1, W.MAX_DIM),
                    rows=_log_int(rng, 1, 300))
        case["n_lo"] = case["n_hi"] = _log_int(rng, 10**4, 10**6)
    elif call == "normal":
        case.update(kind=rng.choice(["peak", "gauss"]), rows=1)
        case["dim"] = rng.randint(5, 10) if case["kind"] == "peak" else rng.randint(3, W.MAX_DIM)
        case["n_lo"] = case["n_hi"] = _log_int(rng, 1000, 1 << 14)
    else:
        case.update(rows=rng.randint(1, 100), jobs=rng.randint(2, 32))
        case["n_lo"], case["n_hi"] = 10**4, rng.choice([10**6, 10**7])
    cost = _mean_budget(case) * case["rows"] * case.get("jobs", 1)
    budget = 1e8 if case["kind"] == "f64" else 0.2 * MAX_SAMPLES
    if cost > budget:
        case["rows"] = max(1, int(case["rows"] * budget / cost))
    return case


# ---------------------------------------------------------------- inputs


def _key(seed):
    return (int(seed) * 0x9E3779B97F4A7C15 + 0x2104) & 0xFFFFFFFFFFFFFFFF


def _row(rng, row, family, dim, n, key, stream):
    lo = rng.uniform(-1.0, 0.0, size=dim)
    hi = lo + rng.uniform(0.5, 2.0, size=dim)
    if family == W.HARMONIC:
        a, b = rng.uniform(0.5, 2.0, size=2)
        W.harmonic(row, a, b, rng.uniform(-30.0, 30.0, size=dim), lo, hi, n, key, stream)
    elif family == W.ABSLIN:
        W.abslin(row, rng.uniform(0.5, 2.0), rng.choice([-1.0, 1.0], size=dim), lo, hi, n, key,
                 stream)
    elif family == W.GAUSS:
        W.gauss(row, 1.0, rng.uniform(0.05, 0.5), rng.uniform(lo, hi), lo, hi, n, key, stream)
    else:
        deg = int(rng.integers(0, 5))
        W.poly(row, rng.standard_normal(size=(dim, deg + 1)), lo, hi, n, key, stream)


def _table(case, seed, job=0):
    rng = np.random.default_rng([int(seed), job, 2104])
    key = _key(int(seed) * 1000 + job)
    kind, rows = case["kind"], int(case["rows"])
    n_lo, n_hi = int(case["n_lo"]), int(case["n_hi"])
    if kind == "fig1":
        t = W.harmonic_fig1(n_lo, seeds=range((rows + 99) // 100))[:rows]
        t["seed"] += np.uint64(key & 0xFFFFFFFF)
    elif kind == "eq2":
        t = W.abslin_eq2(n_lo, gen_seed=int(seed), seed=key)[:rows]
    elif kind == "mixed":
        t = W.mixed_block(rng, rows, key, math.log10(n_lo), math.log10(n_hi))
        return t
    else:
        t = W.empty(rows)
        for i in range(rows):
            dim = int(case["dim"]) or int(rng.integers(1, W.MAX_DIM + 1))
            _row(rng, t[i], FAMILIES[kind], dim, n_lo, key, i)
    if n_hi > n_lo:
        u = rng.uniform(math.log10(n_lo), math.log10(n_hi), size=rows)
        t["n_samples"] = np.round(10.0 ** u).astype(np.uint64)
    return t


def _jobs(case, seed):
    """Tables of growing size, from a few rows to about twice case["rows"]."""
    jobs = int(case["jobs"])
    return [_table({**case, "rows": 1 + (int(case["rows"]) * 2 * (j + 1) - 1) // jobs}, seed, j)
            for j in range(jobs)]


def _lattice(case, seed):
    """Base row, slots and values of a scan: the harmonic's wave vector, or the Gaussian's
    width and first mean."""
    rng = np.random.default_rng([int(seed), 2104])
    dim, n = int(case["dim"]), int(case["n_lo"])
    base = W.empty(1)
    if case["kind"] == "harmonic":
        W.harmonic(base[0], 1.0, 1.0, np.ones(dim), np.zeros(dim), np.ones(dim), n, _key(seed), 3)
        slots = [zmc.slot_p(2 + i) for i in range(dim)]
        values = rng.uniform(-30.0, 30.0, size=(int(case["rows"]), dim))
    else:
        W.gauss(base[0], 1.0, 0.1, np.full(dim, 0.5), np.zeros(dim), np.ones(dim), n, _key(seed), 3)
        slots = [zmc.slot_p(1), zmc.slot_p(2)]
        values = np.stack([rng.uniform(0.05, 0.5, size=int(case["rows"])),
                           rng.uniform(0.0, 1.0, size=int(case["rows"]))], axis=1)
    return base, slots, values


def _user_table(case, seed):
    t = _table({**case, "kind": "harmonic"}, seed)
    t["family"] = W.USER
    return t


def _normal(case, seed):
    """Box, parameters and options of a stratified run."""
    rng = np.random.default_rng([int(seed), 2104])
    dim = int(case["dim"])
    p = np.array([0.25 + rng.uniform(-0.05, 0.05), rng.uniform(0.09, 0.12)])
    opts = dict(divisions=2, depth=2, samples_per_cell=int(case["n_lo"]), sigma_mult=3.0,
                seed=_key(seed) >> 1, max_leaves=8 << 10)
    return np.zeros(dim), np.ones(dim), p, opts


class State:
    """A program's handles and inputs: released in order when the state goes."""

    def __init__(self, case):
        self.call = case["call"]
        self.ctx = self.plan = self.udf = None

    def __del__(self):
        try:
            if self.plan is not None:
                zmc.zmc_plan_destroy(self.plan)
            if self.udf is not None:
                self.udf.close()
            if self.ctx is not None:
                self.ctx.close()
        except Exception:
            pass


def prepare(case, seed):
    s = State(case)
    s.kind = case["kind"]
    serving = s.call == "serving"
    s.ctx = zmc.Context(arena_bytes=(1 << 30) if serving else (256 << 20), serving=serving)
    if s.call in ("integrate", "plan", "moments"):
        s.table = _table(case, seed)
        if s.call == "plan":
            s.plan = zmc.zmc_plan_create(s.ctx.handle, s.table)
        if s.call == "moments":
            s.end = s.table["n_samples"].copy()
            s.begin = s.end // np.uint64(10) * np.uint64(5)  # a multiple of 5, half way
    elif s.call == "functional":
        s.base, s.slots, s.values = _lattice(case, seed)
    elif s.call == "udf":
        s.table = _user_table(case, seed)
        s.udf = zmc.Udf(USER_HARMONIC[case["kind"]], int(case["dim"]),
                        zmc.ZMC_UDF_F32 if case["kind"] == "f32" else zmc.ZMC_UDF_F64,
                        amplitude=4.0)
    elif s.call == "normal":
        s.lo, s.hi, s.p, opts = _normal(case, seed)
        s.opts = zmc.normal_options(**opts)
        if case["kind"] == "peak":
            s.udf = zmc.Udf(USER_PEAK, int(case["dim"]), zmc.ZMC_UDF_F32, amplitude=1.0)
        else:
            s.base = W.empty(1)
            W.gauss(s.base[0], 1.0, s.p[1], np.full(int(case["dim"]), s.p[0]), s.lo, s.hi,
                    2, 0, 0)
    else:
        s.jobs = _jobs(case, seed)
    return s


def _fields(res, names=("estimate", "stderr", "n", "status")):
    return {k: np.ascontiguousarray(res[k]) for k in names}


def run(s):
    h = s.ctx.handle
    if s.call == "integrate":
        return _fields(zmc.zmc_integrate(h, s.table))
    if s.call == "plan":
        zmc.zmc_plan_run(s.plan)
        return _fields(zmc.zmc_plan_results(s.plan, len(s.table)))
    if s.call == "moments":
        return _fields(zmc.zmc_integrate_moments(h, s.table, s.begin, s.end),
                       ("mean", "m2", "n", "status"))
    if s.call == "functional":
        return _fields(zmc.zmc_integrate_functional(h, s.base[0], s.slots, s.values, False))
    if s.call == "udf":
        return _fields(s.udf.integrate(h, s.table))
    if s.call == "normal":
        if s.kind == "peak":
            return s.udf.normal_integrate(h, s.lo, s.hi, s.p, s.opts)
        return zmc.zmc_normal_integrate(h, s.base[0], s.opts)
    ids = [zmc.zmc_submit(h, t) for t in s.jobs]
    out = []
    for j, t in zip(ids, s.jobs):
        st, res = zmc.zmc_poll(h, j, len(t))
        if st != zmc.ZMC_OK:
            raise RuntimeError(f"job {j}: status {st}")
        out.append(res)
    return _fields(np.concatenate(out))


# ---------------------------------------------------------------- work


def work(case):
    """Bytes: the descriptors in, the results out.  Operations, 32-bit integer and FP32: per
    coordinate a fifth of a Philox4x32-10 block (40 operations), its share of the field shifts
    and the mask (1.8) and one multiply-add of the integrand (2); per sample the function
    itself and the two sums."""
    rows = int(case["rows"]) * int(case.get("jobs", 1))
    samples, dim, kind = _mean_budget(case) * rows, _mean_dim(case), case["kind"]
    if case["call"] == "moments":
        samples *= 0.5
    if case["call"] == "normal":  # level 0 of the tree, without any refinement
        samples = float(case["n_lo"]) * 2.0 ** int(case["dim"])
    per_sample = {"harmonic": 12, "fig1": 12, "f32": 12, "f64": 12, "abslin": 2, "eq2": 2,
                  "gauss": 8, "peak": 8, "poly": 4 * dim, "mixed": 10}[kind] + 4
    return {"bytes": rows * (464.0 + 32.0), "flops": samples * (dim * 11.8 + per_sample)}


# ---------------------------------------------------------------- 64-bit results

_BATCH = 1 << 22  # samples evaluated at once


def _philox(sid, block, key):
    """Philox4x32-10 of counter (sid, block lo, block hi, 0), words as int64 tensors."""
    m32 = 0xFFFFFFFF
    c0, c1, c2 = (sid + block * 0), block & m32, (block >> 32) & m32
    c3 = torch.zeros_like(c0)
    k0, k1 = key & m32, (key >> 32) & m32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c2 = ((p1 >> 32) & m32) ^ c1 ^ k0, ((p0 >> 32) & m32) ^ c3 ^ k1
        c1, c3 = p1 & m32, p0 & m32
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return c0, c1, c2, c3


def _uniforms(sid, key, begin, count, dim):
    """u of samples [begin, begin + count), begin a multiple of 5: (streams, count, dim)."""
    first, blocks = begin * dim // 5, (count * dim + 4) // 5
    block = torch.arange(first, first + blocks, device="cuda").reshape(1, -1)
    w0, w1, w2, w3 = _philox(sid.reshape(-1, 1), block, key)
    f = torch.stack([w0, (w0 >> 23) | (w1 << 9), (w1 >> 14) | (w2 << 18), w2 >> 5,
                     (w2 >> 28) | (w3 << 4)], dim=-1)
    u = (f & 0x7FFFFF).double() * 2.0 ** -23
    return u.reshape(len(sid), -1)[:, :count * dim].reshape(len(sid), count, dim)


def _evaluate(kind, deg, x, p):
    """f at x (rows, samples, dim) with parameters p (rows, 40)."""
    d = x.shape[-1]
    q = p[:, None, :]
    if kind == W.HARMONIC:
        phase = (q[..., 2:2 + d] * x).sum(-1)
        return q[..., 0] * torch.cos(phase) + q[..., 1] * torch.sin(phase)
    if kind == W.ABSLIN:
        return q[..., 0] * (q[..., 1:1 + d] * x).sum(-1).abs()
    if kind == W.GAUSS:
        r2 = ((x - q[..., 2:2 + d]) ** 2).sum(-1)
        return q[..., 0] * torch.exp(-r2 / (2.0 * q[..., 1] ** 2))
    prod = torch.ones_like(x[..., 0])
    for i in range(d):
        v = q[..., 5 * i + deg].expand_as(prod)
        for j in range(deg - 1, -1, -1):
            v = v * x[..., i] + q[..., 5 * i + j]
        prod = prod * v
    return prod


def _moments(family, dim, deg, key, streams, lo, hi, p, begin, end):
    """(mean, M2) of each row over samples [begin, end) of its stream."""
    dev = dict(dtype=torch.float64, device="cuda")
    sid = torch.as_tensor(np.asarray(streams, dtype=np.int64), device="cuda")
    lo, w, p = (torch.as_tensor(np.ascontiguousarray(v), **dev) for v in (lo, hi - lo, p))
    rows = len(sid)
    mean, m2 = torch.zeros(rows, **dev), torch.zeros(rows, **dev)
    per = max(1, _BATCH // max(1, min(rows, _BATCH // 1000)) // 5) * 5
    for r in range(0, rows, max(1, _BATCH // per)):
        sl = slice(r, r + max(1, _BATCH // per))
        n = 0
        for b in range(begin, end, per):
            c = min(per, end - b)
            u = _uniforms(sid[sl], key, b, c, dim)
            f = _evaluate(family, deg, lo[sl, None, :] + w[sl, None, :] * u, p[sl])
            mb = f.mean(-1)
            m2b = ((f - mb[:, None]) ** 2).sum(-1)
            delta = mb - mean[sl]
            m2[sl] += m2b + delta ** 2 * (n * c / (n + c))
            mean[sl] += delta * (c / (n + c))
            n += c
    return mean.cpu().numpy(), m2.cpu().numpy()


def _exact_rows(t, begin=None, end=None, family=None):
    """Moments of every row, rows of one shape and key taken together."""
    n = t["n_samples"].astype(np.int64)
    b = np.zeros_like(n) if begin is None else np.asarray(begin, dtype=np.int64)
    e = n if end is None else np.asarray(end, dtype=np.int64)
    fam = t["family"] if family is None else np.full(len(t), family)
    groups = {}
    for i in range(len(t)):
        groups.setdefault((int(fam[i]), int(t["dim"][i]), int(t["deg"][i]), int(t["seed"][i]),
                           int(b[i]), int(e[i])), []).append(i)
    mean, m2 = np.zeros(len(t)), np.zeros(len(t))
    for (f, d, g, key, bb, ee), at in groups.items():
        s = t[at]
        mean[at], m2[at] = _moments(f, d, g, key, s["stream_id"], s["lo"][:, :d], s["hi"][:, :d],
                                    s["p"], bb, ee)
    return mean, m2


def _volume(t):
    active = np.arange(W.MAX_DIM)[None, :] < t["dim"][:, None]
    return np.prod(np.where(active, t["hi"] - t["lo"], 1.0), axis=1)


def _results(t, mean, m2, volume):
    n = t["n_samples"].astype(np.float64)
    return {"estimate": volume * mean, "stderr": volume * np.sqrt(m2 / (n * (n - 1.0))),
            "n": None, "status": None}


def _exact_normal(case, seed):
    """Level-0 cells, then rounds that halve every leaf above sigma_mult mean errors."""
    lo, hi, p, o = _normal(case, seed)
    dim, n, per = len(lo), o["samples_per_cell"], 1 << len(lo)
    par = np.zeros(W.N_PARAM)
    par[0], par[1], par[2:2 + dim] = 1.0, p[1], p[0]
    if case["kind"] == "peak":  # the user function has its parameters in FP32
        par[1], par[2:2 + dim] = np.float64(np.float32(p[1])), np.float64(np.float32(p[0]))
    bits = (np.arange(per)[:, None] >> np.arange(dim)) & 1
    width = (hi - lo) * 0.5
    cells_lo, streams = lo + bits * width, np.arange(per)
    cells_hi = cells_lo + width

    def evaluate(cl, ch, sid):
        q = np.zeros((len(cl), max(W.N_PARAM, 2 + dim)))
        q[:, :W.N_PARAM] = par
        mean, m2 = _moments(W.GAUSS, dim, 0, o["seed"], sid, cl, ch, q, 0, n)
        v = np.prod(ch - cl, axis=1)
        return v * mean, v * np.sqrt(m2 / (n * (n - 1.0)))

    est, err = evaluate(cells_lo, cells_hi, streams)
    leaves, rounds, created = list(zip(cells_lo, cells_hi, est, err)), 0, per
    for _ in range(o["depth"]):
        tau = o["sigma_mult"] * (sum(c[3] for c in leaves) / len(leaves))
        new, count, kept = [], len(leaves), []
        for c in leaves:
            if c[3] > tau and count + per - 1 <= o["max_leaves"]:
                count += per - 1
                w = (c[1] - c[0]) * 0.5
                kept.append(range(len(new), len(new) + per))
                new += [(c[0] + k * w, c[0] + k * w + w) for k in bits]
            else:
                kept.append(c)
        if not new:
            break
        cl, ch = np.array([c[0] for c in new]), np.array([c[1] for c in new])
        est, err = evaluate(cl, ch, created + np.arange(len(new)))
        created += len(new)
        leaves = [x for c in kept for x in
                  ([(cl[k], ch[k], est[k], err[k]) for k in c] if isinstance(c, range) else [c])]
        rounds += 1
    return {"estimate": float(sum(c[2] for c in leaves)),
            "stderr": float(math.sqrt(sum(c[3] ** 2 for c in leaves))),
            "n_samples": None, "n_cells": None, "n_leaves": None, "rounds": None}


def exact(case, seed):
    samples = _mean_budget(case) * int(case["rows"]) * int(case.get("jobs", 1))
    if samples > 2.5e9:
        return None
    call = case["call"]
    if call == "normal":
        return _exact_normal(case, seed)
    if call == "serving":
        t = np.concatenate(_jobs(case, seed))
        return _results(t, *_exact_rows(t), _volume(t))
    if call == "functional":
        base, slots, values = _lattice(case, seed)
        t = np.repeat(base, len(values))
        for k, slot in enumerate(slots):
            t["p"][:, slot] = values[:, k]
        return _results(t, *_exact_rows(t), _volume(t))
    if call == "udf":
        t = _user_table(case, seed)
        if case["kind"] == "f32":  # the box and the parameters reach the function in FP32
            w = (t["hi"] - t["lo"]).astype(np.float32).astype(np.float64)
            volume = _volume(t)
            t["lo"] = t["lo"].astype(np.float32)
            t["hi"] = t["lo"] + w
            t["p"] = t["p"].astype(np.float32)
            return _results(t, *_exact_rows(t, family=W.HARMONIC), volume)
        return _results(t, *_exact_rows(t, family=W.HARMONIC), _volume(t))
    t = _table(case, seed)
    if call == "moments":
        end = t["n_samples"].astype(np.int64)
        mean, m2 = _exact_rows(t, end // 10 * 5, end)
        return {"mean": mean, "m2": m2, "n": None, "status": None}
    return _results(t, *_exact_rows(t), _volume(t))
