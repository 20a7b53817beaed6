"""Measured workloads of the library, through its public entry points: the random field
(mlmc_field_eval), batched multigrid solves (mg_solve_batch) and whole level calls
(mlmc_level_run), over the grids, batches, precisions and options of the six workloads
(workloads.CONFIGS), the tests and the README.

exact() restates each path in plain torch in 64 bits: the Philox feature draw and the
phasor sum of the Fourier fields, the SPDE field by cosine transforms, solves by conjugate
gradients on the seven-point operator (preconditioned by a plain V-cycle) down to the
rounding floor, and the FMG cycle step by step.
"""
import math

import numpy as np
import torch

import paper_1607_03252_gb300 as mg
from paper_1607_03252_gb300.workloads import RUN_SEED, level_n, sample_id

PREC = {"f64": mg.MLMC_PREC_F64, "mixed": mg.MLMC_PREC_MIXED}
ACCEL = {"none": mg.MLMC_ACCEL_NONE, "cg": mg.MLMC_ACCEL_CG, "fmg": mg.MLMC_ACCEL_FMG}
COV = {"gauss": mg.MLMC_COV_GAUSS, "exp": mg.MLMC_COV_EXP, "spde": mg.MLMC_COV_SPDE}
DISC = {"fv": mg.MLMC_DISC_FV, "fe": mg.MLMC_DISC_FE}
QOI = {"mean": mg.MLMC_QOI_MEAN, "point": mg.MLMC_QOI_POINT, "flux": mg.MLMC_QOI_FLUX}
SMOOTH = {"auto": mg.MLMC_SMOOTH_AUTO, "split": mg.MLMC_SMOOTH_SPLIT, "nodal": mg.MLMC_SMOOTH_NODAL}
DTYPE = {"f64": torch.float64, "f32": torch.float32}


def _field(name, n, batch, M, cov, sigma2, ell, dtype="f64"):
    return dict(name=name, kind="field", n=n, batch=batch, M=M, cov=cov, sigma2=sigma2, ell=ell, dtype=dtype)


def _solve(name, n, batch, precision, accel, smoother, rhs, sigma2, ell, disc="fv", nu=2):
    return dict(name=name, kind="solve", n=n, batch=batch, precision=precision, accel=accel, smoother=smoother,
                rhs=rhs, sigma2=sigma2, ell=ell, disc=disc, nu=nu)


def _level(name, level, N, precision, accel, smoother, cov, sigma2, ell, M=256, disc="fv", qoi="mean", nu=2):
    return dict(name=name, kind="level", level=level, N=N, precision=precision, accel=accel, smoother=smoother,
                cov=cov, sigma2=sigma2, ell=ell, M=M, disc=disc, qoi=qoi, nu=nu)


def listed():
    return [
        # one served single-sample request of the coarsest level: the smallest call, all latency
        _level("level0_request", 0, 1, "mixed", "cg", "auto", "gauss", 2.0, 0.1),
        # the coefficient of a finest-level batch of the four-level FP64 workload
        _field("field_129_b8", 129, 8, 256, "gauss", 1.0, 0.3),
        # the paper's covariance by Fourier features on a coarse level, FP32 output, ragged M
        _field("field_exp_33_b103", 33, 103, 200, "exp", 1.0, 0.15, "f32"),
        # the adaptive run's field: 1024 features of a short correlation length
        _field("field_m1024_65_b5", 65, 5, 1024, "gauss", 1.0, 0.05),
        # the paper's own sampler
        _field("field_spde_65_b4", 65, 4, 1, "spde", 1.0, 0.1),
        # caller's buffers with a right-hand side, the default solver as the README calls it
        _solve("solve_f64_65_b19", 65, 19, "f64", "none", "auto", True, 1.0, 0.3),
        # mixed refinement of a middle grid (the serving default)
        _solve("solve_mixed_33_b48", 33, 48, "mixed", "none", "auto", False, 1.0, 0.2),
        # FP32 V-cycle preconditioning FP64 CG on the rough field, the large grid
        _solve("solve_mixed_cg_257_b1", 257, 1, "mixed", "cg", "split", False, 2.0, 0.1),
        # the levels of the four-level FP64 workload: many samples of the smallest grid ...
        _level("level0_f64_n4096", 0, 4096, "f64", "none", "auto", "gauss", 1.0, 0.3),
        # ... and a batch of the finest, on the storage the autotuner picks for it
        _level("level3_f64_n24", 3, 24, "f64", "none", "split", "gauss", 1.0, 0.3),
        # the paper's static run: P1 elements, one FMG-2V(4,4) cycle, the point value
        _level("level2_fe_fmg_n108", 2, 108, "f64", "fmg", "auto", "exp", 1.0, 0.15, disc="fe", qoi="point", nu=4),
        # the mixed-precision workload's finest level
        _level("level4_mixed_cg_n2", 4, 2, "mixed", "cg", "split", "gauss", 2.0, 0.1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["field", "solve", "level"])
    if kind == "field":
        cov = rng.choice(["gauss", "exp", "spde"])
        if cov == "spde":
            n = rng.choice([17, 33, 65])
            return _strip(_field("", n, _log_int(rng, 1, {17: 64, 33: 16, 65: 5}[n]), 1, cov,
                                 round(rng.uniform(0.5, 2.0), 2), round(rng.uniform(0.08, 0.3), 3)))
        n = rng.choice([17, 33, 65, 129])
        return _strip(_field("", n, _log_int(rng, 1, {17: 1500, 33: 300, 65: 48, 129: 8}[n]), _log_int(rng, 60, 1024),
                             cov, round(rng.uniform(0.5, 2.0), 2), round(rng.uniform(0.05, 0.4), 3),
                             rng.choice(["f64", "f64", "f32"])))
    if kind == "solve":
        precision, accel = rng.choice([("f64", "none"), ("f64", "none"), ("mixed", "none"), ("mixed", "cg"), ("f64", "cg")])
        n = rng.choice([9, 17, 33, 65, 129])
        rough = accel == "cg"
        return _strip(_solve("", n, _log_int(rng, 1, {9: 4000, 17: 1200, 33: 220, 65: 36, 129: 6}[n]), precision, accel,
                             rng.choice(["auto", "auto", "split"]), rng.random() < 0.4,
                             2.0 if rough else round(rng.uniform(0.5, 1.2), 2),
                             round(rng.uniform(0.1, 0.2) if rough else rng.uniform(0.25, 0.5), 3),
                             nu=rng.choice([2, 2, 2, 3])))
    fe = rng.random() < 0.3
    level = rng.choice([0, 1, 2, 3])
    if fe:
        return _strip(_level("", level, _log_int(rng, 1, {0: 4123, 1: 688, 2: 108, 3: 16}[level]), "f64", "fmg",
                             rng.choice(["auto", "split"]), rng.choice(["exp", "gauss"]), 1.0,
                             round(rng.uniform(0.1, 0.3), 3), M=_log_int(rng, 100, 512), disc="fe",
                             qoi=rng.choice(["point", "flux"]), nu=4))
    precision, accel = rng.choice([("f64", "none"), ("mixed", "cg")])
    cap = {0: 4096, 1: 900, 2: 150, 3: 20} if precision == "f64" else {0: 1024, 1: 256, 2: 40, 3: 8}
    return _strip(_level("", level, _log_int(rng, 1, cap[level]), precision, accel,
                         rng.choice(["auto", "split"]), "gauss", 1.0 if precision == "f64" else 2.0,
                         round(rng.uniform(0.25, 0.5) if precision == "f64" else rng.uniform(0.1, 0.25), 3),
                         M=_log_int(rng, 100, 512)))


def _strip(case):
    return {k: v for k, v in case.items() if k != "name"}


# ---- inputs and the call -----------------------------------------------------------------
def _first_id(case, seed):
    return sample_id(case.get("level", 9), (seed % (1 << 20)) << 20)


def _ids(case, seed):
    n = case["N"] if case["kind"] == "level" else case["batch"]
    return np.arange(n, dtype=np.uint64) + np.uint64(_first_id(case, seed))


def _coefficient(case, seed):
    """A smooth lognormal coefficient of the case's variance and correlation length from 256
    random cosines, as a user's own sampler would hand it over."""
    B, n, M = case["batch"], case["n"], 256
    gen = torch.Generator().manual_seed(seed)
    w = torch.randn(B, M, 3, generator=gen, dtype=torch.float64) / case["ell"]
    b = 2 * math.pi * torch.rand(B, M, generator=gen, dtype=torch.float64)
    return torch.exp(math.sqrt(2.0 * case["sigma2"] / M) * _cosine_sum(w.cuda(), b.cuda(), n))


def _rhs(case, seed):
    if not case["rhs"]:
        return None
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.rand(_shape(case), generator=gen, dtype=torch.float64, device="cuda") * 2.0 - 1.0


def _shape(case):
    return (case["batch"],) + (case["n"],) * 3


def prepare(case, seed):
    if case["kind"] == "field":
        return dict(kind="field", ids=_ids(case, seed),
                    cfg=mg.field_cfg(RUN_SEED, case["sigma2"], case["ell"], case["M"], COV[case["cov"]]),
                    k=torch.empty(_shape(case), dtype=DTYPE[case["dtype"]], device="cuda"))
    fixed = case["accel"] == "fmg"
    opts = dict(nu1=case["nu"], nu2=case["nu"], rtol=0.0 if fixed else 1e-10, max_cycles=2 if fixed else 300,
                precision=PREC[case["precision"]], smoother=SMOOTH[case["smoother"]], accel=ACCEL[case["accel"]],
                disc=DISC[case["disc"]])
    if case["kind"] == "solve":
        k = _coefficient(case, seed)
        return dict(kind="solve", cfg=mg.mg_cfg(**opts), k=k, f=_rhs(case, seed), u=torch.empty_like(k))
    N = case["N"]
    stream = torch.cuda.Stream()
    cfg = mg.make_mlmc_cfg(RUN_SEED, case["sigma2"], case["ell"], case["M"], n0=17, max_batch=N, stream=stream,
                           cov=COV[case["cov"]], qoi=QOI[case["qoi"]], **opts)
    state = dict(kind="level", level=case["level"], cfg=cfg, stream=stream,
                 ids=torch.from_numpy(_ids(case, seed).view("int64")).cuda(),
                 out=[torch.empty(N, dtype=torch.float64, device="cuda") for _ in range(3)])
    torch.cuda.current_stream().synchronize()  # the level call reads its ids on its own stream
    return state


def run(state):
    if state["kind"] == "field":
        mg.mlmc_field_eval(state["cfg"], state["ids"], state["k"])
        return state["k"]
    if state["kind"] == "solve":
        state["u"].zero_()
        cycles, _, _ = mg.mg_solve_batch(state["cfg"], state["k"], state["u"], state["f"])
        return {"u": state["u"], "cycles": cycles}
    Y, Qf, Qc = state["out"]
    stats = mg.mlmc_level_run(state["cfg"], state["level"], state["ids"], Y_dev=Y, Qf_dev=Qf, Qc_dev=Qc)
    return {"Y": Y, "Qf": Qf, "Qc": Qc, "mean": stats.mean, "var": stats.var_unbiased}


# ---- what a pass cannot do without ---------------------------------------------------------
def _cycles(case):
    return 2 if case["accel"] == "fmg" else 10


def _solve_flops(case, n, batch):
    """About ten V(nu, nu) cycles (two per grid of an FMG cycle): a Gauss-Seidel update is 13
    operations, the residual 14, the transfers and the convergence test about 20 per node."""
    return batch * n ** 3 * (_cycles(case) * (26 * case["nu"] + 34) * 8 / 7 + 60)


def work(case):
    if case["kind"] == "field":
        nodes = case["batch"] * case["n"] ** 3
        per = 200 if case["cov"] == "spde" else 4 * case["M"]
        return {"bytes": nodes * (8 if case["dtype"] == "f64" else 4) + 8 * case["batch"], "flops": nodes * per}
    if case["kind"] == "solve":
        nodes = case["batch"] * case["n"] ** 3
        return {"bytes": 8 * nodes * (3 if case["rhs"] else 2), "flops": _solve_flops(case, case["n"], case["batch"])}
    nf, N = level_n(case["level"]), case["N"]
    flops = N * nf ** 3 * 4 * case["M"] + _solve_flops(case, nf, N)
    if case["level"] > 0:
        flops += _solve_flops(case, level_n(case["level"] - 1), N)
    # a level call reads ids and writes three values a sample; its coefficients and solutions
    # are needed in memory once each
    return {"bytes": N * (32 + 16 * nf ** 3), "flops": flops}


# ---- the same in plain torch, 64 bits ------------------------------------------------------
def _philox(c0, c1, c2, c3, key):
    """Philox4x32-10 on int64 tensors that hold 32-bit words."""
    m = 0xFFFFFFFF
    k0, k1 = key & m, key >> 32
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57  # wrap modulo 2^64: both words survive
        c0, c1, c2, c3 = ((p1 >> 32) & m) ^ c1 ^ k0, p1 & m, ((p0 >> 32) & m) ^ c3 ^ k1, p0 & m
    return c0, c1, c2, c3


def _id_words(ids):
    i = torch.from_numpy(ids.view("int64")).cuda()
    return i & 0xFFFFFFFF, (i >> 32) & 0xFFFFFFFF


def _features(case, ids):
    lo, hi = _id_words(ids)
    m = torch.arange(case["M"], device="cuda").expand(len(ids), -1)
    lo, hi = lo[:, None].expand_as(m), hi[:, None].expand_as(m)
    words = [w for c in range(3) for w in _philox(lo, hi, m, torch.full_like(m, c), RUN_SEED)]
    U = [((words[2 * i] >> 5).double() * 67108864.0 + (words[2 * i + 1] >> 6).double() + 0.5) * 2.0 ** -53
         for i in range(5)]
    r1, r2 = torch.sqrt(-2 * torch.log(U[0])), torch.sqrt(-2 * torch.log(U[2]))
    g = torch.stack([r1 * torch.cos(2 * math.pi * U[1]), r1 * torch.sin(2 * math.pi * U[1]),
                     r2 * torch.cos(2 * math.pi * U[3])], -1)
    scale = torch.full_like(r2, case["ell"])
    if case["cov"] == "exp":
        scale = case["ell"] * torch.abs(r2 * torch.sin(2 * math.pi * U[3]))
    return g / scale[..., None], 2 * math.pi * U[4]


def _cosine_sum(w, b, n):
    """sum_m cos(w_m . x + b_m) at the n^3 nodes, by one phasor per axis."""
    x = torch.arange(n, device=w.device, dtype=torch.float64) / (n - 1)
    out = []
    for s in range(w.shape[0]):
        ph = [w[s, :, a, None] * x + (b[s, :, None] if a == 0 else 0.0) for a in range(3)]
        X, Y, Z = (torch.polar(torch.ones_like(p), p) for p in ph)
        Q = (Z[:, :, None] * Y[:, None, :]).reshape(w.shape[1], -1)  # lines (z, y)
        out.append((Q.real.T @ X.real - Q.imag.T @ X.imag).reshape(n, n, n))
    return torch.stack(out)


def _fma32(a, b, c):
    return (a.double() * b.double() + c.double()).float()


def _log32(s):
    """The SPDE noise's FP32 logarithm: mantissa and exponent, an atanh series."""
    m, e = torch.frexp(s)
    m, e = m * 2, e - 1
    big = m > 1.4142135
    m, e = torch.where(big, 0.5 * m, m), torch.where(big, e + 1, e)
    t = (m - 1.0) / (m + 1.0)
    t2 = t * t
    f = lambda x: torch.full_like(s, x)  # noqa: E731
    p = _fma32(t2, f(1 / 11), f(1 / 9))
    for d in (7, 5, 3, 1):
        p = _fma32(t2, p, f(1 / d))
    fe = e.float()
    return _fma32(fe, f(float.fromhex("0x1.62e400p-1")), _fma32(fe, f(float.fromhex("0x1.7f7d1cp-20")), (2.0 * t) * p))


def _octant_normals(lo, hi, octs):
    """Marsaglia's polar method in FP32 on Philox words, up to 32 attempts an octant."""
    out = torch.zeros(octs.shape, dtype=torch.float32, device="cuda")
    todo = torch.arange(octs.numel(), device="cuda")
    flat, res = octs.reshape(-1), out.reshape(-1)
    for call in range(16):
        o = flat[todo]
        words = _philox(torch.full_like(o, lo), torch.full_like(o, hi), o & 0xFFFFFFFF,
                        0x5D000000 | (call << 8) | (o >> 32), RUN_SEED)
        found = torch.zeros(o.shape, dtype=torch.bool, device="cuda")
        for half in range(2):
            u1, u2 = ((((words[half * 2 + i] >> 8) - 8388608).float() + 0.5) * 2.0 ** -23 for i in range(2))
            sq = _fma32(u1, u1, u2 * u2)
            ok = ~found & (sq > 0) & (sq < 1)
            safe = torch.where(ok, sq, torch.full_like(sq, 0.5))
            v = u1 * torch.sqrt((-2.0 * _log32(safe)) / safe)
            res[todo[ok]] = v[ok]
            found |= ok
        todo = todo[~found]
        if not todo.numel():
            break
    return out


def _spde(case, ids, n, n_noise):
    C, r, h, hf = 2 * (n - 1), (n_noise - 1) // (n - 1), 1.0 / (n - 1), 1.0 / (n_noise - 1)
    Mo, kappa, off = 4 * (n_noise - 1) + 1, 1.0 / case["ell"], (n - 1) // 2
    j = torch.arange(C, device="cuda", dtype=torch.float64)
    V = torch.cos(math.pi * j[None, :] * (j[:, None] + 0.5) / C) * math.sqrt(2.0 / C)
    V[:, 0] /= math.sqrt(2.0)
    lam = 2 - 2 * torch.cos(math.pi * j / C)
    den = kappa ** 2 * h ** 2 + lam[:, None, None] + lam[None, :, None] + lam[None, None, :]
    axis = torch.arange(2 - r, 2 * r * (C - 1) + 2 + r, device="cuda")  # the octants of one axis
    # cell i takes octants 2 r i + 2 - r .. 2 r i + 1 + r: consecutive runs of 2 r
    lo, hi = _id_words(ids)
    out = []
    for s in range(len(ids)):
        W = []
        for z in range(C):
            az = axis[2 * r * z:2 * r * (z + 1)]
            octs = (az[:, None, None] * Mo + axis[None, :, None]) * Mo + axis[None, None, :]
            v = _octant_normals(int(lo[s]), int(hi[s]), octs).double()
            W.append(v.reshape(2 * r, C, 2 * r, C, 2 * r).sum((0, 2, 4)))
        g = torch.stack(W) * (math.sqrt((0.5 * hf) ** 3) / h)
        t = torch.einsum("zyx,za,yb,xc->abc", g, V, V, V) / den
        Zf = torch.einsum("abc,za,yb,xc->zyx", t, V, V, V)
        Zf = Zf[off:off + n, off:off + n, off:off + n]
        out.append(torch.exp(math.sqrt(8 * math.pi * kappa * case["sigma2"]) * Zf))
    return torch.stack(out)


def _field_exact(case, ids, n, n_fine):
    if case["cov"] == "spde":
        return _spde(case, ids, n, n_fine)
    w, b = _features(case, ids)
    return torch.exp(math.sqrt(2.0 * case["sigma2"] / case["M"]) * _cosine_sum(w, b, n))


_I = (slice(None),) + (slice(1, -1),) * 3


def _sh(a, dz, dy, dx):
    """The interior nodes' neighbour at (dz, dy, dx)."""
    n = a.shape[1]
    return a[:, 1 + dz:n - 1 + dz, 1 + dy:n - 1 + dy, 1 + dx:n - 1 + dx]


class _Grid:
    def __init__(self, k, disc):
        n = self.n = k.shape[1]
        self.K = []  # per axis: the face below and the face above every interior node
        for a in range(3):  # 0: z, 1: y, 2: x
            e = [0, 0, 0]
            e[a] = 1
            if disc == "fv":
                face = lambda p, e=e: 2 * _at(k, p) * _at(k, [p[i] + e[i] for i in range(3)]) / (  # noqa: E731
                    _at(k, p) + _at(k, [p[i] + e[i] for i in range(3)]))
            else:
                b, c = [[int(i == q) for i in range(3)] for q in range(3) if q != a]

                def face(p, e=e, b=b, c=c):
                    f = lambda *vs: _at(k, [p[i] + sum(s * v[i] for s, v in vs) for i in range(3)])  # noqa: E731
                    return (f() + f((1, e))) / 4 + (f((1, e), (1, b)) + f((1, e), (1, c)) + f((1, e), (1, b), (1, c)) +
                                                    f((-1, b)) + f((-1, c)) + f((-1, b), (-1, c))) / 12
            self.K.append((face([-x for x in e]), face([0, 0, 0])))
        self.D = sum(lo + hi for lo, hi in self.K)
        q = torch.arange(1, n - 1, device=k.device)
        par = (q[:, None, None] + q[None, :, None] + q[None, None, :]) % 2
        self.red = (par == 0)[None]

    def off(self, u):
        s = 0.0
        for a, (lo, hi) in enumerate(self.K):
            e = [0, 0, 0]
            e[a] = 1
            s = s + lo * _sh(u, *[-x for x in e]) + hi * _sh(u, *e)
        return s

    def residual(self, u, g):
        return g - self.D * u[_I] + self.off(u)

    def smooth(self, u, g, sweeps):
        for _ in range(sweeps):
            for mask in (self.red, ~self.red):
                u[_I] = torch.where(mask, (g + self.off(u)) / self.D, u[_I])


def _at(k, p):
    return _sh(k, *p)


def _pad(v):
    return torch.nn.functional.pad(v, (1,) * 6)


def _restrict(r, disc):
    """g_c of the h^2-scaled coarse system from the fine interior residual."""
    f, nc = _pad(r), (r.shape[1] + 3) // 2

    def at(dz, dy, dx):
        m = nc - 2
        return f[:, 2 + dz:2 + dz + 2 * m:2, 2 + dy:2 + dy + 2 * m:2, 2 + dx:2 + dx + 2 * m:2]

    out = 0.0
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                d = abs(dz) + abs(dy) + abs(dx)
                if disc == "fe" and not (min(dz, dy, dx) >= 0 or max(dz, dy, dx) <= 0):
                    continue
                out = out + at(dz, dy, dx) * (0.5 ** d * 0.5 if disc == "fv" else (0.5 if d == 0 else 0.25))
    return out


def _prolong(e, disc):
    """The coarse function at every node of the fine grid."""
    nc = e.shape[1]
    u = torch.zeros((e.shape[0],) + (2 * nc - 1,) * 3, dtype=e.dtype, device=e.device)
    for dz in (0, 1):
        for dy in (0, 1):
            for dx in (0, 1):
                a = e[:, :nc - dz, :nc - dy, :nc - dx]
                u[:, dz::2, dy::2, dx::2] = 0.5 * (a + e[:, dz:, dy:, dx:]) if disc == "fe" else _mean(e, dz, dy, dx)
    return u


def _mean(e, dz, dy, dx):
    """The mean along each odd axis (trilinear)."""
    if dz:
        e = 0.5 * (e[:, :-1] + e[:, 1:])
    if dy:
        e = 0.5 * (e[:, :, :-1] + e[:, :, 1:])
    if dx:
        e = 0.5 * (e[:, :, :, :-1] + e[:, :, :, 1:])
    return e


class _MG:
    def __init__(self, k, disc):
        self.disc, self.grids = disc, []
        while True:
            self.grids.append(_Grid(k, disc))
            if k.shape[1] == 5:
                break
            k = k[:, ::2, ::2, ::2].contiguous()
        G = self.grids[-1]
        cols = []
        for i in range(27):
            u = torch.zeros(1, 27, dtype=torch.float64, device="cuda")
            u[0, i] = 1.0
            u = _pad(u.reshape(1, 3, 3, 3))
            cols.append((G.D * u[_I] - G.off(u)).reshape(-1, 27))
        self.A = torch.stack(cols, -1)

    def cycle(self, j, u, g, nu):
        G = self.grids[j]
        if j == len(self.grids) - 1:
            return _pad(torch.linalg.solve(self.A, g.reshape(-1, 27)).reshape(-1, 3, 3, 3))
        G.smooth(u, g, nu)
        gc = _restrict(G.residual(u, g), self.disc)
        nc = self.grids[j + 1].n
        e = self.cycle(j + 1, torch.zeros((u.shape[0],) + (nc,) * 3, dtype=u.dtype, device=u.device), gc, nu)
        u[_I] += _prolong(e, self.disc)[_I]
        G.smooth(u, g, nu)
        return u

    def ones(self, j, batch):
        n = self.grids[j].n
        return torch.full((batch,) + (n - 2,) * 3, (1.0 / (n - 1)) ** 2, dtype=torch.float64, device="cuda")

    def fmg(self, batch, nu, cycles):
        L = len(self.grids)
        u = self.cycle(L - 1, None, self.ones(L - 1, batch), nu)
        for j in range(L - 2, -1, -1):
            u = _pad(_prolong(u, self.disc)[_I])
            for _ in range(cycles):
                u = self.cycle(j, u, self.ones(j, batch), nu)
        return u

    def solve(self, g):
        """Conjugate gradients to eight digits, thrice, each on the residual of the one before."""
        G, dims = self.grids[0], (1, 2, 3)
        dot = lambda a, b: (a * b).sum(dims, keepdim=True)  # noqa: E731
        pre = lambda r: self.cycle(0, torch.zeros_like(u), r, 2)[_I]  # noqa: E731
        div = lambda a, b: torch.where(b == 0, torch.zeros_like(a), a / b)  # noqa: E731
        u = _pad(torch.zeros_like(g))
        for _ in range(3):
            r = G.residual(u, g)
            x, start = torch.zeros_like(r), dot(r, r)
            z = pre(r)
            p, rz = z, dot(r, z)
            for _ in range(80):
                q = G.D * p - G.off(_pad(p))
                a = div(rz, dot(p, q))
                x, rn = x + a * p, r - a * q
                if float((dot(rn, rn) / torch.clamp(start, min=1e-300)).max()) < 1e-16:
                    break
                z = pre(rn)
                nz = dot(rn, z)
                p = z + div(nz - dot(r, z), rz) * p
                r, rz = rn, nz
            u[_I] += x
        return u


def _qoi(case, u, k):
    n = u.shape[1]
    h, c = 1.0 / (n - 1), (n - 1) // 4
    if case["qoi"] == "point":
        return u[:, c, c, c]
    if case["qoi"] == "mean":
        m = 2 * c + 1
        w = torch.ones(m, dtype=torch.float64, device=u.device)
        w[0] = w[-1] = 0.5
        return torch.einsum("szyx,z,y,x->s", u[:, c:c + m, c:c + m, c:c + m], w, w, w) * 8 * h ** 3
    total = 0.0  # the flux through the layer of elements below x_2 = 1/4
    corner = lambda a, v: a[:, v[2]:n - 1 + v[2], c - 1 + v[1], v[0]:n - 1 + v[0]]  # noqa: E731
    for path in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
        vs = [[0, 0, 0]]
        for a in path:
            vs.append([x + (i == a) for i, x in enumerate(vs[-1])])
        kbar = sum(corner(k, v) for v in vs) / 4
        at = path.index(1)
        total = total + (kbar * (corner(u, vs[at + 1]) - corner(u, vs[at]))).sum((1, 2))
    return total * h / 6


def exact(case, seed):
    if case["kind"] == "field":
        return _field_exact(case, _ids(case, seed), case["n"], case["n"])
    if case["kind"] == "solve":
        h = 1.0 / (case["n"] - 1)
        m = _MG(_coefficient(case, seed), case["disc"])
        f = _rhs(case, seed)
        g = m.ones(0, case["batch"]) if f is None else h * h * f[_I]
        return {"u": m.solve(g), "cycles": None}
    ids, nf = _ids(case, seed), level_n(case["level"])
    Q = []
    for n in [nf] + ([(nf + 1) // 2] if case["level"] else []):
        parts = []
        step = max(1, (1 << 25) // n ** 3)
        for i in range(0, len(ids), step):
            k = _field_exact(case, ids[i:i + step], n, nf)
            m = _MG(k, case["disc"])
            u = m.fmg(len(k), case["nu"], 2) if case["accel"] == "fmg" else m.solve(m.ones(0, len(k)))
            parts.append(_qoi(case, u, k))
        Q.append(torch.cat(parts))
    Qf, Qc = Q[0], (Q[1] if len(Q) > 1 else torch.zeros_like(Q[0]))
    Y = Qf - Qc
    return {"Y": Y, "Qf": Qf, "Qc": Qc, "mean": float(Y.mean()), "var": float(Y.var()) if len(Y) > 1 else 0.0}
