"""What a user has this library do, as cases that can be timed and compared.

A case is a problem (grid levels, KL modes, precision, solver options) and one
call on it: ``step`` is `Context.sample_levels` on a work list with the
per-sample F asked for, ``solution`` is `Context.sample_solution`, ``estimate``
is Algorithm 1 (`Context.estimate`) and ``mixed`` is `Context.sample_mixed` on
two cycle counts. `prepare` makes what a program keeps between calls (the
context, its output buffers); the seed is the problem's own, so another seed
draws other shifts or other Monte Carlo points and with them other fields.

`exact` restates the method in 64 bits with torch: Philox shifts, the lattice
sequence, the inverse normal distribution, the closed-form KL eigenpairs (or
Nystrom interpolation), the finite-volume FMG and Algorithm 1.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_1806_05619_gb300 as M

BASE = dict(kind="step", n0=8, sigma=1.0, corr_len=0.3, qoi="mean", mu0=2, nu1=2, nu2=2, precision="mixed_tf32",
            rtol=0.0, sampler="lattice", R=16, reuse=True, covariance="sep_exp")
MATERN_NU, MATERN_NODES = 1.5, 16  # smoothness and nodes per side of the Matern cases


def _case(name, **kw):
    return dict(BASE, name=name, **kw)


def listed():
    return [
        # The plain multigrid MLMC run of a small problem, all in FP64: every level is tiny, so launches and
        # the latency of the level-0 factorisation are what a user waits for.
        _case("mc_4_levels_fp64", n_levels=4, n0=4, s=10, qoi="center", precision="fp64", sampler="mc", R=1,
              counts="512,128,32,8"),
        # A new level's first round of an adaptive run: one point for each of the 16 shifts on 128 x 128.
        _case("first_round_128", n_levels=6, s=1000, corr_len=0.05, counts="0,0,0,0,1,0"),
        # One sample whose solutions on all levels are wanted (a plot, a check), refined to 1e-10.
        _case("one_sample_256", kind="solution", n_levels=6, s=200, rtol=1e-10, level=5),
        # MLQMC with recycling on six levels with the counts of one estimate, in FP64 and in the mixed form.
        _case("lattice_6_levels_fp64", n_levels=6, s=100, precision="fp64", counts="1024,512,256,128,64,32"),
        _case("lattice_6_levels_mixed", n_levels=6, s=100, counts="1024,512,256,128,64,32"),
        # Sides that are no powers of two, counts with no common factor, the split-BF16 fields, V(1,1), centre value.
        _case("odd_sizes_bf16x3", n_levels=5, n0=6, s=37, qoi="center", precision="mixed_bf16x3", R=5, nu1=1, nu2=1,
              counts="201,77,33,13,5"),
        # The Matern covariance with Nystrom modes.
        _case("matern_6_levels", n_levels=6, s=100, covariance="matern", counts="256,128,64,32,16,8"),
        # The multi-index variant: differences between two cycle counts on the same samples.
        _case("cycle_differences", kind="mixed", n_levels=4, n0=4, s=10, precision="fp64", R=4, mu0=1,
              counts="256,64,16,4"),
        # A batch on one fine level refined to 1e-10.
        _case("refined_1024", n_levels=8, s=400, corr_len=0.1, rtol=1e-10, counts="0,0,0,0,0,0,0,4"),
        # Algorithm 1 to a tolerance: every round's launches and read-backs, converged and fixed-cycle.
        _case("adaptive_7_levels", kind="estimate", n_levels=7, s=200, rtol=1e-10, eps=3e-4),
        _case("adaptive_9_levels", kind="estimate", n_levels=9, s=1000, corr_len=0.05, eps=2e-4),
        # The large problem: nine levels up to 2048 x 2048, 1000 modes, counts doubling per coarser level.
        _case("step_9_levels", n_levels=9, s=1000, corr_len=0.05, counts="1024,512,256,128,64,32,16,8,4"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _cells(c):
    """Cells of all grids of all samples of one pass."""
    per = np.cumsum([float(c["n0"] << t) ** 2 for t in range(c["n_levels"])])
    if c["kind"] == "solution":
        return per[c["level"]]
    if c["kind"] == "estimate":
        return 0.0
    return sum(int(n) * c["R"] * per[t] for t, n in enumerate(c["counts"].split(",")))


def draw(rng):
    kind = rng.choice(["step"] * 7 + ["solution", "estimate", "mixed"])
    precision = rng.choice(["fp64", "mixed_tf32", "mixed_tf32", "mixed_bf16x3"])
    n0 = rng.choice([8, 8, 8, 4, 6, 10])
    c = dict(BASE, kind=kind, precision=precision, n0=n0, corr_len=round(_log(rng, 0.05, 0.5), 3),
             s=int(_log(rng, 8, 500)), R=rng.choice([16, 16, 8, 5, 20]), qoi=rng.choice(["mean", "mean", "center"]),
             rtol=rng.choice([0.0, 0.0, 0.0, 1e-10]), mu0=rng.choice([2, 2, 1]), nu1=rng.choice([2, 2, 1]),
             nu2=rng.choice([2, 2, 1]), reuse=rng.random() < 0.8)
    if kind == "estimate":
        c.update(precision="mixed_tf32" if precision == "fp64" else precision, n0=8, n_levels=rng.choice([5, 6, 7]),
                 eps=float("%.2g" % _log(rng, 4e-4, 1e-2)), R=16, reuse=True, mu0=2, nu1=2, nu2=2, qoi="mean")
        return c
    if kind == "mixed":
        c.update(mu0=1, rtol=0.0)
    elif rng.random() < 0.15:
        c.update(covariance="matern", s=min(c["s"], 120), corr_len=max(c["corr_len"], 0.2))
    if rng.random() < 0.15:
        c["sampler"] = "mc"
    c["n_levels"] = rng.randint(2, 8 if precision != "fp64" else 7)
    if kind == "solution":
        c["level"] = rng.randint(1, c["n_levels"] - 1)
        return c
    # counts that halve per finer level, give or take; work well inside the largest listed case's
    room = 2e8 / (20 if precision == "fp64" else 1) / (4 if c["rtol"] else 1)
    top, shape = _log(rng, 1, 60), rng.uniform(1.4, 2.6)
    while True:
        counts = [int(top * shape ** (c["n_levels"] - 1 - t) * rng.uniform(0.7, 1.3)) for t in range(c["n_levels"])]
        c["counts"] = ",".join(str(min(max(0, n), 2000)) for n in counts[:-1]) + ",%d" % max(1, counts[-1])
        if _cells(c) <= room and sum(int(n) for n in c["counts"].split(",")) * c["R"] <= 60000:
            return c
        if top < 1 and shape < 1.1:
            c["n_levels"] -= 1
        top, shape = top * 0.7, max(1.0, shape * 0.95)


@functools.lru_cache(maxsize=None)
def _genvec(s, m):
    return M.cbc_genvec(s, m)[0]


def _vector(c):
    """The generating vector of a problem: made for 1024 points where the counts are fixed, and for more points than an
    adaptive run takes (past its points a vector of the construction stops reducing the variance)."""
    return _genvec(c["s"], 13 if c["kind"] == "estimate" else 10) if c["sampler"] == "lattice" else None


def _midpoints(m):
    k = (np.arange(m) + 0.5) / m
    return np.tile(k, m), np.repeat(k, m)


def _matern(c, r):
    """sigma^2 (1 + z) exp(-z), z = sqrt(3) r / corr_len: the Matern covariance of smoothness 3/2."""
    z = math.sqrt(2 * MATERN_NU) * r / c["corr_len"]
    return c["sigma"] ** 2 * (1 + z) * np.exp(-z)


@functools.lru_cache(maxsize=4)
def _matern_modes(s, corr_len, sigma):
    """Nystrom eigenpairs on the midpoint nodes: eigenvalues and nodal values (weights 1/m^2, unit norm)."""
    c = dict(corr_len=corr_len, sigma=sigma)
    x, y = _midpoints(MATERN_NODES)
    cov = _matern(c, np.hypot(x[:, None] - x[None, :], y[:, None] - y[None, :]))
    ev, vec = np.linalg.eigh(cov / MATERN_NODES ** 2)
    return ev[::-1][:s].copy(), np.ascontiguousarray(vec[:, ::-1][:, :s]) * MATERN_NODES


def _context(c, seed, mu0):
    more = {}
    if c["covariance"] == "matern":
        theta, psi = _matern_modes(c["s"], c["corr_len"], c["sigma"])
        more = dict(covariance="matern", matern_nu=MATERN_NU, nystrom_m=MATERN_NODES, nystrom_theta=theta,
                    nystrom_psi=psi)
    return M.Context(c["n_levels"], c["n0"], c["s"], sigma=c["sigma"], corr_len=c["corr_len"], qoi=c["qoi"], mu0=mu0,
                     nu1=c["nu1"], nu2=c["nu2"], precision=c["precision"], refine_rtol=c["rtol"], sampler=c["sampler"],
                     seed=seed, n_shifts=c["R"], genvec=_vector(c), log2_nmax=20, reuse=c["reuse"], **more)


def _work_list(c):
    return [(t, 0, int(n), 0, c["R"]) for t, n in enumerate(c["counts"].split(",")) if int(n) > 0]


def prepare(case, seed):
    state = dict(case=case, ctx=_context(case, seed, case["mu0"]))
    if case["kind"] in ("step", "mixed"):
        work = _work_list(case)
        count = sum((e - b) * (re - rb) for _, b, e, rb, re in work)
        state.update(work=work,
                     sums=torch.zeros(case["n_levels"], case["R"], 2, dtype=torch.float64, device="cuda"),
                     F=torch.zeros(count, case["n_levels"], dtype=torch.float64, device="cuda"))
    if case["kind"] == "mixed":
        state["more"] = _context(case, seed, case["mu0"] + 1)
    if case["kind"] == "solution":
        state.update(r=seed % case["R"], n=seed % 64)
    return state


def run(state):
    c, ctx = state["case"], state["ctx"]
    if c["kind"] == "step":
        state["sums"].zero_()
        ctx.sample_levels(state["work"], state["sums"], state["F"])
        return {"sums": state["sums"], "F": state["F"]}
    if c["kind"] == "mixed":
        state["sums"].zero_()
        state["more"].sample_mixed(ctx, state["work"], state["sums"], state["F"])
        return {"sums": state["sums"], "D": state["F"]}
    if c["kind"] == "solution":
        u, F = ctx.sample_solution(c["level"], state["r"], state["n"])
        return {"u": u, "F": F}
    res = ctx.estimate(c["eps"])
    return {k: v for k, v in res.items() if k not in ("wall_seconds", "gpu_seconds")}


def work(case):
    """Arithmetic of the method: per cell of each grid the KL sum, the faces, the FMG stages that visit the grid
    (sweeps, residual and transfers of mu0 cycles) and the level-0 factorisations. Bytes: the outputs, and the 1D
    (or Nystrom) mode tables and generating vector that are read."""
    nl, s = case["n_levels"], case["s"]
    per_cycle = 10 * (case["nu1"] + case["nu2"]) + 11 + 8
    steps = 4 if case["rtol"] else 1
    n = [case["n0"] << t for t in range(nl)]
    ka = min(s, 8 + int(2.5 * math.sqrt(s)))  # about the 1D modes that the s largest products use
    tables = 8.0 * s * (MATERN_NODES ** 2 if case["covariance"] == "matern" else 1) + 8.0 * ka * sum(n) + 4.0 * s

    def sample(level):
        f = n[0] ** 4 + 4.0 * n[0] ** 3
        for t in range(level + 1):
            kl = 2.0 * s * n[t] ** 2 if case["covariance"] == "matern" else 2.0 * s * n[t] + 2.0 * ka * n[t] ** 2
            cycles = sum(case["mu0"] * steps for top in range(max(t, 1), level + 1))
            f += kl + n[t] ** 2 * (8 + 18 + cycles * per_cycle)
        return f

    if case["kind"] == "solution":
        cells = sum(n[t] ** 2 for t in range(case["level"] + 1))
        return {"bytes": tables + 8.0 * (cells + case["level"] + 1), "flops": sample(case["level"])}
    if case["kind"] == "estimate":  # some 16 doublings per tolerance: a rough size, the counts follow from the run
        return {"bytes": tables + 8.0 * 4 * nl, "flops": sum(case["R"] * 2.0 ** (4 - t) * sample(t) for t in range(4))}
    counts = [int(v) * case["R"] for v in case["counts"].split(",")]
    solves = 1.0 + (case["mu0"] + 1.0) / case["mu0"] if case["kind"] == "mixed" else 1.0
    return {"bytes": tables + 8.0 * (sum(counts) * nl + nl * case["R"] * 2),
            "flops": solves * sum(k * sample(t) for t, k in enumerate(counts))}


# ---- the same in 64 bits, with torch -------------------------------------------------------------------------------

def _philox(j, c1, c2, tag, seed):
    """Philox4x32-10 blocks with counters (j/2, c1, c2, tag) and key `seed`: coordinate j's 64 bits."""
    lo32, u64 = np.uint64(0xFFFFFFFF), np.uint64
    j, c1, c2 = np.broadcast_arrays(*(np.asarray(v, dtype=np.uint64) for v in (j, c1, c2)))
    x = [j >> u64(1), c1.copy(), c2.copy(), np.full(j.shape, tag, dtype=np.uint64)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        p, q = u64(0xD2511F53) * x[0], u64(0xCD9E8D57) * x[2]
        x = [(q >> u64(32)) ^ x[1] ^ u64(k0), q & lo32, (p >> u64(32)) ^ x[3] ^ u64(k1), p & lo32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    odd = (j & u64(1)).astype(bool)
    return np.where(odd, (x[3] << u64(32)) | x[2], (x[1] << u64(32)) | x[0])


def _normals(c, seed, z, level, r, n):
    """y of the samples (level, r[i], n[i]): (samples, s) on the GPU."""
    r, n, j = np.asarray(r)[:, None], np.asarray(n)[:, None], np.arange(c["s"])[None, :]
    if c["sampler"] == "lattice":
        rev = np.array([int("{:032b}".format(int(v))[::-1], 2) for v in n[:, 0]], dtype=np.uint64)[:, None]
        t = (rev * z[None, : c["s"]].astype(np.uint64)) & np.uint64(0xFFFFFFFF)
        shifts = _philox(j, np.arange(c["R"])[:, None], level, 0x53484654, seed)
        with np.errstate(over="ignore"):
            x = (t << np.uint64(32)) + shifts[r[:, 0]]
    else:
        x = _philox(j, n, (r << 8) | level, 0x4D43524E, seed)
    u = ((x >> np.uint64(11)).astype(np.float64) + 0.5) * 2.0 ** -53
    return torch.special.ndtri(torch.from_numpy(u).cuda())


def _modes_1d(corr_len, count):
    """Roots, eigenvalues and norms of exp(-|x - x'| / corr_len) on [0, 1], by bisection."""
    k, cc = np.arange(count), 1.0 / corr_len
    lo, hi = np.maximum(k * math.pi, 1e-300), (k + 1) * math.pi

    def g(w):
        return (w * w - cc * cc) * np.sin(w) - 2 * cc * w * np.cos(w)

    glo = g(lo) < 0
    glo[0] = True  # just right of the trivial root at 0
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        same = (g(mid) < 0) == glo
        lo, hi = np.where(same, mid, lo), np.where(same, hi, mid)
    w = 0.5 * (lo + hi)
    norm = 0.5 * (w * w + cc * cc) + (w * w - cc * cc) * np.sin(2 * w) / (4 * w) + cc * np.sin(w) ** 2
    return w, 2 * cc / (w * w + cc * cc), norm


class _Fields:
    """k = exp(Z) on every level for given normals."""

    def __init__(self, c):
        self.c, s = c, c["s"]
        self.tables = {}
        if c["covariance"] == "matern":
            self.theta, self.psi = _matern_modes(s, c["corr_len"], c["sigma"])
            return
        w, th, self.norm = _modes_1d(c["corr_len"], s)
        self.w = w
        prod = c["sigma"] ** 2 * th[:, None] * th[None, :]
        m, e = np.frexp(prod)
        key = np.ldexp(np.rint(np.ldexp(m, 40)), e - 40).ravel()  # ties in 40 bits go to the smaller a, then b
        order = np.argsort(-key, kind="stable")[:s]
        self.a, self.b = order // s, order % s
        self.theta = prod.ravel()[order]
        self.k1 = int(max(self.a.max(), self.b.max())) + 1

    def table(self, n):
        if n not in self.tables:
            c = self.c
            if c["covariance"] == "matern":
                x, y = _midpoints(n)
                p, q = _midpoints(MATERN_NODES)
                t = _matern(c, np.hypot(x[:, None] - p[None, :], y[:, None] - q[None, :])) @ self.psi
                t /= MATERN_NODES ** 2 * self.theta[None, :]
            else:
                x, w, cc = (np.arange(n) + 0.5) / n, self.w[: self.k1, None], 1.0 / c["corr_len"]
                t = (w * np.cos(w * x) + cc * np.sin(w * x)) / np.sqrt(self.norm[: self.k1, None])
            self.tables[n] = torch.from_numpy(np.ascontiguousarray(t)).cuda()
        return self.tables[n]

    def __call__(self, n, y):
        t, coef = self.table(n), y * torch.from_numpy(np.sqrt(self.theta)).cuda()
        if self.c["covariance"] == "matern":
            return torch.exp((coef @ t.T).view(-1, n, n))
        m = torch.zeros(len(y), self.k1, self.k1, dtype=torch.float64, device="cuda")
        m[:, torch.from_numpy(self.b).cuda(), torch.from_numpy(self.a).cuda()] = coef
        return torch.exp(t.T @ (m @ t))  # [i2, i1]: the second index of a mode goes with x2


class _Grid:
    """Faces, diagonal and colours of one level's batch of fields."""

    def __init__(self, k):
        n = self.n = k.shape[-1]
        self.kx = torch.empty(len(k), n, n + 1, dtype=k.dtype, device=k.device)
        self.ky = torch.empty(len(k), n + 1, n, dtype=k.dtype, device=k.device)
        self.kx[:, :, 1:-1] = 2 * k[:, :, 1:] * k[:, :, :-1] / (k[:, :, 1:] + k[:, :, :-1])
        self.ky[:, 1:-1] = 2 * k[:, 1:] * k[:, :-1] / (k[:, 1:] + k[:, :-1])
        self.kx[:, :, 0], self.kx[:, :, -1] = 2 * k[:, :, 0], 2 * k[:, :, -1]
        self.ky[:, 0], self.ky[:, -1] = 2 * k[:, 0], 2 * k[:, -1]
        self.diag = self.kx[:, :, 1:] + self.kx[:, :, :-1] + self.ky[:, 1:] + self.ky[:, :-1]
        i = torch.arange(n, device=k.device)
        self.red = (i[:, None] + i[None, :]) % 2 == 0

    def off(self, u):
        o = torch.zeros_like(u)
        o[:, :, 1:] += self.kx[:, :, 1:-1] * u[:, :, :-1]
        o[:, :, :-1] += self.kx[:, :, 1:-1] * u[:, :, 1:]
        o[:, 1:] += self.ky[:, 1:-1] * u[:, :-1]
        o[:, :-1] += self.ky[:, 1:-1] * u[:, 1:]
        return o

    def sweep(self, u, b, red_first):
        for red in (red_first, not red_first):
            u = torch.where(self.red if red else ~self.red, (b / self.n ** 2 + self.off(u)) / self.diag, u)
        return u

    def residual(self, u, b):
        return b - self.n ** 2 * (self.diag * u - self.off(u))

    def matrix(self):
        e = torch.eye(self.n ** 2, dtype=self.kx.dtype, device=self.kx.device).view(-1, self.n, self.n)
        cols = [self.n ** 2 * (self.diag * v - self.off(v.expand_as(self.diag))) for v in e]
        return torch.stack([v.flatten(1) for v in cols], -1)


def _interpolate(e):
    """Bilinear cell-centred interpolation (weights 3/4, 1/4 per axis), odd about the boundary."""
    for dim in (1, 2):
        first, last = e.narrow(dim, 0, 1), e.narrow(dim, e.shape[dim] - 1, 1)
        g = torch.cat([-first, e, -last], dim)
        m = e.shape[dim]
        lo, mid, hi = g.narrow(dim, 0, m), g.narrow(dim, 1, m), g.narrow(dim, 2, m)
        e = torch.stack([0.75 * mid + 0.25 * lo, 0.75 * mid + 0.25 * hi], dim + 1).flatten(dim, dim + 1)
    return e


def _cycle(c, grids, chol, t, u, b):
    if t == 0:
        return torch.cholesky_solve(b.flatten(1)[:, :, None], chol)[:, :, 0].view_as(b)
    g = grids[t]
    for _ in range(c["nu1"]):
        u = g.sweep(u, b, True)
    r = torch.nn.functional.avg_pool2d(g.residual(u, b)[:, None], 2)[:, 0]
    u = u + _interpolate(_cycle(c, grids, chol, t - 1, torch.zeros_like(r), r))
    for _ in range(c["nu2"]):
        u = g.sweep(u, b, False)
    return u


def _solve(c, fields, level, y, mu0, keep=False):
    """FMG of the samples with normals y: F_0..F_level and, when asked for, the solutions."""
    F = torch.zeros(len(y), c["n_levels"], dtype=torch.float64, device="cuda")
    grids, sols, u = [], [], None
    for t in range(level + 1):
        n = c["n0"] << t
        grids.append(_Grid(fields(n, y)))
        b = torch.ones(len(y), n, n, dtype=torch.float64, device="cuda")
        if t == 0:
            chol = torch.linalg.cholesky(grids[0].matrix())
            u = _cycle(c, grids, chol, 0, None, b)
        else:
            u = _interpolate(u)
            if c["rtol"]:  # to the solution of the discrete equations, as far as 64 bits go
                for _ in range(12):
                    r = grids[t].residual(u, b)
                    if r.flatten(1).norm(dim=1).max() < 1e-11 * n:
                        break
                    u = u + _cycle(c, grids, chol, t, torch.zeros_like(u), r)
            else:
                for _ in range(mu0):
                    u = _cycle(c, grids, chol, t, u, b)
        h = n // 2
        F[:, t] = u.mean((1, 2)) if c["qoi"] == "mean" else u[:, h - 1: h + 1, h - 1: h + 1].mean((1, 2))
        if keep:
            sols.append(u[0].flatten())
    return (sols, F) if keep else F


def _all_samples(c, seed, z, fields, work_list, mu0):
    """F (samples in work order) with each sample's level and shift."""
    parts, levels, shifts = [], [], []
    for level, b, e, rb, re in work_list:
        r, n = np.repeat(np.arange(rb, re), e - b), np.tile(np.arange(b, e), re - rb)
        fine = c["n0"] << level
        chunk = max(1, int(3e8 / (fine * fine + c["n0"] ** 4 + c["s"])))
        for i in range(0, len(r), chunk):
            parts.append(_solve(c, fields, level, _normals(c, seed, z, level, r[i:i + chunk], n[i:i + chunk]), mu0))
        levels.append(np.full(len(r), level))
        shifts.append(r)
    return torch.cat(parts), torch.from_numpy(np.concatenate(levels)).cuda(), torch.from_numpy(np.concatenate(shifts)).cuda()


def _differences(F, levels):
    d = F.clone()
    d[:, 1:] -= F[:, :-1]
    return torch.where(torch.arange(F.shape[1], device="cuda")[None, :] <= levels[:, None], d, torch.zeros_like(d))


def _sums(c, d, levels, shifts):
    t = torch.arange(c["n_levels"], device="cuda")[None, :]
    used = (levels[:, None] >= t) if c["reuse"] else (levels[:, None] == t)
    d = torch.where(used, d, torch.zeros_like(d))
    out = torch.zeros(c["R"], c["n_levels"], 2, dtype=torch.float64, device="cuda")
    out.index_add_(0, shifts, torch.stack([d, d * d], -1))
    return out.transpose(0, 1).contiguous()


def _algorithm_1(c, seed, z, fields):
    nl, R, inf = c["n_levels"], c["R"], math.inf
    cost = np.cumsum([float(c["n0"] << t) ** 2 for t in range(nl)])
    sums = np.zeros((nl, R, 2))
    N, ybar, V, C, L, rounds, status, alpha, bias, clamped = [0] * nl, [0.0] * nl, [inf] * nl, [0.0] * nl, -1, 0, 0, math.nan, inf, 0

    def finish():
        U = np.array([sums[t, :, 0] / max(1, sum(N[t:L + 1])) for t in range(L + 1)])
        var = ((U - U.mean(1, keepdims=True)) ** 2).sum(1) / (R * (R - 1))
        q = U.sum(0)
        return U.mean(1), var, q.mean(), ((q - q.mean()) ** 2).sum() / (R * (R - 1))

    while True:
        if L >= 2:
            x, v = np.arange(1, L + 1), np.log2(np.abs(ybar[1:L + 1]))
            alpha = -float(np.polyfit(x, v, 1)[0])
            clamped = int(not alpha > 0)
            alpha = 0.5 if clamped else alpha
            bias = abs(ybar[L]) / (2 ** alpha + 1)
            if bias <= c["eps"] / math.sqrt(2):
                break
        if L + 1 >= nl:
            status = 7
            break
        L += 1
        while any(v == inf for v in V[: L + 1]) or finish()[3] > c["eps"] ** 2 / 2:
            ratio = [inf if V[t] == inf else V[t] / C[t] for t in range(L + 1)]
            t = ratio.index(max(ratio))
            begin, N[t] = N[t], max(1, 2 * N[t])
            F, levels, shifts = _all_samples(c, seed, z, fields, [(t, begin, N[t], 0, R)], c["mu0"])
            sums += _sums(c, _differences(F, levels), levels, shifts).cpu().numpy()
            C[t], rounds = float(cost[t]), rounds + 1
            mean, var, _, _ = finish()
            ybar[: t + 1], V[: t + 1] = mean[: t + 1].tolist(), var[: t + 1].tolist()
    _, _, Q, varQ = finish()
    for t in range(L + 1, nl):
        V[t] = inf
    return dict(Q=float(Q), varQ=float(varQ), bias=bias, alpha=alpha, L=L, rounds=rounds, run_status=status,
                alpha_clamped=clamped, N=N, Ybar=ybar, Vell=V, C=C)


def exact(case, seed):
    z, fields = _vector(case), _Fields(case)
    if case["kind"] == "estimate":
        return _algorithm_1(case, seed, z, fields)
    if case["kind"] == "solution":
        y = _normals(case, seed, z, case["level"], [seed % case["R"]], [seed % 64])
        u, F = _solve(case, fields, case["level"], y, case["mu0"], keep=True)
        return {"u": u, "F": F[0, : case["level"] + 1]}
    F, levels, shifts = _all_samples(case, seed, z, fields, _work_list(case), case["mu0"])
    if case["kind"] == "step":
        return {"sums": _sums(case, _differences(F, levels), levels, shifts), "F": F}
    hi, _, _ = _all_samples(case, seed, z, fields, _work_list(case), case["mu0"] + 1)
    D = _differences(hi, levels) - _differences(F, levels)
    return {"sums": _sums(case, D, levels, shifts), "D": D}
