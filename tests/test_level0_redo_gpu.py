"""Level 0 of the mixed forms on samples that the pair factor solves and on samples
that it hands to the FP64 factor, side by side in one call.

One mode: a cross-shaped pattern, two cells of exp(t) within a ring of exp(-t) and
1 elsewhere, t = 8 y with the sample's normal y. Up to t = 5 the pairs' corrections
converge; from t = 8.5 the condition number, about exp(2 t), keeps them from it (found
by restating the pair arithmetic on the host: every t in steps of 1/4, sides 4 to 10)."""
import numpy as np
import pytest

import workloads as W
from test_level0_lanes_gpu import _f0

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
M = pytest.importorskip("paper_1806_05619_gb300")


def _context(n0, qoi):
    cfg = W.scaled(W.LATTICE_6LEVEL, n0=n0, n_levels=2, s=1, R=16, qoi=qoi, log2_nmax=12, precision="mixed_tf32", sigma=1.0,
                   corr_len=0.002)
    z, _ = M.cbc_genvec(1, 12)
    pattern = np.zeros((n0, n0))
    for y, x in ((1, 1), (1, 2)):
        for dy, dx in ((0, 1), (0, -1), (1, 0), (-1, 0)):
            pattern[y + dy, x + dx] = -1.0
    pattern[1, 1:3] = 1.0
    # nodes on the cell centres, a correlation length far below their distance: psi(x_p) = psi_p, z = y psi / n0
    return M.Context.from_config(cfg, genvec=z, covariance="matern", matern_nu=0.5, nystrom_m=n0,
                                 nystrom_theta=np.array([1.0 / n0 ** 2]), nystrom_psi=8.0 * n0 * pattern.reshape(-1, 1))


def _solve(k, n):
    """A u = 1 for fields k, by eliminating cells from the graph of faces: sums, products and quotients of positive
    numbers only, so every component is good to a few hundred roundings whatever the contrast."""
    ns, N = len(k), n * n
    k = k.reshape(ns, n, n).astype(np.float32)

    def face(a, b):
        return (np.float32(2) * a * b / (a + b)).astype(np.float64)

    w = np.zeros((ns, N, n + 1))  # w[p][q]: the face between cells p and p + q
    g = np.zeros((ns, n, n))      # faces on the boundary
    wv = w.reshape(ns, n, n, n + 1)
    wv[:, :, :-1, 1] = face(k[:, :, :-1], k[:, :, 1:])
    wv[:, :-1, :, n] = face(k[:, :-1], k[:, 1:])
    for edge in (np.s_[:, 0], np.s_[:, -1], np.s_[:, :, 0], np.s_[:, :, -1]):
        g[edge] += 2.0 * k[edge].astype(np.float64)
    g, f, d, x = g.reshape(ns, N), np.full((ns, N), 1.0 / N), np.zeros((ns, N)), np.zeros((ns, N))
    for p in range(N):
        d[:, p] = g[:, p] + w[:, p].sum(1)
        for a in range(1, min(n, N - 1 - p) + 1):
            c = w[:, p, a] / d[:, p]
            g[:, p + a] += c * g[:, p]
            f[:, p + a] += c * f[:, p]
            for b in range(a + 1, min(n, N - 1 - p) + 1):
                w[:, p + a, b - a] += c * w[:, p, b]
    for p in range(N - 1, -1, -1):
        m = min(n, N - 1 - p)
        x[:, p] = (f[:, p] + (w[:, p, 1:m + 1] * x[:, p + 1:p + m + 1]).sum(1)) / d[:, p]
    return x


@pytest.mark.parametrize("n0", [4, 6, 8, 10])
@pytest.mark.parametrize("qoi", ["mean", "center"])
@pytest.mark.parametrize("points", [3, 100, 400])  # 48, 1,600 (four lanes per row up to n0 = 8) and 6,400 samples (one)
def test_pairs_and_fp64_redo_side_by_side(n0, qoi, points):
    ctx = _context(n0, qoi)
    F = _f0(ctx, 2, 16, points, 16)
    y = torch.cat([ctx.normals(0, r, 0, points) for r in range(16)])
    t = 8.0 * y.cpu().numpy()[:, 0]
    u = _solve(ctx.fields(0, y).cpu().numpy(), n0)
    m = n0 // 2
    want = u.mean(1) if qoi == "mean" else u.reshape(-1, n0, n0)[:, m - 1:m + 1, m - 1:m + 1].mean((1, 2))
    # Faces within two units of 2^-23 of these move every component by at most 2 N times that (each is a ratio of
    # sums of products of N faces). An FP64 factor's last pivot, about 4 exp(-2 t) of its diagonal, is off by n0 + 2
    # roundings of that diagonal. Beyond t = 12 that bound says nothing any more.
    tol = 2 * n0 * n0 * 2.0 ** -22 + 16 * 2.0 ** -53 * np.exp(2 * np.maximum(t, 0))
    use = t <= 12
    redo, pairs = use & (t >= 8.5), t <= 5
    assert redo.sum() >= points // 3 and pairs.sum() >= points  # of 16 times `points` samples
    scale = u.max(1) if qoi == "center" else want  # the island holds the largest values
    err = np.abs(F.reshape(-1) - want) / scale
    assert (err[use] <= tol[use]).all(), (np.flatnonzero(use & ~(err <= tol))[:5], err[use].max())
    for i in [int(np.flatnonzero(redo)[0]), int(np.flatnonzero(pairs)[0])]:
        sols, _ = ctx.sample_solution(0, i // points, i % points)
        assert (np.abs(sols[0].cpu().numpy() - u[i]) <= tol[i] * u[i].max()).all(), i
    ctx.check_device()
