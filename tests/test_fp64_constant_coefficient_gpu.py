"""FP64 form on constant coefficients of many sizes: the solution is the Poisson
problem's divided by k, so the reciprocals and reciprocal square roots of the faces and
the factor (hardware estimates refined by one step) show in F_0 to its last bits."""
import numpy as np
import pytest

import workloads as W
from test_level0_lanes_gpu import _f0

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
M = pytest.importorskip("paper_1806_05619_gb300")


@pytest.mark.parametrize("n0", [2, 4, 6, 8])
def test_f0_times_k_is_the_poisson_value(n0):
    """k = exp(6 y), 20,800 samples. The condition of the Poisson matrix is below
    n0^2 and all its solution's sums are of positive numbers: n0^2 units of 2^-53 for
    the factor and the solve, 4 for k and the faces."""
    cfg = W.scaled(W.LATTICE_6LEVEL, n0=n0, n_levels=1, s=1, R=16, qoi="mean", log2_nmax=12, precision="fp64", sigma=1.0,
                   corr_len=0.002)
    z, _ = M.cbc_genvec(1, 12)
    # nodes on the cell centres, a correlation length far below their distance: z = y psi / n0
    ctx = M.Context.from_config(cfg, genvec=z, covariance="matern", matern_nu=0.5, nystrom_m=n0,
                                nystrom_theta=np.array([1.0 / n0 ** 2]), nystrom_psi=np.full((n0 * n0, 1), 6.0 * n0))
    F = _f0(ctx, 1, 16, 1300, 16).reshape(-1)
    y = torch.cat([ctx.normals(0, r, 0, 1300) for r in range(16)])
    k = ctx.fields(0, y).cpu().numpy()
    assert (np.abs(k / k[:, :1] - 1) <= 2.0 ** -50).all()  # one value per sample, its cells' exponents apart by a rounding
    N = n0 * n0
    A = np.zeros((N, N))
    for q in range(N):
        for d, edge in ((1, q % n0 == n0 - 1), (-1, q % n0 == 0), (n0, q >= N - n0), (-n0, q < n0)):
            A[q, q] += 2.0 if edge else 1.0
            if not edge:
                A[q, q + d] -= 1.0
    want = np.linalg.solve(A, np.full(N, 1.0 / N)).mean()
    spread = np.abs(k / k.mean(1, keepdims=True) - 1).max(1)
    assert (np.abs(F * k.mean(1) / want - 1) <= (N + 4) * 2.0 ** -53 + spread).all()
    ctx.check_device()
