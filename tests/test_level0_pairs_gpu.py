"""Level 0 of the mixed forms: factor and solve in FP32 pairs, corrected with FP64 residuals."""
import numpy as np
import pytest

import workloads as W
from test_level0_lanes_gpu import _f0
from test_parity_gpu import _pair

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SIDES = [4, 6, 8, 10]


def _context(n0, sigma, qoi="mean", precision="mixed_tf32"):
    return _pair(W.LATTICE_6LEVEL, n0=n0, n_levels=2, s=20, R=16, qoi=qoi, log2_nmax=12, precision=precision, sigma=sigma)[1]


@pytest.mark.parametrize("n0", SIDES)
@pytest.mark.parametrize("sigma", [1.0, 12.0])
def test_same_bits_at_every_batch_size(n0, sigma):
    """One sample, a few (a warp's samples incomplete), calls on either side of the
    line between four lanes per row and one: the same operations per sample (also
    where a contrast of many decades sends samples to the FP64 factor, or FP32
    faces overflow)."""
    ctx = _context(n0, sigma)
    want = _f0(ctx, 2, 16, 385, 16)  # 6,160 samples: one lane per row
    assert (want[np.isfinite(want)] > 0).all()  # the inverse of an M-matrix is positive
    for n_end, r_end in [(1, 1), (1, 16), (3, 1), (127, 16), (128, 16), (3071, 1), (3072, 1)]:
        got = _f0(ctx, 2, 16, n_end, r_end)
        m = min(n_end, 385)
        assert np.array_equal(got[:, :m], want[:r_end, :m], equal_nan=True), (n_end, r_end)


@pytest.mark.parametrize("n0", SIDES)
@pytest.mark.parametrize("qoi", ["mean", "center"])
def test_constant_coefficient_to_fp64(n0, qoi):
    """sigma so small that k = 1 and every face is exact: the five-point Poisson
    matrix, whose condition is below n0^2: FP64 solutions agree to n0^2 units of 2^-53."""
    ctx = _context(n0, 1e-12, qoi)
    N = n0 * n0
    A = np.zeros((N, N))
    for y in range(n0):
        for x in range(n0):
            p = y * n0 + x
            for dy, dx in [(0, 1), (0, -1), (1, 0), (-1, 0)]:
                Y, X = y + dy, x + dx
                inside = 0 <= Y < n0 and 0 <= X < n0
                A[p, p] += 1.0 if inside else 2.0
                if inside:
                    A[p, Y * n0 + X] -= 1.0
    u = np.linalg.solve(A, np.full(N, 1.0 / N))
    sols, F = ctx.sample_solution(0, 0, 0)
    tol = n0 * n0 * 2.0 ** -52
    assert np.abs(sols[0].cpu().numpy() / u - 1).max() <= tol
    m = n0 // 2
    g = u.reshape(n0, n0)
    f = u.mean() if qoi == "mean" else g[m - 1:m + 1, m - 1:m + 1].mean()
    assert abs(float(F[0]) / f - 1) <= tol
    ctx.check_device()
