"""The refinement residual and its norm on levels with constant coefficient, whose
faces are exact (1, and 2 on the boundary), so that the norm can be formed again."""
import numpy as np
import pytest

import workloads as W
from test_parity_gpu import _pair

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _context(n0, levels, rtol):
    return _pair(W.LATTICE_6LEVEL, n0=n0, n_levels=levels, s=12, R=2, log2_nmax=6, precision="mixed_tf32", sigma=1e-12,
                 rtol=rtol, max_cycles=40)[1]


def _norm(u):
    """||1 - A u|| / ||1|| of an n x n grid, beyond FP64."""
    n = u.shape[0]
    v = np.zeros((n + 2, n + 2), dtype=np.longdouble)
    v[1:-1, 1:-1] = u
    c = v[1:-1, 1:-1]
    acc = np.zeros_like(c)
    for part in (v[1:-1, :-2], v[1:-1, 2:], v[:-2, 1:-1], v[2:, 1:-1]):
        acc += c - part
    # a boundary face is twice as heavy
    acc[:, 0] += c[:, 0]
    acc[:, -1] += c[:, -1]
    acc[0, :] += c[0, :]
    acc[-1, :] += c[-1, :]
    r = 1 - n * n * acc
    return float(np.sqrt((r * r).mean()))


@pytest.mark.parametrize("n0,levels", [(16, 2), (2, 5)])
def test_tolerance_just_above_the_rounding_of_fp64_values(n0, levels):
    """32 cells per side: FP64 values of the solution leave a residual of 8.9e-15 (each
    off by half a unit at most, one standard deviation over 1,024 cells 3 %); a
    residual formed with 48 bits reads 1.1e-14 there and would not converge."""
    ctx = _context(n0, levels, 9.8e-15)
    u, _ = ctx.sample_solution(levels - 1, 0, 0)
    ctx.check_device()
    n = n0 << (levels - 1)
    assert _norm(u[-1].cpu().numpy().reshape(n, n)) <= 9.8e-15 * (1 + 1e-3)


@pytest.mark.parametrize("n0,levels", [(6, 5), (10, 5), (10, 6), (6, 7), (14, 6)])
def test_norm_that_ends_the_refinement_holds(n0, levels):
    """96 to 448 cells per side: part and whole tiles of the forms with two and with
    eight rows per strip. The norm formed again is below the tolerance, here some
    hundred times the rounding of the values, to the accuracy of its FP64 form."""
    rtol = 1e-10
    ctx = _context(n0, levels, rtol)
    u, _ = ctx.sample_solution(levels - 1, 1, 3)
    ctx.check_device()
    n = n0 << (levels - 1)
    # FP64's own error in r: 2^-51 of the fluxes n^2 sum |k d| <= 4 n^2 max|u| each
    assert _norm(u[-1].cpu().numpy().reshape(n, n)) <= rtol + 2.0 ** -51 * 4 * n * n * 0.08
