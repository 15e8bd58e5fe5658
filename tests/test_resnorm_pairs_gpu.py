"""The refinement residual from FP32 pairs (levels refined to a tolerance)."""
import pytest

import workloads as W
from test_parity_gpu import _pair

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n0,levels", [(10, 4), (6, 5), (8, 5), (10, 5), (8, 6), (12, 5)])
def test_refined_solution_is_the_fixed_cycle_limit(n0, levels):
    """80 to 256 cells per side (part, whole and several tiles of 128 x 64): the
    refined solution against 40 V-cycles on the one first residual, which another
    kernel forms. Those stagnate at FP32 rounding of the correction (2^-24, up to
    the side's length in accumulation, times |e| / |u| < 0.05: below 1e-6); a
    wrong neighbour or face at a tile's edge moves its cells by about 1/n."""
    kw = dict(n0=n0, n_levels=levels, s=12, R=2, log2_nmax=6, precision="mixed_tf32")
    fixed = _pair(W.LATTICE_6LEVEL, mu0=40, rtol=0.0, **kw)[1]
    refined = _pair(W.LATTICE_6LEVEL, mu0=2, rtol=1e-10, **kw)[1]
    for r, n in [(0, 0), (1, 5)]:
        a, _ = fixed.sample_solution(levels - 1, r, n)
        b, _ = refined.sample_solution(levels - 1, r, n)
        for t in range(levels):
            err = (a[t] - b[t]).abs().max() / a[t].abs().max()
            assert float(err) < 5e-6, (t, float(err))
    fixed.check_device()
    refined.check_device()


@pytest.mark.parametrize("n0,levels", [(6, 5), (8, 5)])
def test_refined_sample_alone_and_beside_converged_ones(n0, levels):
    """A sample that needs more passes than its neighbours (their residual is not
    formed again) has the F that it has alone, to what the tolerance leaves open."""
    cfg, ctx, _ = _pair(W.LATTICE_6LEVEL, n0=n0, n_levels=levels, s=12, R=2, log2_nmax=6, precision="mixed_bf16x3", rtol=1e-10)
    top = levels - 1
    S = torch.zeros(levels * 2 * 2, dtype=torch.float64, device="cuda")
    F = torch.zeros(32 * levels, dtype=torch.float64, device="cuda")
    ctx.sample_levels([(top, 0, 16, 0, 2)], S, F)
    F = F.reshape(32, levels).cpu()
    for i, (r, n) in [(0, (0, 0)), (7, (0, 7)), (16, (1, 0)), (31, (1, 15))]:
        _, f = ctx.sample_solution(top, r, n)
        # the same operations per sample on every level, but the two classes of batch size may differ in their smoother
        assert float((F[i] / f.cpu() - 1).abs().max()) < 1e-9, i
    ctx.check_device()
