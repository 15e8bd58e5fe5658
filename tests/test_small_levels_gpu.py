"""The small levels (up to 64 cells per side) of a sample in one launch: the FMG
stages and the V-cycles' part on them, on every coarsest side the kernels are
built for, at the edges of their classes."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from test_parity_gpu import _pair, _rel

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SIDES = [(4, 2), (4, 6), (6, 3), (6, 5), (8, 2), (8, 5), (10, 3), (10, 4)]  # coarsest side, levels


def _run(ctx, nl, R, work):
    ns = sum((e - b) * (re - rb) for _, b, e, rb, re in work)
    S = torch.zeros(nl * R * 2, dtype=torch.float64, device="cuda")
    F = torch.zeros(ns * nl, dtype=torch.float64, device="cuda")
    ctx.sample_levels(work, S, F)
    torch.cuda.synchronize()
    ctx.check_device()
    return F.cpu().numpy().reshape(ns, nl)


@pytest.mark.parametrize("n0,levels", SIDES)
@pytest.mark.parametrize("nu1,nu2,qoi", [(2, 2, "mean"), (1, 3, "center")])
def test_fp64_samples_of_every_finest_level_match_oracle(n0, levels, nu1, nu2, qoi):
    """FP64 form: one to three samples ending on each level in one call, so that
    every class of the stages' launches and the V-cycles above them run."""
    cfg, ctx, orc = _pair(W.LATTICE_6LEVEL, n0=n0, n_levels=levels, s=12, R=2, qoi=qoi, log2_nmax=6, nu1=nu1, nu2=nu2)
    work = [(lv, 0, 1 + lv % 3, 0, 2) for lv in range(levels)]
    F = _run(ctx, levels, 2, work)
    q = 0
    for lv, b, e, rb, re in work:
        for r in range(rb, re):
            for n in range(b, e):
                ref = orc.sample(lv, r, n)
                assert ref["status"] == O.OK
                assert _rel(F[q, : lv + 1], ref["F"]) < 1e-12, (lv, r, n)
                assert not F[q, lv + 1:].any()
                q += 1


@pytest.mark.parametrize("n0,levels", SIDES)
@pytest.mark.parametrize("precision,rtol", [("mixed_tf32", 0.0), ("mixed_bf16x3", 1e-10)])
def test_mixed_sample_alone_and_in_a_batch(n0, levels, precision, rtol):
    """Mixed forms: a sample's F does not depend on the samples around it (300
    of them, the batch sizes' other class), and its solutions, which the
    single-sample call also writes out, have that F as their mean."""
    cfg, ctx, orc = _pair(W.LATTICE_6LEVEL, n0=n0, n_levels=levels, s=12, R=2, log2_nmax=8, precision=precision, rtol=rtol)
    top = levels - 1
    F = _run(ctx, levels, 2, [(top, 0, 2, 0, 2), (1, 0, 150, 0, 2)])
    for row, (r, n) in [(0, (0, 0)), (3, (1, 1))]:
        u, Fs = ctx.sample_solution(top, r, n)
        Fs = Fs.cpu().numpy()
        # levels whose two classes of batch size may take other smoothers agree to FP32 rounding
        tol = [1e-13 if (n0 << t) <= 64 else 1e-6 for t in range(levels)]
        for t in range(levels):
            assert abs(F[row, t] / Fs[t] - 1) <= tol[t], (t, F[row, t], Fs[t])
            assert abs(float(u[t].mean()) / Fs[t] - 1) <= 1e-13, t
    ctx.check_device()
