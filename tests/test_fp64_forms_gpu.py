"""FP64 fields on both sides of the line where the modes' symmetry is used, and
the reuse sums of calls on both sides of the line between their CTA sizes."""
import numpy as np
import pytest

import workloads as W
from test_parity_gpu import _pair

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n0,levels", [(2, 6), (6, 5), (8, 4), (10, 4)])  # 32 | 64, 48 | 96, 32 | 64, 40 | 80
@pytest.mark.parametrize("s", [1, 2, 37])
def test_fp64_fields_with_and_without_the_symmetry(n0, levels, s):
    cfg, ctx, orc = _pair(W.LATTICE_6LEVEL, n0=n0, n_levels=levels, s=s, R=2, log2_nmax=4, precision="fp64", rtol=0.0)
    Y = W.random_normals(s, 2, tag=s)
    for t in (levels - 2, levels - 1):
        k = ctx.fields(t, torch.from_numpy(Y)).cpu().numpy()
        for i in range(2):
            assert np.max(np.abs(k[i] / orc.field(t, Y[i]) - 1.0)) < 1e-12, (t, i)


@pytest.mark.parametrize("points", [256, 257])  # 4,096 and 4,112 samples
def test_reuse_sums_match_the_samples(points):
    nl, R = 2, 16
    ctx = _pair(W.LATTICE_6LEVEL, n0=4, n_levels=nl, s=8, R=R, log2_nmax=10, precision="fp64", rtol=0.0)[1]
    S = torch.zeros(nl * R * 2, dtype=torch.float64, device="cuda")
    F = torch.zeros(points * R * nl, dtype=torch.float64, device="cuda")
    ctx.sample_levels([(1, 0, points, 0, R)], S, F)
    F = F.cpu().numpy().reshape(R, points, nl)
    d = np.stack([F[:, :, 0], F[:, :, 1] - F[:, :, 0]])
    S = S.cpu().numpy().reshape(nl, R, 2)
    mag = np.abs(d).sum(2)
    # sums of 257 terms in any order: 257 units of 2^-53 of the magnitudes
    assert (np.abs(S[:, :, 0] - d.sum(2)) <= 257 * 2.0 ** -53 * mag).all()
    assert (np.abs(S[:, :, 1] - (d * d).sum(2)) <= 258 * 2.0 ** -53 * (d * d).sum(2)).all()
