"""The level-0 exact solve on several lanes per sample (four or one per row of
the working window, by the call's samples) at the edges of its ranges."""
import numpy as np
import pytest

import workloads as W
from test_parity_gpu import _pair

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _f0(ctx, nl, R, n_end, r_end):
    S = torch.zeros(nl * R * 2, dtype=torch.float64, device="cuda")
    F = torch.zeros(n_end * r_end * nl, dtype=torch.float64, device="cuda")
    ctx.sample_levels([(0, 0, n_end, 0, r_end)], S, F)
    torch.cuda.synchronize()
    ctx.check_device()
    return F.cpu().numpy().reshape(r_end, n_end, nl)[:, :, 0]


@pytest.mark.parametrize("n0", [4, 6, 8, 10])
@pytest.mark.parametrize("qoi", ["mean", "center"])
def test_level0_same_bits_at_every_batch_size(n0, qoi):
    """FP64 form: one sample, a few (a warp's samples incomplete), the last
    call on four lanes per row, the first on one: every sum takes its terms in
    one order, so F_0 is the same to the last bit (and for n0 = 4, 8 the same as
    the thread-per-sample kernel's), and within 1e-12 of the oracle."""
    cfg, ctx, orc = _pair(W.LATTICE_6LEVEL, n0=n0, n_levels=2, s=20, R=16, qoi=qoi, log2_nmax=12, precision="fp64")
    want = _f0(ctx, 2, 16, 81, 16)  # 1,296 samples: one lane per row
    if n0 in (4, 8):  # 24,064 samples: one thread per sample
        assert np.array_equal(_f0(ctx, 2, 16, 1504, 16)[:, :81], want)
    for n_end, r_end in [(1, 1), (1, 16), (3, 1), (79, 16), (1281, 1)]:
        got = _f0(ctx, 2, 16, n_end, r_end)
        m = min(n_end, 81)
        assert np.array_equal(got[:, :m], want[:r_end, :m]), (n_end, r_end)
    for r, n in [(0, 0), (7, 40), (15, 80)]:
        assert abs(want[r, n] / orc.sample(0, r, n)["F"][0] - 1) <= 1e-12
