"""FP64 form: what a sample gives depends on the sample alone, to the last bit, also
where a call's size chooses other kernels for it (one launch per sample or one per
level on the small levels, several lanes or one thread on level 0)."""
import numpy as np
import pytest

import workloads as W
from test_level0_lanes_gpu import _f0
from test_parity_gpu import _pair
from test_small_levels_gpu import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n0,levels", [(4, 5), (4, 6), (6, 5), (8, 4), (8, 5), (10, 4)])  # finest sides 64, 128, 96, 64, 128, 80
@pytest.mark.parametrize("qoi,nu1,nu2", [("mean", 2, 2), ("center", 1, 3)])
def test_samples_of_small_and_large_calls_have_the_same_bits(n0, levels, qoi, nu1, nu2):
    ctx = _pair(W.LATTICE_6LEVEL, n0=n0, n_levels=levels, s=12, R=2, qoi=qoi, log2_nmax=11, precision="fp64", nu1=nu1, nu2=nu2)[1]
    top = levels - 1
    few = _run(ctx, levels, 2, [(top, 0, 3, 0, 2), (1, 0, 2, 0, 2)])
    many = _run(ctx, levels, 2, [(top, 0, 1100, 0, 2), (1, 0, 2, 0, 2)])  # 2,200 samples on every level
    assert few[:6].all()
    assert np.array_equal(few[:6].reshape(2, 3, levels), many[:2200].reshape(2, 1100, levels)[:, :3])
    assert np.array_equal(few[6:], many[2200:])


@pytest.mark.parametrize("n0", [6, 10])  # 4 and 8: test_level0_lanes_gpu.py
@pytest.mark.parametrize("qoi", ["mean", "center"])
def test_level0_of_24064_samples_and_of_few(n0, qoi):
    ctx = _pair(W.LATTICE_6LEVEL, n0=n0, n_levels=2, s=20, R=16, qoi=qoi, log2_nmax=12, precision="fp64")[1]
    assert np.array_equal(_f0(ctx, 2, 16, 1504, 16)[:, :81], _f0(ctx, 2, 16, 81, 16))
