"""Round graphs on either side of the lines at which a call's size changes the list of
its launches: rounds that take turns across a line keep two instantiated graphs, which
the later rounds update, and give the sums and samples of the direct path."""
import numpy as np
import pytest

import workloads as W
from test_round_graphs_gpu import _call

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
M = pytest.importorskip("paper_1806_05619_gb300")


@pytest.mark.parametrize("precision,rtol,levels,below,above", [
    ("mixed_tf32", 0.0, 4, 46, 50),      # 2^18 cells: the faces in one launch, or one per level
    ("fp64", 0.0, 3, 2040, 2060),        # 2,048 samples: small stages per sample, or level by level
    ("fp64", 1e-10, 3, 2040, 2060),      # the same for the V-cycles of the converged form
    ("mixed_tf32", 1e-10, 5, 8, 9),      # the loop's norms, flags and decision in one launch, or two
    ("mixed_tf32", 0.0, 3, 3070, 3074),  # 3,072 samples: four lanes or one per row of level 0
    ("fp64", 0.0, 1, 1278, 1282),        # 1,280 samples: the same in FP64
])
def test_rounds_across_a_line_update_two_graphs(precision, rtol, levels, below, above):
    cfg = W.scaled(W.LATTICE_6LEVEL, n_levels=levels, R=2, s=12, precision=precision, rtol=rtol, max_cycles=30, log2_nmax=13)
    z, _ = M.cbc_genvec(cfg["s"], cfg["log2_nmax"])
    ctx = M.Context.from_config(cfg, genvec=z)
    ctx.set_round_graphs("on")
    top = levels - 1
    rounds = []
    for k in range(3):
        for count in (below, above):
            half = count // 2
            rounds.append([(top, k, k + half, 0, 2)] + [(top, k + half, k + half + 1, 0, 1)] * (count % 2))
    on = [_call(ctx, cfg, work) for work in rounds]
    st = ctx.graph_stats()
    assert st["round_launches"] == len(rounds)
    assert st["round_instantiations"] <= 2 and st["round_updates"] >= 4
    ctx.set_graphs(False)
    for work, a in zip(rounds, on):
        b = _call(ctx, cfg, work)
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]), work
