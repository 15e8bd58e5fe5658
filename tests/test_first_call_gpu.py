"""Mixed forms, device memory at creation: the pools of the levels up to 64 cells per
side are there, so that neither the first call nor the first rounds of Algorithm 1
allocate them; buffers that nothing reads are not."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
M = pytest.importorskip("paper_1806_05619_gb300")


@pytest.mark.parametrize("n0,levels", [(8, 4), (4, 5)])
def test_first_call_of_a_small_context_allocates_no_pool(n0, levels):
    cfg = W.scaled(W.LATTICE_6LEVEL, n0=n0, n_levels=levels, s=24, R=2, precision="mixed_tf32", log2_nmax=12)
    z, _ = M.cbc_genvec(cfg["s"], cfg["log2_nmax"])
    sums = torch.zeros(levels * 2 * 2, dtype=torch.float64, device="cuda")
    warm = M.Context.from_config(cfg, genvec=z)  # the library's own code and tables
    warm.sample_levels([(levels - 1, 0, 4, 0, 2)], sums)
    ctx = M.Context.from_config(cfg, genvec=z)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ctx.sample_levels([(levels - 1, 0, 512, 0, 2)], sums)  # 1,024 samples: more than 200 MB of pools
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] <= 16 << 20
    ctx.check_device()


def test_creation_keeps_no_fp64_factor_that_nothing_reads():
    """Sides whose mixed form factors level 0 in FP32 pairs: of the factors of 65,536
    samples (8 x 8 cells) only the FP32 one, 151 MB, beside 30 MB of points and sums."""
    cfg = W.scaled(W.LATTICE_6LEVEL, n0=8, n_levels=1, s=8, R=2, precision="mixed_tf32", log2_nmax=12)
    z, _ = M.cbc_genvec(cfg["s"], cfg["log2_nmax"])
    warm = M.Context.from_config(cfg, genvec=z)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ctx = M.Context.from_config(cfg, genvec=z)
    assert before - torch.cuda.mem_get_info()[0] <= 256 << 20
    sums = torch.zeros(4, dtype=torch.float64, device="cuda")
    for c in (warm, ctx):
        c.sample_levels([(0, 0, 64, 0, 2)], sums)
        c.check_device()


def test_grown_pools_keep_results_and_are_given_back():
    """Calls that grow a level's pool past creation's 1,024 samples again and again: the
    same samples, and all of the memory back when the context is closed (old blocks are
    kept meanwhile, 64 MB at most)."""
    levels = 3
    cfg = W.scaled(W.LATTICE_6LEVEL, n0=8, n_levels=levels, s=24, R=2, precision="mixed_tf32", log2_nmax=15)
    z, _ = M.cbc_genvec(cfg["s"], 12)
    sums = torch.zeros(levels * 2 * 2, dtype=torch.float64, device="cuda")
    F = torch.zeros(2 * 12000 * levels, dtype=torch.float64, device="cuda")
    warm = M.Context.from_config(cfg, genvec=z)
    warm.sample_levels([(levels - 1, 0, 4, 0, 2)], sums)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ctx = M.Context.from_config(cfg, genvec=z)
    seen = []
    for points in (150, 600, 1500, 3000, 12000):  # more than 256 samples each: one class of batch size
        ctx.sample_levels([(levels - 1, 0, points, 0, 2)], sums, F)
        seen.append(F[: 2 * points * levels].view(2, points, levels)[:, :150].clone())
    assert all(torch.equal(seen[0], q) for q in seen[1:])
    ctx.check_device()
    ctx.close()
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] <= 16 << 20
