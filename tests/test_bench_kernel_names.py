"""Host logic: the kernel that a bucket of the bench's event table is named by."""
import bench


def test_small_levels_in_one_launch_are_not_named_by_the_coarse_solve():
    smoothers = ["gs", "whole", "whole", "whole", "tma"]
    assert bench.kernel_name("coarse", 3, smoothers) == "kb_small_stages, kb_small_vcycle"
    assert bench.kernel_name("coarse", 0, smoothers) == "kb_coarse_fixed"
    assert bench.kernel_name("smooth", 4, smoothers) == "kb_rbgs_tma"
    assert "kb_level0_pairs" in bench.kernel_name("level0", 0, smoothers)
