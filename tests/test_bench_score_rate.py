"""What the benchmark says of stages that its instruction and kernel counts do
not describe: the bounded scoring has a rate and no fraction of a peak, and the
cross-brick stage says how many kernels it is."""
import bench


def test_bounded_scoring_has_no_fraction_of_the_issue_peak():
    r = bench.score_rate(256, 48_000_000, 1.2, 40.0)
    assert "frac" not in r and "achieved" not in r
    assert r["point_hypothesis_pairs_decided_per_s"] == round(256 * 48e6 / 1.2e-3, 1)
    assert r["ms_to_test_every_pair_at_the_fp32_peak"] == round(5 * 256 * 48e6 / 40e12 * 1e3, 4)


def test_the_cross_brick_stage_counts_its_kernels():
    st = {"occupied_voxels": 1000, "steppable_voxels": 600, "bricks_allocated": 10}
    t = bench.kernel_table({"ccl_cross": (0.5, 10), "moments": (0.2, 10)}, st, None, n_points_segment=4000)
    assert t["ccl_cross"]["kernels"] == 3 and t["moments"]["kernels"] == 1
    assert bench.roofline(t)["kernel"] == "ccl_cross"  # one unit of the method
