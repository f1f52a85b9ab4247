"""The benchmark's count of binning launches follows the library's rule for the
form (plan_of in kf_bin.cu)."""
import bench


def test_binning_launches_follow_the_form():
    n = lambda *a: bench.binning_launches(*a, 152)
    assert n(1, 350, 7_000_000) == 1 and n(0, 350, 7_000_000) == 5  # a block a segment (and large ones, order)
    assert n(1, 70, 1_400_000) == 4 and n(0, 70, 1_400_000) == 5    # passes over all hits
    assert n(0, 28, 84_000) == 2 and n(0, 7, 0) == 1
    assert bench.build_step_launches(dict(build_scan=4, bin_unordered=1), 7, 6, 70, 1_400_000, 152) == 1 + 4 + 3
