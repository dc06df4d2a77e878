"""What the bench compares and reports: its cross-check's binary64 arm shares no search kernel
with the timed one."""
import bench
import paper_1310_3437_gb300 as kmc


def test_the_check_is_independent_of_the_timed_search():
    p = bench.check_params(bench.headline_setup(1 << 12))
    assert p.precision == kmc.KMC_FP64
    assert p.search_kernel == kmc.KMC_SEARCH_PARTICLE  # not the tiles that the default takes
    assert p.flags & kmc.KMC_FLAG_NO_SPLIT  # nor the fast-particle search
