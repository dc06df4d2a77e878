"""What the bench compares and reports: its cross-check's binary64 arm shares no search kernel
with the timed one, and the search's roofline is the bound that its profile shows."""
import bench
import paper_1310_3437_gb300 as kmc


def test_the_check_is_independent_of_the_timed_search():
    p = bench.check_params(bench.headline_setup(1 << 12))
    assert p.precision == kmc.KMC_FP64
    assert p.search_kernel == kmc.KMC_SEARCH_PARTICLE  # not the tiles that the default takes
    assert p.flags & kmc.KMC_FLAG_NO_SPLIT  # nor the fast-particle search


def test_the_search_roofline_is_issue_slots():
    r = bench.search_roofline({"dram_bytes_per_particle": 30.0, "issue_active_pct": 71.5}, 1 << 24, 2.0,
                              1e10, 6678.8)
    assert (r["bound"], r["achieved"], r["peak"], r["frac"]) == ("issue", 71.5, 100.0, 0.715)
    assert abs(r["hbm_frac"] - 30.0 * (1 << 24) / 2e-3 / 6678.8e9) < 1e-12
    stale = bench.search_roofline(None, 1 << 24, 2.0, 1e10, 6678.8)
    assert stale["achieved"] is None and stale["frac"] is None and stale["hbm_frac"] is None
