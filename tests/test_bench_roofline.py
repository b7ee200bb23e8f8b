"""The benchmark's roofline is a rate of work that the walk does: race draws, one per neighbour and walker, against the
integer pipes.  The FP64 work of determinants that share their rows is reported beside it, as no fraction of a peak
(counted for each determinant by itself it exceeds what the walk computes, and once exceeded a measured peak)."""
import bench


def test_rate_is_draws_over_time_and_the_only_fraction():
    r = bench.roofline(345000.0, 4096, 13e-3, distinct=684.0, terms=5.0e9, neighbours_once=2.3e8)
    assert abs(r["achieved"] * 1e12 - 345000.0 * 4096 / 13e-3) < 1e-6 * r["achieved"] * 1e12
    assert abs(r["frac"] - r["achieved"] / r["peak"]) < 1e-15 and 0.0 < r["frac"] < 1.0

    def keys(d):
        for k, v in d.items():
            yield k
            if isinstance(v, dict):
                yield from keys(v)

    assert [k for k in keys(r) if "frac" in k] == ["frac"]
    assert r["unshared_work"]["flops_per_step"] == 2.0 * 5.0e9 + 8.0 * 2.3e8


def test_more_terms_do_not_raise_the_rate():
    a = bench.roofline(1e5, 1024, 0.1, distinct=300.0, terms=1e9, neighbours_once=3e7)
    b = bench.roofline(1e5, 1024, 0.1, distinct=300.0, terms=9e9, neighbours_once=3e7)
    assert a["achieved"] == b["achieved"] and a["frac"] == b["frac"]
