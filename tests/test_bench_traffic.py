"""The benchmark's DRAM traffic figure of the FP64 headline: of the kernel that runs (CPU only)."""
import bench


def test_the_headline_has_a_figure_for_its_own_kernel(monkeypatch):
    vh = 1048576
    assert {"tm_fix.cuh", "tm_fix.cu"} <= set(bench.TRAFFIC_SOURCES)   # where k_fx_hop is
    monkeypatch.setitem(bench.TRAFFIC, "src", bench.kernel_source_hash())
    t = bench.traffic_per_launch("f64", 18, vh)
    # links once, a fixed-point field, the re-read input and the output; twice that would be a second read of all
    need = (8 * 18 + 24 + 24) * 8 + 196
    assert 0.9 * need * vh < t < 1.2 * need * vh
    assert bench.traffic_per_launch("f64", 18, vh, fixed=False) is None   # FP64 products: another kernel
