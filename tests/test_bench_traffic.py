"""The bench reports a kernel's DRAM traffic only while its sources are those of
the capture: every recorded digest is that of the present sources, and every
kernel that the bench can ask for has an entry."""
import bench


def test_recorded_traffic_is_of_the_present_sources():
    for (kernel, _), (digest, nbytes) in bench.TRAFFIC.items():
        assert digest == bench.source_digest(kernel), kernel
        assert nbytes > 0
    assert {kernel for kernel, _ in bench.TRAFFIC} == set(bench.KERNEL_SOURCES)


def test_reported_traffic():
    assert bench.traffic_of("bat_rows", "batched_512") == 659.993e6 + 409.877e6
    assert bench.traffic_of("bat_rows", "rotated_d1000") is None
