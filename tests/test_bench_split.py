"""bench.py names the time split that a launch runs: none, every tile's, or a mix of whole and cut tiles (CPU)."""
import pytest


@pytest.fixture(scope="module")
def bench():
    import bench
    import paper_1503_06203_gb300 as xe
    xe.build()
    return bench


@pytest.mark.parametrize("N,F,T,split,name", [
    (256, 256, 16384, 0, "1"),          # whole tiles
    (256, 16, 1024, 0, "152+8x4"),      # 152 whole tiles, 8 cut into four ranges
    (250, 61, 4001, 0, "608+2x32"),
    (64, 1, 7 * 128, 0, "7"),           # every tile cut
    (256, 16, 1024, 4, "4"),            # as the option says
    (256, 16, 1024, 64, "8"),           # not into more ranges than chunks
    (256, 16, 1024, 1, "1"),
])
def test_effective_split(bench, N, F, T, split, name):
    assert bench.effective_split(N, F, T, split, 152) == name


@pytest.mark.parametrize("workload,shape", [("pathfinder", (256, 256, 16384)), ("large_n", (8192, 4, 2048))])
def test_traffic_record(bench, workload, shape):
    split = bench.effective_split(*shape, 0, 152)
    N, F, T = shape
    moved = N * F * T + 4 * N * (N + 1) * F
    r = bench.recorded_traffic(workload, 1, split, 5)  # None once the kernel's source is another one
    assert r is None or 0.9 * moved < r < 1.1 * moved
    assert bench.recorded_traffic(workload, 1, "152+8x4", 5) is None and bench.recorded_traffic(workload, 1, split, 6) is None
