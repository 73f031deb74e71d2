"""Stream priorities of serving slots (CPU): higher, that is more negative, for smaller
maps, within the range that PyTorch's stream pools have (0 to -3)."""
from paper_2510_01785_gb300.serve import GpuExecutor


def test_priority_by_nside():
    p = {n: GpuExecutor.stream_priority(n) for n in (1, 2, 64, 128, 256, 512, 1024, 2048)}
    assert p[2048] == 0 and p[1024] == -1 and p[512] == -2
    assert all(p[n] == -3 for n in (1, 2, 64, 128, 256))
