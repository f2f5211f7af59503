"""bench.py's count of the kernel launches of a mixed call (no GPU)."""
import bench


def test_launches_of_the_two_phase_path_follow_its_event_slices():
    assert bench.launches_per_sigma("ggttgg", 1 << 20) == 1
    assert [bench.launches_per_sigma("ggttggg", n) for n in (1, 8704, 8705, 2 * 8704 + 5, 1 << 20)] == [2, 2, 4, 6, 242]
