"""The benchmark charges the TV prox the bytes its launches move: 44 a voxel per launch, of two iterations.  CPU only."""
import bench


def test_bytes_are_those_of_the_launches():
    assert bench.prox_bytes_per_voxel(50) == 22.0
    assert bench.prox_bytes_per_voxel(1) == 44.0
    assert abs(bench.prox_bytes_per_voxel(5) - 44.0 * 3 / 5) < 1e-12
