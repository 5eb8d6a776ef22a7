"""The bench's bytes of a step: pairs of steps move them once, a step left over once more."""
import bench


def test_bytes_of_a_step():
    assert bench.bytes_per_step(72.0, 10, 1) == 72.0
    assert bench.bytes_per_step(72.0, 10, 2) == 36.0
    assert bench.bytes_per_step(72.0, 5, 2) == 72.0 * 3 / 5
    assert bench.bytes_per_step(72.0, 1, 2) == 72.0


def test_traffic_belongs_to_the_kernel_sources():
    text = open(bench.__file__).read()
    for name in ("lbm_device.cuh", "lbm_kernels.cuh", "lbm_pair.cuh", "lbm_pair.cu"):
        assert f'"{name}"' in text
