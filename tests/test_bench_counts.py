"""The launches that the bench counts follow the steps per launch that the handle reports."""
import bench
from paper_1710_10569_gb300 import workloads as W


def test_step_kernels_by_steps_per_launch():
    f32, f16, f64 = W.STORAGE_F32, W.STORAGE_F16DEV, W.STORAGE_F64
    big, small = 2048 * 1024, 256 * 256
    assert bench.step_kernels(f32, big, 2, 250) == 50 + 50 + 25
    assert bench.step_kernels(f32, big, 2, 101) == 50 + 1  # an odd step is a launch
    assert bench.step_kernels(f32, big, 1, 250) == 250     # tuned to one step per launch
    assert bench.step_kernels(f64, big, 1, 250) == 250
    assert bench.step_kernels(f16, big, 1, 250) == 500     # interior and edge kernel
    assert bench.step_kernels(f16, small, 1, 250) == 250   # one kernel
    assert "k_step_two" in bench.step_kernel_name(f32, big, 2) and "k_step<" in bench.step_kernel_name(f32, big, 1)
    assert "inner" in bench.step_kernel_name(f16, big, 1) and "inner" not in bench.step_kernel_name(f16, small, 1)
