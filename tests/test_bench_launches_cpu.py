"""The kernel count that the benchmark line carries (CPU): one refine kernel a
greedy step and group, from the slots that rsc_encode's timing records."""
import inspect

import bench


def test_reported_count_takes_one_refine_kernel_a_step():
    # one call of 3 stream groups at K = 5: per group the init kernel, 5
    # scoring and 5 refine kernels and the hand-off: 12
    assert bench.REFINE_KERNELS == 1
    assert bench.kernel_launch_count([15, 3, 18], 5, "f16", bench.REFINE_KERNELS) == 36
    # ten calls in one group at K = 3: init, 3 + 3, hand-off
    assert bench.kernel_launch_count([30, 10, 40], 3, "f16", bench.REFINE_KERNELS) == 80
    assert bench.kernel_launch_count([4, 0, 0], 5, "fp32", bench.REFINE_KERNELS) == 4


def test_the_line_is_built_with_it():
    src = inspect.getsource(bench).split('"gpu_launches"')[1][:200]
    assert "REFINE_KERNELS" in src
