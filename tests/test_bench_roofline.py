"""Which time the bench takes for the dominant kernel's (CPU)."""
import bench


def test_kernel_time_is_of_a_launch_that_the_timed_steps_make():
    """Kernel timing of a one-launch forward runs a kernel without the weight layout, which no timed step does."""
    assert bench.kernel_time(1, 0.027, 0.032)[0] == 0.027
    assert bench.kernel_time(2, 0.060, 0.055)[0] == 0.055
    assert bench.kernel_time(1, 0.027, 0.032)[1] != bench.kernel_time(2, 0.060, 0.055)[1]
