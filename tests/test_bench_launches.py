"""The kernel launches that the bench line claims for its timed windows, one
call per step."""
import bench


def test_launches_of_one_step_calls():
    assert bench.step_launches(50, 4, 12288, 9) == 4 * 3 + 2  # steps 50 to 53: two odd
    assert bench.step_launches(51, 3, 12288, 9) == 3 * 3 + 2  # 51, 52, 53
    assert bench.step_launches(51, 3, 12287, 9) == 3 * 3  # too few region warps for a launch of their own
    assert bench.step_launches(0, 500, 0, 0) == 500  # no catalytic node


def test_the_region_launch_needs_what_the_kernels_say():
    src = "constexpr int32_t kUniMinWarps = 7;"
    assert bench.step_launches(1, 1, 7, 1, lambda f: src) == 4
    assert bench.step_launches(1, 1, 6, 1, lambda f: src) == 3
