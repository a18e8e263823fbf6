"""The kernel count of the bench line (no GPU): clips of one length share the launches
of their small solves, up to eight at a time."""
import bench


def test_kernels_per_step_counts():
    # five clips of 200 frames under one C: 5 widen passes + 2 packed launches with their
    # reduces, 13 kernels of the solves + the learned selection, per clip lift 1, subtract 2
    assert bench.kernels_per_step("mlp", 10, clips=5, n=200) == 9 + 14 + 5 * 3 == 38
    # one clip: sketch + reduce, 13, lift 1, subtract 2
    assert bench.kernels_per_step("omp", 10, clips=1, n=200) == 2 + 13 + 1 + 2 == 18
    # 17..32 modes take a second lift launch; a ninth clip a second set of solves
    assert bench.kernels_per_step("omp", 20, clips=1, n=200) == 2 + 13 + 2 + 2
    assert bench.kernels_per_step("omp", 10, clips=9, n=50) == 9 + 2 + 2 * 13 + 9 * 3
