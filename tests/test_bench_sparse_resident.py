"""bench.py's launch count of a solve whose sparse session runs in one launch."""


def test_launch_count_of_a_sparse_resident_solve():
    import bench
    T = 50
    count = lambda steps, resident: bench.launches_per_solve(steps, 2, 2, resident, False, False)
    assert count(T, True) == count(2 * T, True)  # one launch whatever the steps
    assert count(T, True) - count(0, False) == 4  # and three that lay out the couplings
