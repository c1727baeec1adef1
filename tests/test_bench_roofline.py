"""The bench's ceiling of the matrix-free sum: shares of tile classes only where they are known."""
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))


def test_class_shares_only_for_the_set_they_belong_to():
    import bench

    ops, ex2, what = bench.pair_operations(100000)
    assert abs(ops - (0.12 * 8.875 + 0.73 * 5.875) / 2) < 1e-12 and ex2 == 0.425 and "73 %" in what
    for n in (2000, 20000, 99999, 1000000):
        ops, ex2, what = bench.pair_operations(n)
        assert ops == 8.875 / 2 and ex2 == 0.5 and "%" not in what
