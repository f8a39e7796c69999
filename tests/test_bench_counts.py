"""The flop counts bench.py reports, against what a unit cell of the recursion
consists of (8 real flops per complex multiply-add)."""
import bench


def test_executed_count_is_that_of_cell_steps():
    # even N: an inverse, A V and a strip product of K x K, K = N / 2
    for K in (1, 5, 122):
        assert bench.executed_flops_per_cell(2 * K) == 8 * 3 * K ** 3
        assert bench.executed_flops_per_cell(2 * K, pairs=False) == 8 * 4 * 2 * K ** 3
    # odd N: the left half inverts on the odd rows, the right half on the even ones
    KL, KR = 123, 122
    left = KR ** 3 + KR ** 3 + KL * KR ** 2
    right = KL ** 3 + KL ** 3 + KR * KL ** 2
    assert bench.executed_flops_per_cell(245) == 8 * (left + right) / 2
    single = sum(K ** 3 + rows * K * K for rows in (KL, KR) for K in (KL, KL, KR, KR))
    assert bench.executed_flops_per_cell(245, pairs=False) == 8 * single / 2
