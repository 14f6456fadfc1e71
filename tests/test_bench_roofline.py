"""The bench's rate of the level-0 steps counts what the launches do."""
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench
from paper_2407_09848_gb300.amgps import op_coefs, opt4_weights


def test_issued_work_of_a_degree_4_cycle():
    n, nnz, stored = 1000, 6900, 7000
    h, g = op_coefs("cheb4_opt", 4, opt4_weights(4))[2:]
    # one cycle: from zero 7, 7 and 8 instructions a row; the correction 7; then 7, 7, 8
    fl, inst = bench.issued_work(4, 1, 7, 14 * nnz + 7 * n, 7 * stored + 6 * n, n, nnz, stored, h, g)
    assert inst == 51 * n
    # lone first products (-1), a multiply-add each for the last steps' second term (+2)
    assert fl == 12 * nnz + (-1 + 0 + 2 + 12 - 1 + 0 + 2) * n


def test_issued_work_of_the_recurrence():
    n, nnz, stored = 1000, 6900, 7000
    # one degree-2 cycle: a step from zero, the correction, one more step
    plain = (2 * nnz + 5 * n) + (2 * nnz + 4 * n) + (2 * nnz + 5 * n)
    inst = 3 * stored + 9 * n
    assert bench.issued_work(2, 0, 3, plain, inst, n, nnz, stored, [], []) == (
        plain - (2 * nnz + 4 * n) + 13 * n, inst - (stored + 3 * n) + 8 * n)
