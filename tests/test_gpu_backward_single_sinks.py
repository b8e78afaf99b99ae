"""Adjoint blocks of n > 6: sinks that belong to no one-column sink family take an LU of their own (one
exchange of rows per step), and the scatter reads the column labels from shared memory and the cells a
step ahead.  Oracle and tolerances of test_gpu_backward."""
import numpy as np
import pytest

from paper_1411_3691_gb300 import workloads as wl
from test_gpu_backward import M, check_vs_oracle  # noqa: F401  (M: the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, sinks", [([7, 3], [1] * 33), ([8, 7], [1] * 20 + [6, 2]), ([12, 9], [1] * 5 + [9] * 4 + [1] * 30),
                                      ([17, 18], [1] * 9 + [4]), ([18], [1] * 40), ([32, 19], [1] * 3 + [3])])
def test_single_sinks(M, n, sinks):
    L = [max(12 * ((x + 2) // 3) + 12, x + 16) for x in n]
    check_vs_oracle(M, wl.make_workload("ss", n, L, [5, 1, 3], sinks, seed=60 + sum(n), diag=3.0))


def test_two_column_sinks(M):
    w = wl.make_workload("tc", [12, 10], [60, 48], [6, 4], [9, 1, 8, 7, 1, 1, 9], seed=82, diag=3.0,
                         two_row_frac=0.5)
    check_vs_oracle(M, w)


def test_graded_propagators(M):
    w = wl.make_workload("ss", [11, 7], [50, 40], [6, 4], [1] * 35, seed=83, diag=3.0)
    rng = np.random.default_rng(84)
    w.S = [np.ascontiguousarray(s * 10.0 ** rng.uniform(-1, 1, (s.shape[0], 1))) for s in w.S]
    check_vs_oracle(M, w)
