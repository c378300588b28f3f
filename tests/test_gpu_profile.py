"""A profiled solve (opts.profile = 1) runs the kernels of the solve that it stands for."""
import numpy as np
import pytest

from paper_1408_5535_gb300 import native, synth
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def test_a_profiled_solve_runs_the_same_kernels():
    """Vectors too long for the one-launch append: same launches, same bits, and one launch per projected
    eigensolve; with 2, its kernels apart."""
    need_gpu()
    A = synth.random_sparse(60000, 40000, 6.0, 4, values="gaussian", shift=0.0)
    runs = []
    with native.Handle(0) as h:
        for prof in (0, 0, 1, 2):
            o = native.default_opts(block_size=8, profile=prof)
            runs.append(native.phsvds_solve(h, A.m, A.n, A.row_ptr, A.col, A.val, 8, native.LARGEST, 1e-9, opts=o))
    plain, prof, apart = (r[4] for r in runs[1:])
    assert plain["kernel_launches"] == prof["kernel_launches"] < apart["kernel_launches"]
    assert np.array_equal(runs[1][0], runs[2][0]) and np.array_equal(runs[1][2], runs[2][2])
    assert prof["n_class"][5] == prof["jacobi_calls"] and apart["n_class"][5] > apart["jacobi_calls"]
    assert prof["t_class_ms"][5] > 0.0


def test_a_profiled_inner_solve_is_the_one_launch():
    need_gpu()
    A = synth.grid_gradient(40, 1.0, 2)
    launches = []
    with native.Handle(0) as h:
        for prof in (1, 2):
            o = native.default_opts(block_size=4, stage1_inner=1, norm_A=-1.0, profile=prof)
            st = native.phsvds_solve(h, A.m, A.n, A.row_ptr, A.col, A.val, 4, native.SMALLEST, 1e-10,
                                     native.PREC_JACOBI, o)[4]
            assert st["inner_steps"] > st["inner_solves"] > 0
            launches.append(st["kernel_launches"] / st["inner_steps"])
    assert launches[0] < 0.5 * launches[1]
