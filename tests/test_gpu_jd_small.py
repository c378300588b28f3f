"""The inner solve of stage 1 in one cluster launch, through whole solves:
every block size (the padded widths 1, 2, 4, 8), rows beside the thread and
cluster edges, short and long rows of A, the scaled and the plain form, FP32
and FP64, against a dense or shift-invert reference."""
import numpy as np
import pytest
import scipy.sparse.linalg as sla

from paper_1408_5535_gb300 import native, synth
from oracle import phsvds_ref as R
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu
DELTA = 1e-14


@pytest.fixture(scope="module")
def h():
    need_gpu()
    with native.Handle(0) as hh:
        yield hh


def _check(S, got, k):
    sig, U, V, _, st, _ = got
    if S.shape[1] <= 1200:
        nA = np.linalg.norm(S.toarray(), 2)
        ref = np.sort(np.linalg.svd(S.toarray(), compute_uv=False))[:k]
    else:
        nA = sla.svds(S, k=1, return_singular_vectors=False)[0]
        C = (S.T @ S).tocsc()
        ref = np.sqrt(np.sort(sla.eigsh(C, k=k, sigma=0.0, return_eigenvectors=False)))
    assert st["inner_steps"] > 0
    assert np.max(np.abs(np.sort(sig) - ref) / ref) <= 1e-10
    rv, ru = np.linalg.norm(S @ V - U * sig, axis=0), np.linalg.norm(S.T @ U - V * sig, axis=0)
    assert np.all(np.sqrt(rv ** 2 + ru ** 2) <= DELTA * nA * (1 + 1e-6))


@pytest.mark.parametrize("N,b,prec,mixed_inner", [(9, 1, "fp64", 1), (20, 3, "mixed", 2), (24, 5, "fp64", 1), (32, 8, "mixed", 2),
                                                  (33, 7, "fp64", 1), (46, 2, "mixed", 1), (65, 6, "mixed", 2),
                                                  (65, 4, "fp64", 1)])
def test_scaled_form(h, N, b, prec, mixed_inner):
    A = synth.grid_gradient(N, 1.0, 2)
    o = native.default_opts(block_size=b, stage2_inner=1, norm_A=-1.0, time_limit_s=60.0)
    if prec == "mixed":
        o.precision, o.mixed_inner = native.MIXED, mixed_inner
    else:
        o.precision, o.stage1_inner = native.FP64, 1
    got = native.phsvds_solve(h, A.m, A.n, A.row_ptr, A.col, A.val, 6, native.SMALLEST, DELTA, native.PREC_JACOBI, o)
    _check(R.as_scipy(A), got, 6)


@pytest.mark.parametrize("m,n,nnz_row,b", [(300, 150, 6.0, 1), (700, 513, 12.0, 3), (900, 600, 40.0, 5),
                                           (1400, 1025, 6.0, 8)])
def test_plain_form(h, m, n, nnz_row, b):
    A = synth.random_sparse(m, n, nnz_row, 21, values="gaussian", shift=0.05)
    o = native.default_opts(block_size=b, stage1_inner=1, norm_A=-1.0, time_limit_s=60.0)
    got = native.phsvds_solve(h, A.m, A.n, A.row_ptr, A.col, A.val, 4, native.SMALLEST, DELTA, native.PREC_NONE, o)
    _check(R.as_scipy(A), got, 4)
