"""A block's append to the stage-1 basis in one cluster launch, through whole
solves: every block size (padded widths 1, 2, 4, 8), fewer rows than CTAs, rows
beside the CTA and warp edges, long rows, both targets and precisions, the general
form behind its line, and blocks that are dependent on the basis."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_1408_5535_gb300 import native, synth
from oracle import phsvds_ref as R
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu
DELTA = 1e-13


@pytest.fixture(scope="module")
def h():
    need_gpu()
    with native.Handle(0) as hh:
        yield hh


def _check(D, got, k, largest):
    sig, U, V = got[:3]
    s = np.linalg.svd(D, compute_uv=False)
    ref = s[:k] if largest else np.sort(s)[:k]
    assert np.max(np.abs(sig - ref) / ref) <= 1e-10
    res = np.sqrt(np.linalg.norm(D @ V - U * sig, axis=0) ** 2 + np.linalg.norm(D.T @ U - V * sig, axis=0) ** 2)
    assert np.all(res <= DELTA * s[0] * (1 + 1e-6))
    assert np.max(np.abs(V.T @ V - np.eye(k))) <= 1e-11


@pytest.mark.parametrize("prec", [native.FP64, native.MIXED], ids=["fp64", "mixed"])
@pytest.mark.parametrize("m,n,row,b,largest", [(12, 9, 4.0, 1, True), (40, 17, 5.0, 3, False), (130, 129, 6.0, 2, True),
                                               (600, 300, 40.0, 5, False), (1100, 1023, 8.0, 8, True),
                                               (1500, 1025, 8.0, 1, False), (2500, 2050, 6.0, 7, True)])
def test_triplets(h, prec, m, n, row, b, largest):
    A = synth.random_sparse(m, n, row, 5, values="gaussian", shift=0.5)
    maxb = min(35, n)
    k = min(b + 1, 2) if n < 40 else b + 1
    b = min(b, k)
    o = native.default_opts(block_size=b, precision=prec, max_basis=min(maxb, 9 if n < 12 else 16 if n < 40 else 35),
                            min_restart=4 if n < 12 else 8 if n < 40 else 21)
    got = native.phsvds_solve(h, A.m, A.n, A.row_ptr, A.col, A.val, k, native.LARGEST if largest else native.SMALLEST,
                              DELTA, opts=o)
    _check(A.to_dense(), got, k, largest)


def _three_values():
    n, m = 90, 120
    d = np.concatenate([np.full(30, 1.0), np.full(30, 2.0), np.full(30, 3.0)])
    Q = np.linalg.qr(np.random.default_rng(3).standard_normal((m, m)))[0][:, :n]
    S = sp.csr_matrix(Q * d)
    S.sort_indices()
    return synth.Csr(m, n, S.indptr.astype(np.int64), S.indices.astype(np.int32), S.data), S


@pytest.mark.parametrize("b", [4, 8])
def test_blocks_dependent_on_the_basis(h, b):
    """Three distinct singular values: the Krylov space of a block closes after three
    steps, and the columns of the next one have to be replaced.  (Which copies of a
    multiple value a closed space holds is not determined.)"""
    A, S = _three_values()
    o = native.default_opts(block_size=b)
    got = native.phsvds_solve(h, A.m, A.n, A.row_ptr, A.col, A.val, 12, native.LARGEST, DELTA, opts=o)
    sig, U, V = got[:3]
    D = S.toarray()
    assert np.max(np.abs(sig[:, None] - np.array([1.0, 2.0, 3.0])).min(axis=1)) <= 1e-10
    assert abs(sig[0] - 3.0) <= 1e-10
    res = np.sqrt(np.linalg.norm(D @ V - U * sig, axis=0) ** 2 + np.linalg.norm(D.T @ U - V * sig, axis=0) ** 2)
    assert np.all(res <= DELTA * 3.0 * (1 + 1e-6))
    assert np.max(np.abs(V.T @ V - np.eye(12))) <= 1e-11


def test_closed_space_of_one_vector_is_refused(h):
    """Block 1 on the same matrix: all three pairs of the closed space converge at once
    and nothing is left to expand; that is an error with the general form as well."""
    A, _ = _three_values()
    for prof in (0, 1):
        o = native.default_opts(block_size=1, profile=prof)
        with pytest.raises(native.PhsvdsError, match="empty basis"):
            native.phsvds_solve(h, A.m, A.n, A.row_ptr, A.col, A.val, 12, native.LARGEST, DELTA, opts=o)


def test_both_sides_of_the_line_agree(h):
    """The same solve with the fused append and (opts.profile) with the general form."""
    A = synth.random_sparse(4000, 2000, 8.0, 11, values="gaussian", shift=0.0)
    runs = []
    for prof in (0, 1):
        o = native.default_opts(block_size=4, profile=prof)
        runs.append(native.phsvds_solve(h, A.m, A.n, A.row_ptr, A.col, A.val, 6, native.LARGEST, DELTA, opts=o))
    assert runs[0][4]["kernel_launches"] < runs[1][4]["kernel_launches"]
    assert np.max(np.abs(runs[0][0] - runs[1][0]) / runs[1][0]) <= 1e-12
    assert abs(runs[0][4]["matvecs_A"] - runs[1][4]["matvecs_A"]) <= 0.1 * runs[1][4]["matvecs_A"]
    assert runs[0][4]["class_flops"][0] > 0
