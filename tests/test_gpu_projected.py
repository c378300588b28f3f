"""The one-launch projected eigensolve of stage 1 through whole solves: the basis
orders at which its work division changes (odd and even, below and above 32
columns, up to 64), both targets, and multiple eigenvalues, against the dense
SVD."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_1408_5535_gb300 import native, synth
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def h():
    need_gpu()
    with native.Handle(0) as hh:
        yield hh


@pytest.mark.parametrize("maxb,mins,b,largest", [(4, 2, 1, True), (11, 6, 1, False), (17, 9, 3, True), (32, 20, 1, False),
                                                 (33, 19, 5, True), (35, 21, 8, False), (56, 30, 8, True),
                                                 (56, 31, 7, False)])
def test_triplets_for_every_order_of_the_projected_problem(h, maxb, mins, b, largest):
    A = synth.random_sparse(300, 150, 6.0, maxb, values="gaussian", shift=0.05)
    k = min(4, mins - 1)
    o = native.default_opts(block_size=b, max_basis=maxb, min_restart=mins)
    sig, U, V, _, st, _ = native.phsvds_solve(h, A.m, A.n, A.row_ptr, A.col, A.val, k,
                                              native.LARGEST if largest else native.SMALLEST, 1e-14, opts=o)
    D = A.to_dense()
    s = np.linalg.svd(D, compute_uv=False)
    ref = s[:k] if largest else s[::-1][:k]
    assert np.all(np.abs(sig - ref) <= 1e-10 * ref)
    res = np.sqrt(np.linalg.norm(D @ V - U * sig, axis=0) ** 2 + np.linalg.norm(D.T @ U - V * sig, axis=0) ** 2)
    assert np.all(res <= 1e-14 * s[0])
    assert np.max(np.abs(V.T @ V - np.eye(k))) <= 1e-12


def test_multiple_singular_values(h):
    """Blocks of equal and of nearly equal singular values among the targets."""
    sigma = np.concatenate([np.repeat([1.0, 1.1], 3), 1.2 + 1e-9 * np.arange(3), np.linspace(1.5, 3.0, 91)])
    A = synth.givens_diag(200, 100, sigma=sigma, n_rot=150, seed=4)
    o = native.default_opts(block_size=4)
    sig, U, V, _, _, _ = native.phsvds_solve(h, A.m, A.n, A.row_ptr, A.col, A.val, 8, native.SMALLEST, 1e-13, opts=o)
    assert np.all(np.abs(sig - np.sort(sigma)[:8]) <= 1e-10)
    D = A.to_dense()
    assert np.all(np.linalg.norm(D @ V - U * sig, axis=0) <= 3e-13)
    assert np.max(np.abs(V.T @ V - np.eye(8))) <= 1e-11


@pytest.mark.parametrize("mat,start", [(4, 7), (5, 7), (8, 13), (11, 17)])
def test_multiple_singular_values_keep_the_basis_orthonormal(h, mat, start):
    """Equal eigenvalues split by rounding alone must not be rotated against each
    other by a first-order step: the basis would lose its orthogonality for good and
    the solve stop converging.  Without that a solve takes 70 to 80 iterations."""
    sigma = np.concatenate([np.repeat([1.0, 1.1], 3), 1.2 + 1e-9 * np.arange(3), np.linspace(1.5, 3.0, 91)])
    A = synth.givens_diag(200, 100, sigma=sigma, n_rot=150, seed=mat)
    o = native.default_opts(block_size=4, max_restarts=60, seed=start)
    sig, U, V, _, _, _ = native.phsvds_solve(h, A.m, A.n, A.row_ptr, A.col, A.val, 8, native.SMALLEST, 1e-13, opts=o)
    assert np.all(np.abs(sig - np.sort(sigma)[:8]) <= 1e-10)
    assert np.max(np.abs(V.T @ V - np.eye(8))) <= 1e-11


@pytest.mark.parametrize("scale,tiny", [(1.0, 1e-20), (1e3, 1e-60), (1e10, 1e-160)])
def test_gaps_below_the_range_of_fp32(h, scale, tiny):
    """Two columns of A that meet no other and are smaller by 20 to 170 decades: the gap of
    their Ritz values has no reciprocal in FP32, and at last none after scaling in FP64."""
    n, m = 100, 160
    rng = np.random.default_rng(3)
    D = np.zeros((m, n))
    D[:150, :98] = scale * rng.standard_normal((150, 98)) * (rng.random((150, 98)) < 0.2)
    D[150, 98], D[151, 98], D[151, 99] = tiny, 1e-2 * tiny, 3 * tiny
    S = sp.csr_matrix(D)
    x0 = np.zeros((n, 6))
    x0[98, 0] = x0[99, 1] = 1.0
    x0[:98, 2:] = rng.standard_normal((98, 4))
    o = native.default_opts(block_size=2)
    sig = native.phsvds_solve(h, m, n, S.indptr.astype(np.int64), S.indices.astype(np.int32), S.data, 3,
                              native.LARGEST, 1e-13, opts=o, init_V=x0)[0]
    ref = np.linalg.svd(D, compute_uv=False)[:3]
    assert np.all(np.abs(sig - ref) <= 1e-10 * ref)


@pytest.mark.parametrize("largest", [True, False])
@pytest.mark.parametrize("spread", [1e-4, 1e-6, 1e-7])
def test_clusters_wider_than_the_targets(h, spread, largest):
    """16 singular values within spread of one another, 12 of them wanted: the couplings that
    FP32 leaves are above the gaps of the whole cluster.  Every start converges, in about as many
    iterations as with the FP64 solver of the projected problem (51 to 110 here, measured)."""
    k, nc = 12, 16
    t = spread * np.linspace(0, 1, nc)
    sigma = (np.concatenate([np.linspace(1.0, 2.0, 200 - nc), 3.0 * (1 + t)]) if largest
             else np.concatenate([0.5 * (1 + t), np.linspace(1.0, 2.0, 200 - nc)]))
    ref = np.sort(sigma)[::-1][:k] if largest else np.sort(sigma)[:k]
    for mat in (4, 5, 6):
        A = synth.givens_diag(400, 200, sigma=sigma, n_rot=600, seed=mat)
        D = A.to_dense()
        for start in (0, 1):
            o = native.default_opts(block_size=4, max_restarts=60, seed=start)
            sig, U, V, _, st, _ = native.phsvds_solve(h, A.m, A.n, A.row_ptr, A.col, A.val, k,
                                                      native.LARGEST if largest else native.SMALLEST, 1e-13, opts=o)
            assert np.all(np.abs(sig - ref) <= 1e-10)
            assert np.max(np.abs(V.T @ V - np.eye(k))) <= 1e-11
            assert np.all(np.linalg.norm(D @ V - U * sig, axis=0) <= 3e-13 * 3)
