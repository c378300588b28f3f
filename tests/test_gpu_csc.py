"""CSR -> CSC on the device: bit-exact against scipy on columns of every kind
the kernels treat apart (empty, shorter and longer than a lane group's
registers, and columns long enough for the CTA's sorting network)."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_1408_5535_gb300 import native
from tests.gpu_util import torch, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def h():
    need_gpu()
    with native.Handle(0) as hh:
        yield hh


@pytest.mark.parametrize("m,n,row,dense", [(1, 1, 1, 0), (40, 3, 2, 1), (5000, 4095, 1, 0), (5000, 4097, 3, 2),
                                           (3001, 700, 2, 5), (3001, 1499, 8, 1), (2500, 61, 6, 0), (9000, 8193, 20, 1)])
def test_csr_to_csc_column_lengths(h, m, n, row, dense):
    rng = np.random.default_rng(m + n)
    S = sp.random(m, n, density=min(1.0, row / n), format="lil", random_state=rng, data_rvs=rng.standard_normal)
    for c in range(dense):                                # whole columns, some of them with gaps
        rows = rng.permutation(m)[: m - 3 * c * (m > 100)]
        S[rows, (c * 7) % n] = rng.standard_normal((rows.size, 1))
    S = S.tocsr()
    S.sort_indices()
    T = S.tocsc()
    T.sort_indices()
    dev = lambda a, t: torch.from_numpy(np.ascontiguousarray(a.astype(t))).cuda()
    cp = torch.full((n + 1,), -1, dtype=torch.int32, device="cuda")
    ri = torch.full((max(1, S.nnz),), -1, dtype=torch.int32, device="cuda")
    cv = torch.full((max(1, S.nnz),), -1.0, dtype=torch.float64, device="cuda")
    native.phsvds_csr_to_csc(h, m, n, S.nnz, dev(S.indptr, np.int32), dev(S.indices, np.int32),
                             dev(S.data, np.float64), cp, ri, cv)
    native.phsvds_sync(h)
    assert np.array_equal(cp.cpu().numpy(), T.indptr)
    assert np.array_equal(ri.cpu().numpy()[: S.nnz], T.indices)
    assert np.array_equal(cv.cpu().numpy()[: S.nnz], T.data)


@pytest.mark.parametrize("n,stray", [(300, 7), (40, 5000)])
def test_entries_past_the_last_row_are_not_followed(h, n, stray):
    """nnz larger than row_ptr[m] (a buffer with room to spare): the entries past the last
    row have no row, all in column 0 here; the other columns are as they should be, and what
    was in the output buffers is not taken for an index."""
    m = 500
    rng = np.random.default_rng(n)
    S = sp.random(m, n, density=0.05, format="csr", random_state=rng, data_rvs=rng.standard_normal)
    S.sort_indices()
    T = S.tocsc()
    T.sort_indices()
    dev = lambda a, t: torch.from_numpy(np.ascontiguousarray(a.astype(t))).cuda()
    nnz = S.nnz + stray
    cp = torch.full((n + 1,), -1, dtype=torch.int32, device="cuda")
    ri = torch.full((nnz,), -1, dtype=torch.int32, device="cuda")
    cv = torch.full((nnz,), 1e300, dtype=torch.float64, device="cuda")
    ci = np.concatenate([S.indices, np.zeros(stray, S.indices.dtype)])
    va = np.concatenate([S.data, np.ones(stray)])
    native.phsvds_csr_to_csc(h, m, n, nnz, dev(S.indptr, np.int32), dev(ci, np.int32), dev(va, np.float64), cp, ri, cv)
    native.phsvds_sync(h)
    a = T.indptr[1]
    assert np.array_equal(cp.cpu().numpy()[1:], T.indptr[1:] + stray)
    assert np.array_equal(ri.cpu().numpy()[a + stray:], T.indices[a:])
    assert np.array_equal(cv.cpu().numpy()[a + stray:], T.data[a:])
