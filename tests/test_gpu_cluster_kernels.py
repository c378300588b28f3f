"""The one-cluster kernels by themselves (an outer iteration repairs a wrong correction or a wrong
row of the projected matrix, so that whole solves say little about them): the basis append, the
inner MINRES solve and the projected eigensolve, through the library's internal launchers, against
64-bit references of what each returns."""
import ctypes as C

import numpy as np
import pytest
import scipy.sparse as sp

from paper_1408_5535_gb300 import native
from tests.gpu_util import torch, need_gpu

pytestmark = pytest.mark.gpu
L = np.longdouble
LD = 64
EXPAND = "_ZN2ph12expand_smallI%sEEbP11CUstream_stRKNS_10SparseViewIT_EES7_iiiiPKS4_PS4_SA_SA_SA_SA_PdSB_SB_iPiSC_"
SOLVE = ("_ZN2ph14jd_solve_smallI%sEEbP11CUstream_stRKNS_10SparseViewIT_EES7_iibPKS4_S9_S9_PKdPS4_SC_SC_SC_SC_SC_SC_SC"
         "_SC_SC_PdidPi")
EIG = "_ZN2ph8eig_stepEP11CUstream_stiPKdPdibiiiS4_PiS4_S4_S4_S5_PKi"


class View(C.Structure):
    _fields_ = [("nrows", C.c_int), ("ncols", C.c_int), ("nnz", C.c_int64), ("ptr", C.c_void_p), ("idx", C.c_void_p),
                ("val", C.c_void_p), ("skew", C.c_double)]


@pytest.fixture(scope="module")
def lib():
    need_gpu()
    with native.Handle(0):
        yield native.lib()


def _call(lib, name, args, res):
    f = getattr(lib, name)
    f.restype = res
    out = f(C.c_void_p(0), *[C.byref(a) if isinstance(a, View) else a if not torch.is_tensor(a) else
                             C.c_void_p(a.data_ptr()) for a in args])
    torch.cuda.synchronize()
    return out


def _dev(x, dt):
    return torch.from_numpy(np.ascontiguousarray(np.asarray(x).astype(dt))).cuda()


def _views(S, dt):
    keep, out = [], []
    for M in (S.tocsr(), S.T.tocsr()):
        M.sort_indices()
        t = [_dev(M.indptr, np.int32), _dev(M.indices, np.int32), _dev(M.data, dt)]
        keep.append(t)
        out.append(View(M.shape[0], M.shape[1], M.nnz, t[0].data_ptr(), t[1].data_ptr(), t[2].data_ptr(), 1.0))
    return out, keep


def _matrix(rng, m, n, row, long_rows, long_cols, dt):
    S = sp.random(m, n, density=row / n, format="lil", random_state=rng, data_rvs=rng.standard_normal)
    for i, k in enumerate(long_rows):
        S[i * 5 + 3, rng.permutation(n)[:k]] = rng.standard_normal(k)
    for i, k in enumerate(long_cols):
        S[rng.permutation(m)[:k], i * 7 + 1] = rng.standard_normal((k, 1))
    S = (S.tocsr() + sp.eye(m, n)).tocsr()
    S.data = S.data.astype(dt).astype(np.float64)
    return S


def _expand(lib, S, X, nlock, T, dt):
    """Appends the columns of T to X = [Xl | V]: (V, W, Ht, S, sprev) after it."""
    m, n = S.shape
    j, nb = X.shape[1] - nlock, T.shape[1]
    (A, At), keep = _views(S, dt)
    V, W = (torch.zeros((j + nb, n), dtype=torch.float32 if dt == np.float32 else torch.float64, device="cuda")
            for _ in range(2))
    V[:j] = _dev(X[:, nlock:].T, dt)
    Xl, Tb = _dev(X[:, :nlock].T if nlock else np.zeros((1, n)), dt), _dev(T.T, dt)
    xrm, z = (torch.full((k, 8), 7.0, dtype=V.dtype, device="cuda") for k in (n, m))
    Ht, Sm, sprev = (torch.full((LD, LD), -1.0, dtype=torch.float64, device="cuda") for _ in range(3))
    flags = torch.full((48,), -1, dtype=torch.int32, device="cuda")
    ok = _call(lib, EXPAND % ("f" if dt == np.float32 else "d"),
               [A, At, nb, nlock, j, 3, Xl, V, W, Tb, xrm, z, Ht, Sm, sprev, LD, flags,
                C.c_void_p(flags.data_ptr() + 160)], C.c_bool)
    el, Q = np.dtype(dt).itemsize, 1 << (nb - 1).bit_length()
    line = n * (nlock + j + 8) * ((Q + 1) / 2e6 if el == 8 else 1e-6) + 2 * S.nnz * (Q + 2) * el / (26e6 + 4e6 * Q)
    if line > 1.0:                         # the general form's: nothing launched
        assert not ok and flags.eq(-1).all() and not V[j:].any()
        return None
    assert ok and int(flags[40]) == 0 and flags[: nb + 1].eq(0).all()
    return [t.cpu().numpy().T.astype(np.float64) for t in (V, W, Ht, Sm, sprev)]


@pytest.mark.parametrize("dt", [np.float32, np.float64], ids=["f32", "f64"])
@pytest.mark.parametrize("m,n,row,nlock,j,nb,long_rows,long_cols",
                         [(30, 20, 4, 0, 0, 1, [], []), (700, 513, 6, 5, 17, 3, [], []), (2100, 1500, 6, 0, 30, 8, [], []),
                          (5000, 4500, 5, 3, 9, 2, [64, 65, 66, 4096, 4097, 4400], [65, 129, 4500]),
                          (9000, 8000, 10, 2, 12, 5, [256, 257, 300, 8000], [4095, 4098, 9000]),
                          (2600, 2300, 40, 4, 20, 7, [1025, 2300], [1500])])
def test_append(lib, dt, m, n, row, nlock, j, nb, long_rows, long_cols):
    rng = np.random.default_rng(n + nb)
    S = _matrix(rng, m, n, row, long_rows, long_cols, dt)
    eps = float(np.finfo(dt).eps)
    X = np.linalg.qr(rng.standard_normal((n, nlock + j)))[0] if nlock + j else np.zeros((n, 0))
    X = X.astype(dt).astype(np.float64)
    got = _expand(lib, S, X, nlock, rng.standard_normal((n, nb)), dt)
    if got is None:
        return
    V, W, Ht, Sm, sprev = got
    new = V[:, j:]
    assert np.array_equal(V[:, :j], X[:, nlock:])
    assert np.max(np.abs(new.T @ new - np.eye(nb))) <= 32 * eps
    if nlock + j:
        assert np.max(np.abs(X.T @ new)) <= 32 * eps
    # W = A^T (A V): the roundings of a row's and a column's sum, and of Z
    absA = abs(S)
    most = np.max(np.diff(S.indptr)) + np.max(np.diff(S.tocsc().indptr)) + 2
    lim = most * eps * (absA.T @ (absA @ np.abs(new)))
    assert np.all(np.abs(W[:, j:] - S.T @ (S @ new)) <= lim)
    # the new rows and columns of V^T W: in FP32 four products are added plainly, what follows is to
    # twice FP32 (half an eps per rounding); in FP64 a lane's terms, the lanes and the CTAs
    per = 2.5 if dt == np.float32 else n / 256 + 24
    dot = np.array([[np.sum(V[:, r].astype(L) * W[:, j + c]) for c in range(nb)] for r in range(j + nb)])
    mod = np.abs(V).T @ np.abs(W[:, j:])
    mean = dot.copy()
    mean[j:] = 0.5 * (dot[j:] + dot[j:].T)
    slack = mod.copy()
    slack[j:] = np.maximum(mod[j:], mod[j:].T)
    k = j + nb
    assert np.all(np.abs(Ht[:k, j:k] - mean) <= per * eps * slack)
    assert np.array_equal(Ht[j:k, :k], Ht[:k, j:k].T) and np.all(Ht[k:] == -1.0) and np.all(Ht[:j, :j] == -1.0)
    unit = np.full((LD, LD), -1.0)
    unit[:k, j:k] = np.eye(LD)[:k, j:k]
    unit[j:k, :k] = np.eye(LD)[j:k, :k]
    assert np.array_equal(Sm, unit)
    assert np.all(sprev[j:k, :3] == 0.0) and np.all(sprev[:j] == -1.0) and np.all(sprev[k:] == -1.0)


@pytest.mark.parametrize("n", [8191, 16000, 26017, 32000])
def test_append_sums_of_equal_terms_in_fp32(lib, n):
    """Equal terms round the same way at every addition: a plain FP32 sum of the 63 terms of a lane is
    off by up to 15 parts in 2^24, four at a time by no more than the products and three additions."""
    for d in (0.7, 0.83, 0.91, 1.0, 1.13, 1.3):
        S = sp.eye(n, format="csr") * d
        S.data = S.data.astype(np.float32).astype(np.float64)
        V, W, Ht, _, _ = _expand(lib, S, np.zeros((n, 0)), 0, np.ones((n, 1)), np.float32)
        ref = np.sum(V[:, 0].astype(L) * W[:, 0])
        assert abs(Ht[0, 0] - ref) <= 2.5 * 2.0 ** -23 * abs(ref), (n, d, float(Ht[0, 0] / ref - 1))


@pytest.mark.parametrize("dt,tol,lim", [(np.float64, 1e-9, 1e-8), (np.float32, 1e-3, 5e-3)], ids=["f64", "f32"])
@pytest.mark.parametrize("scaled", [False, True])
@pytest.mark.parametrize("m,n,q,nl,long_rows", [(40, 30, 1, 0, []), (700, 600, 3, 4, []), (900, 777, 5, 0, [65, 700]),
                                                (3000, 2600, 8, 6, [64, 2600]), (2200, 2100, 7, 1, []),
                                                (5100, 5000, 2, 3, [5000])])
def test_inner_solve(lib, dt, tol, lim, scaled, m, n, q, nl, long_rows):
    """Every column solves its projected, shifted equation to the tolerance (the recursion's own
    residual, so a few times it is allowed)."""
    rng = np.random.default_rng(n)
    S = _matrix(rng, m, n, 5, long_rows, [], dt)
    S.data *= 0.1
    S = (S + 2 * sp.eye(m, n)).tocsr()
    S.data = S.data.astype(dt).astype(np.float64)
    (A, At), keep = _views(S, dt)
    B = np.linalg.qr(rng.standard_normal((n, nl + q)))[0].astype(dt).astype(np.float64)
    Xl, X = B[:, :nl], B[:, nl:]
    Q = B if scaled else Xl
    theta = -rng.uniform(0.0, 0.5, 8)
    ds = (1.0 / np.sqrt(np.asarray(S.multiply(S).sum(0)).ravel())).astype(dt).astype(np.float64)
    R = rng.standard_normal((n, q))

    def op(c, s):
        if scaled:
            u = ds * s
            u = u - Q @ (Q.T @ u)
            y = S.T @ (S @ u) - theta[c] * u
            return ds * (y - Q @ (Q.T @ y))
        y = S.T @ (S @ s) - theta[c] * s
        y = y - Q @ (Q.T @ y)
        return y - X[:, c] * (X[:, c] @ y)
    if scaled:
        W = np.linalg.qr(Q / ds[:, None])[0]          # the operator's null space
        R = R - W @ (W.T @ R)
    else:
        R = R - Q @ (Q.T @ R)
        R = R - X * np.sum(X * R, axis=0)
    R = R.astype(dt).astype(np.float64)
    b1 = np.zeros(8)
    b1[:q] = np.linalg.norm(R, axis=0)
    sc = np.zeros((17, 8))
    sc[0] = sc[1] = sc[5] = b1
    sc[6], sc[9], sc[15] = -1.0, 1.0, b1 > 0
    tt = torch.float32 if dt == np.float32 else torch.float64
    zeros = lambda k=8: torch.zeros((k, n), dtype=tt, device="cuda")
    v, u, r1, r2, w1, w2, sol, cv = (zeros() for _ in range(8))
    r1[:q] = r2[:q] = _dev(R.T, dt)
    v[:q] = _dev((R / b1[:q]).T, dt)
    xrm, z = (torch.full((k, 8), 7.0, dtype=tt, device="cuda") for k in (n, m))
    done = torch.zeros(1, dtype=torch.int32, device="cuda")
    dq, dx, dd = (_dev(M, dt) for M in (Q.T if Q.shape[1] else np.zeros((1, n)), X.T, ds))
    dth, dsc = _dev(theta, np.float64), _dev(sc, np.float64)
    null = C.c_void_p(0)
    ok = _call(lib, SOLVE % ("f" if dt == np.float32 else "d"),
               [A, At, q, Q.shape[1], C.c_bool(scaled), dq, null if scaled else dx, dd if scaled else null, dth, v,
                u if scaled else v, r1, r2, w1, w2, sol, cv, xrm, z, dsc, 200, C.c_double(tol), done], C.c_bool)
    assert ok and 0 < int(done[0]) < 200
    s = sol.cpu().numpy()[:q].T.astype(np.float64)
    for c in range(q):
        assert np.linalg.norm(R[:, c] - op(c, s[:, c])) <= lim * b1[c], c


def _spectrum(rng, j, kind):
    if kind == "even":
        return rng.uniform(1.0, 4.0, j)
    if kind == "equal":
        return np.concatenate([np.full(min(j, 6), 9.0), rng.uniform(1.0, 4.0, max(0, j - 6))])
    nc = max(1, j // 2)
    return np.concatenate([9.0 * (1 + float(kind) * np.linspace(0, 1, nc)) ** 2, rng.uniform(1.0, 4.0, j - nc)])


@pytest.mark.parametrize("kind", ["even", "equal", "1e-4", "1e-6", "1e-8"])
@pytest.mark.parametrize("j,ntarget,ident", [(1, 1, True), (2, 1, True), (7, 3, False), (28, 5, False), (33, 9, True),
                                             (64, 6, False)])
@pytest.mark.parametrize("largest", [True, False])
def test_projected_eigensolve(lib, kind, j, ntarget, ident, largest):
    """The target rows of S^T H S are diagonal to FP64 rounding, also within a cluster of j / 2 values,
    and S is orthonormal; the warm start is the rotation of a matrix near H."""
    rng = np.random.default_rng(j)
    lam = _spectrum(rng, j, kind) * (1 if largest else -1) + (0 if largest else 20.0)
    Z = np.linalg.qr(rng.standard_normal((j, j)))[0]
    H = (Z * lam) @ Z.T
    H = 0.5 * (H + H.T)
    E = 1e-3 * rng.standard_normal((j, j))
    S0 = np.linalg.eigh(H + E + E.T)[1]
    pad = lambda M: np.pad(M, ((0, LD - j), (0, LD - j)), constant_values=-1.0)
    dH, dS = _dev(pad(H).T, np.float64), _dev(pad(S0).T, np.float64)
    nt = min(ntarget, 8, j)
    th, thc, nrm = (torch.full((k,), -1.0, dtype=torch.float64, device="cuda") for k in (LD, LD, 8))
    order, cnt = (torch.full((k,), -1, dtype=torch.int32, device="cuda") for k in (LD, 8))
    sc = torch.full((LD, LD), -1.0, dtype=torch.float64, device="cuda")
    skip = torch.zeros(1, dtype=torch.int32, device="cuda")
    _call(lib, EIG, [j, dH, dS, LD, C.c_bool(ident), min(ntarget, j), 1 if largest else 0, nt, th, order, sc, thc, nrm, cnt,
                     skip], None)
    S = dS.cpu().numpy().T[:j, :j]
    t, o = th.cpu().numpy()[:j], order.cpu().numpy()[:j]
    eps, nH = 2.0 ** -52, np.abs(lam).max()
    assert np.max(np.abs(S.T @ S - np.eye(j))) <= 16 * eps
    assert sorted(o) == list(range(j)) and np.all(np.diff(t[o]) * (-1 if largest else 1) >= 0)
    F = S.T.astype(L) @ H.astype(L) @ S.astype(L)
    off = np.abs(F - np.diag(np.diag(F))).astype(float)[o[: min(ntarget, j)]]
    assert off.max() <= 32 * eps * nH
    ref = np.sort(lam)[::-1] if largest else np.sort(lam)
    assert np.max(np.abs(t[o[: min(ntarget, j)]] - ref[: min(ntarget, j)])) <= 32 * eps * nH
    assert np.array_equal(sc.cpu().numpy().T[:j, :nt], S[:, o[:nt]]) and np.array_equal(thc.cpu().numpy()[:nt], t[o[:nt]])
    assert nrm.cpu().numpy()[:nt].max() == 0.0


@pytest.mark.parametrize("n1,n2", [(1, 1), (15, 16), (17, 33), (1000, 4097), (5, 100000)])
def test_entries_of_the_fullest_part_of_the_rows(lib, n1, n2):
    rng = np.random.default_rng(n2)
    ptrs, ref = [], []
    for n in (n1, n2):
        rp = np.concatenate([[0], np.cumsum(rng.poisson(3.0, n) * (rng.random(n) < 0.2) * 9)]).astype(np.int64)
        per = -(-n // 16)
        ref.append(max(rp[min(n, (r + 1) * per)] - rp[min(n, r * per)] for r in range(16)))
        ptrs.append(_dev(rp, np.int32))
    out = torch.full((2,), -1, dtype=torch.int32, device="cuda")
    _call(lib, "_ZN2ph9row_partsEP11CUstream_stiPKiiS3_Pi", [n1, ptrs[0], n2, ptrs[1], out], None)
    assert out.tolist() == ref


@pytest.mark.parametrize("dt", [np.float32, np.float64], ids=["f32", "f64"])
def test_append_is_left_to_the_general_form_where_one_part_holds_the_entries(lib, dt):
    """The same sizes with the entries spread (taken) and more and more of them in one sixteenth of
    the rows of A and A^T: the line counts that part, as if all were as full."""
    rng = np.random.default_rng(1)
    n = 4000
    S = _matrix(rng, n, n, 12, [], [], dt)
    (A, At), keep = _views(S, dt)
    t = torch.float32 if dt == np.float32 else torch.float64
    V, W, Tb = (torch.zeros((2, n), dtype=t, device="cuda") for _ in range(3))
    Tb[0] = 1.0
    xrm, z = (torch.zeros((n, 8), dtype=t, device="cuda") for _ in range(2))
    Ht, Sm, sprev = (torch.zeros((LD, LD), dtype=torch.float64, device="cuda") for _ in range(3))
    flags = torch.zeros(48, dtype=torch.int32, device="cuda")
    for skew in (1.0, 4.0, 8.0, 16.0):
        A.skew = At.skew = skew
        ok = _call(lib, EXPAND % ("f" if dt == np.float32 else "d"),
                   [A, At, 1, 0, 0, 0, Tb, V, W, Tb, xrm, z, Ht, Sm, sprev, LD, flags,
                    C.c_void_p(flags.data_ptr() + 160)], C.c_bool)
        line = n * 8 * (2 / 2e6 if dt == np.float64 else 1e-6) + 2 * skew * S.nnz * 3 * np.dtype(dt).itemsize / 30e6
        assert ok == (line <= 1.0) and (ok or skew > 1.0), line
