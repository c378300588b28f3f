"""The FP64 tall products that run as exact digit products on the FP16 tensor
cores (block Gram-Schmidt pass and Out = P Y - Xs diag(theta)), and the
streaming form of the latter: edges of their tiles, both sides of the lines
between the forms, columns of very different size, and values that cannot be
cut into digits.

Bounds (eps = 2^-52).  A digit product is off by at most p 2^-56 of the row's
largest element times the coefficient column's largest (2^-62 per operand, 2
bits for the powers of two, 4 for the kept orders and the final integer),
beside the result's own rounding; a chain of p multiply-adds by (p + 1) eps of
the sum of moduli.  Both lie below (p + 4) eps (row maximum) (column maximum).
"""
import numpy as np
import pytest

from paper_1408_5535_gb300 import native
from tests.gpu_util import torch, need_gpu

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -52
L = np.longdouble


@pytest.fixture(scope="module")
def h():
    need_gpu()
    with native.Handle(0) as hh:
        yield hh


def _dev(x, ld, dt=np.float64):
    """Column-major device copy of x (n x c) with leading dimension ld."""
    buf = np.full((x.shape[1], ld), 7.0, dtype=dt)
    buf[:, : x.shape[0]] = x.T
    return torch.from_numpy(buf).cuda()


def _mm(A, B):
    out = np.zeros((A.shape[0], B.shape[1]), dtype=L)
    for k in range(A.shape[1]):
        out += A[:, k: k + 1].astype(L) * B[k].astype(L)
    return out


def _tall(h, P, Y, Xs=None, th=None, odd=False, inplace=False, fp32=False):
    n, p = P.shape
    r = Y.shape[1]
    dt = np.float32 if fp32 else np.float64
    ld = n + (1 if odd else n % 2)
    Pd = _dev(P, ld, dt)
    Yd = torch.from_numpy(np.ascontiguousarray(Y.T)).cuda()
    Od = Pd if inplace else _dev(np.zeros((n, r)), ld, dt)
    Xd = _dev(Xs, ld, dt) if Xs is not None else None
    td = torch.from_numpy(th).cuda() if th is not None else None
    nrm = torch.zeros(r, dtype=torch.float64, device="cuda")
    native.phsvds_tall_small(h, n, Pd, ld, p, Yd, p, r, Od, ld, Xs=Xd, ldx=ld, theta=td, norms2=nrm, fp32=fp32)
    native.phsvds_sync(h)
    return Od.cpu().numpy()[:r, :n].T.astype(np.float64), nrm.cpu().numpy()


@pytest.mark.parametrize("n,p,r,odd", [(511, 20, 5, False), (512, 8, 3, False), (513, 7, 8, False), (527, 16, 8, True),
                                       (4097, 17, 9, False), (3000, 35, 21, True), (2433, 48, 16, False),
                                       (2431, 49, 17, False), (1300, 64, 32, True), (1301, 64, 64, False),
                                       (700, 35, 1, False), (701, 35, 2, True)])
def test_tall_edges(h, n, p, r, odd):
    rng = np.random.default_rng(n + p)
    P, Y, X, th = (rng.standard_normal(s) for s in ((n, p), (p, r), (n, r), (r,)))
    out, nrm = _tall(h, P, Y, X, th, odd)
    ref = _mm(P, Y) - X.astype(L) * th
    bound = (p + 4) * EPS * (np.abs(P).max(1)[:, None] * np.abs(Y).max(0) + np.abs(X * th))
    assert np.all(np.abs(out - ref) <= bound)
    assert np.allclose(nrm, np.sum(out * out, axis=0), rtol=1e-13, atol=0)
    if r <= p:
        out, _ = _tall(h, P, Y, odd=odd, inplace=True)
        assert np.all(np.abs(out - _mm(P, Y)) <= (p + 4) * EPS * np.abs(P).max(1)[:, None] * np.abs(Y).max(0))


@pytest.mark.parametrize("r", [3, 12])
def test_tall_columns_of_different_size(h, r):
    """Columns from 1 down to 1e-30, and coefficients that pick the small ones:
    each result is as accurate as a chain of FP64 multiply-adds."""
    rng = np.random.default_rng(r)
    n, p = 5000, 24
    s = 10.0 ** np.linspace(0, -30, p)
    P = rng.uniform(0.5, 1.0, (n, p)) * np.where(rng.random((n, p)) < 0.5, -1, 1) * s
    Y = np.zeros((p, r))
    for c in range(r):
        Y[p - 1 - c, c] = 1.5
        Y[:, c] += rng.standard_normal(p) * 1e-3 * s[p - 1 - c] / s * (np.arange(p) < p - 1 - c)
    out, _ = _tall(h, P, Y)
    assert np.all(np.abs(out - _mm(P, Y)) <= (p + 4) * EPS * (np.abs(P) @ np.abs(Y)))


def test_tall_rows_of_different_size_and_special_values(h):
    """Rows scaled over 600 decades, a zero row, signed zeros, values near the
    ends of the range, and rows with Inf and NaN: rows do not touch one another."""
    rng = np.random.default_rng(5)
    n, p, r = 2000, 20, 6
    P = rng.standard_normal((n, p)) * 10.0 ** rng.uniform(-300, 300, (n, 1))
    P[7] = 0.0
    P[8] = -0.0
    P[40:60] = rng.standard_normal((20, p)) * 1e-307
    P[100:110] = rng.standard_normal((10, p)) * 1e300
    P[333, 3] = np.inf
    P[500, 19] = np.nan
    Y = rng.standard_normal((p, r))
    Y[3, 2] = 0.0                                           # Inf * 0 is NaN
    out, _ = _tall(h, P, Y)
    with np.errstate(all="ignore"):
        plain = sum(P[:, k: k + 1] * Y[k] for k in range(p))
    odd = [333, 500]
    assert np.array_equal(np.isnan(out[odd]), np.isnan(plain[odd]))
    assert np.array_equal(out[odd][np.isinf(plain[odd])], plain[odd][np.isinf(plain[odd])])
    ok = np.setdiff1d(np.arange(n), odd)
    bound = (p + 4) * EPS * np.abs(P[ok]).max(1)[:, None] * np.abs(Y).max(0) + 1e-322
    assert np.all(np.abs(out[ok] - _mm(P[ok], Y)) <= bound)
    assert np.all(out[7:9] == 0.0)
    Y[0, 0] = np.inf                                        # coefficients that cannot be cut
    out, _ = _tall(h, P[600:1400], Y)
    assert np.all(~np.isfinite(out[:, 0]))
    ref = _mm(P[600:1400], Y[:, 1:])
    assert np.all(np.abs(out[:, 1:] - ref) <= (p + 4) * EPS * np.abs(P[600:1400]).max(1)[:, None] * 4)


@pytest.mark.parametrize("n,p1,p2,q,odd", [(512, 0, 10, 5, False), (511, 4, 12, 8, False), (700, 3, 13, 8, True),
                                           (8192, 7, 9, 3, False), (8191, 7, 9, 3, False), (8321, 0, 17, 4, True),
                                           (2049, 20, 28, 6, False), (1280, 20, 35, 8, False), (641, 29, 35, 7, True)])
def test_block_cgs_edges(h, n, p1, p2, q, odd):
    rng = np.random.default_rng(n)
    p = p1 + p2
    P = rng.standard_normal((n, p)) * 10.0 ** rng.uniform(-2, 2, p)
    T = rng.standard_normal((n, q)) * 10.0 ** rng.uniform(-3, 3, (n, 1))
    G = rng.standard_normal((p, q))
    P[5] = 0.0
    ld = n + (1 if odd else n % 2)
    Pd, Gd = _dev(P, ld), torch.from_numpy(np.ascontiguousarray(G.T)).cuda()
    for sub, gout, tout in ((True, True, True), (False, True, False), (True, False, True), (True, False, False)):
        Td = _dev(T, ld)
        Go = torch.zeros(p * q, dtype=torch.float64, device="cuda")
        To = torch.zeros(q * q, dtype=torch.float64, device="cuda")
        native.phsvds_block_cgs(h, n, Pd[:p1] if p1 else None, ld, p1, Td, ld, q, Gsub=Gd if sub else None,
                                Gout=Go if gout else None, Tout=To if tout else None, P2=Pd[p1:], ld2=ld, p2=p2)
        native.phsvds_sync(h)
        T2 = Td.cpu().numpy()[:q, :n].T
        ref = T.astype(L) - (_mm(P, G) if sub else 0)
        bound = (p + 4) * EPS * (np.abs(T) + (np.abs(P).max(1)[:, None] * np.abs(G).max(0) if sub else 0))
        assert np.all(np.abs(T2 - ref) <= bound)
        tiles = n / 64 + 16
        for on, buf, A in ((gout, Go, P), (tout, To, T2)):
            if not on:
                assert torch.count_nonzero(buf) == 0
                continue
            got = buf.cpu().numpy().reshape(q, -1).T
            lim = tiles * EPS * (np.abs(A).T @ np.abs(T2)) + 2.0 ** -56 * n * np.outer(np.abs(A).max(0), np.abs(T2).max(0))
            assert np.all(np.abs(got - _mm(A.T, T2)) <= lim)


@pytest.mark.parametrize("where", ["basis", "block", "coefficients"])
def test_block_cgs_values_that_cannot_be_cut(h, where):
    rng = np.random.default_rng(9)
    n, p, q = 3000, 30, 8
    P, T, G = rng.standard_normal((n, p)), rng.standard_normal((n, q)), rng.standard_normal((p, q))
    if where == "basis":
        P[1000, 4] = np.nan
    elif where == "block":
        T[1000, 4] = np.inf
    else:
        G[3, 4] = np.inf
    T[:, 5] *= 1e-306
    Pd, Td, Gd = _dev(P, n), _dev(T, n), torch.from_numpy(np.ascontiguousarray(G.T)).cuda()
    Go = torch.zeros(p * q, dtype=torch.float64, device="cuda")
    native.phsvds_block_cgs(h, n, None, n, 0, Td, n, q, Gsub=Gd, Gout=Go, P2=Pd, ld2=n, p2=p)
    native.phsvds_sync(h)
    T2, g = Td.cpu().numpy().T, Go.cpu().numpy().reshape(q, p).T
    bad_t = np.zeros((n, q), bool)
    if where == "basis":
        bad_t[1000] = True
    elif where == "block":
        bad_t[1000, 4] = True
    else:
        bad_t[:, 4] = True
    assert np.array_equal(~np.isfinite(T2), bad_t)
    ok = ~bad_t.any(0)
    if where == "basis":
        assert not np.isfinite(g).any()
    else:
        assert np.isfinite(g[:, ok]).all() and not np.isfinite(g[:, ~ok]).any()
        ref = _mm(P.T, T2[:, ok])
        assert np.all(np.abs(g[:, ok] - ref) <= 70 * EPS * (np.abs(P).T @ np.abs(T2[:, ok])))


@pytest.mark.parametrize("n,p,r", [(1, 1, 1), (130, 9, 3), (1000, 35, 8), (155649, 35, 8), (77825, 20, 17),
                                   (78000, 43, 30), (40000, 10, 60)])
def test_fp32_streaming(h, n, p, r):
    """FP32 storage: one and several rows per thread, with the norms; in place."""
    rng = np.random.default_rng(n)
    P, X = rng.standard_normal((n, p)).astype(np.float32), rng.standard_normal((n, r)).astype(np.float32)
    Y, th = rng.standard_normal((p, r)), rng.standard_normal(r)
    Y32, t32 = Y.astype(np.float32).astype(np.float64), th.astype(np.float32).astype(np.float64)
    P64, X64 = P.astype(np.float64), X.astype(np.float64)
    out, nrm = _tall(h, P, Y, X, th, fp32=True)
    e32 = 2.0 ** -23
    assert np.all(np.abs(out - (P64 @ Y32 - X64 * t32)) <= (p + 2) * e32 * (np.abs(P64) @ np.abs(Y32) + np.abs(X64 * t32)))
    assert np.allclose(nrm, np.sum(out * out, axis=0), rtol=1e-12, atol=0)
    if r <= p:
        out, _ = _tall(h, P, Y, fp32=True, inplace=True)
        assert np.all(np.abs(out - P64 @ Y32) <= (p + 2) * e32 * (np.abs(P64) @ np.abs(Y32)))


def _peaks(rng, n, p, peak, kind):
    """Rows whose magnitudes differ element by element, not by rows or columns."""
    P = rng.standard_normal((n, p))
    if kind == "one":                                       # one element of each row
        P[np.arange(n), np.arange(n) % p] *= peak
    elif kind == "few":                                     # one element in some tiles
        rows = np.arange(5, n, 37)
        P[rows, rows % p] = peak
    else:                                                   # spread over all decades
        P *= peak ** rng.uniform(-1, 1, (n, p))
    return P


@pytest.mark.parametrize("p,r", [(9, 4), (35, 21), (20, 8), (60, 30)])
@pytest.mark.parametrize("peak", [1e3, 1e6, 1e10, 1e25])
@pytest.mark.parametrize("kind", ["one", "few", "spread"])
def test_tall_peaks_inside_a_row(h, p, r, peak, kind):
    """An output whose terms are far below (row maximum) x (coefficient maximum) is as
    accurate as a chain of multiply-adds: within (p + 4) eps of its sum of moduli."""
    rng = np.random.default_rng(p)
    n = 1000
    P = _peaks(rng, n, p, peak, kind)
    zero = rng.standard_normal((p, r))
    zero[:: 3] = 0.0                                        # some peaks meet a zero coefficient
    for Y in (zero, np.eye(p)[:, :r], np.eye(p)[:, :r] + 1e-3 * rng.standard_normal((p, r))):
        out, _ = _tall(h, P, Y)
        S = np.abs(P) @ np.abs(Y)
        assert np.all(np.abs(out - _mm(P, Y)) <= (p + 4) * EPS * S)


def test_tall_peak_with_a_zero_coefficient(h):
    P = np.ones((600, 11))
    P[300, 0] = 1e25
    Y = np.ones((11, 3))
    Y[0] = 0.0
    out, _ = _tall(h, P, Y)
    assert np.all(out == 10.0)


@pytest.mark.parametrize("n,p,q", [(4000, 12, 5), (4001, 35, 8), (9000, 64, 3), (80001, 35, 6)])
@pytest.mark.parametrize("peak", [1e3, 1e8, 1e25])
@pytest.mark.parametrize("kind", ["one", "few", "spread"])
def test_block_cgs_peaks_inside_a_row_and_a_column(h, n, p, q, peak, kind):
    """The same for T - P Gsub (beside |T|), and for P^T T and T^T T within n / 64 + 64 eps
    of the sums of moduli: single elements of T where P is zero, peaks of P where T is small."""
    rng = np.random.default_rng(n + q)
    P = _peaks(rng, n, p, peak, kind)
    T = rng.standard_normal((n, q)) if kind != "spread" else _peaks(rng, n, q, peak, kind)
    rows = np.arange(11, n, 64)
    P[rows] = 0.0
    T[rows, rows % q] = peak
    G = rng.standard_normal((p, q))
    G[:: 3] = 0.0
    Pd, Gd = _dev(P, n), torch.from_numpy(np.ascontiguousarray(G.T)).cuda()
    for sub in (False, True):
        Td = _dev(T, n)
        Go = torch.zeros(p * q, dtype=torch.float64, device="cuda")
        To = torch.zeros(q * q, dtype=torch.float64, device="cuda")
        native.phsvds_block_cgs(h, n, None, n, 0, Td, n, q, Gsub=Gd if sub else None, Gout=Go, Tout=To, P2=Pd, ld2=n,
                                p2=p)
        native.phsvds_sync(h)
        T2 = Td.cpu().numpy().T
        if sub:
            assert np.all(np.abs(T2 - (T.astype(L) - _mm(P, G))) <= (p + 4) * EPS * (np.abs(T) + np.abs(P) @ np.abs(G)))
        else:
            assert np.array_equal(T2, T)
        for buf, A in ((Go, P), (To, T2)):
            got = buf.cpu().numpy().reshape(q, -1).T
            lim = (n / 64 + 64) * EPS * (np.abs(A).T @ np.abs(T2))
            assert np.all(np.abs(got - _mm(A.T, T2)) <= lim)


@pytest.mark.parametrize("p,r", [(9, 4), (33, 8), (35, 21), (64, 30)])
@pytest.mark.parametrize("small", [0.1, 1e-3, 1e-9, 0.0])
def test_tall_coefficients_with_one_large_entry(h, p, r, small):
    """A coefficient far above the others of its column stays out of the digits: unit vectors with
    noise beside them, some columns of even size, one of zeros, signs, and with peaks in P."""
    rng = np.random.default_rng(p)
    n = 1000
    Y = small * rng.standard_normal((p, r))
    Y[rng.permutation(p)[:r], np.arange(r)] = rng.choice([-1.0, 3.0, 1e-200, 1e200], r)
    Y[:, 1] = rng.standard_normal(p)
    Y[:, 2] = 0.0
    for kind, peak in (("one", 1.0), ("one", 1e6), ("spread", 1e25)):
        P = _peaks(rng, n, p, peak, kind)
        out, _ = _tall(h, P, Y)
        S = np.abs(P) @ np.abs(Y)
        assert np.all(np.abs(out - _mm(P, Y)) <= (p + 4) * EPS * S + 1e-300)
