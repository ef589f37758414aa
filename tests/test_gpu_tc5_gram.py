"""The Grams of the option fp64_tc above width 8 (tcgen05, exact digits) at the edges of their 64-bit frame: a
128-row tile whose columns are constant just below a power of two, where the sum of a digit stack comes close to
the frame's end; and the entries of an unconjugated Gram, sum re re' - sum im im', where the two nearly cancel: on the
diagonal, and beside it where columns are correlated.

Bounds: the factor xi_0 of the residual's Cholesky QR satisfies xi^H xi = R^H R; with unit-variance rows the Gram
and its Cholesky factor are accurate to a few hundred roundings (p n-term sums, condition below 10): 1e-12 of the
largest entry.  X after one iteration: the 1e-10 of the option's own parity test."""
import numpy as np
import pytest

import oracle.blcoc_oracle as O
from paper_1601_05362_gb300 import problems as P
from gpu_common import need_gpu, rel, to_dev

pytestmark = pytest.mark.gpu

# (left column, right column) of a tile: their product summed over 128 rows reaches the frame's end
PAIRS = [(0.999, 1 - 1e-13), (0.9961, 1 - 1e-12), (-0.9961, 1 - 1e-12), (0.9980, -(1 - 2.0**-53)), (1 - 2.0**-53, 1 - 2.0**-53)]


def _near_full_scale(n, p, imag, seed):
    """Random columns whose first 128 rows are constants of PAIRS, in places of every 16-column block pair."""
    B = P.complex_normal(n, p, seed=seed)
    places = [(0, 1), (2, p - 1), (p - 3, p - 2), (3, 5), (4, 6)]
    for (a, b), (i, j) in zip(PAIRS, places):
        B[:128, i] = a * (1j if imag else 1)
        B[:128, j] = b * (1j if imag else 1)
    return B


def _identity_on_the_first_tile(n, seed):
    """diag(I_128, a random complex symmetric matrix): A W keeps W's first 128 rows."""
    import scipy.sparse as sp
    R = P.random_complex_symmetric(n - 128, 5, seed=seed)
    return sp.csr_matrix(sp.block_diag([sp.identity(128, dtype=np.complex128), R.to_scipy()], format="csr"))


@pytest.mark.parametrize("imag", [False, True])
@pytest.mark.parametrize("p", [9, 16, 24, 32])
@pytest.mark.parametrize("method", ["cocr_rq", "cocg_rq"])
def test_constant_columns_near_full_scale(method, p, imag):
    torch = need_gpu()
    from paper_1601_05362_gb300 import blcoc
    n = 1024
    A = _identity_on_the_first_tile(n, p)
    Bh = _near_full_scale(n, p, imag, seed=p)
    with blcoc.Handle(n, A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data) as h:
        h.set_option("fp64_tc", 1)
        B = to_dev(torch, Bh)
        X = torch.zeros_like(B)
        assert h.solve(B, X, method=method, tol=0.0, maxit=0) == blcoc.BLCOC_NOT_CONVERGED
        xi = h.xi(p).astype(np.clongdouble)
        G = np.conj(Bh.astype(np.clongdouble)).T @ Bh.astype(np.clongdouble)
        assert float(np.max(np.abs(np.conj(xi).T @ xi - G)) / np.max(np.abs(G))) < 1e-12
        assert h.solve(B, X, method=method, tol=0.0, maxit=1) == blcoc.BLCOC_NOT_CONVERGED
    f = O.bl_cocr_rq if method == "cocr_rq" else O.bl_cocg_rq
    assert rel(X.cpu().numpy(), f(A, Bh, tol=0.0, maxit=1).X) < 1e-10


def _cancelling(n, p, method, seed):
    """Columns of disjoint support whose Gram V^T V (bl_cocg_rq) or V^T A V (bl_cocr_rq), A diagonal, has diagonal
    entries of about 0.02 although sum re^2 and sum im^2 are in the thousands; entries of 30 bits, so that every sum up
    to re - im is exact.  The other Gram that the first iterate depends on, V^T A V or V^T A^2 V, does not cancel.
    Returns the rows' values, A's diagonal, the columns and the exact diagonals of both."""
    rng = np.random.default_rng(seed)
    m = n // 2
    k = rng.integers(2**28, 2**30, m)
    cocg = method == "cocg_rq"
    k2 = np.minimum(np.rint(k * (1 + 1e-3 * rng.standard_normal(m)) / (1 if cocg else np.sqrt(2))), 2.0**30 - 1)
    z, a = np.empty(n, np.complex128), np.empty(n, np.complex128)
    z[0::2], z[1::2] = k, (1j if cocg else 1 + 1j) * k2
    a[0::2], a[1::2] = 1, -1 if cocg else 1j
    col = np.arange(m) % p
    k2 = k2.astype(np.int64)
    G, H = np.empty(p), np.empty(p, np.complex128)
    for j in range(p):
        x, y = (sum(int(v) ** 2 for v in w[col == j]) for w in (k, k2))
        G[j] = (x - (y if cocg else 2 * y)) / 2**60
        H[j] = (x + y) / 2**60 if cocg else complex(x / 2**60, -2 * y / 2**60)
    return z * 2.0**-30, a, np.repeat(col, 2), G, H


@pytest.mark.parametrize("p", [9, 17, 32])
@pytest.mark.parametrize("method", ["cocg_rq", "cocr_rq"])
def test_diagonal_of_an_unconjugated_gram_keeps_its_small_part(method, p):
    """X_1 = V diag(G / H): the error of G's diagonal is read off X_1 (G is small, so that all other roundings are, too:
    some 1e-16 of 0.02).  Bound 2e-15 rms over the columns: each of at most 304 CTAs rounds four differences of its
    stacks, below 0.1, i.e. sqrt(304 * 4) * 0.1 * 2^-54 = 2e-16 rms, with a factor of ten, which also holds the rounding
    of 1563 tiles to 2^-54 of the scales (sqrt(1563 / 12) * 2^-54 = 6e-16).  Sums rounded before the difference miss it by
    a factor of five: emulated, 1.4e-14."""
    torch = need_gpu()
    from paper_1601_05362_gb300 import blcoc
    n = 200064
    z, a, col, G, H = _cancelling(n, p, method, seed=p)
    Bh = np.zeros((n, p), np.complex128)
    Bh[np.arange(n), col] = z
    with blcoc.Handle(n, np.arange(n + 1, dtype=np.int32), np.arange(n, dtype=np.int32), a) as h:
        h.set_option("fp64_tc", 1)
        B = to_dev(torch, Bh)
        X = torch.zeros_like(B)
        assert h.solve(B, X, method=method, tol=0.0, maxit=1) == blcoc.BLCOC_NOT_CONVERGED
        M = (torch.sum(B.conj() * X, 0) / torch.sum(B.abs().square(), 0)).cpu().numpy()
    assert np.sqrt(np.mean(np.abs(M * H - G) ** 2)) < 2e-15


def _gram_exact(v):
    """v^T v of integers below 2^45 in Python integers: pieces of 15 bits, whose sums FP64 holds."""
    w = [((v >> 30)).astype(np.float64), ((v >> 15) & 0x7FFF).astype(np.float64), (v & 0x7FFF).astype(np.float64)]
    p = v.shape[1]
    G = [[0] * p for _ in range(p)]
    for a in range(3):
        for b in range(3):
            P = w[a].T @ w[b]
            for i in range(p):
                for j in range(p):
                    G[i][j] += int(P[i, j]) << (15 * (4 - a - b))
    return G


def _correlated(n, p, method, seed):
    """As _cancelling, but every column has every row, and all of them share a part u (correlation one half): now the
    entries beside the diagonal cancel too.  Entries of 44 bits, so that a tile's sums are rounded; both Grams exact."""
    rng = np.random.default_rng(seed)
    m = n // 2
    cocg = method == "cocg_rq"
    x = rng.integers(-2**43, 2**43, (m, 1)) + rng.integers(-2**43, 2**43, (m, p))
    d = (1 + 1e-3 * rng.standard_normal((m, 1))) / (1 if cocg else np.sqrt(2))
    y = np.clip(np.rint(x * d), -2.0**44, 2.0**44).astype(np.int64)
    gx, gy = _gram_exact(x), _gram_exact(y)
    G, H = np.empty((p, p)), np.empty((p, p), np.complex128)
    for i in range(p):
        for j in range(p):
            a, b = gx[i][j], gy[i][j]
            G[i, j] = (a - (b if cocg else 2 * b)) / 2**88
            H[i, j] = (a + b) / 2**88 if cocg else complex(a / 2**88, -2 * b / 2**88)
    B = np.empty((n, p), np.complex128)
    B[0::2], B[1::2] = x, (1j if cocg else 1 + 1j) * y
    diag = np.empty(n, np.complex128)
    diag[0::2], diag[1::2] = 1, -1 if cocg else 1j
    return B * 2.0**-44, diag, G, H


@pytest.mark.parametrize("p", [9, 17, 32])
@pytest.mark.parametrize("method", ["cocg_rq", "cocr_rq"])
def test_an_unconjugated_gram_of_correlated_columns_keeps_its_small_part(method, p):
    """X_1 = B H^-1 G: the error of G is H M - G with M from X_1 = B M.  Bound 1e-14 rms over the entries: 1563 tiles
    rounded to 2^-54 of the scales are 6e-16 rms, and the p x p stages, of condition p, round G (below 0.5) by
    p * 0.5 * 2^-53, 2e-15 at p = 32: a factor of four.  Real and imaginary parts summed apart reach 50 to 100 in a CTA's
    sums, whose rounding in three adds is 0.3 * 7e-15 * (2 * 3 * 304)^(1/2) = 9e-14."""
    torch = need_gpu()
    from paper_1601_05362_gb300 import blcoc
    n = 200064
    Bh, a, G, H = _correlated(n, p, method, seed=p)
    with blcoc.Handle(n, np.arange(n + 1, dtype=np.int32), np.arange(n, dtype=np.int32), a) as h:
        h.set_option("fp64_tc", 1)
        B = to_dev(torch, Bh)
        X = torch.zeros_like(B)
        assert h.solve(B, X, method=method, tol=0.0, maxit=1) == blcoc.BLCOC_NOT_CONVERGED
        M = torch.linalg.solve(B.conj().T @ B, B.conj().T @ X).cpu().numpy()
    assert np.sqrt(np.mean(np.abs(H @ M - G) ** 2)) < 1e-14
