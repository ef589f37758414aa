"""The Grams of the option fp64_tc above width 8 (tcgen05, exact digits) at the edges of their 64-bit frame: a
128-row tile whose columns are constant just below a power of two, where the sum of a digit stack comes close to
the frame's end.

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
