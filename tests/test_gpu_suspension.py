"""A Cholesky QR that fails in mid-solve: the solve suspends itself for the shifted-CholQR3 fallback (at p <= 4 from
the stage inside a pass, before the QR).  Whatever way the fallback is launched, in a suspended solve, as launches that
every iteration carries (option graph_conditional), without graphs or in a batch, the results are the same bits.

The systems lose rank at the first QR after the setup's: column 2 of B is A times column 1 plus 1e-9 of a random
vector, so that the next block has a column of that size, which the fallback still resolves (the Gram does not)."""
import numpy as np
import pytest

import oracle.blcoc_oracle as O
from paper_1601_05362_gb300 import problems as P
from gpu_common import need_gpu, rel, to_dev

pytestmark = pytest.mark.gpu

M = 4   # iterations


def _system(n, p, seed):
    A = P.random_complex_symmetric(n, 5, seed=seed)
    B = P.complex_normal(n, p, seed=seed + 1)
    B[:, 1] = A.to_scipy() @ B[:, 0] + 1e-9 * B[:, 1]
    return A, B


def _run(torch, blcoc, A, Bh, method, options, batch=False):
    with blcoc.Handle.from_csr(A) as h:
        for key, value in options.items():
            h.set_option(key, value)
        B = to_dev(torch, Bh)
        X = torch.zeros_like(B)
        if batch:   # beside a system that needs no fallback
            A2 = P.random_complex_symmetric(90, 5, seed=9)
            with blcoc.Handle.from_csr(A2) as h2:
                B2 = to_dev(torch, P.complex_normal(90, 2, seed=9))
                blcoc.solve_batched([h2, h], [B2, B], [torch.zeros_like(B2), X], method=method, tol=0.0, maxit=M, autotune=False)
            st = None
        else:
            st = h.solve(B, X, method=method, tol=0.0, maxit=M)
        info = h.info()
        return st, X.cpu().numpy(), np.asarray(info["hist"]), info["iters"], h.stat("qr_fallbacks")


@pytest.mark.parametrize("method", ["cocr_rq", "cocg_rq"])
@pytest.mark.parametrize("p,tc", [(2, 0), (3, 0), (4, 0), (8, 0), (8, 1), (12, 1), (16, 1), (24, 1)])
def test_fallback_in_mid_solve(method, p, tc):
    torch = need_gpu()
    from paper_1601_05362_gb300 import blcoc
    n = 40 * p + 3
    A, B = _system(n, p, seed=p)
    base = {"fp64_tc": tc}
    want = _run(torch, blcoc, A, B, method, base)
    assert want[0] == blcoc.BLCOC_NOT_CONVERGED and want[3] == M and want[4] >= 1
    for options in ({"poll": 1}, {"graph": 0}, {"graph_conditional": 1}, {"graph_conditional": 1, "graph": 0}):
        got = _run(torch, blcoc, A, B, method, {**base, **options})
        assert got[0] == want[0] and got[3:] == want[3:], options
        assert np.array_equal(got[1], want[1]) and np.array_equal(got[2], want[2]), options
    got = _run(torch, blcoc, A, B, method, base, batch=True)
    assert got[3:] == want[3:] and np.array_equal(got[1], want[1]) and np.array_equal(got[2], want[2])
    # the column of size 1e-9 carries 1e-7 of relative accuracy
    f = O.bl_cocr_rq if method == "cocr_rq" else O.bl_cocg_rq
    assert rel(want[1], f(A.to_scipy(), B, tol=0.0, maxit=M).X) < 1e-6


@pytest.mark.parametrize("method", ["cocr_rq", "cocg_rq"])
@pytest.mark.parametrize("p,tc", [(2, 0), (4, 0), (8, 0), (16, 1)])
def test_without_the_fallback_it_is_a_breakdown(method, p, tc):
    torch = need_gpu()
    from paper_1601_05362_gb300 import blcoc
    A, B = _system(40 * p + 3, p, seed=p)
    base = {"fp64_tc": tc, "qr_fallback": 0}
    want = _run(torch, blcoc, A, B, method, base)
    assert want[0] == blcoc.BLCOC_BREAKDOWN and want[4] == 0
    for options in ({"poll": 1}, {"graph": 0}, {"graph_conditional": 1}):
        got = _run(torch, blcoc, A, B, method, {**base, **options})
        assert got[0] == want[0] and got[3:] == want[3:], options
        assert np.array_equal(got[1], want[1]) and np.array_equal(got[2], want[2]), options
    got = _run(torch, blcoc, A, B, method, base, batch=True)
    assert got[3:] == want[3:] and np.array_equal(got[1], want[1]) and np.array_equal(got[2], want[2])


@pytest.mark.parametrize("method,after", [("cocr_rq", ["spmm_gram", "cocr_passC", "small_beta"]), ("cocg_rq", ["spmm_gram", "cocg_pass2"])])
@pytest.mark.parametrize("graph", [0, 1])
def test_kernel_times_leave_out_what_returned_at_once(method, after, graph):
    """Option timing, suspended in the first of M iterations: the kernels behind that QR returned at once and are run
    again untimed, so M - 1 of each are counted, and M of those before it."""
    torch = need_gpu()
    from paper_1601_05362_gb300 import blcoc
    A, Bh = _system(323, 8, seed=8)
    with blcoc.Handle.from_csr(A) as h:
        h.set_option("timing", 1)
        h.set_option("graph", graph)
        B = to_dev(torch, Bh)
        assert h.solve(B, torch.zeros_like(B), method=method, tol=0.0, maxit=M) == blcoc.BLCOC_NOT_CONVERGED
        assert h.stat("qr_fallbacks") == 1
        assert h.stat("kt_n.small_alpha") == h.stat("kt_n.small_chol") == M
        assert [h.stat("kt_n." + k) for k in after] == [M - 1] * len(after)
