"""The counter "launches" of fp64_tc above width 8, whose passes are one or two kernels, against the launches of a
solve that ends at its first stopping test, counted by hand.  (Small n: every reduction but the residual's runs
inside its pass.)"""
import pytest

from paper_1601_05362_gb300 import problems as P
from gpu_common import need_gpu, to_dev

pytestmark = pytest.mark.gpu

RESIDUAL = 2 + 1 + 1            # R and norms, its Grams; their reduction; the QR of R_0
TRUE_RESIDUAL = 1 + 1 + 1       # norms only; their reduction; the norm
COCR_SETUP = 2 + 1 + 2          # product and Gram; H_0; first pass C and its Gram
COCG_SETUP = 1 + 2              # first pass 2; product and Gram
COCR = 1 + 2 + 1 + 2 + 1 + 2    # alpha, pass A + Gram, QR, product + Gram, beta, pass C + Gram
COCR_U = COCR - 1 + 2           # pass C without a Gram, second product + Gram
COCG = 1 + 2 + 1 + 1 + 2        # alpha, pass 1 + Grams, QR, pass 2, product + Gram


@pytest.mark.parametrize("method,uexpl,count", [("cocr_rq", 0, COCR_SETUP + COCR), ("cocr_rq", 1, COCR_SETUP + COCR_U),
                                                ("cocg_rq", 0, COCG_SETUP + COCG)])
@pytest.mark.parametrize("graph", [0, 1])
def test_launches_of_the_tensor_core_set(method, uexpl, count, graph):
    torch = need_gpu()
    from paper_1601_05362_gb300 import blcoc
    A = P.random_complex_symmetric(1000, 6, seed=1)
    B = to_dev(torch, P.complex_normal(1000, 16, seed=2))
    with blcoc.Handle.from_csr(A) as h:
        for key, value in (("fp64_tc", 1), ("u_explicit", uexpl), ("poll", 1), ("graph", graph)):
            h.set_option(key, value)
        assert h.solve(B, torch.zeros_like(B), method=method, tol=0.0, maxit=0) == blcoc.BLCOC_NOT_CONVERGED
        assert h.stat("launches") == RESIDUAL + count + TRUE_RESIDUAL
