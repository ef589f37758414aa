"""The cache of the SpMM's timed row bundle: a single solve and a batch of the same shape share an entry only where
bundle 1 is the same kernel for both (at 5 <= p <= 16 a single FP64 solve runs it as two launches), so that a bundle
timed for one is not taken over by the other."""
import pytest

from paper_1601_05362_gb300 import problems as P
from gpu_common import need_gpu, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,shared", [(4, True), (8, False), (16, False), (24, True)])
def test_batch_and_single_solves_time_their_own_kernels(p, shared):
    torch = need_gpu()
    from paper_1601_05362_gb300 import blcoc
    n = 2300 + p   # sizes of this test alone: the cache is the process's
    A = P.random_complex_symmetric(n, 6, seed=p)
    B = to_dev(torch, P.complex_normal(n, p, seed=1))
    with blcoc.Handle.from_csr(A) as h:
        h.set_option("spmm_split", 0)

        def batch():
            blcoc.solve_batched([h], [B], [torch.zeros_like(B)], tol=0.0, maxit=3, autotune=False)
            return h.stat("spmm_sweeps")

        def single():
            h.solve(B, torch.zeros_like(B), tol=0.0, maxit=3)
            return h.stat("spmm_sweeps")

        assert batch() == 1
        assert single() == (1 if shared else 2)
        assert batch() == single() == (1 if shared else 2)
