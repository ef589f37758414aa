"""A solve whose kernel gave up a wait: it returns BLCOC_ERR_TIMEOUT, and whatever call comes next on the handle
starts with clean arrival counters of the fused reductions, so that its results are those of a fresh handle, bit
for bit.  The failure is made on the host (option lost_wait): no kernel waits in vain here."""
import numpy as np
import pytest

from paper_1601_05362_gb300 import problems as P
from gpu_common import need_gpu, to_dev

pytestmark = pytest.mark.gpu

FORMS = ["solve", "solve_tc", "mixed", "graph_batch", "persistent_batch", "residual_norm"]


def _call(torch, blcoc, form, h, B):
    X = torch.zeros_like(B)
    if form == "residual_norm":
        return [h.residual_norm(B, B * 0.25)]
    if form in ("graph_batch", "persistent_batch"):
        blcoc.solve_batched([h], [B], [X], tol=0.0, maxit=6, autotune=False, persistent=form == "persistent_batch")
    elif form == "mixed":
        h.solve(B, X, method="cocr_rq_mixed", tol=1e-11, maxit=60)
    else:
        h.set_option("fp64_tc", 1 if form == "solve_tc" else 0)
        h.solve(B, X, tol=0.0, maxit=6)
        h.set_option("fp64_tc", 0)
    return [X.cpu().numpy(), np.asarray(h.info()["hist"]), np.asarray(h.info()["relres_true"])]


@pytest.mark.parametrize("p", [3, 8, 16])
@pytest.mark.parametrize("form", FORMS)
def test_next_call_after_a_lost_wait(form, p):
    torch = need_gpu()
    from paper_1601_05362_gb300 import blcoc
    A = P.random_complex_symmetric(1501, 6, seed=p)
    B = to_dev(torch, P.complex_normal(1501, p, seed=3))
    with blcoc.Handle.from_csr(A) as h:
        want = _call(torch, blcoc, form, h, B)
    for lost in FORMS[:-1]:
        with blcoc.Handle.from_csr(A) as h:
            h.set_option("lost_wait", 1)
            with pytest.raises(blcoc.BlcocError) as e:
                _call(torch, blcoc, lost, h, B)
            assert e.value.status == blcoc.BLCOC_ERR_TIMEOUT
            h.set_option("fp64_tc", 0)
            for got in (_call(torch, blcoc, form, h, B), _call(torch, blcoc, form, h, B)):
                for g, w in zip(got, want):
                    assert np.array_equal(g, w)
