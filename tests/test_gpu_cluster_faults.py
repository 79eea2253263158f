"""GPU: the bounded waits of the cluster's exchanges, made to run out.

As the other faults of the tests, made on the host: a limit of 1 ms, and a first exchange that
waits for more bytes than are sent (a number beyond what an mbarrier counts included). The whole cycle of these small quadtrees runs in the
cluster, so no grid barrier runs out before it. The call returns AMG_ERR_TIMEOUT, every CTA
goes through its remaining steps without exchanges and leaves together with the others, and
the next call on the same hierarchy gives the same bits as before.
"""
import numpy as np
import pytest

from paper_1209_5421_gb300.meshes import p1_poisson

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def amg():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("a CUDA device is required for -m gpu tests")
    from paper_1209_5421_gb300 import amg as A
    from paper_1209_5421_gb300 import build

    build.build()
    return A


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("n,extra", [(9, 1), (34, 1), (34, 2**31 - 1)])
def test_cluster_wait_timeout_then_recovery(amg, prec, n, extra):
    prob = p1_poisson(n, jitter=0.2, seed=n, rhs="normal")
    kw = dict(cycle_prec=amg.FP32, outer=amg.OUTER_FGMRES) if prec == "fp32" else {}
    H = amg.Hierarchy.from_problem(prob, coarsest_max=4, **kw)
    z0 = H.apply_cycle(0, prob.b)
    x0, it0, _, st0 = H.solve(prob.b, 1e-8)
    assert st0 == amg.OK
    for call in (lambda: H.apply_cycle(0, prob.b), lambda: H.solve(prob.b, 1e-8)):
        H.debug_barrier_fault(limit_ns=1_000_000, extra=extra)
        with pytest.raises(amg.AmgError) as ei:
            call()
        assert ei.value.status == amg.ERR_TIMEOUT
        H.debug_barrier_fault(0, 0)
        assert np.array_equal(H.apply_cycle(0, prob.b), z0)
        x1, it1, _, st1 = H.solve(prob.b, 1e-8)
        assert st1 == amg.OK and it1 == it0 and np.array_equal(x1, x0)
    H.close()
