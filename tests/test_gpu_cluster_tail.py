"""GPU: the coarse levels in a thread-block cluster, against the FP64 CPU oracle.

One application of B^_0 (Alg. 2) at the sizes where the cluster's code takes another branch:
only the dense level in the cluster; one and several swept levels; strips of unequal size,
empty cells and children in another strip (disks); nine and more colours; the coarsest
inverse in place of the dense level (a dense level too large, or FP64 in 3D); one to four
Alg. 1 steps; several smoothing sweeps; levels above the cluster left to the grid.

Bars, as everywhere: FP64 within 1e-11 relative (the order of FP64 sums is the only
difference), the FP32 cycle within 1e-5.
"""
import numpy as np
import pytest

from paper_1209_5421_gb300.meshes import disk_poisson, p1_poisson, p1_poisson_3d

pytestmark = pytest.mark.gpu

CASES = [
    ("square", 20, {}), ("square", 33, {}), ("square", 65, dict(aux_level=6)),
    ("square", 130, {}), ("square", 97, dict(kcycle_n=1)), ("square", 97, dict(kcycle_n=3)),
    ("square", 97, dict(kcycle_n=4, nu_pre=2)), ("square", 97, dict(nu_pre=3, nu_post=2)),
    ("square", 101, dict(coarsest_max=7)), ("square", 129, dict(coarsest_max=256)),
    ("square", 257, {}), ("square", 300, dict(coarsest_max=16)),
    ("disk", 51, {}), ("disk", 203, {}), ("disk", 160, dict(coarsest_max=250, kcycle_n=3)),
    ("graded", 129, {}), ("cube", 9, {}), ("cube", 17, {}), ("cube", 30, {}),
    ("cube", 26, dict(coarsest_max=8, kcycle_n=1)),
]


@pytest.fixture(scope="module")
def amg():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("a CUDA device is required for -m gpu tests")
    from paper_1209_5421_gb300 import amg as A
    from paper_1209_5421_gb300 import build

    build.build()
    return A


def _problem(mesh, n):
    if mesh == "disk":
        return disk_poisson(n, jitter=0.2, seed=n)
    if mesh == "cube":
        return p1_poisson_3d(n, seed=n)
    if mesh == "graded":
        return p1_poisson(n, jitter=0.1, graded=True, kappa_blocks=16, seed=n, rhs="normal")
    return p1_poisson(n, jitter=0.2, seed=n, rhs="normal")


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("mesh,n,opts", CASES)
def test_cycle_matches_oracle(amg, prec, mesh, n, opts):
    from oracle import oracle

    prob = _problem(mesh, n)
    O = oracle.Hierarchy.from_problem(prob, **opts)
    G = amg.Hierarchy.from_problem(prob, cycle_prec=amg.FP32 if prec == "fp32" else amg.FP64, **opts)
    f = np.random.default_rng(n).standard_normal(prob.n)
    z, zo = G.apply_cycle(0, f), O.bhat(0, f)
    rel = np.linalg.norm(z - zo) / np.linalg.norm(zo)
    assert rel <= (1e-11 if prec == "fp64" else 1e-5), (G.nlev, rel)
    assert np.array_equal(G.apply_cycle(0, f), z)  # the same bits every time
    G.close()
