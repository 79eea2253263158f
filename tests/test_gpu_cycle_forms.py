"""GPU: the four instances of the grid's cycle kernel, against the FP64 CPU oracle.

The instance follows the finest level: blocks of a few rows or of several (the lane-parallel
block smoother), with big blocks (more than 16 rows, graded nodes) or without. One
application of B^_0 each, with the grid's launches and the cluster's in turn.

Bars, as everywhere: FP64 within 1e-11 relative (the order of FP64 sums is the only
difference), the FP32 cycle within 1e-5.
"""
import dataclasses

import numpy as np
import pytest

from paper_1209_5421_gb300.meshes import p1_poisson, p1_poisson_3d

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


def _problem(dim, several, big):
    """Graded by the coordinates alone; the auxiliary grid's depth sets the rows per block."""
    n = 33 if dim == 3 else 90 if several else 129
    prob = p1_poisson(n, jitter=0.2, seed=n) if dim == 2 else p1_poisson_3d(n, seed=n)
    if big:
        xyz = {k: np.abs(getattr(prob, k)) ** (2.0 if dim == 2 else 1.5) for k in ("x", "y", "z")[:dim]}
        prob = dataclasses.replace(prob, **xyz)
    depth = {(2, False): 7, (2, True): 5, (3, False): 5, (3, True): 4}[dim, several]
    return prob, depth


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("big", [False, True])
@pytest.mark.parametrize("several", [False, True])
@pytest.mark.parametrize("dim", [2, 3])
def test_cycle_matches_oracle(amg, dim, several, big, prec):
    from oracle import oracle

    prob, depth = _problem(dim, several, big)
    O = oracle.Hierarchy.from_problem(prob, aux_level=depth)
    rows = np.bincount(O.level(0).agg)
    rows = rows[rows > 0]
    assert (rows.mean() >= 6) == several
    assert (rows.max() > 16) == big
    G = amg.Hierarchy.from_problem(prob, aux_level=depth,
                                   cycle_prec=amg.FP32 if prec == "fp32" else amg.FP64)
    f = np.random.default_rng(7).standard_normal(prob.n)
    z, zo = G.apply_cycle(0, f), O.bhat(0, f)
    rel = np.linalg.norm(z - zo) / np.linalg.norm(zo)
    assert rel <= (1e-11 if prec == "fp64" else 1e-5), (G.nlev, rel)
    assert np.array_equal(G.apply_cycle(0, f), z)  # the same bits every time
    G.close()
