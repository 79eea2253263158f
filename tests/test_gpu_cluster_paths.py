"""GPU: which levels run in the cluster, and the paths that only some of them reach.

* the whole cycle of small quadtrees runs in the cluster, larger finest levels and the octree's
  on the grid with the coarse levels in the cluster;
* a quadtree with blocks of several rows (the lane-parallel block smoother) whose finest level
  is on the grid;
* a device without room for the cluster (host-set): every level on the grid;
* a right-hand side so small that (p, A p) of Alg. 1 is subnormal;
* the bounded waits made to run out on either path (a host-set limit of 1 ms and a first wait
  for more than comes): AMG_ERR_TIMEOUT, then the same bits as before.

Bars against the FP64 CPU oracle, as everywhere: FP64 within 1e-11 relative, the FP32 cycle
within 1e-5.
"""
import numpy as np
import pytest

from paper_1209_5421_gb300.meshes import disk_poisson, p1_poisson, p1_poisson_3d

pytestmark = pytest.mark.gpu

PRECS = ["fp64", "fp32"]


@pytest.fixture(scope="module")
def amg():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("a CUDA device is required for -m gpu tests")
    from paper_1209_5421_gb300 import amg as A
    from paper_1209_5421_gb300 import build

    build.build()
    return A


def _square(n):
    return p1_poisson(n, jitter=0.2, seed=n, rhs="normal")


def _hierarchy(amg, prob, prec, **kw):
    if prec == "fp32":
        kw.update(cycle_prec=amg.FP32, outer=amg.OUTER_FGMRES)
    return amg.Hierarchy.from_problem(prob, **kw)


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("mesh,n,whole", [
    (_square, 20, True), (_square, 34, True), (_square, 65, True),
    (lambda n: disk_poisson(n, jitter=0.2, seed=n), 51, True),
    (_square, 180, False), (_square, 257, False),
    (lambda n: disk_poisson(n, jitter=0.2, seed=n), 203, False),
    (lambda n: p1_poisson_3d(n, seed=n), 17, False),
])
def test_first_level_in_the_cluster(amg, mesh, n, whole, prec):
    prob = mesh(n)
    H = _hierarchy(amg, prob, prec)
    H.apply_cycle(0, prob.b)
    tl = H.debug_cluster_level()
    assert tl == 0 if whole else 1 <= tl < H.nlev, (tl, H.nlev)
    H.close()


@pytest.mark.parametrize("prec", PRECS)
def test_blocks_of_several_rows_on_the_grid(amg, prec):
    from oracle import oracle

    prob = _square(200)  # 39,204 rows over 64 x 64 cells
    O = oracle.Hierarchy.from_problem(prob, aux_level=6)
    rows = np.bincount(O.level(0).agg)
    assert rows[rows > 0].mean() >= 6 and rows.max() <= 16
    H = _hierarchy(amg, prob, prec, aux_level=6)
    z, zo = H.apply_cycle(0, prob.b), O.bhat(0, prob.b)
    assert 1 <= H.debug_cluster_level() < H.nlev
    rel = np.linalg.norm(z - zo) / np.linalg.norm(zo)
    assert rel <= (1e-11 if prec == "fp64" else 1e-5), rel
    H.close()


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("n,whole", [(34, True), (180, False)])
def test_timeout_on_either_path(amg, n, whole, prec):
    prob = _square(n)
    H = _hierarchy(amg, prob, prec)
    x0, it0, _, st0 = H.solve(prob.b, 1e-8)
    assert st0 == amg.OK and (H.debug_cluster_level() == 0) == whole
    H.debug_barrier_fault(limit_ns=1_000_000, extra=1)
    with pytest.raises(amg.AmgError) as ei:
        H.solve(prob.b, 1e-8)
    assert ei.value.status == amg.ERR_TIMEOUT
    H.debug_barrier_fault(0, 0)
    x1, it1, _, st1 = H.solve(prob.b, 1e-8)
    assert st1 == amg.OK and it1 == it0 and np.array_equal(x1, x0)
    H.close()


@pytest.fixture
def no_cluster(amg):
    amg.debug_no_cluster(True)
    yield
    amg.debug_no_cluster(False)


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("mesh,n", [
    (_square, 34), (_square, 257), (lambda n: disk_poisson(n, jitter=0.2, seed=n), 51),
    (lambda n: p1_poisson_3d(n, seed=n), 17)])
def test_every_level_on_the_grid(amg, no_cluster, mesh, n, prec):
    from oracle import oracle

    prob = mesh(n)
    O = oracle.Hierarchy.from_problem(prob)
    H = _hierarchy(amg, prob, prec)
    z, zo = H.apply_cycle(0, prob.b), O.bhat(0, prob.b)
    assert H.debug_cluster_level() == H.nlev
    rel = np.linalg.norm(z - zo) / np.linalg.norm(zo)
    assert rel <= (1e-11 if prec == "fp64" else 1e-5), rel
    x, it, _, st = H.solve(prob.b, 1e-8)
    assert st == amg.OK
    if prec == "fp64":  # the plain method: the oracle's iteration count within one
        assert abs(it - O.solve(prob.b, 1e-8)[1]) <= 1
    H.close()


@pytest.mark.parametrize("n,opts", [(34, {}), (34, dict(kcycle_n=3)), (257, {}), (257, dict(kcycle_n=3))])
def test_subnormal_energy(amg, n, opts):
    # B^ is homogeneous, so B^[c f] / c is B^[f], with c chosen so that (p, A p) is about
    # 2^-1030: a sum of n products, each rounded by at most 2^-1075, has a relative error of
    # n 2^-45 (5e-10 at the cluster's 16,384 rows); a few such sums in turn: bar 1e-6
    prob = _square(n)
    H = _hierarchy(amg, prob, "fp64", **opts)
    f = np.ones(prob.n)
    z = H.apply_cycle(0, f)
    c = 2.0 ** np.floor((-1030 - np.log2(f @ z)) / 2)
    zc = H.apply_cycle(0, c * f) / c
    assert np.isfinite(zc).all()
    assert np.linalg.norm(zc - z) <= 1e-6 * np.linalg.norm(z)
    H.close()
