"""GPU: the order of the cluster's steps, with warps that are late now and then.

What keeps the steps of k_cluster_tail in order are counted exchanges, not barriers over the
cluster, so a missing wait shows only when some warp is slower than usual. The checking build
(libamg_gb300_bc.so) makes some warps of every step wait for a few microseconds, another set each
step. One application of B^_0 each on that build, in a child process: the whole cycle in the
cluster (small quadtrees) and coarse levels only, strips of unequal size, children in another
strip, one to three Alg. 1 steps.

Bars, as everywhere: FP64 within 1e-11 relative of the FP64 CPU oracle (the order of FP64 sums
is the only difference), the FP32 cycle within 1e-5; the same bits every time; no flag set.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HEAD = r"""
import numpy as np
from oracle import oracle
from paper_1209_5421_gb300 import amg
from paper_1209_5421_gb300.meshes import disk_poisson, p1_poisson, p1_poisson_3d
assert amg.LIB_PATH.endswith("libamg_gb300_bc.so"), amg.LIB_PATH
square = lambda n: p1_poisson(n, jitter=0.2, seed=n, rhs="normal")
"""
LATE = r"""
cases = [(square(20), {}), (square(34), {}), (square(34), dict(kcycle_n=3)),
         (square(65), dict(aux_level=6)), (square(65), dict(nu_pre=2, nu_post=2)),
         (square(130), {}), (square(150), dict(kcycle_n=3)),
         (disk_poisson(51, jitter=0.2, seed=1), {}), (disk_poisson(203, jitter=0.2, seed=2), {}),
         (p1_poisson_3d(17, seed=3), {})]
"""
# fewer than 16 rows in every colour of the swept levels: CTAs without rows, hence without
# neighbours, which only the sums and gathers over the cluster hold to the others
EMPTY = r"""
cases = [(p, dict(coarsest_max=m, kcycle_n=k))
         for p in (square(6), square(7), square(9), disk_poisson(9, jitter=0.2, seed=4),
                   p1_poisson_3d(7, seed=5))
         for m in (1, 3) for k in (1, 2, 3)]
"""
TAIL = r"""
for k, (p, opts) in enumerate(cases):
    f = np.random.default_rng(k).standard_normal(p.n)
    zo = oracle.Hierarchy.from_problem(p, **opts).bhat(0, f)
    for prec, bar in ((amg.FP64, 1e-11), (amg.FP32, 1e-5)):
        G = amg.Hierarchy.from_problem(p, cycle_prec=prec, **opts)
        z = G.apply_cycle(0, f)
        assert np.linalg.norm(z - zo) <= bar * np.linalg.norm(zo), (k, prec)
        for _ in range(4):
            assert np.array_equal(G.apply_cycle(0, f), z), (k, prec)
        G.close()
assert amg.bounds_flags() == 0
print("late warps ok")
"""


def _run(cases):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("a CUDA device is required for -m gpu tests")
    from paper_1209_5421_gb300 import build

    path = build.build(bounds_check=True)
    env = dict(os.environ, AMG_GB300_LIBRARY=path)
    r = subprocess.run([sys.executable, "-c", HEAD + cases + TAIL], cwd=ROOT, env=env,
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-3000:]
    assert "late warps ok" in r.stdout


def test_late_warps_change_nothing():
    _run(LATE)


def test_ctas_without_rows():
    _run(EMPTY)
