"""The work a user of this library has it do, as cases that can be timed and compared.

A case is a dict of plain values: a family of matrices with its size, the arithmetic of the
cycle, and what the program does with the library:

* ``once``   set up a new matrix, solve one right-hand side, release it;
* ``solve``  keep the hierarchy, solve a further right-hand side;
* ``apply``  keep the hierarchy, apply the cycle once (a preconditioner in a Krylov loop of
             the program's own);
* ``batch``  keep many hierarchies, solve all their systems in one call.

Matrices are P1 stiffness matrices of jittered Kuhn triangulations (two triangles per square,
six tetrahedra per cube) with zero Dirichlet data, as the library's workloads: quasi-uniform
squares, squares graded by x -> x^2 with a coefficient that jumps between 16 x 16 blocks,
disks cut from a square, cubes. The jitter, the coefficient and the right-hand side come from
the seed. A pass returns the solution and the iteration counts; the residual norm that the
library reports beside them is left out, as it is a norm of the solution's error.

The graded meshes are solved with the FP64 cycle only: they take about a hundred iterations,
and with the FP32 cycle their number depends on the rounding of the cycle's sums.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_1209_5421_gb300 import amg

TOL = 1e-8


# --- the cases -----------------------------------------------------------------------------

def _case(name, do, mesh, n, prec, outer, aux=0, **more):
    return dict(name=name, do=do, mesh=mesh, n=n, prec=prec, outer=outer, aux=aux, **more)


def listed():
    return [
        # smallest calls, where launches and latency are all there is: a small model set up
        # and solved once (the plain FP64 method), and one more right-hand side on a smaller
        _case("once_square_65_fp64", "once", "square", 65, "fp64", "fcg", aux=6),
        _case("solve_square_34_fp64", "solve", "square", 34, "fp64", "fcg"),
        # ordinary sizes: a mid-size square, a disk (empty auxiliary cells, ragged rows), and
        # the cycle alone as the preconditioner of the caller's own iteration
        _case("solve_square_257_fp64", "solve", "square", 257, "fp64", "fcg"),
        _case("solve_disk_641_fp32", "solve", "disk", 641, "fp32", "fgmres"),
        _case("apply_square_513_fp64", "apply", "square", 513, "fp64", "fcg"),
        # a graded mesh with coefficient jumps: many iterations, cells of many unknowns
        _case("solve_graded_513_fp64", "solve", "graded", 513, "fp64", "fcg"),
        # a million unknowns on a 1024 x 1024 auxiliary grid: the FP32 cycle inside FP64
        # FGMRES, with setup and without, and the plain FP64 method
        _case("once_square_1025_fp32", "once", "square", 1025, "fp32", "fgmres", aux=10),
        _case("solve_square_1025_fp32", "solve", "square", 1025, "fp32", "fgmres", aux=10),
        _case("solve_square_1025_fp64", "solve", "square", 1025, "fp64", "fcg", aux=10),
        # two million unknowns in 3D (octree)
        _case("solve_cube_129_fp32", "solve", "cube", 129, "fp32", "fgmres"),
        # many systems at once: a full batch of uneven systems in the launch shape the library
        # picks, and a server's handful in a fixed shape
        _case("batch_256_fp32", "batch", "square", 450, "fp32", "fcg", systems=256, nmin=45,
              threads=0),
        _case("batch_12_fp64", "batch", "square", 225, "fp64", "fcg", systems=12, nmin=45,
              threads=1024),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    mesh, prec, outer = "square", "fp64", "fcg"
    do = rng.choice(["once", "solve", "solve", "apply", "batch"])
    more = {}
    if do == "batch":
        n = _log_int(rng, 90, 400)
        more = dict(systems=_log_int(rng, 2, 200), nmin=rng.choice([20, 45]),
                    threads=rng.choice([0, 1024]))
        prec = rng.choice(["fp64", "fp32"])
    else:
        mesh = rng.choice(["square", "square", "disk", "cube", "graded"])
        n = _log_int(rng, *{"square": (24, 1000), "disk": (40, 1000), "cube": (12, 110),
                            "graded": (33, 420)}[mesh])
        if mesh != "graded" and do != "apply":
            prec, outer = rng.choice([("fp64", "fcg"), ("fp32", "fgmres")])
    case = _case("", do, mesh, n, prec, outer, **more)
    del case["name"]
    return case


# --- meshes and matrices -------------------------------------------------------------------

def _sizes(case):
    """Nodes per side of a batch's systems: log-uniform, the largest first (the same for every
    seed: a server's users keep their meshes)."""
    count, lo, hi = case["systems"], case["nmin"], case["n"]
    u = (np.arange(count) + 0.5) / count
    return [int(v) for v in np.rint(np.exp(math.log(lo) + u * math.log(hi / lo)))][::-1]


def _shape(case, n):
    """(unknowns, stored entries) of a system of n nodes per side, about (disk: by area)."""
    if case["mesh"] == "cube":
        m = n - 2
        return m ** 3, 15 * m ** 3
    m2 = (n - 2) ** 2 * (math.pi / 4 if case["mesh"] == "disk" else 1.0)
    return int(m2), int(7 * m2)


def _matrix(mesh, n, gen):
    """rowptr, col, val and the unknowns' coordinates of one system, on the GPU."""
    dim = 3 if mesh == "cube" else 2
    f64 = dict(dtype=torch.float64, device="cuda")
    h = 1.0 / (n - 1)
    inner = tuple(slice(1, n - 1) for _ in range(dim))
    axis = torch.arange(n, **f64) * h
    xyz, grid = [], []  # coordinate arrays indexed [(k,) j, i]; the nodes before the jitter
    for d in range(dim):
        grid.append(axis.view([n if a == dim - 1 - d else 1 for a in range(dim)]).expand([n] * dim))
        c = grid[d].clone()
        width = {"cube": 0.15, "graded": 0.1}.get(mesh, 0.2) * h
        c[inner] += (2.0 * torch.rand([n - 2] * dim, generator=gen, **f64) - 1.0) * width
        xyz.append(c * c if mesh == "graded" else c)
    kappa = torch.ones([n - 1] * dim, **f64)
    if mesh == "graded":
        block = 10.0 ** (2.0 * torch.rand(16, 16, generator=gen, **f64) - 1.0)
        at = (torch.arange(n - 1, device="cuda") * 16) // (n - 1)
        kappa = block[at][:, at]

    def cells(off):  # the node at offset `off` (x, y(, z)) of every cell
        return tuple(slice(off[dim - 1 - a], n - 1 + off[dim - 1 - a]) for a in range(dim))

    def cross(a, b):
        return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]

    stencil = {}
    for perm in itertools.permutations(range(dim)):  # one simplex of every cell
        offs = [[0] * dim]
        for a in perm:
            offs.append([o + (k == a) for k, o in enumerate(offs[-1])])
        v = [[c[cells(o)] for c in xyz] for o in offs]
        e = [[p - q for p, q in zip(w, v[0])] for w in v[1:]]
        if dim == 2:
            det = e[0][0] * e[1][1] - e[0][1] * e[1][0]
            g = [[e[1][1], -e[1][0]], [-e[0][1], e[0][0]]]
        else:
            g = [cross(e[1], e[2]), cross(e[2], e[0]), cross(e[0], e[1])]
            det = sum(p * q for p, q in zip(e[0], g[0]))
        g = [[-sum(t) for t in zip(*g)]] + g  # gradients of the barycentric coordinates x det
        scale = kappa / ((2.0 if dim == 2 else 6.0) * det.abs())
        for a in range(dim + 1):
            for b in range(a, dim + 1):
                k = scale * sum(p * q for p, q in zip(g[a], g[b]))
                for s, t in {(a, b), (b, a)}:
                    key = tuple(q - p for p, q in zip(offs[s], offs[t]))
                    if key not in stencil:
                        stencil[key] = torch.zeros([n] * dim, **f64)
                    stencil[key][cells(offs[s])] += k
    keep = torch.zeros([n] * dim, dtype=torch.bool, device="cuda")
    keep[inner] = True
    if mesh == "disk":  # by the nodes before the jitter: the same unknowns for every seed
        keep &= (grid[0] - 0.5) ** 2 + (grid[1] - 0.5) ** 2 < 0.25
    nodes = keep.view(-1).nonzero().view(-1)
    uid = torch.full((n ** dim,), -1, dtype=torch.int64, device="cuda")
    uid[nodes] = torch.arange(len(nodes), device="cuda")
    lin = {key: sum(o * n ** d for d, o in enumerate(key)) for key in stencil}
    keys = sorted(stencil, key=lin.get)  # ascending columns
    cols = torch.stack([uid[nodes + lin[key]] for key in keys], 1)
    vals = torch.stack([stencil[key].view(-1)[nodes] for key in keys], 1)
    ok = cols >= 0
    rowptr = torch.zeros(len(nodes) + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(ok.sum(1), 0, out=rowptr[1:])
    return (rowptr.to(torch.int32), cols[ok].to(torch.int32), vals[ok],
            [c.reshape(-1)[nodes] for c in xyz])


def _system(case, seed):
    """The case's matrix (a batch's: one block-diagonal matrix, with row offsets) and b."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    sizes = _sizes(case) if case["do"] == "batch" else [case["n"]]
    parts = [_matrix(case["mesh"], n, gen) for n in sizes]
    rows = np.cumsum([0] + [len(p[0]) - 1 for p in parts])
    nnz = np.cumsum([0] + [len(p[1]) for p in parts])
    rowptr = torch.cat([p[0][:-1] + int(z) for p, z in zip(parts, nnz)] + [parts[-1][0][-1:] + int(nnz[-2])])
    col = torch.cat([p[1] + int(r) for p, r in zip(parts, rows)])
    val = torch.cat([p[2] for p in parts])
    xyz = [torch.cat(c) for c in zip(*[p[3] for p in parts])]
    b = torch.randn(int(rows[-1]), dtype=torch.float64, device="cuda", generator=gen)
    return rows, rowptr, col, val, xyz, b


# --- what the program does -----------------------------------------------------------------

def _options(case):
    o = dict(cycle_prec=amg.FP32 if case["prec"] == "fp32" else amg.FP64)
    if case["do"] != "batch":
        o.update(aux_level=case["aux"],
                 outer=amg.OUTER_FGMRES if case["outer"] == "fgmres" else amg.OUTER_FCG)
    return o


def _hierarchy(state):
    rowptr, col, val, xyz = state["matrix"]
    return amg.Hierarchy(rowptr, col, val, xyz[0], xyz[1], z=xyz[2] if len(xyz) == 3 else None,
                         **_options(state["case"]))


def prepare(case, seed):
    rows, rowptr, col, val, xyz, b = _system(case, seed)
    state = dict(case=case, matrix=(rowptr, col, val, xyz), b=b)
    if case["do"] == "batch":
        together = (rows, rowptr, col, val, xyz[0], xyz[1])
        if case["threads"]:  # a server's: hierarchies of its own, a fixed launch shape
            state["kept"] = amg.setup_many(concatenated=together, **_options(case))
            state["batch"] = amg.Batch.over(state["kept"], threads=case["threads"])
        else:  # the launch shape is chosen by the first solve
            state["batch"] = amg.Batch(concatenated=together, **_options(case))
            state["batch"].solve(b, TOL)
        state["matrix"] = None
    elif case["do"] != "once":
        state["h"] = _hierarchy(state)
        state["matrix"] = None
    return state


def run(state):
    do = state["case"]["do"]
    if do == "batch":
        x, iters, _, status = state["batch"].solve(state["b"], TOL)
        return x, iters, status
    if do == "apply":
        return state["h"].apply_cycle(0, state["b"])
    h = _hierarchy(state) if do == "once" else state["h"]
    x, iters, _, status = h.solve(state["b"], TOL)
    if do == "once":
        h.close()
    return x, iters, status


def work(case):
    """The matrix (once: as CSR with coordinates; kept: its values and columns), b and x once;
    one product with the matrix."""
    sizes = _sizes(case) if case["do"] == "batch" else [case["n"]]
    n, nnz = (sum(v) for v in zip(*[_shape(case, s) for s in sizes]))
    more = (4 + 8 * (3 if case["mesh"] == "cube" else 2)) * n if case["do"] == "once" else 0
    return {"bytes": 12 * nnz + 16 * n + more, "flops": 2 * nnz}


def exact(case, seed):
    """The solution, by conjugate gradients with the diagonal as preconditioner in 64 bits,
    corrected twice by its own residual."""
    if case["do"] == "apply":
        return None
    rows, rowptr, col, val, _, b = _system(case, seed)
    n = len(b)
    A = torch.sparse_csr_tensor(rowptr, col, val, size=(n, n))
    line = torch.repeat_interleave(torch.arange(n, device="cuda"), (rowptr[1:] - rowptr[:-1]).long())
    dinv = 1.0 / val[line == col]
    bn = float(b.norm())
    x = torch.zeros_like(b)
    for _ in range(3):
        r = b - A @ x
        goal, e = 1e-14 * bn, torch.zeros_like(b)
        z = dinv * r
        p, rz = z.clone(), torch.dot(r, z)
        for k in range(30000):
            q = A @ p
            alpha = rz / torch.dot(p, q)
            e.addcmul_(alpha.expand(n), p)
            r.addcmul_(alpha.expand(n), q, value=-1.0)
            if k % 100 == 99 and float(r.norm()) <= goal:
                break
            torch.mul(dinv, r, out=z)
            rz, old = torch.dot(r, z), rz
            p.mul_(rz / old).add_(z)
        x += e
    if float((b - A @ x).norm()) > 1e-11 * bn:
        return None
    return x, None, None
