"""The mixed solvers on operators whose records and plans the cube meshes' numbering does not reach.

Rows of several records (25 and 1501 slots), 32-bit columns (a mesh numbered at random: the columns of a
slot span the whole vector), and the sizes around the largest edge system that is held on chip: with
152 SMs 32^3 fits with the polynomial's vectors, 33^3 without them (both solvers are set up, and take
turns on the same exchange words), 34^3 not any more; likewise the node system at 64^3.

The FP64 residual of each solution is formed on the CPU with the library's own operators: it may
exceed the tolerance by its own rounding only (10%).
"""
import numpy as np
import pytest
import scipy.sparse as sp
import torch

from paper_2103_06737_gb300 import inputs as I

pytestmark = pytest.mark.gpu

F = pytest.importorskip("paper_2103_06737_gb300.fem_pic")
TOL = 1e-10
EDGES, NODES = F.FP_SYS_NEWMARK, F.FP_SYS_GAUSS


def fan(n):
    """n tets around one edge, in which 3 n + 1 edges meet."""
    rng = np.random.default_rng(n)
    t = 2 * np.pi * (np.arange(n) + rng.uniform(-0.2, 0.2, n)) / n
    ring = np.stack([np.cos(t), np.sin(t), rng.uniform(-0.1, 0.1, n)], 1)
    k = np.arange(n)
    return (np.concatenate([[[0.0, 0.0, -0.5], [0.0, 0.0, 0.5]], ring]),
            np.stack([0 * k, 0 * k + 1, 2 + k, 2 + (k + 1) % n], 1).astype(np.int32))


def twelve(n):
    """n^3 hexes of the unit cube, each cut into twelve tets around its centre: rows of up to 25 edges."""
    cube = I.cube_mesh(n)
    k, j, i = (a.ravel() for a in np.meshgrid(*(np.arange(n),) * 3, indexing="ij"))
    centre = (n + 1) ** 3 + i + n * (j + n * k)
    node = lambda d: (i + d[0]) + (n + 1) * ((j + d[1]) + (n + 1) * (k + d[2]))
    tets = []
    for axis in range(3):
        for side in (0, 1):
            def corner(p, q):
                d = [p, q]
                d.insert(axis, side)
                return node(d)
            for mid in ((1, 0), (0, 1)):
                tets.append(np.stack([centre, corner(0, 0), corner(*mid), corner(1, 1)], 1))
    xyz = np.concatenate([cube.xyz, (np.stack([i, j, k], 1) + 0.5) / n])
    return xyz, np.concatenate(tets).astype(np.int32)


def cube(n, renumbered=False):
    m = I.cube_mesh(n, 1.0, 0.1, seed=1)
    if not renumbered:
        return m.xyz, m.tets
    p = np.random.default_rng(n).permutation(m.n_nodes)      # new id of each node
    xyz = np.empty_like(m.xyz)
    xyz[p] = m.xyz
    return xyz, p[m.tets].astype(np.int32)


def check(mesh, dt, systems, bc, runs, width=None):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    lib = F.FemPic(*mesh, F.FP_FP32)
    F.fem_pic_field_setup(lib.h, dt, bc=bc)
    for system in systems:
        rp, col, val = F.fem_pic_field_matrix(lib.h, 2 if system == EDGES else 3)
        assert width is None or np.diff(rp).max() == width
        rows = len(rp) - 1
        A = sp.csr_matrix((val, col, rp), shape=(rows, rows))
        b = np.random.default_rng(rows + system).uniform(-1.0, 1.0, rows)
        if bc == F.FP_BC_PEC:
            b[(np.diff(rp) == 1) & (val[rp[:-1]] == 1.0)] = 0.0     # PEC rows: the identity
        bd = torch.as_tensor(b, device="cuda")
        if any(pc == F.FP_PC_LEARNED for _, pc in runs):
            F.fem_pic_learned_select(lib.h, system)
            F.fem_pic_learned_init_model(lib.h, seed=4, sample_capacity=1, model=F.FP_LEARNED_PRECOND)
            P = F.fem_pic_learned_params(lib.h)
            P[-130:] = 0.0
            P[-66] = -0.1                  # Delta~ = -0.1 A~ off the diagonal: positive definite
            F.fem_pic_learned_params(lib.h, P)
            F.fem_pic_learned_build(lib.h)
        seen = {}
        for degree, pc in runs:
            F.fem_pic_field_poly(lib.h, system, degree, 30.0)
            x = torch.as_tensor(0.01 * A.diagonal(), device="cuda")
            st, info = F.fem_pic_field_solve(lib.h, system, bd, x, tol=TOL, precond=pc)
            assert st == F.FP_OK and info["rel_res"] <= TOL and info["fell_back"] == 0, (system, degree, pc, info)
            got = x.cpu().numpy()
            assert np.linalg.norm(b - A @ got) <= 1.1 * TOL * np.linalg.norm(b), (system, degree, pc)
            # the same bits whenever the same solver runs, whatever ran before it
            assert np.array_equal(seen.setdefault((degree, pc), got), got), (system, degree, pc)
    assert lib.status() == F.FP_OK
    lib.close()


ALL = [(1, F.FP_PC_JACOBI), (4, F.FP_PC_JACOBI), (1, F.FP_PC_LEARNED)]


def test_rows_of_many_records():
    check(fan(500), 1e-9, [EDGES], F.FP_BC_NEUMANN, ALL, width=1501)


def test_rows_of_two_records():
    check(twelve(30), 1e-10, [EDGES], F.FP_BC_PEC, ALL, width=25)


def test_columns_of_32_bits():
    check(cube(41, renumbered=True), 0.2 * I.gyro_period(0.1), [EDGES, NODES], F.FP_BC_PEC, ALL)


@pytest.mark.parametrize("n,systems", [(32, [EDGES]), (33, [EDGES]), (34, [EDGES]), (64, [NODES])])
def test_solvers_take_turns(n, systems):
    check(cube(n), 0.2 * I.gyro_period(0.1), systems, F.FP_BC_PEC, ALL + [(1, F.FP_PC_JACOBI), (4, F.FP_PC_JACOBI)] + ALL)
