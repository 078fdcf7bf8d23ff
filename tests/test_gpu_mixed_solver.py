"""The mixed solvers: on chip (operator and vectors in shared memory) and streamed, with sums on the
grid's arrivals.

Sizes at their edges: one block (at most 1024 rows) and just above it, a few blocks, every SM with
several slices per warp, partial last slices, the first edge systems that no longer fit on chip
(41, 44: streamed); Jacobi, the Chebyshev polynomial and a learned
correction; both boundary conditions; a start that is not zero and a second solve right after.
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


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2103_06737_gb300 import build
    build.build()


@pytest.mark.parametrize("n", [2, 4, 5, 9, 10, 17, 23, 32, 41, 44])
@pytest.mark.parametrize("bc", [F.FP_BC_PEC, F.FP_BC_NEUMANN])
def test_mixed_solves_reach_the_tolerance(n, bc):
    m = I.cube_mesh(n, 1.0, 0.1, seed=1)
    lib = F.FemPic(m.xyz, m.tets, F.FP_FP32)
    F.fem_pic_field_setup(lib.h, 0.2 * I.gyro_period(0.1), bc=bc)
    for system in (F.FP_SYS_NEWMARK, F.FP_SYS_GAUSS):
        rp, col, val = F.fem_pic_field_matrix(lib.h, 2 if system == F.FP_SYS_NEWMARK else 3)
        rows = len(rp) - 1
        A = sp.csr_matrix((val, col, rp), shape=(rows, rows))
        rng = np.random.default_rng(100 * n + system)
        b = rng.uniform(-1.0, 1.0, rows)
        if bc == F.FP_BC_PEC:
            b[(np.diff(rp) == 1) & (val[rp[:-1]] == 1.0)] = 0.0     # PEC rows: the identity
        elif system == F.FP_SYS_GAUSS:
            b -= b.mean()                  # the natural boundary's Laplacian: zero row sums
        F.fem_pic_learned_select(lib.h, system)
        F.fem_pic_learned_init_model(lib.h, seed=4, sample_capacity=1, model=F.FP_LEARNED_PRECOND)
        P = F.fem_pic_learned_params(lib.h)
        P[-130:] = 0.0
        P[-66] = -0.1                      # Delta~ = -0.1 A~ off the diagonal: positive definite
        F.fem_pic_learned_params(lib.h, P)
        F.fem_pic_learned_build(lib.h)
        for degree, pc, start in ((1, F.FP_PC_JACOBI, 0.0), (2, F.FP_PC_JACOBI, 1.0), (8, F.FP_PC_JACOBI, 0.0),
                                  (1, F.FP_PC_LEARNED, 1.0)):
            F.fem_pic_field_poly(lib.h, system, degree, 30.0)
            x = torch.as_tensor(start * A.diagonal() * 0.01, device="cuda")
            bd = torch.as_tensor(b, device="cuda")
            for again in range(2):
                st, info = F.fem_pic_field_solve(lib.h, system, bd, x, tol=TOL, precond=pc)
                assert st == F.FP_OK and info["rel_res"] <= TOL and info["fell_back"] == 0, (n, system, degree, info)
                r = b - A @ x.cpu().numpy()
                assert np.linalg.norm(r) <= 1.1 * TOL * np.linalg.norm(b), (n, system, degree, pc)
            assert info["iters"] == 0      # the second solve starts from the first one's solution
    assert lib.status() == F.FP_OK
    lib.close()


def test_sums_that_leave_the_expected_range():
    """A right-hand side of one entry: the first sums of the inner CG fall by many orders of
    magnitude, so the blocks add their partials one by one; the same bits on every run."""
    m = I.cube_mesh(12, 1.0, 0.1, seed=1)
    lib = F.FemPic(m.xyz, m.tets, F.FP_FP32)
    F.fem_pic_field_setup(lib.h, 0.2 * I.gyro_period(0.1))
    rp, col, val = F.fem_pic_field_matrix(lib.h, 2)
    rows = len(rp) - 1
    A = sp.csr_matrix((val, col, rp), shape=(rows, rows))
    b = np.zeros(rows)
    b[np.nonzero(np.diff(rp) > 1)[0][0]] = 1e-30
    F.fem_pic_field_poly(lib.h, F.FP_SYS_NEWMARK, 16, 100.0)
    out = []
    for _ in range(3):
        x = torch.zeros(rows, dtype=torch.float64, device="cuda")
        st, info = F.fem_pic_field_solve(lib.h, F.FP_SYS_NEWMARK, torch.as_tensor(b, device="cuda"), x, tol=TOL)
        assert st == F.FP_OK
        out.append(x.cpu().numpy())
    assert np.linalg.norm(b - A @ out[0]) <= 1.1 * TOL * np.linalg.norm(b)
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])
    lib.close()
