"""A field solve that ends without a solution says so: in the returned status where info is asked
for, in the status word where it is not."""
import numpy as np
import pytest
import torch

from paper_2103_06737_gb300 import inputs as I

pytestmark = pytest.mark.gpu

F = pytest.importorskip("paper_2103_06737_gb300.fem_pic")


def _lib(n):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    m = I.cube_mesh(n, 1.0, 0.1, seed=1)
    lib = F.FemPic(m.xyz, m.tets, F.FP_FP32)
    F.fem_pic_field_setup(lib.h, 0.2 * I.gyro_period(0.1))
    return lib


# one block, on chip over several blocks, streamed; and the FP64 solver
@pytest.mark.parametrize("n,pc", [(2, F.FP_PC_JACOBI), (9, F.FP_PC_JACOBI), (36, F.FP_PC_JACOBI),
                                  (9, F.FP_PC_JACOBI_FP64)])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), 1e200])
def test_no_finite_residual_is_no_convergence(n, pc, bad):
    lib = _lib(n)
    rp, _, _ = F.fem_pic_field_matrix(lib.h, 2)
    rhs = torch.zeros(lib.n_edges, dtype=torch.float64, device="cuda")
    rhs[int(np.nonzero(np.diff(rp) > 1)[0][0])] = bad
    x = torch.zeros_like(rhs)
    st, info = F.fem_pic_field_solve(lib.h, F.FP_SYS_NEWMARK, rhs, x, tol=1e-10, precond=pc)
    assert st == F.FP_ENOCONV and not info["rel_res"] <= 1e-10 and info["iters"] == 0
    assert lib.status() == F.FP_ENOCONV
    x.zero_()
    F.fem_pic_field_solve(lib.h, F.FP_SYS_NEWMARK, rhs, x, tol=1e-10, precond=pc, info=False)
    assert lib.status() == F.FP_ENOCONV
    rhs.zero_()
    x.zero_()
    st, info = F.fem_pic_field_solve(lib.h, F.FP_SYS_NEWMARK, rhs, x, tol=1e-10, precond=pc)
    assert st == F.FP_OK and info["rel_res"] == 0.0 and float(x.abs().max()) == 0.0
    assert lib.status() == F.FP_OK
    lib.close()


# on chip over several blocks, streamed
@pytest.mark.parametrize("n", [9, 36])
def test_abandoned_exchange_is_reported_and_reset(n):
    """An exchange that a block leaves unfinished: the solves after it give up at once and say so
    (not with the numbers of the solve before), and fem_pic_status puts the handle back."""
    lib = _lib(n)
    rp, col, val = F.fem_pic_field_matrix(lib.h, 2)
    rhs = np.random.default_rng(n).uniform(-1.0, 1.0, lib.n_edges)
    rhs[np.diff(rp) == 1] = 0.0
    rhs = torch.as_tensor(rhs, device="cuda")
    vec = lambda k: torch.zeros(k, dtype=torch.float64, device="cuda")
    solve = lambda x, **kw: F.fem_pic_field_solve(lib.h, F.FP_SYS_NEWMARK, rhs, x, tol=1e-10, **kw)
    x0 = vec(lib.n_edges)
    st, info = solve(x0)
    assert st == F.FP_OK and info["iters"] > 0
    assert F.fem_pic_field_last_info(lib.h)[0]["iters"] == info["iters"]
    F.fem_pic_selftest_wait(lib.h, 1e-3)
    with pytest.raises(F.FemPicError, match="gave up waiting"):
        F.fem_pic_field_last_info(lib.h)       # good output words beside the mark are not taken either
    with pytest.raises(F.FemPicError, match="gave up waiting"):
        solve(vec(lib.n_edges))
    solve(vec(lib.n_edges), info=False)
    E = [vec(lib.n_edges) for _ in range(3)]
    with pytest.raises(F.FemPicError, match="gave up waiting"):
        F.fem_pic_field_step(lib.h, E[0], E[1], E[2], None, None, None,
                             torch.zeros(lib.n_nodes, dtype=torch.float32, device="cuda"), tol=1e-10)
    assert lib.status() == F.FP_ECUDA and lib.status() == F.FP_OK
    x1 = vec(lib.n_edges)
    st, again = solve(x1)
    assert st == F.FP_OK and torch.equal(x0, x1)
    assert (again["iters"], again["outer"], again["rel_res"]) == (info["iters"], info["outer"], info["rel_res"])
    assert lib.status() == F.FP_OK
    lib.close()


@pytest.mark.parametrize("model", [F.FP_LEARNED_GUESS, F.FP_LEARNED_PRECOND])
def test_failed_learned_init_leaves_no_network(model):
    """A network whose sample store does not fit on any device: the system is left without one, so
    that a step that asks for it is refused, and everything else works on."""
    lib = _lib(9)
    with pytest.raises(F.FemPicError):
        F.fem_pic_learned_init_model(lib.h, seed=1, sample_capacity=2**31 - 1, model=model)
    E = [torch.zeros(lib.n_edges, dtype=torch.float64, device="cuda") for _ in range(3)]
    Q = torch.zeros(lib.n_nodes, dtype=torch.float32, device="cuda")
    step = lambda pc: F.fem_pic_field_step(lib.h, E[0], E[1], E[2], None, None, None, Q, tol=1e-10, precond=pc)
    with pytest.raises(F.FemPicError, match="learned_init"):
        step(F.FP_PC_LEARNED)
    with pytest.raises(F.FemPicError):
        F.fem_pic_learned_params(lib.h)
    assert step(F.FP_PC_JACOBI)[0] == F.FP_OK
    F.fem_pic_learned_init_model(lib.h, seed=1, sample_capacity=1, model=model)
    if model == F.FP_LEARNED_PRECOND:
        F.fem_pic_learned_build(lib.h)
    assert step(F.FP_PC_LEARNED)[0] == F.FP_OK and lib.status() == F.FP_OK
    lib.close()


def test_solvers_without_exchanges_work_beside_the_mark():
    """A system of one block and the FP64 solver exchange nothing through the words: they go on."""
    lib = _lib(9)
    rhs = torch.zeros(lib.n_edges, dtype=torch.float64, device="cuda")
    rp, _, _ = F.fem_pic_field_matrix(lib.h, 2)
    rhs[int(np.nonzero(np.diff(rp) > 1)[0][0])] = 1.0
    F.fem_pic_selftest_wait(lib.h, 1e-3)
    x = torch.zeros_like(rhs)
    st, info = F.fem_pic_field_solve(lib.h, F.FP_SYS_NEWMARK, rhs, x, tol=1e-10, precond=F.FP_PC_JACOBI_FP64)
    assert st == F.FP_OK and info["rel_res"] <= 1e-10
    g = torch.zeros(lib.n_nodes, dtype=torch.float64, device="cuda")     # 1,000 nodes: one block
    rp, _, _ = F.fem_pic_field_matrix(lib.h, 3)
    g[int(np.nonzero(np.diff(rp) > 1)[0][0])] = 1.0
    st, info = F.fem_pic_field_solve(lib.h, F.FP_SYS_GAUSS, g, torch.zeros_like(g), tol=1e-10)
    assert st == F.FP_OK and info["rel_res"] <= 1e-10
    assert lib.status() == F.FP_ECUDA and lib.status() == F.FP_OK
    lib.close()
