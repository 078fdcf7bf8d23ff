"""The mixed solvers start the field step's Newmark solve from the residual that comes with its
right-hand side; the FP64 solver forms its own.  Both stop at a relative residual of 1e-10, so their
fields agree within 1e-8 (the condition margin of the field tests), on chip and streamed, under
both boundaries, from fields that are not zero on the boundary, and from zero.
"""
import numpy as np
import pytest
import torch

from paper_2103_06737_gb300 import inputs as I

pytestmark = pytest.mark.gpu

F = pytest.importorskip("paper_2103_06737_gb300.fem_pic")


@pytest.mark.parametrize("bc", ["pec", "neumann"])
@pytest.mark.parametrize("n", [2, 5, 13, 42])
def test_mixed_step_matches_fp64_solver(n, bc):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    m = I.cube_mesh(n, 1.0, 0.1, seed=1)
    lib = F.FemPic(m.xyz, m.tets, F.FP_FP64)
    F.fem_pic_field_setup(lib.h, 0.2 / n / I.C_LIGHT, bc=F.FP_BC_NEUMANN if bc == "neumann" else None)
    g = torch.Generator(device="cuda").manual_seed(n)
    rand = lambda k, a: (2 * torch.rand(k, dtype=torch.float64, device="cuda", generator=g) - 1) * a
    ne, nn = lib.n_edges, lib.n_nodes
    for scale in (1.0, 0.0):
        Ep, Ec = rand(ne, scale), rand(ne, scale)
        dGh, dGp, Q = rand(ne, 1e-12 * scale), rand(ne, 1e-12 * scale), rand(nn, 1e-12 * scale)
        out = []
        for pc in (F.FP_PC_JACOBI, F.FP_PC_JACOBI_FP64):
            En = torch.full((ne,), 7.0, dtype=torch.float64, device="cuda")
            st, info = F.fem_pic_field_step(lib.h, Ep, Ec, En, None, dGh, dGp, Q, tol=1e-10, precond=pc)
            assert st == F.FP_OK, info
            assert info[0]["rel_res"] <= 1e-10 and info[1]["rel_res"] <= 1e-10
            out.append(En.cpu().numpy())
        assert np.abs(out[0] - out[1]).max() <= 1e-8 * np.abs(out[1]).max()
        assert scale > 0 or np.abs(out[0]).max() == 0.0
    assert lib.status() == F.FP_OK
    lib.close()
