"""The FP64 push: particles that stay (deposits summed per run in shared memory) and that leave their
tet (queued per warp and walked together), at the sizes where the queue and the last warp are
partly filled, with none, some and all particles leaving, aggregated or not, against the oracle.
"""
import numpy as np
import pytest
import torch

from paper_2103_06737_gb300 import inputs as I
from helpers import EPS, TOL, assert_deposit_close

pytestmark = pytest.mark.gpu

F = pytest.importorskip("paper_2103_06737_gb300.fem_pic")
O = pytest.importorskip("oracle")


@pytest.fixture(scope="module")
def setup():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2103_06737_gb300 import build
    build.build()
    m = I.cube_mesh(4, 1.0, 0.1, seed=1)
    lib = F.FemPic(m.xyz, m.tets, F.FP_FP64)
    orc = O.Oracle(m.xyz, m.tets)
    e, b = orc.project_uniform((0.05, -0.02, 0.03), (0.1, 0.0, 0.5))
    yield m, lib, orc, e, b
    lib.close()


@pytest.mark.parametrize("n", [1, 31, 33, 256, 257, 5001])
@pytest.mark.parametrize("dt", [0.01, 0.05, 0.3, 5.0])
@pytest.mark.parametrize("flags", [0, F.FP_NO_AGGREGATE])
def test_push64_matches_the_oracle(setup, n, dt, flags):
    m, lib, orc, e, b = setup
    sp = I.uniform_species(m, n, 7, 0.5, -1.0, 1.0, 1.0)
    order = np.argsort(sp.cell, kind="stable")          # runs of particles in one tet
    cell, X, V = sp.cell[order], sp.X[order], sp.V[order]
    ref = orc.step(cell, X, V, e, b, sp.q, sp.m, sp.w, dt, touch=True)
    d = lib.species(cell, X, V, sp.q, sp.m, sp.w)
    dG = torch.empty(lib.n_edges, dtype=torch.float64, device="cuda")
    Q = torch.empty(lib.n_nodes, dtype=torch.float64, device="cuda")
    lib.push_deposit(torch.as_tensor(e, device="cuda"), torch.as_tensor(b, device="cuda"), d, dt, dG, Q, flags=flags)
    assert lib.status() == F.FP_OK
    assert np.array_equal(d.cell.cpu().numpy(), ref["cell"])
    for got, k in ((dG, "dG"), (Q, "Q")):
        assert_deposit_close(got.cpu().numpy(), ref[k], np.abs(ref[k]), TOL["fp64"], k, ref[k + "_touch"], EPS["fp64"])
