"""The Faraday update that the field step takes from E^N, before the projection, against
b - dt/2 D1 (E_next + E_cur) with the projected E_next that the step returns (D1 D0 = 0).

Tolerance: the two differ by roundings only.  E_next = E^N - D0 d is rounded once per edge, so a
face's sum of three edges differs by at most a few ulp of |E^N| and of |d|; E^N and D0 d are each
bounded by the field norms below, d by D0 d along a path of at most 3 n edges; b adds its own ulp.
"""
import numpy as np
import pytest
import torch

from paper_2103_06737_gb300 import inputs as I
import oracle as O

pytestmark = pytest.mark.gpu

F = pytest.importorskip("paper_2103_06737_gb300.fem_pic")


@pytest.mark.parametrize("q", [torch.float32, torch.float64])
@pytest.mark.parametrize("n", [1, 2, 5])
@pytest.mark.parametrize("bc", ["pec", "neumann"])
def test_faraday_from_the_unprojected_field(q, n, bc):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    m = I.cube_mesh(n, 1.0, 0.1 if n > 2 else 0.0, seed=1)
    cx = O.Complex(m.xyz, m.tets)
    lib = F.FemPic(m.xyz, m.tets, F.FP_FP32 if q is torch.float32 else F.FP_FP64)
    F.fem_pic_field_setup(lib.h, 1e-10, bc=F.FP_BC_NEUMANN if bc == "neumann" else None)
    rng = np.random.default_rng(n)
    free = np.ones(cx.n_edges) if bc == "neumann" else ~cx.boundary_edge
    Ep, Ec = (rng.uniform(-1, 1, cx.n_edges) * free for _ in range(2))
    b = rng.uniform(-1e-10, 1e-10, cx.n_faces)
    Q = torch.as_tensor(rng.uniform(-1e-12, 1e-12, cx.n_nodes), device="cuda").to(q)
    out = []
    for with_b in (True, False):
        En = torch.empty(cx.n_edges, dtype=torch.float64, device="cuda")
        bd = torch.as_tensor(b.copy(), device="cuda")
        st, info = F.fem_pic_field_step(lib.h, torch.as_tensor(Ep, device="cuda"), torch.as_tensor(Ec, device="cuda"),
                                        En, bd if with_b else None, None, None, Q, tol=1e-10)
        assert st == F.FP_OK, info
        out.append(En.cpu().numpy())
        if with_b:
            b1 = bd.cpu().numpy()
    lib.close()
    assert np.array_equal(out[0], out[1])
    D1 = cx.D1().astype(np.float64)
    ref = b - 0.5e-10 * (D1 @ (out[0] + Ec))
    size = np.linalg.norm(out[0]) + 2 * np.linalg.norm(Ec) + np.linalg.norm(Ep)
    eps = np.finfo(np.float64).eps
    tol = eps * (4 * np.abs(b).max() + 0.5e-10 * 12 * (1 + 3 * n) * size)
    assert np.abs(b1 - ref).max() <= tol
