"""The cell sort through records: in random order (records), nearly sorted and dead particles
(straight), at sizes around the threshold, both precisions, with extra columns, against a stable
sort: every particle's row moves as a whole, cells ascending, dead ones last.
"""
import numpy as np
import pytest
import torch

from paper_2103_06737_gb300 import inputs as I

pytestmark = pytest.mark.gpu

F = pytest.importorskip("paper_2103_06737_gb300.fem_pic")


@pytest.mark.parametrize("precision", [F.FP_FP32, F.FP_FP64])
@pytest.mark.parametrize("n", [(1 << 17) - 1, 1 << 17, 200_003])
@pytest.mark.parametrize("order", ["random", "sorted", "half"])
@pytest.mark.parametrize("ncols", [0, 3, 18])
def test_sort_moves_whole_rows(precision, n, order, ncols):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    m = I.cube_mesh(6, 1.0, 0.1, seed=1)
    lib = F.FemPic(m.xyz, m.tets, precision)
    rng = np.random.default_rng(n + ncols)
    cell = rng.integers(-1, m.n_tets, n).astype(np.int32)
    if order != "random":
        cell = np.sort(cell)
        if order == "half":
            k = rng.random(n) < 0.5
            cell[k] = rng.permutation(cell[k])
    real = np.float32 if precision == F.FP_FP32 else np.float64
    rows = rng.standard_normal((6 + ncols, n)).astype(real)
    rows[0] = np.arange(n)          # tells the particles apart (exact in float)
    t = torch.as_tensor(rows, device="cuda")
    src = F.Species(torch.as_tensor(cell, device="cuda"), t[:3].contiguous(), t[3:6].contiguous(), -1.0, 1.0, 1.0)
    dst = src.empty_like()
    if ncols:
        cols = t[6:].contiguous()
        out = torch.empty_like(cols)
        lib.sort_columns(src, dst, cols, out, ncols)
    else:
        lib.sort(src, dst)
    assert lib.status() == F.FP_OK
    got = [dst.off, dst.vel] + ([out] if ncols else [])
    got = torch.cat(got).cpu().numpy()
    c = dst.cell.cpu().numpy()
    key = np.where(c < 0, m.n_tets, c)
    assert (np.diff(key) >= 0).all()
    who = got[0].astype(np.int64)
    assert np.array_equal(np.sort(who), np.arange(n))
    assert np.array_equal(c, cell[who]) and np.array_equal(got, rows[:, who])
    lib.close()
